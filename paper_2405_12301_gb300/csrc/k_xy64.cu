// k_xy64.cu -- fused x+y residual kernel of the FP64 WENO5-JS scheme for 2D grids
// and for each z-plane of 3D grids.
//
// A CTA owns a tile of at most 16 x 8 cells of one plane, one cell per thread, and
// the plus-shaped halo around it (three ghost layers per side in x and in y, Sec.
// 4.5).  Phases, all through shared memory:
//   A+F. every point of the tile and halo is loaded once (boundary rule applied to
//      ghost indices) and its LF split fluxes f(+/-) (Sec. 2.2) are formed in the
//      directions that need them: own points in x and y, halo points in the halo's;
//   W. every x- and y-interface flux of the tile is reconstructed once, as sliding
//      runs of at most 9 faces along tile columns and rows (weights in FP32 pairs,
//      rough windows in triples from the list), WENO(+) and WENO(-) kept apart;
//   C. each thread forms -(dF/dx) - (dG/dy) for its cell (Sec. 4.1) and either
//      stores it (3D: the z sweep adds its part and runs the stage), writes L(U),
//      or applies the SSP-RK3 stage combination (Eq. tt-ssprk3 without rounding)
//      and publishes the wavespeed max of the new state.
//
// The FP64 pipe bounds it (an SM issues one FP64 warp instruction per ~20 cycles,
// however many lanes are active), so what a tile computes for nobody costs time.
// The tile's extents are fitted to the grid (plan_xy64): tiles of equal size, none
// beyond the grid's edge, whose cells, halo points and runs fill their warps and whose
// number fills the SMs.
#include <algorithm>

#include "weno_dev.cuh"
#include "weno_internal.h"

namespace wg {

namespace xy64 {
constexpr int MW = 32, MH = 16, MNT = 256;  // bounds of a tile's extents and cells (one per thread)
constexpr int RUN = 9;

// Sizes of the shared arrays of a w x h tile, in elements per component and sign
struct Sizes {
    int px, nxp, nyp, pxi, nxi, nyi;
    __host__ __device__ Sizes(int w, int h)
        : px((w + 6) | 1), nxp(px * h), nyp(w * (h + 6)), pxi(w + 1), nxi(pxi * h), nyi(w * (h + 1))
    {
    }  // (odd pitch: the rows of neighbouring lanes' x-runs lie in distinct banks)
    int points() const { return nxp + nyp; }
    int faces() const { return nxi + nyi; }
};
}  // namespace xy64

template <int D, int EPI, bool PD>
__global__ void __launch_bounds__(xy64::MNT, 2) k_xy64(const SweepArgs a)
{
    using namespace xy64;
    constexpr int NF = D + 2;
    const int NT = blockDim.x, TW = a.txy.w;
    const Sizes Z(TW, a.txy.s);
    extern __shared__ __align__(16) unsigned char smem[];
    double *Fx = reinterpret_cast<double *>(smem);  // [2][NF][s][w+1]
    double *Fy = Fx + 2 * NF * Z.nxi;               // [2][NF][s+1][w]
    double *fx = Fy + 2 * NF * Z.nyi;               // [2][NF][s][px]
    double *fy = fx + 2 * NF * Z.nxp;               // [2][NF][s+6][w]
    __shared__ int s_rough;
    const RoughList rough{&s_rough, reinterpret_cast<unsigned *>(fy + 2 * NF * Z.nyp)};
    if (threadIdx.x == 0) s_rough = 0;

    const double dt = a.ctl->dt;
    if (a.check_dt && __double_as_longlong(dt) == 0) return;
    const double alpha = __longlong_as_double((long long)a.ctl->alpha[a.slot_in]);
    // LF constants of the x and y splittings: the global alpha, or per direction
    const double alx = PD ? __longlong_as_double((long long)a.ctl->alpha_dir[a.slot_in][0]) : alpha;
    const double aly = PD ? __longlong_as_double((long long)a.ctl->alpha_dir[a.slot_in][1]) : alpha;

    const int nx = a.n[0], ny = a.n[1];
    const long long N = a.N;
    const int x0 = blockIdx.x * TW, y0 = blockIdx.y * a.txy.s;
    const int W = min(TW, nx - x0), H = min(a.txy.s, ny - y0);
    const long long zoff = (long long)blockIdx.z * a.stride[2];
    const int tid = threadIdx.x, ty = tid / W, tx = tid - ty * W;
    const bool own = ty < H;
    const long long cell = zoff + (long long)(y0 + ty) * nx + (x0 + tx);

    // the stage combination needs U^n at this thread's cell: issue the loads now
    double un[NF];
    if (EPI == EPI_STAGE && a.stage > 0 && own) {
#pragma unroll
        for (int f = 0; f < NF; ++f) un[f] = __ldg(a.Un + f * N + cell);
    }

    // interior tiles (halo inside the grid) skip the boundary rule
    const bool interior = x0 >= 3 && y0 >= 3 && x0 + W + 3 <= nx && y0 + H + 3 <= ny;
    auto load_point = [&](int lx, int ly, double *q) {
        int cx = x0 + lx, cy = y0 + ly;
        bool fx_ = false, fy_ = false;
        if (!interior) {
            int inx, iny;
            cx = ghost_map(cx, nx, a.bc[0][0], a.bc[0][1], fx_, inx);
            cy = ghost_map(cy, ny, a.bc[1][0], a.bc[1][1], fy_, iny);
            if (inx >= 0 || iny >= 0) {  // a ghost of an inflow side holds the given state
                const double *st = inx >= 0 ? a.bc_state[0][inx] : a.bc_state[1][iny];
#pragma unroll
                for (int f = 0; f < NF; ++f) q[f] = st[f];
                return;
            }
        }
        const double *src = a.U + zoff + (long long)cy * nx + cx;
#pragma unroll
        for (int f = 0; f < NF; ++f) q[f] = __ldg(src + f * N);
        if (fx_) q[1] = -q[1];
        if (fy_) q[2] = -q[2];
    };
    // halo point t: rows -3..-1 and H..H+2 of every column, then columns -3..-1 and W..W+2 of every row
    const int nhy = 6 * W, nhalo = nhy + 6 * H;
    auto halo_at = [&](int t, int &hx, int &hy) -> bool {
        if (t < nhy) {
            const int k = t / W;
            hx = t - k * W;
            hy = k < 3 ? k - 3 : H + k - 3;
            return false;
        }
        t -= nhy;
        hy = t / 6;
        const int k = t - hy * 6;
        hx = k < 3 ? k - 3 : W + k - 3;
        return true;
    };
    const double gm1 = a.gamma - 1.0;
    // split flux (twice, see below) of a point in one direction, stored at its slot of fx / fy
    auto flux_x = [&](const double *q, int lx, int ly) {
        double fp[NF], fm[NF];
        split_flux_f64<D, 0, true>(q, alx, gm1, fp, fm);
        const int o = ly * Z.px + lx + 3;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            fx[f * Z.nxp + o] = fp[f];
            fx[(NF + f) * Z.nxp + o] = fm[f];
        }
    };
    auto flux_y = [&](const double *q, int lx, int ly) {
        double fp[NF], fm[NF];
        split_flux_f64<D, 1, true>(q, aly, gm1, fp, fm);
        const int o = (ly + 3) * TW + lx;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            fy[f * Z.nyp + o] = fp[f];
            fy[(NF + f) * Z.nyp + o] = fm[f];
        }
    };

    // ---- phase A+F: halo points are dealt from the last thread down, so that threads
    // without a cell take them first
    double uk[NF];  // U^(k) at the own cell, kept for the stage combination
    {
        double qh[NF];
        int t = NT - 1 - tid, hx = 0, hy = 0;
        bool dirx = false;
        if (own) load_point(tx, ty, uk);
        if (t < nhalo) {
            dirx = halo_at(t, hx, hy);
            load_point(hx, hy, qh);
        }
        if (own) {
            flux_x(uk, tx, ty);
            flux_y(uk, tx, ty);
        }
        while (t < nhalo) {
            if (dirx) flux_x(qh, hx, hy);
            else flux_y(qh, hx, hy);
            t += NT;
            if (t < nhalo) {
                dirx = halo_at(t, hx, hy);
                load_point(hx, hy, qh);
            }
        }
    }
    __syncthreads();

    // ---- phase W: runs of a column's H + 1 faces and of a row's W + 1 in nseg segments,
    // one code path.  The shared arrays hold 2 f(+/-):
    // reconstruct with 4 eps (twice the WENO5 value)
    {
        const PairEps P = pair_eps(4.0 * a.eps);
        const int nseg = a.txy.nseg, len = (W + nseg) / nseg;
        const int nry = 2 * NF * W, nrx = 2 * NF * nseg * H;
#pragma unroll 1
        for (int run = tid; run < nry + nrx; run += NT) {
            int po, oo, st, fs, cnt;  // offsets from fx and Fx (fy and Fy follow them)
            if (run < nry) {
                fs = run / W;
                const int lx = run - fs * W;
                po = 2 * NF * Z.nxp + fs * Z.nyp + lx;
                oo = 2 * NF * Z.nxi + fs * Z.nyi + lx;
                st = TW;
                cnt = H + 1;
            } else {
                const int u = run - nry, r = u / H, ly = u - r * H;
                fs = r / nseg;
                const int j0 = (r - fs * nseg) * len;
                po = fs * Z.nxp + ly * Z.px + j0;
                oo = fs * Z.nxi + ly * Z.pxi + j0;
                st = 1;
                cnt = min(len, W + 1 - j0);
                if (cnt <= 0) continue;
            }
            if (fs >= NF) {  // WENO(-): the same run read backwards from the far end
                po += (cnt + 4) * st;
                oo += (cnt - 1) * st;
                st = -st;
            }
            weno5_slide_pair(fx, po, st, P, Fx, oo, st, cnt, TW, rough);
        }
        __syncthreads();
        rough_windows(rough, TW, fx, Fx, P);
    }
    __syncthreads();

    // ---- phase C: the cell's residual -(dF/dx) - (dG/dy) and the epilogue.
    // Face fluxes are twice F^ = WENO(+) + WENO(-): the halving rides on 1/h
    double out[NF];
    if (own) {
        const double ihx = 0.5 * a.inv_h[0], ihy = 0.5 * a.inv_h[1];
        const double *FxM = Fx + NF * Z.nxi, *FyM = Fy + NF * Z.nyi;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const int ox = f * Z.nxi + ty * Z.pxi + tx, oy = f * Z.nyi + ty * TW + tx;
            const double dx = (Fx[ox + 1] + FxM[ox + 1]) - (Fx[ox] + FxM[ox]);
            const double dy = (Fy[oy + TW] + FyM[oy + TW]) - (Fy[oy] + FyM[oy]);
            const double r = -dx * ihx - dy * ihy;
            if (EPI == EPI_STORE) reinterpret_cast<double *>(a.acc)[f * N + cell] = r;
            else if (EPI == EPI_RHS) a.Rout[f * N + cell] = r;
            else a.Uout[f * N + cell] = out[f] = stage_combine(a.stage, un[f], uk[f], r, dt);
        }
    }
    if constexpr (EPI == EPI_STAGE)
        speed_max_publish_f64<D, PD ? 1 + D : 1>(
            [&](long long, double *q) {
#pragma unroll
                for (int f = 0; f < NF; ++f) q[f] = out[f];
            },
            0, own ? 1 : 0, 1, a.gamma, a.gg_f, &a.ctl->alpha[a.slot_out], a.ctl->alpha_dir[a.slot_out], &a.ctl->status);
}

double tile64_cycles(long long tiles, const Tile64 &t, int regs, int cells, double cell, int halo, int runs, int longest)
{
    auto warps = [](int k) { return 4 * ((k + 127) / 128); };
    const int k = (runs + t.nt - 1) / t.nt, w = t.nt / 32;
    const double work = cell * warps(cells) + 22.0 * warps(halo) + 7.0 * k * w * (longest + 1) + 40.0;
    const long long most = 227 * 1024, per_sm = (tiles + sm_count() - 1) / sm_count();
    const long long res = std::min(most / (t.smem + 1024), 65536ll / (regs * t.nt));  // resident CTAs
    if (res < 1) return -1.0;
    const double rounds = (double)((per_sm + res - 1) / res), ctas = (double)std::min(res, per_sm);
    const double chain = k * (longest + 1) + 4;
    return std::max(20.0 * work * (double)per_sm, 1000.0 * chain * rounds) * (1.0 + 0.15 / ctas + 4.0 / (ctas * w)) +
           300.0 * chain;
}

// The estimate's choice and the best of ~30 tiles measured (us): 256 x 256, 12 stages,
// 14 x 16 the best; 1000 x 777 (one L(U)) 16 x 16 the best; 400 x 300 16 x 16 72, 8 x 8
// 70; 120 x 150 15 x 8 the best; 97 x 83 x 61 25 x 8 543, 11 x 14 528; 64^3 13 x 6 329,
// 16 x 13 324; 40 x 53 x 37 10 x 11 151, 10 x 14 147 (32 x 8 of 256 threads, fixed: up to
// 12% more).  Blocks of 3 or 5 warps are left out: an SM's FP64 units are its four
// sub-partitions', and such blocks load them unevenly (8 x 8 cells, 64 / 96 / 128
// threads: 622 / 737 / 659).
Tile64 plan_xy64(int dim, const long long n[3])
{
    using namespace xy64;
    const int nf = dim + 2;
    Tile64 best{};
    double least = -1.0;
    for (int mw = (int)std::min(8ll, n[0]); mw <= MW; ++mw)  // (whole sectors)
        for (int mh = 1; mh <= MH; ++mh)
            for (int run : {std::max(4, std::min(RUN, mh + 1)), mh + 1})  // (faces of an x-run)
                for (int nt = 128; nt <= MNT; nt += 128) {
                    Tile64 t{mw, mh, 0, 0, nt, 0};
                    if (fit_extent(n[0], mw) != mw || fit_extent(n[1], mh) != mh) break;
                    const Sizes Z(mw, mh);
                    t.nseg = (mw + run) / run;
                    t.len = (mw + t.nseg) / t.nseg;
                    t.smem = (unsigned)(2 * nf * (8 * Z.points() + 12 * Z.faces()));
                    const long long gy = (n[1] + mh - 1) / mh, tiles = (n[0] + mw - 1) / mw * gy * n[2];
                    if (mw * mh > nt || gy > 65535 || 2 * nf * std::max(Z.points(), Z.faces()) > 8192) continue;
                    const double c = tile64_cycles(tiles, t, 112, mw * mh, dim == 2 ? 75.0 : 85.0, 6 * (mw + mh),
                                                   2 * nf * (mw + t.nseg * mh), std::max(mh + 1, t.len));
                    if (c >= 0.0 && (least < 0.0 || c < least)) {
                        least = c;
                        best = t;
                    }
                }
    return best;
}

template <int D, int EPI, bool PD> static cudaError_t launch_xy64_t(const SweepArgs &a, cudaStream_t s)
{
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_xy64<D, EPI, PD>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    const Tile64 &t = a.txy;
    if (t.nt == 0) return cudaErrorInvalidConfiguration;
    dim3 grid((unsigned)((a.n[0] + t.w - 1) / t.w), (unsigned)((a.n[1] + t.s - 1) / t.s), (unsigned)a.n[2]);
    k_xy64<D, EPI, PD><<<grid, t.nt, t.smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_xy64(int dim, int epi, const SweepArgs &a, cudaStream_t s)
{
#define X(D, E) \
    if (dim == D && epi == E) return a.per_dir ? launch_xy64_t<D, E, true>(a, s) : launch_xy64_t<D, E, false>(a, s);
    X(2, EPI_RHS) X(2, EPI_STAGE) X(3, EPI_STORE)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace wg
