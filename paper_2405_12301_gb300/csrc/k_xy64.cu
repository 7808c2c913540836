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
// The FP64 pipe bounds it, so what a tile computes for nobody costs time: the tile
// is fitted to the grid (tiles of equal size, none beyond the grid's edge; on grids
// of a few tiles per SM the height whose fullest SM has least to do), and small
// tiles, 4 (3D planes: 3) to an SM, even out rough and smooth ones.
#include "weno_dev.cuh"
#include "weno_internal.h"

namespace wg {

namespace xy64 {
constexpr int MW = 16, MH = 8;           // tile bounds
constexpr int PX = MW + 6;               // row pitch of the x-flux points: 8 rows x 2 runs of a half-warp, distinct banks
constexpr int NXP = PX * MH;             // x-flux points
constexpr int NYP = MW * (MH + 6);       // y-flux points (row pitch MW)
constexpr int PXI = MW + 1;
constexpr int NXI = PXI * MH;            // x interfaces
constexpr int NYI = MW * (MH + 1);       // y interfaces
constexpr int RUN = MH + 1;              // most faces of a run

// 2 NF MW y runs and 2 NF MH 2 x runs: 2 per thread in 2D (256) and in 3D planes (320)
template <int D> struct Layout {
    static constexpr int NF = D + 2, NT = D == 2 ? 128 : 160, CTAS = D == 2 ? 4 : 3;
    static constexpr size_t fx_off = sizeof(double) * 2 * NF * (NXI + NYI);
    static constexpr size_t rough_off = fx_off + sizeof(double) * 2 * NF * (NXP + NYP);
    static constexpr size_t bytes = rough_off + sizeof(unsigned) * 2 * NF * (NXI + NYI);  // (every window)
    static_assert(2 * NF * (NXP + NYP) <= 8192 && 2 * NF * (NXI + NYI) <= 8192, "offsets of a RoughList entry");
    static_assert(MW * MH <= NT, "one cell per thread");
};
}  // namespace xy64

template <int D, int EPI, bool PD>
__global__ void __launch_bounds__(xy64::Layout<D>::NT, xy64::Layout<D>::CTAS) k_xy64(const SweepArgs a)
{
    using namespace xy64;
    using L = Layout<D>;
    constexpr int NF = L::NF, NT = L::NT;
    extern __shared__ __align__(16) unsigned char smem[];
    double *Fx = reinterpret_cast<double *>(smem);              // [2][NF][MH][PXI]
    double *Fy = Fx + 2 * NF * NXI;                             // [2][NF][MH+1][MW]
    double *fx = reinterpret_cast<double *>(smem + L::fx_off);  // [2][NF][MH][PX]
    double *fy = fx + 2 * NF * NXP;                             // [2][NF][MH+6][MW]
    __shared__ int s_rough;
    const RoughList rough{&s_rough, reinterpret_cast<unsigned *>(smem + L::rough_off)};
    if (threadIdx.x == 0) s_rough = 0;

    const double dt = a.ctl->dt;
    if (a.check_dt && __double_as_longlong(dt) == 0) return;
    const double alpha = __longlong_as_double((long long)a.ctl->alpha[a.slot_in]);
    // LF constants of the x and y splittings: the global alpha, or per direction
    const double alx = PD ? __longlong_as_double((long long)a.ctl->alpha_dir[a.slot_in][0]) : alpha;
    const double aly = PD ? __longlong_as_double((long long)a.ctl->alpha_dir[a.slot_in][1]) : alpha;

    const int nx = a.n[0], ny = a.n[1];
    const long long N = a.N;
    const int x0 = blockIdx.x * a.tile_w, y0 = blockIdx.y * a.tile_s;
    const int W = min(a.tile_w, nx - x0), H = min(a.tile_s, ny - y0);
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
        const int o = ly * PX + lx + 3;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            fx[f * NXP + o] = fp[f];
            fx[(NF + f) * NXP + o] = fm[f];
        }
    };
    auto flux_y = [&](const double *q, int lx, int ly) {
        double fp[NF], fm[NF];
        split_flux_f64<D, 1, true>(q, aly, gm1, fp, fm);
        const int o = (ly + 3) * MW + lx;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            fy[f * NYP + o] = fp[f];
            fy[(NF + f) * NYP + o] = fm[f];
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

    // ---- phase W: runs of equal length (H + 1 faces of a column; a row's W + 1 faces
    // in segments no longer), one code path.  The shared arrays hold 2 f(+/-):
    // reconstruct with 4 eps (twice the WENO5 value)
    {
        const PairEps P = pair_eps(4.0 * a.eps);
        const int most = max(H + 1, 4), nseg = (W + most) / most, len = (W + nseg) / nseg;
        const int nry = 2 * NF * W, nrx = 2 * NF * nseg * H;
#pragma unroll 1
        for (int run = tid; run < nry + nrx; run += NT) {
            int po, oo, st, fs, cnt;  // offsets from fx and Fx (fy and Fy follow them)
            if (run < nry) {
                fs = run / W;
                const int lx = run - fs * W;
                po = 2 * NF * NXP + fs * NYP + lx;
                oo = 2 * NF * NXI + fs * NYI + lx;
                st = MW;
                cnt = H + 1;
            } else {
                const int u = run - nry, r = u / H, ly = u - r * H;
                fs = r / nseg;
                const int j0 = (r - fs * nseg) * len;
                po = fs * NXP + ly * PX + j0;
                oo = fs * NXI + ly * PXI + j0;
                st = 1;
                cnt = min(len, W + 1 - j0);
            }
            if (fs >= NF) {  // WENO(-): the same run read backwards from the far end
                po += (cnt + 4) * st;
                oo += (cnt - 1) * st;
                st = -st;
            }
            weno5_slide_pair(fx, po, st, P, Fx, oo, st, cnt, MW, rough);
        }
        __syncthreads();
        rough_windows(rough, MW, fx, Fx, P);
    }
    __syncthreads();

    // ---- phase C: the cell's residual -(dF/dx) - (dG/dy) and the epilogue.
    // Face fluxes are twice F^ = WENO(+) + WENO(-): the halving rides on 1/h
    double out[NF];
    if (own) {
        const double ihx = 0.5 * a.inv_h[0], ihy = 0.5 * a.inv_h[1];
        const double *FxM = Fx + NF * NXI, *FyM = Fy + NF * NYI;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const int ox = f * NXI + ty * PXI + tx, oy = f * NYI + ty * MW + tx;
            const double dx = (Fx[ox + 1] + FxM[ox + 1]) - (Fx[ox] + FxM[ox]);
            const double dy = (Fy[oy + MW] + FyM[oy + MW]) - (Fy[oy] + FyM[oy]);
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
            0, own ? 1 : 0, 1, a.gamma, &a.ctl->alpha[a.slot_out], a.ctl->alpha_dir[a.slot_out], &a.ctl->status);
}

template <int D, int EPI, bool PD> static cudaError_t launch_xy64_t(SweepArgs a, cudaStream_t s)
{
    using namespace xy64;
    using L = Layout<D>;
    static bool attr = false;
    if (!attr) {
        cudaError_t e =
            cudaFuncSetAttribute(k_xy64<D, EPI, PD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    a.tile_w = fit_extent(a.n[0], MW);
    const long long gx = (a.n[0] + a.tile_w - 1) / a.tile_w;
    const int w = a.tile_w;
    // FP64 instructions of a tile: ~75 for a cell's fluxes and update, ~22 for a halo
    // point's flux, ~8 for a window
    a.tile_s = fit_tile(a.n[1], MH, gx * a.n[2], [&](int h) {
        return 75.0 * w * h + 132.0 * (w + h) + 16.0 * L::NF * (w * (h + 1) + h * (w + 1));
    });
    dim3 grid((unsigned)gx, (unsigned)((a.n[1] + a.tile_s - 1) / a.tile_s), (unsigned)a.n[2]);
    k_xy64<D, EPI, PD><<<grid, L::NT, L::bytes, s>>>(a);
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
