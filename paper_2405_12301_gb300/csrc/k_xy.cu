// k_xy.cu -- fused x+y residual kernel of the FP32-bulk WENO5-JS scheme for the
// z-planes of 3D grids (2D FP32-bulk: k_xy2.cu; FP64: k_xy64.cu).
//
// A CTA (256 threads) owns a TX x TY = 32 x 8 tile of one plane, one cell per
// thread, and the plus-shaped halo around it (three ghost layers per side in x
// and in y, Sec. 4.5).  Phases, all through shared memory:
//   A+F. every point of the tile and halo is loaded once (boundary rule applied
//      to ghost indices), its difference from the tile's reference state taken,
//      and its LF split fluxes f(+/-) (Sec. 2.2) formed in the directions that
//      need them: each thread its own point in x and y, and one halo point in the
//      halo's direction;
//   W. every x- and y-interface flux of the tile is reconstructed once, WENO(+)
//      plus mirrored WENO(-): each thread its cell's left and bottom faces for
//      every component, a face's two windows as one f32x2 pair, and the tile's
//      last column/row faces spread over the threads;
//   C. each thread stores -(dF/dx) - (dG/dy) of its cell (Sec. 4.1); the z sweep
//      adds its part and runs the stage.
// Compared with one launch per direction, each point is loaded and split once
// per stage.
#include "bulk_load.cuh"
#include "weno_dev.cuh"
#include "weno_internal.h"

namespace wg {

namespace xy {
constexpr int NT = 256;
constexpr int TX = 32, TY = 8;
constexpr int BX = TX + 6, BY = TY + 6;     // row and column extents with halo
constexpr int BXP = BX + 3;                 // row pitch of the x-flux points
constexpr int NXP = BXP * TY;               // x-flux points: 38 (pitch 41) x 8
constexpr int NYP = TX * BY;                // y-flux points: 32 x 14
constexpr int NXI = (TX + 1) * TY;          // x interfaces: 33 x 8
constexpr int NYI = TX * (TY + 1);          // y interfaces: 32 x 9
constexpr int NHY = 6 * TX;                 // y-halo points (rows -3..-1, TY..TY+2)
constexpr int NHALO = NHY + 6 * TY;         // plus x-halo points: 240

constexpr int D = 3, NF = D + 2;
constexpr size_t fx_off = (sizeof(float) * NF * (NXI + NYI) + 15) & ~size_t(15);
constexpr size_t fy_off = fx_off + sizeof(float) * 2 * NF * NXP;
constexpr size_t ref_off = (fy_off + sizeof(float) * 2 * NF * NYP + 15) & ~size_t(15);
constexpr size_t bytes = ref_off + sizeof(RefState<D>);
}  // namespace xy

// Held to 48 registers so that 5 CTAs (40 warps) share an SM; its shared memory
// allows that many.  ST: the stage, which selects where the stencil state comes
// from -- the split of U (stage 1, L(U)) or the stored split of U^n plus Delta_k
// (stages 2 and 3, the stage state of k_xy2.cu).
template <bool PD, int ST>
__global__ void __launch_bounds__(xy::NT, 5) k_xy(const SweepArgs a)
{
    using namespace xy;
    extern __shared__ __align__(16) unsigned char smem[];
    float *Fx = reinterpret_cast<float *>(smem);           // [NF][TY][TX+1]
    float *Fy = Fx + NF * NXI;                             // [NF][TY+1][TX]
    float *fx = reinterpret_cast<float *>(smem + fx_off);  // [2][NF][TY][BXP]
    float *fy = reinterpret_cast<float *>(smem + fy_off);  // [2][NF][BY][TX]
    RefState<D> &ref = *reinterpret_cast<RefState<D> *>(smem + ref_off);

    const long long dtbits = __double_as_longlong(a.ctl->dt);
    if (a.check_dt && dtbits == 0) return;
    const double alpha = __longlong_as_double((long long)a.ctl->alpha[a.slot_in]);
    // LF constants of the x and y splittings: the global alpha, or per direction
    const double alx = PD ? __longlong_as_double((long long)a.ctl->alpha_dir[a.slot_in][0]) : alpha;
    const double aly = PD ? __longlong_as_double((long long)a.ctl->alpha_dir[a.slot_in][1]) : alpha;

    const int nx = a.n[0], ny = a.n[1];
    const long long N = a.N;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const long long zoff = (long long)blockIdx.z * a.stride[2];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int gx = x0 + tx, gy = y0 + ty;
    const bool own = gx < nx && gy < ny;
    const long long cell = zoff + (long long)(gy < ny ? gy : ny - 1) * nx + (gx < nx ? gx : nx - 1);

    // interior tiles (halo inside the grid) skip the boundary rule
    const bool interior = x0 >= 3 && y0 >= 3 && x0 + TX + 3 <= nx && y0 + TY + 3 <= ny;

    // A point's hi/lo state (boundary rule on ghost indices)
    auto load_point_b = [&](int lx, int ly, float *h, float *l) {
        int cx = x0 + lx, cy = y0 + ly;
        bool fx_ = false, fy_ = false;
        if (!interior) {
            int inx, iny;
            cx = cx < nx + 2 ? cx : nx + 2;
            cy = cy < ny + 2 ? cy : ny + 2;
            cx = ghost_map(cx, nx, a.bc[0][0], a.bc[0][1], fx_, inx);
            cy = ghost_map(cy, ny, a.bc[1][0], a.bc[1][1], fy_, iny);
            if (inx >= 0 || iny >= 0) {
                bulk_state<NF>(inx >= 0 ? a.bc_state[0][inx] : a.bc_state[1][iny], h, l);
                return;
            }
        }
        bulk_point<NF, (ST > 0)>(a, zoff + (long long)cy * nx + cx, h, l);
        if (fx_) { h[1] = -h[1]; l[1] = -l[1]; }
        if (fy_) { h[2] = -h[2]; l[2] = -l[2]; }
    };

    // ---- phase A+F: own point (x and y fluxes) and one halo point per thread;
    // their loads go out before the reference state's barrier, so their latency
    // overlaps warp 0's work on the reference
    float hq[NF], lq[NF];         // the own point's hi/lo
    load_point_b(tx, ty, hq, lq);
    const bool halo = threadIdx.x < NHALO;
    int hx = 0, hy = 0;
    bool hdirx = false;
    float hh[NF], lh[NF];
    if (halo) {
        int t = threadIdx.x;
        if (t < NHY) {     // y halo: rows -3..-1 and TY..TY+2 of every tile column
            hx = t & 31;
            const int k = t >> 5;
            hy = k < 3 ? k - 3 : TY + k - 3;
        } else {           // x halo: columns -3..-1 and TX..TX+2 of every tile row
            t -= NHY;
            hy = t / 6;
            const int k = t - hy * 6;
            hx = k < 3 ? k - 3 : TX + k - 3;
            hdirx = true;
        }
        load_point_b(hx, hy, hh, lh);
    }

    // ---- reference state of the tile: its first cell (inside the grid); the LF
    // constants in FP32, converted once per block (on the integer pipe: a cvt issues
    // at FP64 rate on this GPU)
    __shared__ float2 s_al;
    if (threadIdx.x < 32) {
        float h0[NF], l0[NF];
        load_point_b(0, 0, h0, l0);
        RefState<D> r;
        make_ref_hl<D>(h0, l0, a.gm1_f, r);
        if (threadIdx.x == 0) {
            ref = r;
            const float ax = f64_to_f32(alx);
            s_al = make_float2(ax, PD ? f64_to_f32(aly) : ax);
        }
    }
    __syncthreads();
    const float alX = s_al.x, alY = s_al.y;

    // split flux of a point in direction x or y, stored at its slot of fx / fy
    auto flux_store = [&](const float *q, bool dirx, int lx, int ly) {
        float fp[NF], fm[NF];
        if (dirx) {
            split_flux_diff<D, 0, true>(q, ref, alX, a.gm1_f, fp, fm);
            const int o = ly * BXP + (lx + 3);
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                fx[f * NXP + o] = fp[f];
                fx[(NF + f) * NXP + o] = fm[f];
            }
        } else {
            split_flux_diff<D, 1, true>(q, ref, alY, a.gm1_f, fp, fm);
            const int o = (ly + 3) * TX + lx;
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                fy[f * NYP + o] = fp[f];
                fy[(NF + f) * NYP + o] = fm[f];
            }
        }
    };

    {
        float q[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) q[f] = (hq[f] - ref.hi[f]) + (lq[f] - ref.lo[f]);
        flux_store(q, true, tx, ty);
        flux_store(q, false, tx, ty);
    }
    if (halo) {
        float q[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) q[f] = (hh[f] - ref.hi[f]) + (lh[f] - ref.lo[f]);
        flux_store(q, hdirx, hx, hy);
    }
    __syncthreads();

    // ---- phase W: the own left x face and bottom y face for every component, plus
    // one of the remaining faces (top of the tile's top row, right of its last
    // column).  The shared arrays hold 2 f(+/-): reconstruct with 4 eps (twice the WENO5 value)
    const float eps = 4.0f * a.eps_f;
    float fxl[NF], fyb[NF];
    // WENO(+) and the mirrored WENO(-) of a face as one f32x2 pair
    auto face_x = [&](int f, int ly, int j) -> float {  // between local columns j-1 and j of row ly
        const float *P = fx + f * NXP + ly * BXP;
        const float *M = fx + (NF + f) * NXP + ly * BXP;
        return weno5_pm(make_float2(P[j], M[j + 5]), make_float2(P[j + 1], M[j + 4]),
                        make_float2(P[j + 2], M[j + 3]), make_float2(P[j + 3], M[j + 2]),
                        make_float2(P[j + 4], M[j + 1]), eps);
    };
    auto face_y = [&](int f, int lx, int j) -> float {  // between local rows j-1 and j of column lx
        const float *P = fy + f * NYP + lx;
        const float *M = fy + (NF + f) * NYP + lx;
        return weno5_pm(make_float2(P[j * TX], M[(j + 5) * TX]), make_float2(P[(j + 1) * TX], M[(j + 4) * TX]),
                        make_float2(P[(j + 2) * TX], M[(j + 3) * TX]), make_float2(P[(j + 3) * TX], M[(j + 2) * TX]),
                        make_float2(P[(j + 4) * TX], M[(j + 1) * TX]), eps);
    };
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        fxl[f] = face_x(f, ty, tx);
        Fx[f * NXI + ty * (TX + 1) + tx] = fxl[f];
        fyb[f] = face_y(f, tx, ty);
        Fy[f * NYI + ty * TX + tx] = fyb[f];
    }
    if (threadIdx.x < NF * (TX + TY)) {
        const int t = threadIdx.x;
        if (t < NF * TX) {
            const int f = t >> 5, lx = t & 31;
            Fy[f * NYI + TY * TX + lx] = face_y(f, lx, TY);
        } else {
            const int u = t - NF * TX;
            const int f = u >> 3, ly = u & 7;
            Fx[f * NXI + ly * (TX + 1) + TX] = face_x(f, ly, TX);
        }
    }
    __syncthreads();

    // ---- phase C: the cell's residual -(dF/dx) - (dG/dy); face fluxes are twice F^:
    // the halving rides on 1/h
    if (!own) return;
    const float ihx = 0.5f * a.inv_h_f[0], ihy = 0.5f * a.inv_h_f[1];
    float *acc = reinterpret_cast<float *>(a.acc);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const float dx = Fx[f * NXI + ty * (TX + 1) + tx + 1] - fxl[f];
        const float dy = Fy[f * NYI + (ty + 1) * TX + tx] - fyb[f];
        acc[f * N + cell] = -dx * ihx - dy * ihy;
    }
}

template <bool PD, int ST> static cudaError_t launch_xy_t(const SweepArgs &a, cudaStream_t s)
{
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_xy<PD, ST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)xy::bytes);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    dim3 grid((unsigned)((a.n[0] + xy::TX - 1) / xy::TX), (unsigned)((a.n[1] + xy::TY - 1) / xy::TY),
              (unsigned)a.n[2]);
    k_xy<PD, ST><<<grid, xy::NT, xy::bytes, s>>>(a);
    return cudaGetLastError();
}

// The stage selects the stencil-state source (a handle's stage state exists only
// inside a step; L(U) reads U like stage 1)
cudaError_t launch_xy(const SweepArgs &a, cudaStream_t s)
{
    if (a.N >= (1ll << 32)) return cudaErrorInvalidValue;  // the stage state is indexed in 32 bits
    const int st = a.hl == nullptr ? 0 : a.stage < 2 ? a.stage : 2;
#define X(P, S) \
    if ((a.per_dir != 0) == P && st == S) return launch_xy_t<P, S>(a, s);
    X(false, 0) X(false, 1) X(false, 2) X(true, 0) X(true, 1) X(true, 2)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace wg
