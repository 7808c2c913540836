// k_z.cu -- z direction of the FP64 WENO5-JS residual for 3D grids, ending the
// residual of a stage (the x and y directions run in k_xy64.cu; FP32-bulk's z
// direction is k_z2.cu).
#include <algorithm>

#include "weno_dev.cuh"
#include "weno_internal.h"

namespace wg {

// A CTA owns a tile of x- and z-cells of one y-row, one cell per thread, plus the
// 3 + 3 halo z-planes of its columns; the tile is fitted to the grid as in k_xy64.cu
// (plan_z).  Phases: split fluxes of every point, sliding WENO runs along the columns
// (one run per column, component and sign), then each cell's flux difference is added
// to the x+y part left in the accumulator by k_xy64<3>, and the epilogue writes L(U) or
// applies the SSP-RK3 stage combination and publishes the wavespeed max.
namespace zs {
constexpr int MW = 32, MH = 24, MNT = 256;  // bounds of a tile's extents and cells
constexpr int NF = 5;
}  // namespace zs

template <int EPI, bool PD>
__global__ void __launch_bounds__(zs::MNT, 2) k_z(const SweepArgs a)
{
    using namespace zs;
    extern __shared__ __align__(16) unsigned char smem[];
    const int NT = blockDim.x, TW = a.tz.w, NZP = TW * (a.tz.s + 6), NZI = TW * (a.tz.s + 1);
    double *Fz = reinterpret_cast<double *>(smem);  // [2][NF][s+1][w]
    double *fz = Fz + 2 * NF * NZI;                 // [2][NF][s+6][w]
    __shared__ int s_rough;
    const RoughList rough{&s_rough, reinterpret_cast<unsigned *>(fz + 2 * NF * NZP)};
    if (threadIdx.x == 0) s_rough = 0;

    const double dt = a.ctl->dt;
    if (a.check_dt && __double_as_longlong(dt) == 0) return;
    const double alpha = PD ? __longlong_as_double((long long)a.ctl->alpha_dir[a.slot_in][2])
                            : __longlong_as_double((long long)a.ctl->alpha[a.slot_in]);

    const int nx = a.n[0], nz = a.n[2];
    const long long N = a.N, sz = a.stride[2];
    // z-tiles are the fastest grid index, so that tiles sharing halo planes run
    // close together and find those planes in L2
    const int zt = (nz + a.tz.s - 1) / a.tz.s, xt = blockIdx.x / zt;
    const int x0 = xt * TW, z0 = (blockIdx.x - xt * zt) * a.tz.s;
    const int W = min(TW, nx - x0), H = min(a.tz.s, nz - z0);
    const long long yoff = (long long)blockIdx.y * a.stride[1];
    const int tid = threadIdx.x, tz = tid / W, tx = tid - tz * W;
    const bool own = tz < H;
    const long long cell = yoff + (long long)(z0 + tz) * sz + (x0 + tx);

    double un[NF];
    if (EPI == EPI_STAGE && a.stage > 0 && own) {
#pragma unroll
        for (int f = 0; f < NF; ++f) un[f] = __ldg(a.Un + f * N + cell);
    }
    const double gm1 = a.gamma - 1.0;
    const bool interior = z0 >= 3 && z0 + H + 3 <= nz;

    auto load_point = [&](int lx, int lz, double *q) {
        int cz = z0 + lz;
        bool fz_ = false;
        if (!interior) {
            int inz;
            cz = ghost_map(cz, nz, a.bc[2][0], a.bc[2][1], fz_, inz);
            if (inz >= 0) {  // a ghost of an inflow side holds the given state
#pragma unroll
                for (int f = 0; f < NF; ++f) q[f] = a.bc_state[2][inz][f];
                return;
            }
        }
        const double *src = a.U + yoff + (long long)cz * sz + (x0 + lx);
#pragma unroll
        for (int f = 0; f < NF; ++f) q[f] = __ldg(src + f * N);
        if (fz_) q[3] = -q[3];
    };
    auto flux_store = [&](const double *q, int lx, int lz) {
        double fp[NF], fm[NF];
        split_flux_f64<3, 2, true>(q, alpha, gm1, fp, fm);
        const int o = (lz + 3) * TW + lx;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            fz[f * NZP + o] = fp[f];
            fz[(NF + f) * NZP + o] = fm[f];
        }
    };

    // the halo's 6 W points (no more than threads) are dealt from the last thread down
    double uk[NF], qd[NF];
    if (own) load_point(tx, tz, uk);
    const int t = NT - 1 - tid, hk = t / W, hx = t - hk * W, hz = hk < 3 ? hk - 3 : H + hk - 3;
    if (hk < 6) load_point(hx, hz, qd);
    if (own) flux_store(uk, tx, tz);
    if (hk < 6) flux_store(qd, hx, hz);
    __syncthreads();

    {
        // the shared arrays hold 2 f(+/-): reconstruct with 4 eps (twice the WENO5 value)
        const PairEps P = pair_eps(4.0 * a.eps);
#pragma unroll 1
        for (int run = tid; run < 2 * NF * W; run += NT) {
            const int fs = run / W, lx = run - fs * W;
            int po = fs * NZP + lx, oo = fs * NZI + lx, st = TW;
            if (fs >= NF) {  // WENO(-): the same run read backwards from the far end
                po += (H + 5) * TW;
                oo += H * TW;
                st = -TW;
            }
            weno5_slide_pair(fz, po, st, P, Fz, oo, st, H + 1, TW, rough);
        }
        __syncthreads();
        rough_windows(rough, TW, fz, Fz, P);
    }
    __syncthreads();

    const double ihz = 0.5 * a.inv_h[2];  // face fluxes are twice F^
    const double *acc = reinterpret_cast<const double *>(a.acc);
    const double *FzM = Fz + NF * NZI;
    double out[NF];
    if (own) {
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const int o = f * NZI + tz * TW + tx;
            const double dz = (Fz[o + TW] + FzM[o + TW]) - (Fz[o] + FzM[o]);
            const double r = acc[f * N + cell] + (-dz * ihz);
            if (EPI == EPI_RHS) a.Rout[f * N + cell] = r;
            else a.Uout[f * N + cell] = out[f] = stage_combine(a.stage, un[f], uk[f], r, dt);
        }
    }
    if constexpr (EPI == EPI_STAGE)
        speed_max_publish_f64<3, PD ? 4 : 1>(
            [&](long long, double *q) {
#pragma unroll
                for (int f = 0; f < NF; ++f) q[f] = out[f];
            },
            0, own ? 1 : 0, 1, a.gamma, a.gg_f, &a.ctl->alpha[a.slot_out], a.ctl->alpha_dir[a.slot_out], &a.ctl->status);
}

// Measured at 97 x 83 x 61, L(U) (us): 11 x 11 580, 9 x 11 587, 25 x 9 597, 17 x 13 604.
Tile64 plan_z(const long long n[3])
{
    using namespace zs;
    Tile64 best{};
    double least = -1.0;
    for (int mw = (int)std::min(8ll, n[0]); mw <= MW; ++mw)
        for (int mh = 1; mh <= MH; ++mh)
            for (int nt = 128; nt <= MNT; nt += 128) {
                Tile64 t{mw, mh, 0, 0, nt, 0};
                if (fit_extent(n[0], mw) != mw || fit_extent(n[2], mh) != mh) break;
                const int points = mw * (mh + 6), faces = mw * (mh + 1);
                t.smem = (unsigned)(2 * NF * (8 * points + 12 * faces));
                if (mw * mh > nt || 6 * mw > nt || 2 * NF * points > 8192) continue;
                const long long tiles = (n[0] + mw - 1) / mw * ((n[2] + mh - 1) / mh) * n[1];
                const double c = tile64_cycles(tiles, t, 96, mw * mh, 62.0, 6 * mw, 2 * NF * mw, mh + 1);
                if (c >= 0.0 && (least < 0.0 || c < least)) {
                    least = c;
                    best = t;
                }
            }
    return best;
}

template <int EPI, bool PD>
static cudaError_t launch_z_t(const SweepArgs &a, cudaStream_t s)
{
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_z<EPI, PD>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    const Tile64 &t = a.tz;
    if (t.nt == 0) return cudaErrorInvalidConfiguration;
    const long long gx = (a.n[0] + t.w - 1) / t.w, gz = (a.n[2] + t.s - 1) / t.s;
    k_z<EPI, PD><<<dim3((unsigned)(gx * gz), (unsigned)a.n[1]), t.nt, t.smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_z(int epi, const SweepArgs &a, cudaStream_t s)
{
#define X(E, P) \
    if (epi == E && (a.per_dir != 0) == P) return launch_z_t<E, P>(a, s);
    X(EPI_RHS, false) X(EPI_STAGE, false) X(EPI_RHS, true) X(EPI_STAGE, true)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace wg
