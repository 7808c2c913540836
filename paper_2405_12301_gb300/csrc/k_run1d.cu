// k_run1d.cu -- whole SSP-RK3 steps of a small 1D FP64 Euler grid in one launch.
//
// A 1D grid of some hundred cells is all latency: three stage kernels and two
// control kernels per step, each a few microseconds of launch and of dependent
// FP64 instructions (~76 cycles each per warp, the FP64 pipe's width) on three
// SMs.  Here one thread-block cluster of 8 CTAs keeps the state in shared memory
// for as many steps as the launch is given; a stage is one pass and one cluster
// barrier, after which a CTA reads its neighbours' edge cells and all CTAs'
// wavespeed maxima through distributed shared memory.  The state is double
// buffered, so one barrier per stage separates the reads of a stage from the
// writes of the next.
//   256 cells, 64 steps: 2.36 ms as five kernels per step, 1.14 ms here.
// Up to 2048 cells (256 per CTA, one cell per thread); larger grids have more
// FP64 work than 8 SMs do in the time of the launches saved.
// The arithmetic is that of k_sweep and of the step control (k_aux.cu), bit for bit.
#include <cooperative_groups.h>

#include "weno_dev.cuh"
#include "weno_internal.h"

namespace wg {

namespace cg = cooperative_groups;

namespace r1 {
constexpr int NT = 256, NCL = 8;     // threads (and cells at most) per CTA, CTAs per cluster
constexpr int NF = 3;
constexpr int NP = NT + 6;           // points of a CTA with its halo
constexpr int NI = NT + 1;           // interfaces
}  // namespace r1

template <bool PD>
__global__ void __launch_bounds__(r1::NT) k_run1d(const SweepArgs a, double *U, int nsteps)
{
    using namespace r1;
    constexpr int K = PD ? 2 : 1;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tid = threadIdx.x;
    const int n = a.n[0], chunk = (n + NCL - 1) / NCL;
    const int lo = min(rank * chunk, n), cnt = min(n, lo + chunk) - lo;

    __shared__ double q[2][NF][NT];                  // the CTA's cells, double buffered
    __shared__ double sf[2 * NF][NP];                // split fluxes f(+), then f(-)
    __shared__ double sF[2 * NF][NI];                // WENO values at the interfaces
    __shared__ unsigned list[2 * NF * NI];
    __shared__ int s_rough, s_bad;
    __shared__ unsigned long long s_max[2][K];       // wavespeed maxima of the state in the same buffer
    __shared__ double s_al[K], s_dt, s_tn;
    const RoughList rough{&s_rough, list};
    const PairEps P = pair_eps(a.eps);
    const double gm1 = a.gamma - 1.0;

    // the run's control values: every CTA advances its own copy, rank 0 stores it
    double t = a.ctl->t;
    const double t_end = a.ctl->t_end, dt_req = a.ctl->dt_req, cfl_h = a.ctl->cfl_h;
    const long long steps0 = a.ctl->steps, max_steps = a.ctl->max_steps;
    long long steps = steps0;
    double dt = 0.0, tn = t, al[K];
    al[0] = __longlong_as_double((long long)a.ctl->alpha[0]);
    if (PD) al[K - 1] = __longlong_as_double((long long)a.ctl->alpha_dir[0][0]);

    double un[NF], uk[NF];
    if (tid < cnt) {
#pragma unroll
        for (int f = 0; f < NF; ++f) q[0][f][tid] = uk[f] = U[f * a.N + lo + tid];
    }
    int buf = 0;
    cl.sync();

    for (int st = 0; st < nsteps; ++st) {
        if (tid == 0) {
            if (next_dt(t, t_end, dt_req, cfl_h, al[0], steps, max_steps, s_dt, s_tn) && rank == 0)
                atomicOr(&a.ctl->status, ST_NONPHYSICAL);
        }
        __syncthreads();
        dt = s_dt;
        tn = s_tn;
        if (!(dt > 0.0)) break;  // the same on every CTA: the rest of the launch is no-ops
#pragma unroll
        for (int f = 0; f < NF; ++f) un[f] = uk[f];
#pragma unroll 1
        for (int stage = 0; stage < 3; ++stage) {
            const double alx = al[K - 1];
            // split fluxes of the CTA's cells and of three cells on either side
            for (int p = tid; p < cnt + 6 && cnt > 0; p += NT) {
                double s[NF], fp[NF], fm[NF];
                bool flip;
                int inflow;
                const int c = ghost_map(lo + p - 3, n, a.bc[0][0], a.bc[0][1], flip, inflow);
                const int owner = c / chunk;
                const double *src = &q[buf][0][0];
                if (owner != rank) src = cl.map_shared_rank(src, owner);
#pragma unroll
                for (int f = 0; f < NF; ++f) s[f] = inflow >= 0 ? a.bc_state[0][inflow][f] : src[f * NT + c - owner * chunk];
                if (flip) s[1] = -s[1];
                split_flux_f64<1, 0>(s, alx, gm1, fp, fm);
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    sf[f][p] = fp[f];
                    sf[NF + f][p] = fm[f];
                }
            }
            if (tid == 0) s_rough = 0;
            __syncthreads();
            // the interfaces' WENO(+) and WENO(-) values, in runs as short as the threads allow
            if (cnt > 0) {
                const int len = (2 * NF * (cnt + 1) + NT - 1) / NT, nseg = (cnt + len) / len;
                for (int u = tid; u < 2 * NF * nseg; u += NT) {
                    const int fs = u / nseg, j0 = (u - fs * nseg) * len, m = min(len, cnt + 1 - j0);
                    const bool minus = fs >= NF;
                    if (m > 0)
                        weno5_slide_pair(&sf[0][0], fs * NP + (minus ? j0 + m + 4 : j0), minus ? -1 : 1, P, &sF[0][0],
                                            fs * NI + (minus ? j0 + m - 1 : j0), minus ? -1 : 1, m, 1, rough);
                }
            }
            __syncthreads();
            rough_windows(rough, 1, &sf[0][0], &sF[0][0], P);
            __syncthreads();
            const bool own = tid < cnt;
            if (own) {
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    const double r = -((sF[f][tid + 1] + sF[NF + f][tid + 1]) - (sF[f][tid] + sF[NF + f][tid])) * a.inv_h[0];
                    uk[f] = stage_combine(stage, un[f], uk[f], r, dt);
                    q[buf ^ 1][f][tid] = uk[f];
                }
            }
            buf ^= 1;
            speed_max_block_f64<1, K>(
                [&](long long, double *s) {
#pragma unroll
                    for (int f = 0; f < NF; ++f) s[f] = uk[f];
                },
                0, own ? 1 : 0, 1, a.gamma, a.gg_f, s_max[buf], &s_bad);
            __syncthreads();
            if (tid == 0 && s_bad) atomicOr(&a.ctl->status, ST_NONPHYSICAL);
            cl.sync();
            if (tid < 32) {  // the maximum over the CTAs, on the integer pipe
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    unsigned long long m = tid < NCL ? *cl.map_shared_rank(&s_max[buf][k], tid) : 0ull;
                    const unsigned mh = __reduce_max_sync(0xFFFFFFFFu, (unsigned)(m >> 32));
                    const unsigned ml = __reduce_max_sync(0xFFFFFFFFu, (unsigned)(m >> 32) == mh ? (unsigned)m : 0u);
                    if (tid == 0) s_al[k] = __hiloint2double((int)mh, (int)ml);
                }
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < K; ++k) al[k] = s_al[k];
        }
        t = tn;
        ++steps;
    }
    cl.sync();  // no CTA leaves while another may still read its cells
    if (steps != steps0 && tid < cnt) {
#pragma unroll
        for (int f = 0; f < NF; ++f) U[f * a.N + lo + tid] = uk[f];
    }
    if (rank == 0 && tid == 0) {
        a.ctl->t = t;
        a.ctl->t_next = t;
        a.ctl->dt = dt;
        a.ctl->steps = steps;
        a.ctl->alpha[0] = (unsigned long long)__double_as_longlong(al[0]);
        if (PD) a.ctl->alpha_dir[0][0] = (unsigned long long)__double_as_longlong(al[K - 1]);
    }
}

bool run1d_takes(long long n) { return n <= r1::NT * r1::NCL; }

cudaError_t launch_run1d(const SweepArgs &a, double *U, int nsteps, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(r1::NCL);
    cfg.blockDim = dim3(r1::NT);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = r1::NCL;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return a.per_dir ? cudaLaunchKernelEx(&cfg, k_run1d<true>, a, U, nsteps)
                     : cudaLaunchKernelEx(&cfg, k_run1d<false>, a, U, nsteps);
}

}  // namespace wg
