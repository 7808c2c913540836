// k_aux.cu -- small kernels around the residual sweeps: the global
// wavespeed max (LF alpha, Sec. 4.3), the device-side time-step control
// (dt = lambda h / alpha with the last step shortened to land on t_end,
// Eq. cfl-other), and the fixed-order FP64 conservation sums.
#include <algorithm>
#include <climits>

#include "weno_dev.cuh"
#include "weno_internal.h"

namespace wg {

// Start of a step: dt from alpha(U^n) (or the fixed dt), shortened so that the
// time lands exactly on t_end; zero when the time is up or the step budget of
// the current call is spent.  Clears the stage alpha slots 1..3.  (Values in
// registers: one thread runs this, and every dependent load costs it ~0.4 us.)
__device__ __forceinline__ void step_begin(Ctl *c, double t, double t_end, double dt_req, double cfl_h,
                                           unsigned long long alpha, long long steps, long long max_steps)
{
    double dt, tn;
    if (next_dt(t, t_end, dt_req, cfl_h, __longlong_as_double((long long)alpha), steps, max_steps, dt, tn))
        atomicOr(&c->status, ST_NONPHYSICAL);
    c->dt = dt;
    c->t_next = tn;
    c->bdt[0] = f64_to_f32x2(dt);
    c->bdt[1] = f64_to_f32x2(0.25 * dt);
    c->bdt[2] = f64_to_f32x2(2.0 / 3.0 * dt);
    for (int k = 1; k < 4; ++k) {
        c->alpha[k] = 0ull;
        for (int e = 0; e < 3; ++e) c->alpha_dir[k][e] = 0ull;
    }
}

// The end of every block of an alpha kernel; the last block's takes the maxima to slot
// 0, clears them for the next launch and does what follows -- launches of one thread
// each (clear, set the run, begin, copy out) before.
__device__ void alpha_done(Ctl *c, const AlphaThen &then)
{
    __syncthreads();
    if (threadIdx.x != 0) return;
    const double t = c->t;
    const long long steps = c->steps;
    __threadfence();
    if (atomicAdd(&c->ticket, 1u) != gridDim.x - 1) return;
    __threadfence();
    c->ticket = 0u;
    unsigned long long m[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) m[e] = __ldcg(&c->alpha_new[e]);
    c->alpha[0] = m[0];
#pragma unroll
    for (int e = 0; e < 4; ++e) c->alpha_new[e] = 0ull;
#pragma unroll
    for (int e = 0; e < 3; ++e) c->alpha_dir[0][e] = m[1 + e];
    if (then.out) *then.out = __longlong_as_double((long long)m[0]);
    if (!then.set_run) return;
    const long long max_steps = (then.max_steps > LLONG_MAX - steps) ? LLONG_MAX : steps + then.max_steps;
    c->t_end = then.t_end;
    c->dt_req = then.dt_req;
    c->cfl_h = then.cfl_h;
    c->max_steps = max_steps;
    if (then.begin) step_begin(c, t, then.t_end, then.dt_req, then.cfl_h, m[0], steps, max_steps);
}

// alpha of an FP64 state (PD: and the per-direction speeds).  Bound by the FP64
// pipe if every cell's speed is formed there (84% busy at 97 x 83 x 61); the FP32
// estimates leave it a handful of cells per block, so few large blocks: at 97 x 83 x 61
// 1216 blocks of 256 threads took 27 us, 304 of 512 take 17.
constexpr int ALPHA_NT = 512;
template <int D, bool PD>
__global__ void __launch_bounds__(ALPHA_NT, 2) k_alpha(const double *__restrict__ U, long long N, double gamma, float gg,
                                                       Ctl *ctl, const AlphaThen then)
{
    speed_max_publish_f64<D, PD ? 1 + D : 1>(
        [&](long long i, double *q) {
#pragma unroll
            for (int f = 0; f < D + 2; ++f) q[f] = __ldg(U + f * N + i);
        },
        (long long)blockIdx.x * blockDim.x + threadIdx.x, N, (long long)gridDim.x * blockDim.x, gamma, gg, &ctl->alpha_new[0],
        &ctl->alpha_new[1], &ctl->status);
    alpha_done(ctl, then);
}

// The same for the FP32-bulk mode: FP32 speeds, their maximum widened exactly.  Bound
// by memory: a thread loads four cells before it uses the first (one cell at a time
// took 45 us at 2048 x 2048, 3 TB/s; now 28).
template <int D>
__global__ void __launch_bounds__(256, 4) k_alpha_bulk(const double *__restrict__ U, long long N, float gamma, float gm1,
                                                       Ctl *ctl, int per_dir, const AlphaThen then)
{
    constexpr int NF = D + 2, UN = 4;
    float mf = 0.0f, mdf[D];
#pragma unroll
    for (int e = 0; e < D; ++e) mdf[e] = 0.0f;
    bool bad = false;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += UN * step) {
        double u[UN][NF];
#pragma unroll
        for (int k = 0; k < UN; ++k) {
#pragma unroll
            for (int f = 0; f < NF; ++f) u[k][f] = i + k * step < N ? __ldg(U + f * N + i + k * step) : 0.0;
        }
#pragma unroll
        for (int k = 0; k < UN; ++k) {
            if (i + k * step >= N) break;
            float qf[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) qf[f] = f64_to_f32(u[k][f]);
            bool b;
            mf = fmaxf(mf, wavespeed_f32<D>(qf, gamma, gm1, b));
            if (per_dir) {
                float sd[D];
                dirspeeds_f32<D>(qf, gamma, gm1, sd);
#pragma unroll
                for (int e = 0; e < D; ++e) mdf[e] = fmaxf(mdf[e], b ? 0.0f : sd[e]);
            }
            bad |= b;
        }
    }
    block_max_publish_f32(mf, bad, &ctl->alpha_new[0], &ctl->status);
    if (per_dir) {
#pragma unroll
        for (int e = 0; e < D; ++e) block_max_publish_f32(mdf[e], false, &ctl->alpha_new[1 + e], &ctl->status);
    }
    alpha_done(ctl, then);
}

// Scalar laws: alpha = max |f'(u)| (1 for advection, |u| for Burgers).
template <int M>
__global__ void __launch_bounds__(256) k_alpha_scalar(const double *__restrict__ U, long long N, Ctl *ctl, const AlphaThen then)
{
    double m = 0.0;
    bool bad = false;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        const double u = __ldg(U + i);
        bad |= !isfinite(u);
        m = fmax(m, M == MODEL_ADVECT ? 1.0 : fabs(u));
    }
    block_max_publish(m, bad, &ctl->alpha_new[0], &ctl->status);
    alpha_done(ctl, then);
}

// End of a step: advance the time and carry alpha(U^{n+1}) into slot 0; within a run
// also the start of the next.
__global__ void k_step_end(Ctl *c, int begin)
{
    const double dt = c->dt, t0 = c->t, tn = c->t_next;
    const double t_end = c->t_end, dt_req = c->dt_req, cfl_h = c->cfl_h;
    const long long s0 = c->steps, max_steps = c->max_steps;
    const unsigned long long a0 = c->alpha[0], a3 = c->alpha[3];
    unsigned long long ad[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) ad[e] = c->alpha_dir[3][e];
    const bool took = dt > 0.0;
    if (took) {
        c->t = tn;
        c->steps = s0 + 1;
        c->alpha[0] = a3;
#pragma unroll
        for (int e = 0; e < 3; ++e) c->alpha_dir[0][e] = ad[e];
    }
    if (begin) step_begin(c, took ? tn : t0, t_end, dt_req, cfl_h, took ? a3 : a0, took ? s0 + 1 : s0, max_steps);
}

// Two-level fixed-order sums: block b reduces a fixed contiguous chunk of
// cells with a fixed tree; one block then reduces the partials in order.
constexpr int SUM_NT = 256;

__device__ __forceinline__ double block_sum_fixed(double v, double *sh)
{
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = SUM_NT / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(SUM_NT) k_sums_partial(const double *__restrict__ U, int nf, long long N,
                                                         long long chunk, double *partials)
{
    __shared__ double sh[SUM_NT];
    const long long b0 = (long long)blockIdx.x * chunk;
    const long long b1 = b0 + chunk < N ? b0 + chunk : N;
    for (int f = 0; f < nf; ++f) {
        double s = 0.0;
        for (long long i = b0 + threadIdx.x; i < b1; i += SUM_NT) s += U[f * N + i];
        s = block_sum_fixed(s, sh);
        if (threadIdx.x == 0) partials[(long long)blockIdx.x * nf + f] = s;
    }
}

__global__ void __launch_bounds__(SUM_NT) k_sums_final(const double *partials, int nblocks, int nf, double *out)
{
    __shared__ double sh[SUM_NT];
    for (int f = 0; f < nf; ++f) {
        double s = 0.0;
        for (int b = threadIdx.x; b < nblocks; b += SUM_NT) s += partials[(long long)b * nf + f];
        s = block_sum_fixed(s, sh);
        if (threadIdx.x == 0) out[f] = s;
    }
}

int sums_blocks(long long N)
{
    const long long b = (N + 4095) / 4096;
    return (int)(b < 1024 ? (b < 1 ? 1 : b) : 1024);
}

cudaError_t launch_sums(const double *U, int nf, long long N, double *partials, int nblocks, double *out,
                        cudaStream_t s)
{
    const long long chunk = (N + nblocks - 1) / nblocks;
    k_sums_partial<<<nblocks, SUM_NT, 0, s>>>(U, nf, N, chunk, partials);
    k_sums_final<<<1, SUM_NT, 0, s>>>(partials, nblocks, nf, out);
    return cudaGetLastError();
}

int sm_count()
{
    static int cache[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
    if (cache[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 152;
        cache[dev] = n;
    }
    return cache[dev];
}

cudaError_t launch_alpha(int model, int dim, bool bulk, const double *U, long long N, double gamma, Ctl *ctl,
                         int per_dir, const AlphaThen &then, cudaStream_t s)
{
    int blocks = (int)((N + 255) / 256);
    if (blocks > sm_count() * 8) blocks = sm_count() * 8;
    if (blocks < 1) blocks = 1;
    if (model == MODEL_ADVECT) k_alpha_scalar<MODEL_ADVECT><<<blocks, 256, 0, s>>>(U, N, ctl, then);
    if (model == MODEL_BURGERS) k_alpha_scalar<MODEL_BURGERS><<<blocks, 256, 0, s>>>(U, N, ctl, then);
    if (model != MODEL_EULER) return cudaGetLastError();
    const float gm1 = speed_gm1(gamma), gg = (float)(gamma * (gamma - 1.0));
    const int big = (int)std::min<long long>((N + ALPHA_NT - 1) / ALPHA_NT, 2 * sm_count());
#define X(D)                                                                                        \
    if (dim == D && bulk)                                                                           \
        k_alpha_bulk<D><<<blocks < sm_count() * 4 ? blocks : sm_count() * 4, 256, 0, s>>>(U, N, (float)gamma, gm1, ctl, per_dir, then); \
    else if (dim == D && per_dir) k_alpha<D, true><<<big, ALPHA_NT, 0, s>>>(U, N, gamma, gg, ctl, then);   \
    else if (dim == D) k_alpha<D, false><<<big, ALPHA_NT, 0, s>>>(U, N, gamma, gg, ctl, then);
    X(1) X(2) X(3)
#undef X
    return cudaGetLastError();
}

cudaError_t launch_step_end(Ctl *ctl, bool begin, cudaStream_t s)
{
    k_step_end<<<1, 1, 0, s>>>(ctl, begin ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace wg
