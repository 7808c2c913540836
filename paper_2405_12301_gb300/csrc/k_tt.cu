// k_tt.cu -- batched TT-rounding of 3D tensor trains in FP64 (Sec. 3
// "TT-rounding", the two-pass algorithm of Oseledets 2011, Algorithm 2), the
// rounding behind every stage of Eq. (tt-ssprk3).
//
// Building blocks, each a batched kernel over independent problems:
//   * k_qr_factor: Householder QR of a tall-skinny m x k matrix (k <= 96),
//     a TSQR tree.  A chunk of rows is factored by one CTA as a flat tree:
//     a plain Householder QR of its first b rows, then for every further
//     sub-block B of b rows the structured QR of [R; B] whose reflectors are
//     [e_j; y_j].  The chunk R factors are stacked and factored the same way
//     by further launches, a few R's per CTA, until one is left; there the first
//     block is an R already and reflector j of the others has j + 1 rows.
//     Reflectors overwrite the matrix; taus are kept.
//   * k_qr_apply: Q [X; 0] for a k x p block X, replaying the reflectors of a
//     chunk in reverse (eight lanes per column of X, four columns per warp,
//     no block barrier inside a sub-block); writes the rows through a general row map so that results
//     land directly in TT-core layout.
//   * k_svd_jacobi: SVD T = V S U^T of a k x q triangular factor by a QR with
//     column pivoting and one-sided Jacobi (round-robin pair ordering); picks the
//     truncation rank from the singular values and writes V's kept columns and
//     (U S)'s kept columns.  The rows that Jacobi rotates are spread over the CTAs
//     of a cluster: a rotation acts on every row alone, only the dot products that
//     choose the angles are sums over all of them.
//   * k_tt_build / k_tt_contract / k_tt_gemm_tr: the TT sum's first and last
//     unfoldings, the block-diagonal middle core times a triangular factor, and
//     a small dense product.
// All sums, factors and vectors are FP64.  FP32 only steers: the pivot norms and the
// tangents of the Jacobi angles (k_svd_jacobi), and the seeds of Newton iterations.
#include <algorithm>
#include <cfloat>

#include <cooperative_groups.h>

#include "weno_dev.cuh"
#include "weno_internal.h"
#include "tt_internal.h"

namespace wg {

namespace cg = cooperative_groups;

constexpr int TT_NT = 256, TT_NW = TT_NT / 32;

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// The update loops below give each column of a reflector update to a group of
// LPC lanes (CPW = 32 / LPC columns per warp, a lane every LPC-th row).  On
// this GPU every FP64 warp instruction holds the FP64 pipe however many lanes
// it serves, so the group's shuffle adds (log2 LPC per lane), the redundant
// w = tau (dot + x_j) on every lane of the group and the one-lane diagonal
// update are pure overhead on top of the 2 FMAs per row: 4 lanes keep it near
// 15% (8 lanes cost about 35%).  Sub-blocks are stored with a pitch of b + 4
// (b a multiple of 32), so a half-warp's 4 columns x 4 rows hit 16 distinct
// banks.
constexpr int LPC = 4, CPW = 32 / LPC, LDPAD = 4;

__device__ __forceinline__ double group_sum(double v)
{
#pragma unroll
    for (int o = LPC / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// 1 / sqrt(s) of a normal s: an FP32 seed on the mantissa (scaled by an even power
// of two to [1, 4)), two Newton-Raphson steps y (3 - s y^2) / 2.
__device__ __forceinline__ double rsqrt_f64(double s)
{
    const int h = __double2hiint(s), e2 = ((h >> 20) - 1023) & ~1;  // the even exponent
    const double m = __hiloint2double(h - (e2 << 20), __double2loint(s));
    float f;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(f64_to_f32(m)));
    double y = f32_to_f64_nz(f);
#pragma unroll
    for (int k = 0; k < 2; ++k) y = fma(0.5 * y, fma(-m * y, y, 1.0), y);
    return __hiloint2double(__double2hiint(y) - ((e2 / 2) << 20), __double2loint(y));
}

// The turn of a warp in taking column groups, from its distance to the warp that is
// ahead: the warps that do not share its sub-partition first, itself last.
__device__ __forceinline__ int turn(int dist) { return (0x54362107 >> ((dist & 7) * 4)) & 7; }

// Householder vector of x = (x0, y) with ||y||^2 = sig: H = I - tau v v^T,
// v = (1, y / (x0 - beta)), H x = (beta, 0).  sig == 0 gives tau = 0.  Every column
// waits for this chain of dependent FP64 operations (68 cycles each), so it takes
// one reciprocal square root and one reciprocal by Newton's method (18 operations;
// with sqrt and two divisions ~40).
__device__ __forceinline__ void householder(double x0, double sig, double &beta, double &tau, double &scale)
{
    beta = x0;
    tau = 0.0;
    scale = 0.0;
    if (sig > 0.0) {
        const double s = fma(x0, x0, sig);
        if (s > 1e-280 && s < 1e280) {
            const double y = rsqrt_f64(s);
            double b = s * y;
            b = fma(fma(-b, b, s), 0.5 * y, b);
            beta = -copysign(b, x0);
            tau = fma(-x0, -copysign(y, x0), 1.0);  // 1 - x0 / beta
            scale = rcp_f64(x0 - beta);
        } else {
            beta = -copysign(sqrt(s), x0);
            tau = (beta - x0) / beta;
            scale = 1.0 / (x0 - beta);
        }
    }
}

size_t qr_factor_smem(int k, int b) { return sizeof(double) * ((size_t)k * (b + LDPAD) + (size_t)k * (k + 1) + k); }
size_t qr_apply_smem(int k, int b, int p)
{
    return sizeof(double) * ((size_t)k * (b + LDPAD) + (size_t)p * (b + LDPAD) + (size_t)p * (k + 1) + k);
}
constexpr int SV_MAXCL = 8;  // CTAs per SVD at most
size_t svd_smem(int pk, int q, int ncl)
{
    const size_t m = (size_t)pk * ((2 * ((pk + ncl - 1) / ncl)) | 1);
    return sizeof(double) * ((size_t)pk * (q | 1) + 2 * ncl * 3 * (TT_KMAX / 2) + (m > 8 * (size_t)(q | 1) ? m : 8 * (size_t)(q | 1)));
}

// CTAs per matrix: as many as the GPU has SMs for, at most 8 and at least 6 rows
// each; two where one CTA's shared memory would not do.
constexpr int SV_ONE = 88;  // largest matrix of a single CTA
int svd_cluster(int n, int max_pk)
{
    int ncl = SV_MAXCL;
    const int least = max_pk > SV_ONE ? 2 : 1;
    while (ncl > least && ((long long)n * ncl > sm_count() || max_pk / ncl < 6)) ncl /= 2;
    return ncl;
}

// The column loop keeps one reflector ahead: while the other warps apply reflector
// j to their columns, one warp applies it to column j + 1 and forms reflector j + 1
// from it, so that chain (~35 dependent FP64 operations) runs beside the updates
// and a column takes one barrier.  The other column groups go first to the warps of
// the other three sub-partitions: a sub-partition issues an FP64 instruction every 64
// cycles, whatever its warps.  A 64-row sub-block
// of 64 columns takes 185 us (195 with the updates before the next reflector), a
// triangular merge of 58 columns 158.
__global__ void __launch_bounds__(TT_NT) k_qr_factor(const QRDesc *descs)
{
    const QRDesc &d = descs[blockIdx.y];
    const int chunk = blockIdx.x;
    if (chunk >= d.chunks || d.m <= 0) return;
    extern __shared__ double sm[];
    const int k = d.k, b = d.tri ? k : d.b, ldb = d.b + LDPAD, ldr = k + 1;
    double *B = sm;                       // sub-block, column-major [k][ldb]
    double *R = B + (size_t)k * ldb;      // running R, column-major [k][ldr]
    double *ts = R + (size_t)k * ldr;     // taus of the current sub-block
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = lane / LPC, sub = lane % LPC;
    const long long r0 = (long long)chunk * d.chunk_rows;
    const long long r1 = min(d.m, r0 + d.chunk_rows);

    for (int s = 0;; ++s) {
        const long long s0 = r0 + (long long)s * b;
        if (s0 >= r1) break;
        const int bs = (int)min((long long)b, r1 - s0);
        for (int e = threadIdx.x; e < bs * k; e += TT_NT) {
            const int i = e / k, c = e - i * k;
            B[c * ldb + i] = d.A[(s0 + i) * d.lda + c];
        }
        for (int j = threadIdx.x; j < k; j += TT_NT) ts[j] = 0.0;
        __syncthreads();
        const bool plain = s == 0;
        const int kk = plain ? (d.tri ? 0 : min(bs, k)) : k;  // reflectors
        // reflector j: the top element (plain: row j of B, else row j of R) and rows
        // i0 .. i1 of B's column j
        auto top = [&](int c, int j) -> double & { return plain ? B[c * ldb + j] : R[c * ldr + j]; };
        auto first = [&](int j) { return plain ? j + 1 : 0; };
        auto last = [&](int j) { return d.tri && !plain ? min(j + 1, bs) : bs; };
        auto generate = [&](int j) {  // one warp
            double *x = B + j * ldb;
            const int i0 = first(j), i1 = last(j);
            double sig = 0.0;
            for (int i = i0 + lane; i < i1; i += 32) sig = fma(x[i], x[i], sig);
            sig = warp_sum_d(sig);
            double beta, tau, scale;
            householder(top(j, j), sig, beta, tau, scale);
            for (int i = i0 + lane; i < i1; i += 32) x[i] *= scale;
            __syncwarp();  // every lane has read the top element
            if (lane == 0) {
                top(j, j) = beta;
                ts[j] = tau;
            }
        };
        if (warp == 0 && kk > 0) generate(0);
        __syncthreads();
        for (int j = 0; j < kk; ++j) {
            const double tau = ts[j];
            const double *v = B + j * ldb;
            const int i0 = first(j), i1 = last(j), ahead = j & (TT_NW - 1);
            if (warp == ahead && j + 1 < k) {
                if (tau != 0.0) {
                    double *col = B + (j + 1) * ldb;
                    double w = 0.0;
                    for (int i = i0 + lane; i < i1; i += 32) w = fma(v[i], col[i], w);
                    w = (warp_sum_d(w) + top(j + 1, j)) * tau;
                    for (int i = i0 + lane; i < i1; i += 32) col[i] = fma(-v[i], w, col[i]);
                    __syncwarp();
                    if (lane == 0) top(j + 1, j) -= w;
                    __syncwarp();
                }
                if (j + 1 < kk) generate(j + 1);
            }
            if (tau != 0.0) {
                for (int c0 = j + 2 + turn(warp - ahead) * CPW; c0 < k; c0 += TT_NW * CPW) {
                    const int c = c0 + grp;
                    const bool ok = c < k;
                    double *col = B + (ok ? c : 0) * ldb;
                    double w = 0.0, w1 = 0.0;
                    if (ok) {
                        int i = i0 + sub;
                        for (; i + LPC < i1; i += 2 * LPC) {
                            w = fma(v[i], col[i], w);
                            w1 = fma(v[i + LPC], col[i + LPC], w1);
                        }
                        if (i < i1) w = fma(v[i], col[i], w);
                    }
                    w = (group_sum(w + w1) + (ok ? top(c, j) : 0.0)) * tau;
                    if (ok)
                        for (int i = i0 + sub; i < i1; i += LPC) col[i] = fma(-v[i], w, col[i]);
                    __syncwarp();
                    if (ok && sub == 0) top(c, j) -= w;
                }
            }
            __syncthreads();
        }
        if (plain) {
            for (int e = threadIdx.x; e < k * k; e += TT_NT) {
                const int c = e / k, j = e - c * k;
                R[c * ldr + j] = (j <= c && j < min(bs, k)) ? B[c * ldb + j] : 0.0;
            }
        }
        if (kk > 0) {
            for (int e = threadIdx.x; e < bs * k; e += TT_NT) {
                const int i = e / k, c = e - i * k;
                d.A[(s0 + i) * d.lda + c] = B[c * ldb + i];
            }
        }
        for (int j = threadIdx.x; j < k; j += TT_NT) d.tau[((long long)chunk * d.sub_per_chunk + s) * k + j] = ts[j];
        __syncthreads();
    }
    for (int e = threadIdx.x; e < k * k; e += TT_NT) {
        const int j = e / k, c = e - j * k;
        d.Rout[(long long)chunk * k * k + e] = R[c * ldr + j];
    }
}

__global__ void __launch_bounds__(TT_NT) k_qr_apply(const QApplyDesc *descs)
{
    const QApplyDesc &d = descs[blockIdx.y];
    const int chunk = blockIdx.x;
    if (chunk >= d.chunks || d.m <= 0 || d.p <= 0) return;
    extern __shared__ double sm[];
    const int k = d.k, b = d.tri ? k : d.b, p = d.p, ldb = d.b + LDPAD, ldx = k + 1;
    double *Y = sm;                        // reflectors of a sub-block, column-major [k][ldb]
    double *Z = Y + (size_t)k * ldb;       // output block, column-major [p][ldb]
    double *X = Z + (size_t)p * ldb;       // running top rows, column-major [p][ldx]
    double *ts = X + (size_t)p * ldx;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = lane / LPC, sub = lane % LPC;
    const long long r0 = (long long)chunk * d.chunk_rows;
    const long long r1 = min(d.m, r0 + d.chunk_rows);
    const int nsub = (int)((r1 - r0 + b - 1) / b);
    const int b1 = (int)min((long long)b, r1 - r0);
    const int kk = min(b1, k);  // rows of X (k unless the chunk is shorter than k)
    const double *Xin = d.X ? d.X + (long long)chunk * d.x_chunk_stride : nullptr;  // null: identity
    for (int e = threadIdx.x; e < kk * p; e += TT_NT) {
        const int j = e / p, q = e - j * p;
        X[q * ldx + j] = Xin ? Xin[(long long)j * d.ldx + q] : (j == q ? 1.0 : 0.0);
    }
    __syncthreads();
    auto store = [&](long long row0, int rows) {
        for (int e = threadIdx.x; e < rows * p; e += TT_NT) {
            const int i = e / p, q = e - i * p;
            const long long row = row0 + i;
            d.out[(row % d.P) * d.sP + (row / d.P) * d.sQ + (long long)q * d.sC] = Z[q * ldb + i];
        }
    };
    for (int s = nsub - 1; s >= 1; --s) {
        const long long s0 = r0 + (long long)s * b;
        const int bs = (int)min((long long)b, r1 - s0);
        for (int e = threadIdx.x; e < bs * k; e += TT_NT) {
            const int i = e / k, c = e - i * k;
            Y[c * ldb + i] = d.A[(s0 + i) * d.lda + c];
        }
        for (int e = threadIdx.x; e < bs * p; e += TT_NT) Z[(e / bs) * ldb + e % bs] = 0.0;
        for (int j = threadIdx.x; j < k; j += TT_NT) ts[j] = d.tau[((long long)chunk * d.sub_per_chunk + s) * k + j];
        __syncthreads();
        for (int q0 = warp * CPW; q0 < p; q0 += TT_NW * CPW) {
            const int q = q0 + grp;
            const bool ok = q < p;
            double *zq = Z + (ok ? q : 0) * ldb;
            double *xq = X + (ok ? q : 0) * ldx;
            for (int j = k - 1; j >= 0; --j) {
                const double tau = ts[j];
                if (tau == 0.0) continue;
                const double *y = Y + j * ldb;
                const int i1 = d.tri ? min(j + 1, bs) : bs;
                double w = 0.0, w1 = 0.0;
                if (ok) {
                    int i = sub;
                    for (; i + LPC < i1; i += 2 * LPC) {
                        w = fma(y[i], zq[i], w);
                        w1 = fma(y[i + LPC], zq[i + LPC], w1);
                    }
                    if (i < i1) w = fma(y[i], zq[i], w);
                }
                w = (group_sum(w + w1) + (ok ? xq[j] : 0.0)) * tau;
                if (ok)
                    for (int i = sub; i < i1; i += LPC) zq[i] = fma(-y[i], w, zq[i]);
                __syncwarp();
                if (ok && sub == 0) xq[j] -= w;
                __syncwarp();
            }
        }
        __syncthreads();
        store(s0, bs);
        __syncthreads();
    }
    // first sub-block: plain reflectors below the diagonal, acting on [X; 0] (none
    // where it is an R already)
    for (int e = threadIdx.x; e < b1 * k; e += TT_NT) {
        const int i = e / k, c = e - i * k;
        Y[c * ldb + i] = d.A[(r0 + i) * d.lda + c];
    }
    for (int e = threadIdx.x; e < b1 * p; e += TT_NT) {
        const int q = e / b1, i = e - q * b1;
        Z[q * ldb + i] = i < kk ? X[q * ldx + i] : 0.0;
    }
    for (int j = threadIdx.x; j < k; j += TT_NT) ts[j] = d.tau[(long long)chunk * d.sub_per_chunk * k + j];
    __syncthreads();
    for (int q0 = warp * CPW; q0 < p; q0 += TT_NW * CPW) {
        const int q = q0 + grp;
        const bool ok = q < p;
        double *zq = Z + (ok ? q : 0) * ldb;
        for (int j = kk - 1; j >= 0; --j) {
            const double tau = ts[j];
            if (tau == 0.0) continue;
            const double *v = Y + j * ldb;
            double w = 0.0;
            if (ok)
                for (int i = j + 1 + sub; i < b1; i += LPC) w = fma(v[i], zq[i], w);
            w = (group_sum(w) + (ok ? zq[j] : 0.0)) * tau;
            if (ok)
                for (int i = j + 1 + sub; i < b1; i += LPC) zq[i] = fma(-v[i], w, zq[i]);
            __syncwarp();
            if (ok && sub == 0) zq[j] -= w;
            __syncwarp();
        }
    }
    __syncthreads();
    store(r0, b1);
}

// SVD of T (pk x q row-major, pk <= q): one-sided Jacobi, preconditioned by a QR with
// column pivoting.  T^T P = Q R, Jacobi makes the columns of the lower triangular
// R^T orthogonal, R^T J = Z, so T = P R^T Q^T = (P Z) (Q J)^T: the left vectors are
// the columns of P Z over their norms sigma, and sigma u = Q J sigma.  On R^T Jacobi
// takes 5 sweeps where it takes 8 to 10 on T^T itself (the nearly dependent columns
// of a TT sum; 64 x 64).
//   1. pivoted Householder QR of T^T, every CTA of the cluster the same;
//   2. Jacobi: each CTA holds all columns of a slice of Z's and J's rows.  Per round
//      of disjoint pairs: partial dot products over the slice (a lane per pair, a
//      warp per quantity), pushed to every CTA; one cluster barrier; the sums of the
//      partials, the angle (a lane per pair, every CTA the same); the rotations of
//      the slice (a lane per pair, a warp per row).  The tangent of the angle is formed in FP32
//      (with Newton steps for cos = 1 / sqrt(1 + t^2)): it only steers, the rotation
//      is orthogonal to FP64 rounding whatever t is.  Every pair beyond 4 eps is
//      rotated; the sweeps end when no pair's cosine was above 8 max(pk, q) eps.
//   3. each CTA applies Q to its share of the columns of J sigma.
// A round is a chain of latencies (FP64 68 cycles each, a cluster barrier), not
// work: 10 matrices of 50..64, 5.1 ms on one CTA each without the QR, 3.6 ms on 8
// CTAs with pulled partials and no QR, 1.3 - 1.8 ms here.
// Cluster size 1..8 (svd_cluster): fewer CTAs where the batch fills the GPU.
__global__ void __launch_bounds__(TT_NT) k_svd_jacobi(const SvdDesc *descs)
{
    cg::cluster_group cl = cg::this_cluster();
    const int ncl = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const SvdDesc &d = descs[blockIdx.y];
    const int pk = d.pk, q = d.q;
    if (pk <= 0) return;  // the same for every CTA of the cluster
    extern __shared__ double sm[];
    constexpr int NPR = TT_KMAX / 2;
    __shared__ double sig[TT_KMAX], ts[TT_KMAX], s_cs[NPR], s_sn[NPR], s_tot[3][NPR];
    __shared__ float nrm[TT_KMAX];
    __shared__ int s_uv[NPR][2], ord[TT_KMAX], perm[TT_KMAX], rotated, s_rank, s_exp;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = lane / LPC, sub = lane % LPC;
    const int pa = rank * pk / ncl, pn = (rank + 1) * pk / ncl - pa;   // rows of Z and of J
    const int lda = q | 1, ldm = (2 * pn) | 1;
    double *A = sm;                          // [pk][lda]: T^T column-major, then its reflectors and R
    // the CTAs' partial dot products (z_u . z_u, z_v . z_v, z_u . z_v), double buffered:
    // part + ((par * ncl + CTA) * 3 + k) * NPR
    double *part = A + (size_t)pk * lda;
    double *M = part + 2 * ncl * 3 * NPR;    // [pk][ldm]: pn rows of Z, then pn rows of J
    if (threadIdx.x == 0) s_exp = 0;
    __syncthreads();
    for (int e = threadIdx.x; e < pk * q; e += TT_NT) {
        const int t = e / q, i = e - t * q;
        const double x = d.T[(long long)t * d.ldt + i];
        A[t * lda + i] = x;
        atomicMax(&s_exp, (__double2hiint(x) >> 20) & 0x7FF);
    }
    for (int t = threadIdx.x; t < pk; t += TT_NT) perm[t] = t;
    __syncthreads();
    // T over a power of four near its largest entry, so that the squares that Jacobi
    // works on stay normal whatever T's scale is (a T of norm 1e-146 left its small
    // columns, of norms below 2^-511, unrotated; exact, so no bit of the result moves
    // where nothing underflowed); the singular values are scaled back at the end
    const int e4 = max(-1000, min(1000, (s_exp - 1023) & ~1));
    const double down = __hiloint2double((1023 - e4) << 20, 0), up = __hiloint2double((1023 + e4) << 20, 0);
    for (int e = threadIdx.x; e < pk * q; e += TT_NT) A[(e / q) * lda + e % q] *= down;
    __syncthreads();
    // FP32 value of x over the power of two of T's largest entry (0 below 2^-60 of it)
    const int eoff = s_exp - 1023 - e4;
    auto relative = [&](double x) {
        const int h = __double2hiint(x), ex = ((h >> 20) & 0x7FF) - eoff;
        const unsigned b = ((unsigned)(ex - 896) << 23) | (((unsigned)h & 0xFFFFFu) << 3) | ((unsigned)__double2loint(x) >> 29);
        return ex < 963 ? 0.0f : __uint_as_float(b);
    };

    // ---- 1. QR with column pivoting (the pivot by FP32 norms of what is left: it only
    // has to be near the largest)
    for (int j = 0; j < pk; ++j) {
        for (int c = j + warp * CPW + grp; c < pk + grp; c += TT_NW * CPW) {  // (whole warps: c - grp < pk)
            float s = 0.0f;
            if (c < pk)
                for (int i = j + sub; i < q; i += LPC) {
                    const float x = relative(A[c * lda + i]);
                    s = fmaf(x, x, s);
                }
#pragma unroll
            for (int o = LPC / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
            if (c < pk && sub == 0) nrm[c] = s;
        }
        __syncthreads();
        if (warp == 0) {
            float best = -1.0f;
            int bc = j;
            for (int c = j + lane; c < pk; c += 32)
                if (nrm[c] > best) {
                    best = nrm[c];
                    bc = c;
                }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float ob = __shfl_xor_sync(0xFFFFFFFFu, best, o);
                const int oc = __shfl_xor_sync(0xFFFFFFFFu, bc, o);
                if (ob > best || (ob == best && oc < bc)) {
                    best = ob;
                    bc = oc;
                }
            }
            if (bc != j)
                for (int i = lane; i < q; i += 32) {
                    const double x = A[j * lda + i];
                    A[j * lda + i] = A[bc * lda + i];
                    A[bc * lda + i] = x;
                }
            __syncwarp();
            double *x = A + j * lda;
            double s = 0.0;
            for (int i = j + 1 + lane; i < q; i += 32) s = fma(x[i], x[i], s);
            s = warp_sum_d(s);
            double beta, tau, scale;
            householder(x[j], s, beta, tau, scale);
            for (int i = j + 1 + lane; i < q; i += 32) x[i] *= scale;
            __syncwarp();  // every lane has read x[j]
            if (lane == 0) {
                x[j] = beta;
                ts[j] = tau;
                const int p = perm[j];
                perm[j] = perm[bc];
                perm[bc] = p;
            }
        }
        __syncthreads();
        const double tau = ts[j];
        if (tau != 0.0) {
            const double *v = A + j * lda;
            for (int c0 = j + 1 + warp * CPW; c0 < pk; c0 += TT_NW * CPW) {
                const int c = c0 + grp;
                const bool ok = c < pk;
                double *col = A + (ok ? c : 0) * lda;
                double w = 0.0, w1 = 0.0;
                if (ok) {
                    int i = j + 1 + sub;
                    for (; i + LPC < q; i += 2 * LPC) {
                        w = fma(v[i], col[i], w);
                        w1 = fma(v[i + LPC], col[i + LPC], w1);
                    }
                    if (i < q) w = fma(v[i], col[i], w);
                }
                w = (group_sum(w + w1) + (ok ? col[j] : 0.0)) * tau;
                if (ok)
                    for (int i = j + 1 + sub; i < q; i += LPC) col[i] = fma(-v[i], w, col[i]);
                __syncwarp();
                if (ok && sub == 0) col[j] -= w;
            }
        }
        __syncthreads();
    }

    // ---- 2. Z = R^T (column t of Z is row t of R), J = identity
    for (int e = threadIdx.x; e < pk * pn; e += TT_NT) {
        const int t = e / pn, i = e - t * pn, c = pa + i;
        M[t * ldm + i] = c >= t ? A[c * lda + t] : 0.0;
        M[t * ldm + pn + i] = c == t ? 1.0 : 0.0;
    }
    if (threadIdx.x == 0) rotated = 0;
    cl.sync();  // every CTA has started: partials may be pushed
    const int n = pk + (pk & 1);  // round-robin over an even count; index pk (odd case) is a bye
    const int npairs = n / 2;
    const double eps_cos = 8.0 * (double)max(pk, q) * DBL_EPSILON;  // cosine below which a pair counts as orthogonal
    int par = 0;
    // this CTA's partial sums over its rows of column pairs, into every CTA's part
    double *dst[SV_MAXCL];
#pragma unroll
    for (int r = 0; r < SV_MAXCL; ++r) dst[r] = cl.map_shared_rank(part + rank * 3 * NPR, r < ncl ? r : 0);
    // (quantity k of a pair: z_x . z_x, z_y . z_y, z_x . z_y -- a warp each, on sub-partitions
    // of their own: one issues an FP64 instruction every 64 cycles)
    auto push = [&](int k, int slot, int x, int y) {
        double s0 = 0.0, s1 = 0.0;
        if (x < pk && y < pk) {
            const double *zx = M + (k == 1 ? y : x) * ldm, *zy = M + (k == 0 ? x : y) * ldm;
            int i = 0;
            for (; i + 1 < pn; i += 2) {
                s0 = fma(zx[i], zy[i], s0);
                s1 = fma(zx[i + 1], zy[i + 1], s1);
            }
            if (i < pn) s0 = fma(zx[i], zy[i], s0);
            s0 += s1;
        }
        const int o = (par * ncl * 3 + k) * NPR + slot;
#pragma unroll
        for (int r = 0; r < SV_MAXCL; ++r)
            if (r < ncl) dst[r][o] = s0;
    };
    auto total = [&](int k, int slot) {  // over the CTAs, in a fixed order
        const double *p = part + (par * ncl * 3 + k) * NPR + slot;
        if (ncl == 1) return p[0];
        double s[SV_MAXCL];
#pragma unroll
        for (int r = 0; r < SV_MAXCL; ++r) s[r] = r < ncl ? p[r * 3 * NPR] : 0.0;
        const double lo = (s[0] + s[1]) + (s[2] + s[3]);
        return ncl <= 4 ? lo : lo + ((s[4] + s[5]) + (s[6] + s[7]));
    };
    // warps 0, 1, 2 (pairs 0..31) and 4, 5, 6 (pairs 32..47) form the quantities 0, 1, 2
    const int quantity = warp & 3, qslot = lane + (warp >> 2) * 32;
    const bool qactive = quantity < 3 && qslot < npairs;
    // a round's pair of slot t: the players at places t and n - 1 - t of a circle; player
    // 0 stays, the others move one place a round
    int px = qslot < npairs ? qslot : 0, py = n - 1 - px;
    for (int sweep = 0; sweep < 60 && n > 1; ++sweep) {
        for (int round = 0; round < n - 1; ++round, par ^= 1) {
            const int slot = qslot, x = px, y = py;
            if (qactive) push(quantity, slot, x, y);
            cl.sync();
            if (qactive) s_tot[quantity][slot] = total(quantity, slot);
            px = px == 0 ? 0 : px + 1 < n ? px + 1 : 1;
            py = py == 0 ? 0 : py + 1 < n ? py + 1 : 1;
            __syncthreads();
            if (quantity == 0 && slot < npairs) {
                const double a = s_tot[0][slot], b = s_tot[1][slot], c = s_tot[2][slot];
                double cs = 1.0, sn = 0.0;
                // (byes have zero sums; NaNs and columns below 2^-511 are left alone)
                const int eh = max(__double2hiint(a), __double2hiint(b)) & 0x7FF00000;
                if (c != 0.0 && eh >= 0x00100000 && eh < 0x7FE00000) {
                    // over the power of two of the larger norm, in FP32: the tangent of
                    // the angle (0 below 2^-126)
                    auto rel = [&](double v) {
                        const int h = __double2hiint(v), ex = ((h & 0x7FF00000) - eh) >> 20;
                        const unsigned m = ((unsigned)h & 0x800FFFFFu) | (unsigned)((ex + 127) << 20);
                        return ex < -126 ? 0.0f
                                         : __uint_as_float((m & 0x80000000u) | ((m & 0x0FFFFFFFu) << 3) |
                                                           ((unsigned)__double2loint(v) >> 29));
                    };
                    const float cf = rel(c), len = sqrt_approx(rel(a)) * sqrt_approx(rel(b));
                    if (fabsf(cf) > 4.0f * (float)DBL_EPSILON * len || cf == 0.0f) {
                        float t;
                        if (cf == 0.0f) {
                            t = (float)(c / (b - a));
                        } else {
                            const float zeta = 0.5f * rel(b - a) * fast_rcp(cf);
                            t = fabsf(zeta) < 1e15f
                                    ? copysignf(fast_rcp(fabsf(zeta) + sqrt_approx(fmaf(zeta, zeta, 1.0f))), zeta)
                                    : 0.5f * fast_rcp(zeta);
                        }
                        if (fabsf(t) > 1e-37f) {
                            const double td = f32_to_f64_nz(t);
                            cs = rsqrt_f64(fma(td, td, 1.0));
                            sn = cs * td;
                            // (len == 0: a norm ratio below 2^-63)
                            if (len > 0.0f ? fabsf(cf) > (float)eps_cos * len : c * c > eps_cos * eps_cos * a * b) rotated = 1;
                        }
                    }
                }
                s_cs[slot] = cs;
                s_sn[slot] = sn;
                s_uv[slot][0] = x;
                s_uv[slot][1] = y;
            }
            __syncthreads();
            for (int g = lane; g < npairs; g += 32) {
                if (s_sn[g] == 0.0) continue;
                const double cs = s_cs[g], sn = s_sn[g];
                double *mu = M + s_uv[g][0] * ldm, *mv = M + s_uv[g][1] * ldm;
                for (int i = warp; i < 2 * pn; i += TT_NW) {
                    const double u = mu[i], v = mv[i];
                    mu[i] = cs * u - sn * v;
                    mv[i] = sn * u + cs * v;
                }
            }
            __syncthreads();
        }
        const bool more = rotated != 0;  // the same on every CTA: all form the same angles
        __syncthreads();
        if (threadIdx.x == 0) rotated = 0;
        if (!more) break;
    }
    // ---- singular values (the norms of Z's columns), their descending order (ties by
    // index), norm, rank
    for (int t0 = 0; t0 < pk; t0 += NPR, par ^= 1) {  // (as pairs of a column with itself)
        if (threadIdx.x < NPR && t0 + threadIdx.x < pk) push(0, threadIdx.x, t0 + threadIdx.x, t0 + threadIdx.x);
        cl.sync();
        if (threadIdx.x < NPR && t0 + threadIdx.x < pk) sig[t0 + threadIdx.x] = sqrt(total(0, threadIdx.x));
    }
    for (int t = threadIdx.x; t < pk; t += TT_NT) ord[t] = t;  // every entry stays an index, also with NaNs
    __syncthreads();
    for (int t = threadIdx.x; t < pk; t += TT_NT) {
        int r = 0;
        for (int u = 0; u < pk; ++u) r += (sig[u] > sig[t]) || (sig[u] == sig[t] && u < t);
        ord[r] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double delta;
        if (d.set_delta) {
            double s2 = 0.0;
            for (int t = pk - 1; t >= 0; --t) s2 += sig[ord[t]] * sig[ord[t]];
            delta = d.eps / sqrt(2.0) * sqrt(s2);
            if (rank == 0) {
                d.delta[0] = delta * up;
                d.delta[1] = sqrt(s2) * up;
            }
        } else {
            delta = d.delta[0] * down;
        }
        // smallest r >= 1 whose discarded singular values have a 2-norm <= delta
        int r = pk;
        double tail = 0.0;
        while (r > 1) {
            const double s = sig[ord[r - 1]];
            const double nt = fma(s, s, tail);
            if (sqrt(nt) > delta) break;
            tail = nt;
            --r;
        }
        if (r > d.rmax) r = d.rmax;
        s_rank = r;
        if (rank == 0) d.rank[0] = r;
    }
    __syncthreads();
    const int r = s_rank;
    if (rank == 0)
        for (int t = threadIdx.x; t < pk; t += TT_NT) d.sv[t] = sig[ord[t]] * up;
    // left vectors: rows P of Z over sigma.  A zero column (only kept when T has fewer
    // nonzero singular values than the rank) gets an orthonormal direction below.
    for (int e = threadIdx.x; e < pn * r; e += TT_NT) {
        const int i = e / r, c = e - i * r, t = ord[c];
        const double s = sig[t];
        d.Vsel[(long long)perm[pa + i] * d.ld_out + c] = s > 0.0 ? M[t * ldm + i] / s : 0.0;
        d.Wt[(long long)(pa + i) * d.ld_out + c] = M[t * ldm + pn + i] * (s * up);
    }
    __threadfence();
    cl.sync();  // J sigma is complete (and no CTA reads another's shared memory any more)
    // ---- 3. columns c = rank, rank + ncl, .. of Q [J sigma; 0], in place of J sigma
    double *X = M;  // [..][lda] columns (M is free)
    const int nc = (r - rank + ncl - 1) / ncl;
    constexpr int CB = 8;
    for (int c0 = 0; c0 < nc; c0 += CB) {
        const int w = min(CB, nc - c0);
        for (int e = threadIdx.x; e < w * q; e += TT_NT) {
            const int i = e / w, c = e - i * w;
            X[c * lda + i] = i < pk ? __ldcg(d.Wt + (long long)i * d.ld_out + rank + (c0 + c) * ncl) : 0.0;
        }
        __syncthreads();
        if (warp < w) {  // a warp per column: no barrier between reflectors
            double *x = X + warp * lda;
            for (int j = pk - 1; j >= 0; --j) {
                const double tau = ts[j];
                if (tau == 0.0) continue;
                const double *v = A + j * lda;
                double s = 0.0;
                for (int i = j + 1 + lane; i < q; i += 32) s = fma(v[i], x[i], s);
                s = (warp_sum_d(s) + x[j]) * tau;
                for (int i = j + 1 + lane; i < q; i += 32) x[i] = fma(-v[i], s, x[i]);
                __syncwarp();
                if (lane == 0) x[j] -= s;
                __syncwarp();
            }
        }
        __syncthreads();
        for (int e = threadIdx.x; e < w * q; e += TT_NT) {
            const int i = e / w, c = e - i * w;
            d.Wt[(long long)i * d.ld_out + rank + (c0 + c) * ncl] = X[c * lda + i];
        }
        __syncthreads();
    }
    // ---- zero singular values among the kept ones: complete the left vectors to an
    // orthonormal set (their sigma u is zero) by Gram-Schmidt on unit vectors
    if (rank == 0 && warp == 0) {
        int e0 = 0;
        for (int c = 0; c < r; ++c) {
            if (sig[ord[c]] > 0.0) continue;
            for (; e0 < pk; ++e0) {
                for (int pass = 0; pass < 2; ++pass) {
                    for (int i = lane; i < pk; i += 32)
                        if (pass == 0) X[i] = i == e0 ? 1.0 : 0.0;
                    __syncwarp();
                    for (int u = 0; u < c; ++u) {
                        double s = 0.0;
                        for (int i = lane; i < pk; i += 32) s = fma(__ldcg(d.Vsel + (long long)i * d.ld_out + u), X[i], s);
                        s = warp_sum_d(s);
                        for (int i = lane; i < pk; i += 32) X[i] = fma(-s, __ldcg(d.Vsel + (long long)i * d.ld_out + u), X[i]);
                        __syncwarp();
                    }
                }
                double s = 0.0;
                for (int i = lane; i < pk; i += 32) s = fma(X[i], X[i], s);
                s = warp_sum_d(s);
                if (s * pk < 0.25) continue;  // some unit vector keeps at least 1 / pk of its square
                for (int i = lane; i < pk; i += 32) d.Vsel[(long long)i * d.ld_out + c] = X[i] / sqrt(s);
                __threadfence();
                __syncwarp();
                ++e0;
                break;
            }
        }
    }
}

// First-core unfolding C1 [n1][R1] (coefficient folded in) and transposed
// last-core unfolding MA [n3][R2] of the TT sum.
__global__ void k_tt_build(const TTSumDesc *descs)
{
    const TTSumDesc &d = descs[blockIdx.y];
    const long long e1 = (long long)d.n[0] * d.R1, e3 = (long long)d.n[2] * d.R2;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < e1 + e3;
         e += (long long)gridDim.x * blockDim.x) {
        if (e < e1) {
            const int i = (int)(e / d.R1), a = (int)(e - (long long)i * d.R1);
            int t = 0;
            while (t + 1 < d.nt && a >= d.a0[t + 1]) ++t;
            d.C1[e] = d.coef[t] * d.core[t][0][(long long)i * d.r1[t] + (a - d.a0[t])];
        } else {
            const long long f = e - e1;
            const int i = (int)(f / d.R2), bb = (int)(f - (long long)i * d.R2);
            int t = 0;
            while (t + 1 < d.nt && bb >= d.b0[t + 1]) ++t;
            d.MA[f] = d.core[t][2][(long long)i * d.r2[t] + (bb - d.b0[t])];
        }
    }
}

// MB[(j k3 + c) R1 + a] = sum_b G2_t[j][a - a0_t][b] TA[c][b0_t + b]  (t = term of a):
// the block-diagonal middle core of the sum times TA^T on its right rank,
// written as the (n2 k3) x R1 unfolding of the next QR.
__global__ void k_tt_contract(const TTSumDesc *descs)
{
    const TTSumDesc &d = descs[blockIdx.y];
    const long long tot = (long long)d.n[1] * d.k3 * d.R1;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < tot;
         e += (long long)gridDim.x * blockDim.x) {
        const int a = (int)(e % d.R1);
        const long long jc = e / d.R1;
        const int c = (int)(jc % d.k3), j = (int)(jc / d.k3);
        int t = 0;
        while (t + 1 < d.nt && a >= d.a0[t + 1]) ++t;
        const double *g = d.core[t][1] + ((long long)j * d.r1[t] + (a - d.a0[t])) * d.r2[t];
        const double *ta = d.TA + (long long)c * d.R2 + d.b0[t];
        double s = 0.0;
        for (int bb = 0; bb < d.r2[t]; ++bb) s = fma(g[bb], ta[bb], s);
        d.MB[e] = s;
    }
}

// out[i][c] = sum_a L[i][a] Rt[c][a]  (out = L Rt^T; L [rows][ka], Rt [cols][ka], row-major)
__global__ void k_tt_gemm_tr(const GemmDesc *descs)
{
    const GemmDesc &d = descs[blockIdx.y];
    const long long tot = (long long)d.rows * d.cols;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < tot;
         e += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(e % d.cols);
        const long long i = e / d.cols;
        const double *l = d.L + i * d.ka;
        const double *r = d.Rt + (long long)c * d.ka;
        double s = 0.0;
        for (int a = 0; a < d.ka; ++a) s = fma(l[a], r[a], s);
        d.out[e] = s;
    }
}

static bool tt_attrs_set = false;

static cudaError_t tt_set_attributes()
{
    if (tt_attrs_set) return cudaSuccess;
    const int mx = (int)qr_apply_smem(TT_KMAX, TT_KMAX, TT_KMAX);
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_qr_factor, cudaFuncAttributeMaxDynamicSharedMemorySize, mx)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_qr_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, mx)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_svd_jacobi, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)std::max(svd_smem(SV_ONE, TT_KMAX, 1), svd_smem(TT_KMAX, TT_KMAX, 2)))) != cudaSuccess) return e;
    tt_attrs_set = true;
    return cudaSuccess;
}

cudaError_t launch_qr_factor(const QRDesc *d, int n, int max_chunks, size_t smem, cudaStream_t s)
{
    cudaError_t e = tt_set_attributes();
    if (e != cudaSuccess) return e;
    k_qr_factor<<<dim3(max_chunks, n), TT_NT, smem, s>>>(d);
    return cudaGetLastError();
}

cudaError_t launch_qr_apply(const QApplyDesc *d, int n, int max_chunks, size_t smem, cudaStream_t s)
{
    cudaError_t e = tt_set_attributes();
    if (e != cudaSuccess) return e;
    k_qr_apply<<<dim3(max_chunks, n), TT_NT, smem, s>>>(d);
    return cudaGetLastError();
}

cudaError_t launch_svd_jacobi(const SvdDesc *d, int n, int ncl, size_t smem, cudaStream_t s)
{
    cudaError_t e = tt_set_attributes();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ncl, n);
    cfg.blockDim = dim3(TT_NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ncl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_svd_jacobi, d);
}

cudaError_t launch_tt_build(const TTSumDesc *d, int n, cudaStream_t s)
{
    k_tt_build<<<dim3(64, n), 256, 0, s>>>(d);
    return cudaGetLastError();
}

cudaError_t launch_tt_contract(const TTSumDesc *d, int n, cudaStream_t s)
{
    k_tt_contract<<<dim3((unsigned)sm_count(), n), 256, 0, s>>>(d);
    return cudaGetLastError();
}

cudaError_t launch_tt_gemm_tr(const GemmDesc *d, int n, cudaStream_t s)
{
    k_tt_gemm_tr<<<dim3(64, n), 256, 0, s>>>(d);
    return cudaGetLastError();
}

}  // namespace wg
