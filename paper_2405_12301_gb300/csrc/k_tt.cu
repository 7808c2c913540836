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
//   * k_svd_jacobi: one-sided Jacobi SVD (round-robin pair ordering) of the
//     transpose of a k x q triangular factor T: T^T V = U S gives T = V S U^T;
//     picks the truncation rank from the singular values and writes V's kept
//     columns and (U S)'s kept columns.  The rows of T^T and of V are spread over
//     the CTAs of a cluster: a rotation acts on every row alone, only the dot
//     products that choose the angles are sums over all of them.
//   * k_tt_build / k_tt_contract / k_tt_gemm_tr: the TT sum's first and last
//     unfoldings, the block-diagonal middle core times a triangular factor, and
//     a small dense product.
// All arithmetic is FP64.
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
size_t svd_smem(int pk, int q, int ncl)
{
    return sizeof(double) * ((size_t)pk * (((q + ncl - 1) / ncl + (pk + ncl - 1) / ncl) | 1) + pk);
}

// CTAs per matrix: as many as the GPU has SMs for, at most 8 and at least ~8 rows each.
int svd_cluster(int n, int max_pk)
{
    int ncl = 8;
    while (ncl > 1 && ((long long)n * ncl > sm_count() || max_pk / ncl < 6)) ncl /= 2;
    return ncl;
}

// The column loop keeps one reflector ahead: while the other warps apply reflector
// j to their columns, one warp applies it to column j + 1 and forms reflector j + 1
// from it, so that chain (~35 dependent FP64 operations) runs beside the updates
// and a column takes one barrier.  64 columns of a 64-row sub-block: 195 -> QRSUB us.
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
                for (int c0 = j + 2 + ((warp - ahead - 1) & (TT_NW - 1)) * CPW; c0 < k; c0 += TT_NW * CPW) {
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

// One-sided Jacobi on the pk columns of M = T^T (column t = row t of T, length q).
// A sweep of 64 columns is 63 rounds of 32 disjoint pairs; per round an SM did ~790
// FP64 instructions (7.2 us).  Here each CTA of the cluster holds all columns of a
// slice of M's and V's rows.  Per round: partial dot products m_u . m_u, m_v . m_v
// and m_u . m_v over the slice (a lane per pair; the three chains overlap, and
// norms carried from round to round lose all digits on nearly dependent columns),
// one cluster barrier, the sum of all partials and the angle (a lane per pair,
// every CTA the same), the rotations of the slice (a lane per pair, a warp per
// row).  The tangent of the angle is formed in FP32 (with Newton steps for cos =
// 1 / sqrt(1 + t^2)): it only steers, the rotation is orthogonal to FP64 rounding
// whatever t is, and a pair counts as orthogonal by its FP64 dot products.  64 x 64, 10 matrices: 4.8 -> SVDT ms.
// cluster size 1..8 (svd_cluster): fewer CTAs where the batch fills the GPU.
__global__ void __launch_bounds__(TT_NT) k_svd_jacobi(const SvdDesc *descs)
{
    cg::cluster_group cl = cg::this_cluster();
    const int ncl = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const SvdDesc &d = descs[blockIdx.y];
    const int pk = d.pk, q = d.q;
    if (pk <= 0) return;  // the same for every CTA of the cluster
    extern __shared__ double sm[];
    constexpr int NPR = TT_KMAX / 2, NPART = 4;
    // this CTA's partial dot products (m_u . m_u, m_v . m_v, m_u . m_v; double buffered) and norms
    __shared__ double part[2][NPART][3][NPR], norm_part[NPART][TT_KMAX];
    __shared__ double s_nrm[TT_KMAX], s_cs[NPR], s_sn[NPR];
    __shared__ int s_uv[NPR][2], ord[TT_KMAX], rotated, s_rank;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int qa = rank * q / ncl, qn = (rank + 1) * q / ncl - qa;     // rows of M
    const int pa = rank * pk / ncl, pn = (rank + 1) * pk / ncl - pa;   // rows of V
    const int ldm = (qn + pn) | 1;
    double *M = sm;                          // [pk][ldm]: qn rows of M, then pn rows of V
    double *sig = M + (size_t)pk * ldm;      // [pk]
    for (int e = threadIdx.x; e < pk * qn; e += TT_NT) {
        const int t = e / qn, i = e - t * qn;
        M[t * ldm + i] = d.T[(long long)t * d.ldt + qa + i];
    }
    for (int e = threadIdx.x; e < pk * pn; e += TT_NT) {
        const int t = e / pn, i = e - t * pn;
        M[t * ldm + qn + i] = (pa + i == t) ? 1.0 : 0.0;
    }
    __syncthreads();
    const int n = pk + (pk & 1);  // round-robin over an even count; index pk (odd case) is a bye
    const int npairs = n / 2;
    const double tol = 8.0 * (double)max(pk, q) * DBL_EPSILON;  // cosine below which a pair counts as orthogonal
    const int nd = min(NPART, max(1, qn / 8));  // warps per column or pair that form partial sums, ~8+ rows each

    // squared norms of all columns, summed over the cluster in a fixed order into s_nrm
    auto norms = [&]() {
        for (int u = warp; u < nd * ((pk + 31) / 32); u += TT_NW) {
            const int w = u % nd, t = (u / nd) * 32 + lane;
            if (t < pk) {
                double a = 0.0;
                for (int i = w; i < qn; i += nd) a = fma(M[t * ldm + i], M[t * ldm + i], a);
                norm_part[w][t] = a;
            }
        }
        cl.sync();
        for (int t = threadIdx.x; t < pk; t += TT_NT) {
            double a = 0.0;
            for (int c = 0; c < ncl; ++c) {
                const double *np = cl.map_shared_rank(&norm_part[0][0], c);
                const int ndc = min(NPART, max(1, ((c + 1) * q / ncl - c * q / ncl) / 8));
                for (int w = 0; w < ndc; ++w) a += np[w * TT_KMAX + t];
            }
            s_nrm[t] = a;
        }
        cl.sync();  // the partials may be written again
    };
    int par = 0;
    for (int sweep = 0; sweep < 60 && n > 1; ++sweep) {
        if (threadIdx.x == 0) rotated = 0;  // (set after the next barrier at the earliest)
        for (int round = 0; round < n - 1; ++round, par ^= 1) {
            auto idx = [&](int t) { return t == 0 ? 0 : 1 + (t - 1 + round) % (n - 1); };
            for (int u = warp; u < nd * ((npairs + 31) / 32); u += TT_NW) {
                const int w = u % nd, slot = (u / nd) * 32 + lane;
                if (slot < npairs) {
                    const int x = idx(slot), y = idx(n - 1 - slot);
                    double a = 0.0, b = 0.0, c = 0.0;
                    if (x < pk && y < pk)
                        for (int i = w; i < qn; i += nd) {
                            const double u = M[x * ldm + i], v = M[y * ldm + i];
                            a = fma(u, u, a);
                            b = fma(v, v, b);
                            c = fma(u, v, c);
                        }
                    part[par][w][0][slot] = a;
                    part[par][w][1][slot] = b;
                    part[par][w][2][slot] = c;
                }
            }
            cl.sync();
            for (int slot = threadIdx.x; slot < npairs; slot += TT_NT) {
                const int x = idx(slot), y = idx(n - 1 - slot);
                double a = 0.0, bb = 0.0, c = 0.0;
                for (int r = 0; r < ncl; ++r) {
                    const double *pp = cl.map_shared_rank(&part[par][0][0][0], r) + slot;
                    const int ndc = min(NPART, max(1, ((r + 1) * q / ncl - r * q / ncl) / 8));
                    for (int w = 0; w < ndc; ++w, pp += 3 * NPR) {
                        a += pp[0];
                        bb += pp[NPR];
                        c += pp[2 * NPR];
                    }
                }
                double cs = 1.0, sn = 0.0;
                // (byes have zero sums; NaNs and columns below 2^-511 are left alone)
                const int eh = max(__double2hiint(a), __double2hiint(bb)) & 0x7FF00000;
                if (c != 0.0 && eh >= 0x00100000 && eh < 0x7FE00000) {
                    // scaled by the power of two that takes the larger norm to [1, 2)
                    const double sc = __hiloint2double(0x7FE00000 - eh, 0);
                    const double as = a * sc, bs = bb * sc, cs_ = c * sc;
                    if (cs_ * cs_ > tol * tol * as * bs) {
                        // tangent of the angle in FP32
                        const float df = f64_to_f32(bs - as), cf = f64_to_f32(cs_);
                        float t;
                        if (cf == 0.0f) {
                            t = (float)(c / (bb - a));
                        } else {
                            const float zeta = 0.5f * df / cf;
                            t = fabsf(zeta) < 1e15f ? copysignf(1.0f, zeta) / (fabsf(zeta) + sqrtf(fmaf(zeta, zeta, 1.0f)))
                                                    : 0.5f / zeta;
                        }
                        const double td = (double)t;
                        if (td != 0.0) {
                            cs = rsqrt_f64(fma(td, td, 1.0));
                            sn = cs * td;
                            rotated = 1;
                        }
                    }
                }
                s_cs[slot] = cs;
                s_sn[slot] = sn;
                s_uv[slot][0] = x;
                s_uv[slot][1] = y;
            }
            __syncthreads();
            for (int u = warp; u < (qn + pn) * ((npairs + 31) / 32); u += TT_NW) {
                const int i = u % (qn + pn), slot = (u / (qn + pn)) * 32 + lane;
                if (slot < npairs && s_sn[slot] != 0.0) {
                    const double cs = s_cs[slot], sn = s_sn[slot];
                    double *mu = M + s_uv[slot][0] * ldm + i, *mv = M + s_uv[slot][1] * ldm + i;
                    const double x = *mu, y = *mv;
                    *mu = cs * x - sn * y;
                    *mv = sn * x + cs * y;
                }
            }
            __syncthreads();
        }
        if (!rotated) break;  // the same on every CTA: all form the same angles
        __syncthreads();
    }
    // singular values, their descending order (ties by index), norm, rank
    norms();
    for (int t = threadIdx.x; t < pk; t += TT_NT) {
        sig[t] = sqrt(s_nrm[t]);
        ord[t] = t;  // (every entry stays an index, also when NaNs leave the order undefined)
    }
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
                d.delta[0] = delta;
                d.delta[1] = sqrt(s2);
            }
        } else {
            delta = d.delta[0];
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
        for (int t = threadIdx.x; t < pk; t += TT_NT) d.sv[t] = sig[ord[t]];
    for (int e = threadIdx.x; e < pn * r; e += TT_NT) {
        const int i = e / r, c = e - i * r;
        d.Vsel[(long long)(pa + i) * d.ld_out + c] = M[ord[c] * ldm + qn + i];
    }
    for (int e = threadIdx.x; e < qn * r; e += TT_NT) {
        const int i = e / r, c = e - i * r;
        d.Wt[(long long)(qa + i) * d.ld_out + c] = M[ord[c] * ldm + i];
    }
    cl.sync();  // no CTA leaves while another may still read its partial sums
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
                                  (int)svd_smem(TT_KMAX, TT_KMAX, 1))) != cudaSuccess) return e;
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
