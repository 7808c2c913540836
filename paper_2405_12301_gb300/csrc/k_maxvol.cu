// k_maxvol.cu -- batched maxvol (the maximum-volume row selection that picks
// the cross indices of TT-cross, Sec. 3 "TT-cross Interpolation"), FP64, five
// launches per batch (three for small matrices):
//   1. the r pivot rows I of Gaussian elimination with partial pivoting on a
//      working copy W (largest remaining |W[i][j]| of column j, ties to the
//      smaller row); the multipliers L[i][j] overwrite column j of W, and the
//      unit lower triangular L[I] is inverted;
//   2. B = A A[I]^{-1} = L L[I]^{-1} (A = P L U, so the U factor cancels; the
//      rows I get the unit vectors exactly), spread over many CTAs per matrix;
//   3. while max |B[i][j]| > 1 + delta (ties to the first entry in row-major
//      order): row i replaces I[j] and B -= B[:, j] (B[i, :] - e_j) / B[i][j],
//      on a copy of B in FP32 pairs hi + lo (about 47 bits);
//   4. if rows were swapped, B[I]^{-1} of the B of 2 and the new rows I, FP64;
//   5. then B := B B[I]^{-1} = A A[I]^{-1}, FP64.
// Forming B from L rather than from an inverse of A[I] keeps it accurate when
// A is ill-conditioned: |L| <= 1 under partial pivoting, and the scale of
// A's columns stays in U.  The swaps only choose rows: their rank-one updates
// would hold the FP64 pipe for n r instructions each (12000 x 32: 15 us a swap
// on 8 SMs).  Entries closer than the pairs' 2^-46 may be taken in another order than
// FP64 swaps would; equal rows stay equal bit for bit, so ties go to the first entry, and
// a delta too small for pairs takes FP64 swaps.  The final B is one FP64 product of the
// accurate B of step 2 with the inverse of its rows I, without the swaps' accumulated
// rounding: the inverse's entries are those of the final B (1 + delta at most once the
// swaps have ended), so its error is that of a sum of r products of B's entries, bounded
// by the elimination's growth as B's own error is.  Phases 1 and 3 are sequences of (argmax, rank-one
// update) steps.  Each matrix gets a thread-block cluster whose CTAs own
// contiguous slices of its rows, held in shared memory as far as they fit (a slice
// in L2 costs a round trip per step and column batch) and in W beyond.  Per step
// every CTA finds the best entry of its slice, in the pass that updates it, and
// stashes that entry's row in a shared-memory slot; after one cluster barrier
// every CTA reduces the slots (read through distributed shared memory) to the
// same winner and copies the winner's row from its owner.  Slots alternate
// between two buffers, so the writes of step t + 1 never meet the reads of
// step t, and the stash lets the owner update the winning row in place while
// others still read it.  Slices are column-major, so a warp's row-parallel
// accesses coalesce.
//   16 matrices of 256..12000 x 4..32: pivot 1.10 -> 0.41 ms, swaps 1.82 -> 0.47 ms.
#include <algorithm>
#include <climits>
#include <type_traits>

#include <cooperative_groups.h>

#include "weno_dev.cuh"
#include "weno_internal.h"
#include "tt_internal.h"

namespace wg {

namespace cg = cooperative_groups;

constexpr int MV_NT = 512, MV_NW = MV_NT / 32;
constexpr int MV_ROWS = 64;  // rows that a CTA of a cluster gets at least (launch_maxvol)
// A pivot |w| <= MV_RANK_TOL r max_i |A[i][j]| counts as zero: the residual
// of a column that lies in the span of the earlier ones is a few rounding
// errors of the column's own scale (a full-rank matrix reaches it only with a
// condition number near 1 / (r MV_RANK_TOL) ~ 1e13).
constexpr double MV_RANK_TOL = 4.0 * 2.220446049250313e-16;

// |x| as an unsigned integer: for finite x its order is the order of |x|, so
// argmaxes run on the integer pipe (FP64 compares issue at the FP64 rate).
__device__ __forceinline__ unsigned long long absbits(double x)
{
    return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

__device__ __forceinline__ bool better(unsigned long long k, long long i, unsigned long long bk, long long bi)
{
    return k > bk || (k == bk && i < bi);
}

// Block-wide argmax of (key, i): largest key, smallest i among equal keys.
__device__ __forceinline__ void block_argmax_u(unsigned long long &k, long long &i, unsigned long long *sk, long long *si)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long ok = __shfl_xor_sync(0xFFFFFFFFu, k, o);
        const long long oi = __shfl_xor_sync(0xFFFFFFFFu, i, o);
        if (better(ok, oi, k, i)) {
            k = ok;
            i = oi;
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) {
        sk[warp] = k;
        si[warp] = i;
    }
    __syncthreads();
    k = sk[0];
    i = si[0];
    for (int w = 1; w < MV_NW; ++w)
        if (better(sk[w], si[w], k, i)) {
            k = sk[w];
            i = si[w];
        }
}

// One CTA's candidate of a step: its best key, the entry's index and the
// entry's row (all r columns of W).
struct MvSlot {
    unsigned long long key;
    long long e;
    double row[MV_RMAX];
};

// Per-CTA state of a cluster-wide argmax step.
struct MvStep {
    MvSlot slot[2];
    double row[MV_RMAX];            // the winner's row, copied from its owner's slot
    unsigned long long sk[MV_NW];
    long long si[MV_NW];
    unsigned long long win_key;
    long long win_e;
    int win_rank;
};

// The cluster-wide step: publish this CTA's candidate (k, e) -- stash(slot,
// k, e) copies the candidate's row into the slot -- then agree on the winner
// (st.win_*).  Every CTA of the cluster makes the same sequence of calls (the
// barrier inside is cluster-wide); par alternates between consecutive calls.
template <class Stash>
__device__ __forceinline__ const MvSlot *cluster_argmax(cg::cluster_group &cl, MvStep &st, int par, int ncl,
                                                        unsigned long long k, long long e, Stash stash)
{
    block_argmax_u(k, e, st.sk, st.si);
    MvSlot &s = st.slot[par];
    if (threadIdx.x == 0) {
        s.key = k;
        s.e = e;
    }
    stash(s, k, e);
    cl.sync();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        unsigned long long bk = 0ull;
        long long be = LLONG_MAX;
        int br = 0;
        if (lane < ncl) {
            const MvSlot *rs = cl.map_shared_rank(&s, lane);
            bk = rs->key;
            be = rs->e;
            br = lane;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long ok = __shfl_xor_sync(0xFFFFFFFFu, bk, o);
            const long long oe = __shfl_xor_sync(0xFFFFFFFFu, be, o);
            const int orr = __shfl_xor_sync(0xFFFFFFFFu, br, o);
            if (better(ok, oe, bk, be)) {
                bk = ok;
                be = oe;
                br = orr;
            }
        }
        if (lane == 0) {
            st.win_key = bk;
            st.win_e = be;
            st.win_rank = br;
        }
    }
    __syncthreads();
    return cl.map_shared_rank(&s, st.win_rank);  // the winner's slot
}

__device__ __forceinline__ void row_slice(int n, int rank, int ncl, int &lo, int &hi)
{
    lo = (int)((long long)rank * n / ncl);
    hi = (int)((long long)(rank + 1) * n / ncl);
}

// The element (row t of the slice, column c) of a slice whose first `cap` rows are
// in shared memory and whose others are in W: p[c * ld].
template <class V> struct MvRow {
    V *p;
    int ld;
};
template <class V>
__device__ __forceinline__ MvRow<V> mv_row(V *sh, int cap, V *W, int n, int lo, int t)
{
    return t < cap ? MvRow<V>{sh + t, cap} : MvRow<V>{W + lo + t, n};
}

// Phase 1: pivot rows and multipliers (the whole cluster), then L[I]^{-1}
// (rank 0 alone, in dynamic shared memory).
__global__ void __launch_bounds__(MV_NT) k_maxvol_pivot(const MaxvolDesc *descs, int smem_doubles)
{
    cg::cluster_group cl = cg::this_cluster();
    const MaxvolDesc &d = descs[blockIdx.y];
    const int n = d.n, r = d.r, ncl = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    int lo, hi;
    row_slice(n, rank, ncl, lo, hi);
    __shared__ MvStep st;
    __shared__ int I[MV_RMAX];
    // rows of this slice already picked: a slice has MV_NMAX / 8 rows at most on 8 CTAs or
    // more, and fewer than 2 MV_ROWS r on a cluster that launch_maxvol halved below 8
    static_assert(2 * MV_ROWS * MV_RMAX <= MV_NMAX / 8, "chosen holds a slice's rows");
    __shared__ unsigned chosen[MV_NMAX / 8 / 32];
    __shared__ int s_fail;
    __shared__ unsigned long long cbits[MV_RMAX];  // this CTA's column maxima of |A| (bit patterns)
    __shared__ double ctol[MV_RMAX];
    extern __shared__ double G[];
    double *W = d.W;
    const int m = hi - lo, cap = min(m, smem_doubles / r);
    if (threadIdx.x == 0) s_fail = 0;
    for (int e = threadIdx.x; e < (m + 31) / 32; e += MV_NT) chosen[e] = 0u;
    for (int c = threadIdx.x; c < r; c += MV_NT) cbits[c] = 0ull;
    for (int e = threadIdx.x; e < m * r; e += MV_NT) {  // column-major copy of the slice
        const int t = e / r, c = e - t * r;
        const MvRow<double> w = mv_row(G, cap, W, n, lo, t);
        w.p[(long long)c * w.ld] = d.A[(long long)lo * r + e];
    }
    __syncthreads();
    // the scale of every column, max_i |A[i][c]|, over the whole cluster: a
    // pivot at or below MV_RANK_TOL of its column's scale means rank < r
    for (int c = threadIdx.x >> 5; c < r; c += MV_NW) {
        unsigned long long k = 0ull;
        for (int t = threadIdx.x & 31; t < m; t += 32) {
            const MvRow<double> w = mv_row(G, cap, W, n, lo, t);
            k = max(k, absbits(w.p[(long long)c * w.ld]));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) k = max(k, __shfl_xor_sync(0xFFFFFFFFu, k, o));
        if ((threadIdx.x & 31) == 0) cbits[c] = k;
    }
    cl.sync();
    for (int c = threadIdx.x; c < r; c += MV_NT) {
        unsigned long long k = 0ull;
        for (int q = 0; q < ncl; ++q) k = max(k, *cl.map_shared_rank(&cbits[c], q));
        ctol[c] = MV_RANK_TOL * r * __longlong_as_double((long long)k);
    }
    __syncthreads();

    // 1. partial pivoting; only the columns after j are updated (earlier ones
    // are never read again); the pass that updates column j + 1 finds its argmax
    unsigned long long kmax = 0ull;  // 0 marks "no row"
    long long bi = LLONG_MAX;
    for (int t = threadIdx.x; t < m; t += MV_NT) {
        const unsigned long long k = absbits(*mv_row(G, cap, W, n, lo, t).p) + 1ull;
        if (k > kmax) {  // t grows per thread, so equal keys keep the first
            kmax = k;
            bi = lo + t;
        }
    }
    for (int j = 0; j < r; ++j) {
        // the slot's row: the candidate's W[j..r) (entries before j are stale)
        const MvSlot *ws = cluster_argmax(cl, st, j & 1, ncl, kmax, bi, [&](MvSlot &s, unsigned long long k, long long e) {
            if (k != 0ull) {
                const MvRow<double> w = mv_row(G, cap, W, n, lo, (int)(e - lo));
                for (int c = j + threadIdx.x; c < r; c += MV_NT) s.row[c] = w.p[(long long)c * w.ld];
            }
        });
        for (int c = j + threadIdx.x; c < r; c += MV_NT) st.row[c] = ws->row[c];
        const int p = (int)st.win_e;
        if (threadIdx.x == 0) {
            I[j] = p;
            if (p >= lo && p < hi) chosen[(p - lo) >> 5] |= 1u << ((p - lo) & 31);
        }
        __syncthreads();
        kmax = 0ull;
        bi = LLONG_MAX;
        const double wp = st.row[j];
        const bool zero = !(fabs(wp) > ctol[j]);
        if (zero && threadIdx.x == 0) s_fail = 1;  // every CTA sees the same pivot and scale
        const double inv = zero ? 0.0 : 1.0 / wp;
        for (int t = threadIdx.x; t < m; t += MV_NT) {
            if ((chosen[t >> 5] >> (t & 31)) & 1u) continue;
            const MvRow<double> w = mv_row(G, cap, W, n, lo, t);
            double *wj = w.p + (long long)j * w.ld;
            if (!zero) {
                const double f = *wj * inv;
                *wj = f;  // L[i][j]
                double *wc = wj + w.ld;
#pragma unroll 8
                for (int c = j + 1; c < r; ++c, wc += w.ld) *wc = fma(-f, st.row[c], *wc);
            }
            if (j + 1 < r) {
                const unsigned long long k = absbits(wj[w.ld]) + 1ull;
                if (k > kmax) {
                    kmax = k;
                    bi = lo + t;
                }
            }
        }
        // (the next step's block argmax starts with a barrier before st is written again)
    }
    __syncthreads();
    for (int e = threadIdx.x; e < cap * r; e += MV_NT) {  // the multipliers of the rows in shared memory
        const int c = e / cap, t = e - c * cap;
        W[(long long)c * n + lo + t] = G[e];
    }
    cl.sync();  // no CTA leaves while another may still read its slots
    if (rank != 0) return;

    // L[I]^{-1}: L[I] is unit lower triangular, row k holding the multipliers
    // of row I[k] from the steps before k (other slices' rows are read from L2:
    // they were written before the barrier above)
    double *Lt = G;                       // [r][r]
    double *Li = G + (size_t)r * r;       // [r][r]
    for (int e = threadIdx.x; e < r * r; e += MV_NT) {
        const int k = e / r, m = e - k * r;
        Lt[e] = m < k ? __ldcg(W + (long long)m * n + I[k]) : (m == k ? 1.0 : 0.0);
    }
    __syncthreads();
    // column c of the inverse by forward substitution, one thread per column
    for (int c = threadIdx.x; c < r; c += MV_NT) {
        for (int k = 0; k < c; ++k) Li[k * r + c] = 0.0;
        Li[c * r + c] = 1.0;
        for (int k = c + 1; k < r; ++k) {
            double acc = 0.0;
            for (int m = c; m < k; ++m) acc = fma(Lt[k * r + m], Li[m * r + c], acc);
            Li[k * r + c] = -acc;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) d.status[0] = s_fail;
    if (s_fail) return;
    for (int e = threadIdx.x; e < r * r; e += MV_NT) d.Linv[e] = Li[e];
    for (int j = threadIdx.x; j < r; j += MV_NT) d.idx[j] = I[j];
}

// B = L L[I]^{-1} (L: the multipliers in W, column-major), spread over many
// CTAs per matrix; the pivot rows get the unit vectors.
__global__ void __launch_bounds__(256) k_maxvol_b(const MaxvolDesc *descs)
{
    const MaxvolDesc &d = descs[blockIdx.y];
    if (d.status[0]) return;
    const int n = d.n, r = d.r;
    __shared__ double Li[MV_RMAX * MV_RMAX];
    __shared__ unsigned piv[MV_NMAX / 32];  // rows in I
    __shared__ int I[MV_RMAX];
    for (int e = threadIdx.x; e < r * r; e += blockDim.x) Li[e] = d.Linv[e];
    for (int w = threadIdx.x; w < (n + 31) / 32; w += blockDim.x) piv[w] = 0u;
    for (int k = threadIdx.x; k < r; k += blockDim.x) I[k] = d.idx[k];
    __syncthreads();
    for (int k = threadIdx.x; k < r; k += blockDim.x) atomicOr(&piv[I[k] >> 5], 1u << (I[k] & 31));
    __syncthreads();
    const double *W = d.W;
    const long long nr = (long long)n * r;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < nr; e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e / r), c = (int)(e - (long long)i * r);
        double acc = 0.0;
        if ((piv[i >> 5] >> (i & 31)) & 1u) {
            acc = I[c] == i ? 1.0 : 0.0;
        } else {
            for (int k = c; k < r; ++k) acc = fma(W[(long long)k * n + i], Li[k * r + c], acc);
        }
        d.B[e] = acc;
    }
}

// Phase 3, the swaps (the whole cluster), on a column-major copy of B in FP32
// pairs (the slice's first rows in shared memory, the others in W).
__device__ __forceinline__ unsigned pair_low_order(float2 v)  // orders the low parts of equal |high| parts
{
    const unsigned b = __float_as_uint(v.x < 0.0f ? -v.y : v.y);
    return b & 0x80000000u ? ~b : b | 0x80000000u;
}

// F64: on FP64 values, whose rounding the result keeps: B is written back and phases 4
// and 5 are left out.
template <bool F64>
__global__ void __launch_bounds__(MV_NT) k_maxvol_swap(const MaxvolDesc *descs, double delta, int max_iters, int smem_doubles)
{
    cg::cluster_group cl = cg::this_cluster();
    const MaxvolDesc &d = descs[blockIdx.y];
    if (d.status[0]) return;  // the same value for every CTA of the cluster
    const int n = d.n, r = d.r, ncl = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    int lo, hi;
    row_slice(n, rank, ncl, lo, hi);
    using V = typename std::conditional<F64, double, float2>::type;
    __shared__ MvStep st;
    __shared__ V s_row[MV_RMAX];
    __shared__ int I[MV_RMAX];
    extern __shared__ double mv_smem[];
    V *P = reinterpret_cast<V *>(mv_smem), *W = reinterpret_cast<V *>(d.W);
    const int m = hi - lo, cap = min(m, smem_doubles / r);
    for (int j = threadIdx.x; j < r; j += MV_NT) I[j] = d.idx[j];
    for (int e = threadIdx.x; e < m * r; e += MV_NT) {
        const int t = e / r, c = e - t * r;
        const MvRow<V> w = mv_row(P, cap, W, n, lo, t);
        if constexpr (F64) w.p[(long long)c * w.ld] = d.B[(long long)lo * r + e];
        else w.p[(long long)c * w.ld] = pr_norm(split_sat(d.B[(long long)lo * r + e]));
    }
    __syncthreads();
    // an entry's key: |hi|, then the low part's order; e = i r + c grows per thread,
    // so equal keys keep the first
    unsigned long long key = 0ull;
    long long be = LLONG_MAX;
    auto consider = [&](V v, long long e) {
        if constexpr (F64) {
            const unsigned long long x = absbits(v);
            if (be == LLONG_MAX || x > key) {
                key = x;
                be = e;
            }
        } else {
            const unsigned h = __float_as_uint(v.x) & 0x7FFFFFFFu;
            if (h < (unsigned)(key >> 32) && be != LLONG_MAX) return;
            const unsigned long long x = (unsigned long long)h << 32 | pair_low_order(v);
            if (be == LLONG_MAX || x > key) {
                key = x;
                be = e;
            }
        }
    };
    for (int t = threadIdx.x; t < m; t += MV_NT) {
        const MvRow<V> w = mv_row(P, cap, W, n, lo, t);
        for (int c = 0; c < r; ++c) consider(w.p[(long long)c * w.ld], (long long)(lo + t) * r + c);
    }
    int it = 0;
    for (; it < max_iters; ++it) {
        const MvSlot *ws = cluster_argmax(cl, st, it & 1, ncl, key, be,
                                          [&](MvSlot &s, unsigned long long, long long e) {
            if (e != LLONG_MAX) {
                const MvRow<V> w = mv_row(P, cap, W, n, lo, (int)(e / r - lo));
                for (int c = threadIdx.x; c < r; c += MV_NT) reinterpret_cast<V *>(s.row)[c] = w.p[(long long)c * w.ld];
            }
        });
        const long long we = st.win_e;
        const int i0 = (int)(we / r), j0 = (int)(we - (long long)i0 * r);
        const V piv = reinterpret_cast<const V *>(ws->row)[j0];
        double pv;
        if constexpr (F64) pv = piv;
        else pv = (double)piv.x + (double)piv.y;
        if (!(fabs(pv) > 1.0 + delta)) break;  // the same decision everywhere
        if (threadIdx.x < r) {  // (row_i0 - e_j0) / piv, one residual correction of an approximate quotient
            V v = reinterpret_cast<const V *>(ws->row)[threadIdx.x];
            if constexpr (F64) {
                s_row[threadIdx.x] = (threadIdx.x == j0 ? v - 1.0 : v) / piv;
            } else {
                if (threadIdx.x == j0) v = pr_norm(pr_sub(v, make_float2(1.0f, 0.0f)));
                const float q = fast_rcp(piv.x), x = __fmul_rn(v.x, q);
                const float rem = __fadd_rn(__fmaf_rn(-x, piv.x, v.x), __fmaf_rn(-x, piv.y, v.y));
                s_row[threadIdx.x] = make_float2(x, __fmul_rn(rem, q));
            }
        }
        if (threadIdx.x == 0) I[j0] = i0;
        __syncthreads();
        // B -= B[:, j0] (row_i0 - e_j0) / piv over the slice, with the next argmax
        key = 0ull;
        be = LLONG_MAX;
        for (int t = threadIdx.x; t < m; t += MV_NT) {
            const MvRow<V> w = mv_row(P, cap, W, n, lo, t);
            const V f = w.p[(long long)j0 * w.ld];
            V *wc = w.p;
            const long long e0 = (long long)(lo + t) * r;
#pragma unroll 4
            for (int c = 0; c < r; ++c, wc += w.ld) {
                V v;
                if constexpr (F64) v = fma(-f, s_row[c], *wc);
                else v = pr_norm(pr_sub(*wc, pr_mul(f, s_row[c])));
                *wc = v;
                consider(v, e0 + c);
            }
        }
    }
    if (F64 && it > 0) {  // (the rows I exactly the unit vectors)
        __syncthreads();
        for (int e = threadIdx.x; e < m * r; e += MV_NT) {
            const int t = e / r, c = e - t * r;
            const MvRow<V> w = mv_row(P, cap, W, n, lo, t);
            if constexpr (F64) d.B[(long long)lo * r + e] = w.p[(long long)c * w.ld];
        }
        __syncthreads();
        for (int e = threadIdx.x; e < r * r; e += MV_NT) {
            const int j = e / r, c = e - j * r;
            if (I[j] >= lo && I[j] < hi) d.B[(long long)I[j] * r + c] = c == j ? 1.0 : 0.0;
        }
    }
    cl.sync();  // no CTA leaves while another may still read its slots
    if (rank == 0) {
        for (int j = threadIdx.x; j < r; j += MV_NT) d.idx[j] = I[j];
        if (threadIdx.x == 0) d.swaps[0] = it;
    }
}

// Phase 4: Linv := B[I]^{-1} for the final rows I (Gauss-Jordan with partial
// pivoting in shared memory), one CTA per matrix whose rows changed.
__global__ void __launch_bounds__(256) k_maxvol_inverse(const MaxvolDesc *descs)
{
    const MaxvolDesc &d = descs[blockIdx.x];
    if (d.status[0] || d.swaps[0] == 0) return;
    const int r = d.r, ld = 2 * r + 1;
    extern __shared__ double G[];  // [r][B[I] | identity], pitch 2 r + 1
    __shared__ double col[MV_RMAX];
    __shared__ int s_piv;
    for (int e = threadIdx.x; e < r * r; e += blockDim.x) {
        const int k = e / r, c = e - k * r;
        G[k * ld + c] = d.B[(long long)d.idx[k] * r + c];
        G[k * ld + r + c] = k == c ? 1.0 : 0.0;
    }
    __syncthreads();
    for (int j = 0; j < r; ++j) {
        if (threadIdx.x < 32) {
            unsigned long long k = 0ull;
            int best = j;
            for (int i = j + threadIdx.x; i < r; i += 32) {
                const unsigned long long x = absbits(G[i * ld + j]) + 1ull;
                if (x > k) {
                    k = x;
                    best = i;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long ok = __shfl_xor_sync(0xFFFFFFFFu, k, o);
                const int ob = __shfl_xor_sync(0xFFFFFFFFu, best, o);
                if (ok > k || (ok == k && ob < best)) {
                    k = ok;
                    best = ob;
                }
            }
            if (threadIdx.x == 0) s_piv = best;
        }
        __syncthreads();
        const int p = s_piv;
        const double inv = 1.0 / G[p * ld + j];
        __syncthreads();
        for (int c = threadIdx.x; c < 2 * r; c += blockDim.x) {  // swap rows j and p, scale the pivot row
            const double x = G[j * ld + c], y = G[p * ld + c];
            if (p != j) G[p * ld + c] = x;
            G[j * ld + c] = y * inv;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < r; i += blockDim.x) col[i] = i == j ? 0.0 : G[i * ld + j];
        __syncthreads();
        // (the columns before j of the left half are unit vectors already)
        for (int e = threadIdx.x; e < r * (2 * r - j); e += blockDim.x) {
            const int i = e / (2 * r - j), c = j + e - i * (2 * r - j);
            if (i != j) G[i * ld + c] = fma(-col[i], G[j * ld + c], G[i * ld + c]);
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < r * r; e += blockDim.x) d.Linv[e] = G[(e / r) * ld + r + e % r];
}

// Phase 5: B := B B[I]^{-1}, the rows I exactly the unit vectors.  A block takes
// 64 rows at a time, staged in shared memory (the product overwrites them).
__global__ void __launch_bounds__(256) k_maxvol_final(const MaxvolDesc *descs)
{
    const MaxvolDesc &d = descs[blockIdx.y];
    if (d.status[0] || d.swaps[0] == 0) return;
    const int n = d.n, r = d.r;
    constexpr int RB = 64;
    if ((int)blockIdx.x * RB >= n) return;
    extern __shared__ double G[];  // [r][r] the inverse, then [RB][r] rows
    double *T = G + r * r;
    __shared__ int I[MV_RMAX];
    for (int e = threadIdx.x; e < r * r; e += blockDim.x) G[e] = d.Linv[e];
    for (int k = threadIdx.x; k < r; k += blockDim.x) I[k] = d.idx[k];
    for (int i0 = blockIdx.x * RB; i0 < n; i0 += gridDim.x * RB) {
        const int rows = min(RB, n - i0);
        __syncthreads();
        for (int e = threadIdx.x; e < rows * r; e += blockDim.x) T[e] = d.B[(long long)i0 * r + e];
        __syncthreads();
        for (int e = threadIdx.x; e < rows * r; e += blockDim.x) {
            const int t = e / r, c = e - t * r;
            double acc = 0.0;
            for (int k = 0; k < r; ++k) acc = fma(T[t * r + k], G[k * r + c], acc);
            d.B[(long long)i0 * r + e] = acc;
        }
        __syncthreads();
        for (int k = 0; k < r; ++k)
            if (I[k] >= i0 && I[k] < i0 + rows)
                for (int c = threadIdx.x; c < r; c += blockDim.x) d.B[(long long)I[k] * r + c] = c == k ? 1.0 : 0.0;
    }
}

// Largest matrices first, so that their clusters start in the first wave.
void maxvol_order(MaxvolDesc *d, int n)
{
    std::stable_sort(d, d + n, [](const MaxvolDesc &a, const MaxvolDesc &b) {
        return (double)a.n * a.r * a.r > (double)b.n * b.r * b.r;
    });
}

template <class K, class... Args>
static cudaError_t launch_cluster(K kern, int ncl, int n, size_t smem, cudaStream_t s, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ncl, n);
    cfg.blockDim = dim3(MV_NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ncl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// Dynamic shared memory of a cluster kernel at most (the static part is ~12 KB).
constexpr int MV_SMEM = 200 * 1024;

static cudaError_t maxvol_attributes()
{
    static bool done = false;
    if (done) return cudaSuccess;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_maxvol_pivot, cudaFuncAttributeMaxDynamicSharedMemorySize, MV_SMEM)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(k_maxvol_swap<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, MV_SMEM)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(k_maxvol_swap<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, MV_SMEM)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(k_maxvol_inverse, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(double) * MV_RMAX * (2 * MV_RMAX + 1))) != cudaSuccess ||
        (e = cudaFuncSetAttribute(k_maxvol_final, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(double) * 2 * MV_RMAX * MV_RMAX)) != cudaSuccess)
        return e;
    done = true;
    return e;
}

// Cluster size: 16 CTAs where the device schedules clusters that large, else 8.
static int maxvol_cluster_size()
{
    static int ncl = 0;
    if (ncl) return ncl;
    if (maxvol_attributes() != cudaSuccess) return 8;
    ncl = 8;
    if (cudaFuncSetAttribute(k_maxvol_pivot, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaFuncSetAttribute(k_maxvol_swap<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaFuncSetAttribute(k_maxvol_swap<false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(16, 1);
        cfg.blockDim = dim3(MV_NT);
        cfg.dynamicSmemBytes = MV_SMEM;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 16;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int c1 = 0, c2 = 0, c3 = 0;
        if (cudaOccupancyMaxActiveClusters(&c1, k_maxvol_pivot, &cfg) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&c2, k_maxvol_swap<true>, &cfg) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&c3, k_maxvol_swap<false>, &cfg) == cudaSuccess && c1 > 0 && c2 > 0 && c3 > 0)
            ncl = 16;
    }
    cudaGetLastError();  // a refused query leaves no sticky state; clear the last error
    return ncl;
}

// FP64 swaps: for small matrices (launch_maxvol), and where delta is within 2^10 of the
// pairs' 2^-46 -- an entry of a selected row, 1 but for its rounding, would pass for a swap.
static bool maxvol_in_f64(long long max_nr, double delta)
{
    return delta < 0x1p-36 || max_nr <= 4096ll * maxvol_cluster_size();
}
int maxvol_launches(long long max_nr, double delta) { return maxvol_in_f64(max_nr, delta) ? 3 : 5; }

// max_nr: the largest n r of the batch.  Shared memory for a slice: what the
// largest slice takes, and no more than lets the batch's CTAs run together.
cudaError_t launch_maxvol(const MaxvolDesc *d, int n, int max_r, long long max_nr, double delta, int max_iters,
                          cudaStream_t s)
{
    cudaError_t e = maxvol_attributes();
    if (e != cudaSuccess) return e;
    // at least MV_ROWS rows to a CTA: below, the cluster barriers of a step cost more than its
    // pass over the rows
    int ncl = maxvol_cluster_size();
    while (ncl > 2 && max_nr < (long long)MV_ROWS * ncl * max_r) ncl /= 2;
    const long long per_sm = std::min(3ll, std::max(1ll, ((long long)n * ncl + sm_count() - 1) / sm_count()));
    const long long want = sizeof(double) * std::max((max_nr + ncl - 1) / ncl + max_r, 2ll * max_r * max_r);
    const long long least = sizeof(double) * 2ll * max_r * max_r;  // L[I] and its inverse
    const size_t smem = (size_t)std::max(least, std::min(want, MV_SMEM / per_sm));
    const int doubles = (int)(smem / sizeof(double));
    e = launch_cluster(k_maxvol_pivot, ncl, n, smem, s, d, doubles);
    if (e != cudaSuccess) return e;
    k_maxvol_b<<<dim3(64, n), 256, 0, s>>>(d);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // Small slices swap in FP64: an entry then costs a swap ~14 cycles of 32 lanes more
    // than in pairs, but the inverse and the final product (18-23 us) fall away; at 4096
    // entries a CTA that is ~1 us a swap.  A call on 8 matrices of up to 1233 x 9: 176 us in
    // pairs, 147 in FP64.
    if (maxvol_in_f64(max_nr, delta)) return launch_cluster(k_maxvol_swap<true>, ncl, n, smem, s, d, delta, max_iters, doubles);
    e = launch_cluster(k_maxvol_swap<false>, ncl, n, smem, s, d, delta, max_iters, doubles);
    if (e != cudaSuccess) return e;
    k_maxvol_inverse<<<n, 256, sizeof(double) * max_r * (2 * max_r + 1), s>>>(d);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int blocks = std::max(8, std::min(128, 8 * sm_count() / n));
    k_maxvol_final<<<dim3(blocks, n), 256, sizeof(double) * (max_r * max_r + 64 * max_r), s>>>(d);
    return cudaGetLastError();
}

}  // namespace wg
