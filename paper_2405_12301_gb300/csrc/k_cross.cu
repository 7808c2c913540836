// k_cross.cu -- pointwise WENO5-JS residual at TT-cross sample points
// (Sec. 4.2-4.3, Algorithms 1 and 2), evaluated from TT cores (Eq. TT_def).
//
// A fiber set of one instance is every sample (l, i, r): left multi-index l
// over the modes before the sweep mode m, index i of mode m, right
// multi-index r over the modes after it.  The value of field f at a sample is
// L_l G_m(i) R_r with L_l = G_0(.)..G_{m-1}(.) and R_r = G_{m+1}(.)..G_2(.).
// The residual in flux direction fd needs the 7-point stencil along fd, which
// moves the left vector (fd < m), the core index i (fd = m) or the right
// vector (fd > m).
//
// Two launches:
//   k_cross_vecs  contracts every left and right vector of every set once,
//                 the 7 shifted ones where the stencil moves that side (FP32:
//                 stored as differences from the centre vector, so rounding
//                 scales with the variation along the stencil);
//   k_cross       persistent; a work item is a chunk of rows i of the core and a
//                 block of up to eight indices of the side the stencil does not
//                 move (r for fd <= m, l for fd > m), small enough that the items
//                 of the largest fiber set do not outlast the rest (cross_plan).
//                 It contracts the core rows G_m(i) with the block's vectors once
//                 into shared memory; every sample (v, i) of the other side's
//                 index v then needs only 7 dot products per field, followed by
//                 the LF split fluxes at the 7 points and WENO5(+/-) at the two
//                 interfaces of the sample.  Where the stencil moves along the
//                 fiber (fd = m) neighbouring samples share points and interfaces,
//                 so those are formed once per chunk and varying index.
// Ghost rows (Sec. 4.5) are mapped by the boundary rule of fd.
//
// Bound by the latency of the core rows' loads and by the shared-memory pipe.  On the
// FP32 workload of 64 instances (15 million samples) what brought it from 4.13 to
// 2.95 ms: all loads of a matrix piece before their first use, a thread per entry where
// rows have one entry, no reloads of the set's description behind stores, columns that
// fill the buffer at small ranks, and the samples' stencil values as a register-tiled
// product through shared memory (thread per sample: 280 float4 loads, now ~110).
#include <algorithm>
#include <type_traits>

#include "weno_dev.cuh"
#include "weno_internal.h"
#include "cross_internal.h"

namespace wg {

constexpr int XT = 256;       // threads per CTA of k_cross_vecs
constexpr int VP = 32;        // padded vector length (largest rank)
constexpr int CS = VP + 4;    // shared-memory row stride: float4 reads of 8 consecutive rows hit distinct banks
// fixed indices per work item at most; with fd = m, where a chunk's points carry a
// 6-point halo, 4 (FP32) or 1
constexpr int cross_jb(bool f64) { return f64 ? 4 : 8; }
constexpr int JB1 = 4;
// Row pitch of the contracted rows of clen entries: a multiple of 4 that is odd in
// float4s, so that float4 reads of 8 consecutive rows hit distinct banks; shorter rows
// leave room for more columns.
__host__ __device__ constexpr int cross_cs(bool f64, int clen)
{
    return f64 ? 36 : ((clen + 3) / 4 | 1) * 4;
}
constexpr int SP = 9;         // pitch of a warp's staged 32 x 8 piece of a core row's matrix
constexpr int FLS = 11;       // values per point of the fiber path's split fluxes (10, padded odd:
                              // consecutive points of a warp fall on distinct banks)
// k_cross is compiled for several (threads per CTA, samples per chunk) pairs;
// the autotuner of api_cross.cu picks one, and the persistent grid size, per
// workload class.  Until then variant 7 at 2 CTAs per SM runs (FP32: held to 128
// registers, no spills; the 64-instance workload takes 2.95 ms, variant 5 at 80
// registers 3.3); FP64, bound by its pipe, takes the variant whose shared memory
// lets two CTAs share an SM.  minb > 1 asks the compiler for registers that fit
// minb CTAs per SM.
struct CrossVariant { int threads, chunk, minb; };
constexpr CrossVariant kCrossVariants[] = {{256, 64, 1}, {256, 32, 1}, {128, 64, 1}, {128, 32, 1},
                                           {256, 128, 1}, {256, 64, 3}, {128, 64, 6}, {256, 64, 2}};
// rows of an FP64 chunk: at most 96 (shared memory)
constexpr int variant_chunk(bool f64, int v)
{
    return f64 && kCrossVariants[v].chunk > 96 ? 96 : kCrossVariants[v].chunk;
}
constexpr int kNumCrossVariants = sizeof(kCrossVariants) / sizeof(kCrossVariants[0]);
static_assert(kCrossVariants[7].threads == 256 && kCrossVariants[7].chunk == 64 && kCrossVariants[7].minb == 2,
              "cross_default names variant 7");

template <typename T> __device__ __forceinline__ T cvtf(float x) { return (T)x; }

// Index along mode m after the boundary rule of that mode.
__device__ __forceinline__ int xmap(const CrossInst &in, int m, int c, bool &flip)
{
    return ghost_source(c, in.n[m], in.bc[m][0], in.bc[m][1], flip);
}

// Entry a of the left vector of field f for multi-index lidx (modes < mode),
// with the index of mode fd moved by s (s = 0: the centre).
template <typename T>
__device__ T left_entry(const CrossInst &in, int mode, const int *lidx, int f, int a, int fd, int s, bool &flip)
{
    flip = false;
    int i0 = lidx[0];
    if (fd == 0 && s != 0) i0 = xmap(in, 0, i0 + s, flip);
    const int r1 = in.r[0];
    if (mode == 1) return cvtf<T>(__ldg(in.core[f][0] + (long long)i0 * r1 + a));
    int i1 = lidx[1];
    if (fd == 1 && s != 0) i1 = xmap(in, 1, i1 + s, flip);
    const int r2 = in.r[1];
    const float *g0 = in.core[f][0] + (long long)i0 * r1;
    const float *g1 = in.core[f][1] + (long long)i1 * r1 * r2 + a;
    T acc = T(0);
    for (int b = 0; b < r1; ++b) acc += cvtf<T>(__ldg(g0 + b)) * cvtf<T>(__ldg(g1 + b * r2));
    return acc;
}

// Entry b of the right vector of field f for multi-index ridx (modes > mode).
template <typename T>
__device__ T right_entry(const CrossInst &in, int mode, const int *ridx, int f, int b, int fd, int s, bool &flip)
{
    flip = false;
    const int r1 = in.r[0], r2 = in.r[1];
    if (mode == 1) {
        int k = ridx[0];
        if (fd == 2 && s != 0) k = xmap(in, 2, k + s, flip);
        return cvtf<T>(__ldg(in.core[f][2] + (long long)k * r2 + b));
    }
    int j = ridx[0], k = ridx[1];
    if (fd == 1 && s != 0) j = xmap(in, 1, j + s, flip);
    if (fd == 2 && s != 0) k = xmap(in, 2, k + s, flip);
    const float *g1 = in.core[f][1] + (long long)j * r1 * r2 + (long long)b * r2;
    const float *g2 = in.core[f][2] + (long long)k * r2;
    T acc = T(0);
    for (int c = 0; c < r2; ++c) acc += cvtf<T>(__ldg(g1 + c)) * cvtf<T>(__ldg(g2 + c));
    return acc;
}

// ---------------------------------------------------------------- vectors
// Lvec of a set: [n_left][nsl][5][VP], Rvec: [n_right][nsr][5][VP]; ns = 7
// holds s = -3..3 (centre at 3), ns = 1 the centre only.  gridDim.y CTAs per set
// share its vectors (one CTA per set took 0.96 ms on the 64-instance workload,
// the largest set's ~10^5 entries in one CTA; a thread forms an entry's centre
// once for all its shifted copies).
template <bool F64>
__global__ void __launch_bounds__(XT) k_cross_vecs(const CrossArgs A)
{
    using T = typename std::conditional<F64, double, float>::type;
    const CrossSet &S = A.sets[blockIdx.x];
    const CrossInst &in = A.inst[S.inst];
    const int mode = S.mode, fd = S.fd;
    T *vec = reinterpret_cast<T *>(A.vecs);
    __shared__ int bad;
    if (threadIdx.x == 0) bad = 0;
    __syncthreads();
    // index check: a bad multi-index marks the set (its samples are skipped, never read)
    for (long long u = threadIdx.x; u < S.n_left * mode; u += XT)
        if ((unsigned)S.left[u] >= (unsigned)in.n[u % mode]) bad = 1;
    for (long long u = threadIdx.x; u < S.n_right * (2 - mode); u += XT)
        if ((unsigned)S.right[u] >= (unsigned)in.n[mode + 1 + u % (2 - mode)]) bad = 1;
    __syncthreads();
    if (threadIdx.x == 0 && blockIdx.y == 0) A.bad[blockIdx.x] = bad;
    if (bad) {
        if (threadIdx.x == 0) atomicOr(A.status, ST_BADINDEX);
        return;
    }
    const int rl = mode == 0 ? 1 : in.r[mode - 1];
    const int rr = mode == 2 ? 1 : in.r[mode];
    for (int side = 0; side < 2; ++side) {
        const long long nidx = side == 0 ? S.n_left : S.n_right;
        const int ns = side == 0 ? S.nsl : S.nsr;
        const int len = side == 0 ? rl : rr;
        const bool empty = (side == 0 && mode == 0) || (side == 1 && mode == 2);
        T *out = vec + (side == 0 ? S.lvec_off : S.rvec_off);
        for (long long u = blockIdx.y * XT + threadIdx.x; u < nidx * 5 * VP; u += gridDim.y * XT) {
            const int a = (int)(u % VP);
            const int f = (int)((u / VP) % 5);
            const long long idx = u / (5 * VP);
            auto entry = [&](int s, bool &fl) {
                return side == 0 ? left_entry<T>(in, mode, S.left + idx * mode, f, a, fd, s, fl)
                                 : right_entry<T>(in, mode, S.right + idx * (2 - mode), f, a, fd, s, fl);
            };
            const bool live = a < len;
            bool f0;
            const T c = !live ? T(0) : empty ? T(1) : entry(0, f0);  // an empty side is the 1 x 1 identity
            T *o = out + idx * ns * 5 * VP + f * VP + a;
            for (int k = 0; k < ns; ++k) {
                const int s = ns == 7 ? k - 3 : 0;
                T v = c;
                if (s != 0 && live) {
                    bool fl;
                    v = entry(s, fl);
                    if (fl && f == 1 + fd) v = -v;  // mirrored ghost row: normal momentum negated
                    if (!F64) v -= c;
                }
                o[(long long)k * 5 * VP] = v;
            }
        }
    }
}

// ------------------------------------------------------------------- main
// Shared memory of k_cross in elements of T.
template <bool F64, int XT, int CH> struct CrossSmem {
    static constexpr int JB = cross_jb(F64);
    static constexpr int CP = CH + 6;               // columns of a chunk, with the stencil halo of fd = m
    static constexpr int c = 0;                     // [5][CP][CS] (as [5][cap][cs]) contracted core rows
    static constexpr int cref = c + 5 * CP * CS;    // [5][JB1][CS] the chunk's reference row (FP32, fd = m)
    static constexpr int fixv = cref + 5 * JB1 * CS;  // [5][VP][JB] the item's fixed vectors
    static constexpr int fl = fixv + 5 * VP * JB;   // [XT][FLS]   fd = m: split fluxes of a block's points
    static constexpr int stage = fl;                // [XT / 32][32][SP] (before fl is written) staged core pieces
    static constexpr int ff = fl + (XT * FLS > XT * SP ? XT * FLS : XT * SP);  // [5][XT] face fluxes (doubled)
    static constexpr int ct = ff + 5 * XT;          // [XT / 7 + 1][5] reference values (row i0)
    static constexpr int q7 = fl;                   // fd != m, FP32: [5][7][XT] stencil differences of a block of samples
    static constexpr int t1 = ct + 5 * (XT / 7 + 1), t7 = q7 + (F64 ? 0 : 35 * XT);
    static constexpr int total = t1 > t7 ? t1 : t7;
};

// RefState of a sample's centre (FP32), whose primitives multiply differences only.
__device__ __forceinline__ void cross_ref(const float *ctr, float gm1, RefState<3> &rs)
{
#pragma unroll
    for (int f = 0; f < 5; ++f) { rs.hi[f] = ctr[f]; rs.lo[f] = 0.0f; }
    const float ir = 1.0f / ctr[0];
    float ke = 0.0f;
    rs.rho = ctr[0];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        rs.m[e] = ctr[1 + e];
        rs.u[e] = ctr[1 + e] * ir;
        ke += rs.m[e] * rs.u[e];
    }
    rs.H = ctr[4] + gm1 * (ctr[4] - 0.5f * ke);
}

// Twice the split fluxes of one stencil point: q the state (FP64) or its difference from rs (FP32).
__device__ __forceinline__ void cross_flux(int fd, const float *q, const RefState<3> &rs, float alpha, double gm1, float *a5, float *b5)
{
    if (fd == 0) split_flux_diff<3, 0, true>(q, rs, alpha, (float)gm1, a5, b5);
    else if (fd == 1) split_flux_diff<3, 1, true>(q, rs, alpha, (float)gm1, a5, b5);
    else split_flux_diff<3, 2, true>(q, rs, alpha, (float)gm1, a5, b5);
}
__device__ __forceinline__ void cross_flux(int fd, const double *q, const RefState<3> &, double alpha, double gm1, double *a5, double *b5)
{
    if (fd == 0) split_flux_f64<3, 0, true>(q, alpha, gm1, a5, b5);
    else if (fd == 1) split_flux_f64<3, 1, true>(q, alpha, gm1, a5, b5);
    else split_flux_f64<3, 2, true>(q, alpha, gm1, a5, b5);
}

// Twice the flux of the face whose f(+) window is P[0], P[s], .., P[4 s] and whose
// mirrored f(-) window is M[5 s], M[4 s], .., M[s] (FP32: one f32x2 pair).
__device__ __forceinline__ float cross_face(const float *P, const float *M, int s, float eps, const PairEps &)
{
    return weno5_pm(make_float2(P[0], M[5 * s]), make_float2(P[s], M[4 * s]), make_float2(P[2 * s], M[3 * s]),
                    make_float2(P[3 * s], M[2 * s]), make_float2(P[4 * s], M[s]), eps);
}
__device__ __forceinline__ double cross_face(const double *P, const double *M, int s, double, const PairEps &E)
{
    return weno5_pair(P[0], P[s], P[2 * s], P[3 * s], P[4 * s], E) + weno5_pair(M[5 * s], M[4 * s], M[3 * s], M[2 * s], M[s], E);
}

// Six times -(F_hi - F_lo) of a sample along fd, FP32, for its five fields: q[(7 f + k)
// stride] is the difference of field f at stencil point k from the centre (k = 3),
// whose state it holds there.  The primitives' differences are formed once per point;
// a field's two faces share their differences and indicators (the run of two windows
// of weno5d_cells2, WENO(+) in lane x, the mirrored WENO(-) in lane y).
template <class Put>
__device__ __forceinline__ void cross_sample(const float *q, int stride, int fd, float alpha, float gm1, float Geps_, Put put)
{
    float ctr[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) ctr[f] = q[(7 * f + 3) * stride];
    RefState<3> rs;
    cross_ref(ctr, gm1, rs);
    const float un = fd == 0 ? rs.u[0] : fd == 1 ? rs.u[1] : rs.u[2];
    float du[7], dp[7];  // of the normal velocity and the pressure (split_flux_diff)
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        du[k] = dp[k] = 0.0f;
        if (k == 3) continue;
        const float d0 = q[k * stride], ir = fast_rcp(rs.rho + d0);
        float dk = 0.0f;
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            const float dm = q[(7 * (1 + e) + k) * stride], d = (dm - rs.u[e] * d0) * ir;
            dk += dm * (rs.u[e] + d) + rs.m[e] * d;
            if (e == fd) du[k] = d;
        }
        dp[k] = gm1 * (q[(28 + k) * stride] - 0.5f * dk);
    }
    const float2 kk = bc2((float)(13.0 / 3.0)), Geps = bc2(Geps_), al = make_float2(alpha, -alpha);
#pragma unroll
    for (int f = 0; f < 5; ++f) {
        float2 s[7];  // twice the split fluxes f(+), f(-), less the centre's
#pragma unroll
        for (int k = 0; k < 7; ++k) {
            if (k == 3) {
                s[k] = bc2(0.0f);
                continue;
            }
            const float d = q[(7 * f + k) * stride];
            float F;
            if (f == 0) {
                F = q[(7 * (1 + fd) + k) * stride];
            } else if (f < 4) {
                F = d * (un + du[k]) + rs.m[f < 4 ? f - 1 : 0] * du[k] + (f == 1 + fd ? dp[k] : 0.0f);
            } else {
                const float dH = d + dp[k];
                F = du[k] * (rs.H + dH) + un * dH;
            }
            s[k] = fma2(al, bc2(d), bc2(F));
        }
        float2 D[5];
#pragma unroll
        for (int k = 0; k < 5; ++k)
            D[k] = mul2(bc2(0.5f), sub2(make_float2(s[k + 1].x, s[5 - k].y), make_float2(s[k].x, s[6 - k].y)));
        float2 t[4], A[4], C[2];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            t[k] = sub2(D[k + 1], D[k]);
            A[k] = fma2(mul2(kk, t[k]), t[k], Geps);
        }
        const float2 e[3] = {sub2(t[0], t[1]), sub2(t[1], t[2]), sub2(t[2], t[3])};
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const float2 s0 = fma2(bc2(-3.0f), D[m + 2], D[m + 3]), s1 = add2(D[m + 1], D[m + 2]),
                         s2 = fma2(bc2(-3.0f), D[m + 1], D[m]);
            float2 g0 = fma2(s0, s0, A[m + 2]), g1 = fma2(s1, s1, A[m + 1]), g2 = fma2(s2, s2, A[m]);
            g0 = mul2(g0, g0);
            g1 = mul2(g1, g1);
            g2 = mul2(g2, g2);
            const float2 w0 = mul2(g1, g2), w1 = mul2(g0, g2), w2 = mul2(g0, g1);  // times 3, 6, 1
            const float2 sw = fma2(bc2(3.0f), w0, fma2(bc2(6.0f), w1, w2));
            const float2 num = fma2(w0, mul2(bc2(3.0f), e[m + 1]), mul2(w2, add2(e[m], e[m])));
            C[m] = fma2(num, make_float2(fast_rcp(sw.x), fast_rcp(sw.y)), fma2(bc2(2.0f), D[m + 2], D[m + 1]));
        }
        const float2 r = fma2(bc2(6.0f), D[2], sub2(C[1], C[0]));  // (lane y: of the mirrored run)
        put(f, r.y - r.x);
    }
}

// Dot product of two zero-padded rows of l4 entries.  FP32: even and odd entries
// accumulate in the two lanes of an f32x2 (one issue slot per two FMAs).
__device__ __forceinline__ float row_dot(const float *x, const float *y, int, int l4)
{
    float2 s = bc2(0.0f);
    for (int e = 0; e < l4; e += 4) {
        const float4 p = *reinterpret_cast<const float4 *>(x + e), q = *reinterpret_cast<const float4 *>(y + e);
        s = fma2(make_float2(p.z, p.w), make_float2(q.z, q.w), fma2(make_float2(p.x, p.y), make_float2(q.x, q.y), s));
    }
    return s.x + s.y;
}
__device__ __forceinline__ double row_dot(const double *x, const double *y, int l, int)
{
    double s = 0.0;
    for (int e = 0; e < l; ++e) s = fma(x[e], y[e], s);
    return s;
}

template <bool F64, int XT, int CH, int MINB>
__global__ void __launch_bounds__(XT, MINB) k_cross(const CrossArgs A)
{
    using T = typename std::conditional<F64, double, float>::type;
    using SM = CrossSmem<F64, XT, CH>;
    constexpr int CP = SM::CP, JB = SM::JB, NWARP = XT / 32;
    constexpr int NC = MINB > 2 ? 2 : 4;
    extern __shared__ __align__(16) unsigned char dyn[];
    T *base = reinterpret_cast<T *>(dyn);
    T *C = base + SM::c, *Cref = base + SM::cref, *fixv = base + SM::fixv;
    T *FL = base + SM::fl, *FF = base + SM::ff, *CT = base + SM::ct;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T *stage = base + SM::stage + warp * 32 * SP;
    __shared__ long long s_item;
    __shared__ const float *s_core[5];
    const T eps = T(4) * (T)A.eps;  // split fluxes are formed doubled: 4 eps gives twice the WENO5 value
    PairEps E{};
    if constexpr (F64) E = pair_eps(4.0 * A.eps);
    const double gm1 = A.gamma - 1.0;
    const T *vecs = reinterpret_cast<const T *>(A.vecs);

    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(A.counter, 1ull);
        __syncthreads();
        const long long item = s_item;
        if (item >= A.n_work) break;
        int lo = 0, hi = A.n_sets - 1;  // the set holding this item
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (A.sets[mid].work_begin <= item) lo = mid;
            else hi = mid - 1;
        }
        if (A.bad[lo]) continue;
        // what the loops below read of the set and its instance, by value: a store to the
        // output would have them read again
        const CrossSet S = A.sets[lo];
        const CrossInst &in = A.inst[S.inst];
        const int mode = S.mode, fd = S.fd, n = S.n_mode;
        const int n_fd = in.n[fd], bc_lo = in.bc[fd][0], bc_hi = in.bc[fd][1];
        if (threadIdx.x < 5) s_core[threadIdx.x] = in.core[threadIdx.x][mode];
        const long long plane = S.n_left * n * S.n_right;  // samples of a field
        const int role = fd < mode ? 0 : (fd == mode ? 1 : 2);  // stencil moves: L / the core index / R
        const int rl = mode == 0 ? 1 : in.r[mode - 1];
        const int rr = mode == 2 ? 1 : in.r[mode];
        const int clen = role == 2 ? rr : rl;                    // length of a contracted row
        const int cl4 = (clen + 3) & ~3;
        const int cs = cross_cs(F64, clen), cap = CP * CS / cs;  // row pitch and columns of C
        const long long nvar = role == 2 ? S.n_right : S.n_left;
        const long long nfix = role == 2 ? S.n_left : S.n_right;
        const T *var = vecs + (role == 2 ? S.rvec_off : S.lvec_off);  // the varying side's vectors
        const int nsv = role == 2 ? S.nsr : S.nsl;
        const T alpha = (T)in.alpha;
        const T ih = (T)(0.5 / in.h[fd]);  // halves the doubled face fluxes
        // the item: rows i0 .. i0 + cn, fixed indices j0 .. j0 + jn
        const int jb = S.jb;
        const long long njb = S.njb, w = item - S.work_begin;
        const int i0 = (int)(w / njb) * S.rows;
        const long long j0 = (w - (w / njb) * njb) * jb;
        const int jn = nfix - j0 < jb ? (int)(nfix - j0) : jb;
        const int cn = n - i0 < S.rows ? n - i0 : S.rows;
        for (int u = threadIdx.x; u < 5 * VP * JB; u += XT) {  // the fixed side's centre vectors
            const int jj = u / (5 * VP), x = u - jj * 5 * VP;
            const T *src = vecs + (role == 2 ? S.lvec_off + ((j0 + jj) * S.nsl + (S.nsl == 7 ? 3 : 0)) * 5 * VP
                                             : S.rvec_off + ((j0 + jj) * S.nsr + (S.nsr == 7 ? 3 : 0)) * 5 * VP);
            fixv[x * JB + jj] = jj < jn ? src[x] : T(0);
        }
        const long long outstride_v = role == 2 ? 1 : (long long)n * S.n_right;   // along the varying index
        const long long outstride_j = role == 2 ? (long long)n * S.n_right : 1;   // along the fixed index
        T *out = reinterpret_cast<T *>(S.out);
        __syncthreads();

        // One core row's matrix against the fixed vectors, by one warp, lane x the
        // row entry.  Role 2: sum_y fixv[y] G[y][x], coalesced as it stands.
        // Otherwise sum_y G[x][y] fixv[y] (of G - G0 if there is a G0): pieces of 8
        // columns go through the warp's stage, so that the loads take whole 32-byte
        // sectors (a lane reading its own row touched 32 lines per load, and these
        // loads were 85% of the kernel's L1 traffic).  An entry's sums for all fixed
        // indices are formed at once (FP32: in f32x2 pairs of indices).
        T acc[JB];
        auto contract_n = [&](auto nq, int f, const float *g, const float *g0) {
            constexpr int NQ = decltype(nq)::value;  // fixed indices (1, or a multiple of 4)
#pragma unroll
            for (int q = 0; q < JB; ++q) acc[q] = T(0);
            const T *fv = fixv + f * VP * JB;
            auto add = [&](T v, int y) {
                const T *r = fv + y * JB;
                if constexpr (NQ == 1) {
                    acc[0] = fma(v, r[0], acc[0]);
                } else if constexpr (F64) {
#pragma unroll
                    for (int q = 0; q < NQ; ++q) acc[q] = fma(v, r[q], acc[q]);
                } else {
#pragma unroll
                    for (int q = 0; q < NQ; q += 4) {
                        const float4 r4 = *reinterpret_cast<const float4 *>(r + q);
                        const float2 lo2 = fma2(bc2(v), make_float2(r4.x, r4.y), make_float2(acc[q], acc[q + 1]));
                        const float2 hi2 = fma2(bc2(v), make_float2(r4.z, r4.w), make_float2(acc[q + 2], acc[q + 3]));
                        acc[q] = lo2.x;
                        acc[q + 1] = lo2.y;
                        acc[q + 2] = hi2.x;
                        acc[q + 3] = hi2.y;
                    }
                }
            };
            if (role == 2) {
                for (int y0 = 0; y0 < rl; y0 += 8) {
                    T v[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) v[k] = y0 + k < rl && lane < rr ? cvtf<T>(__ldg(g + (y0 + k) * rr + lane)) : T(0);
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (y0 + k < rl) add(v[k], y0 + k);
                }
            } else if (rr == 1) {
                add(lane < rl ? cvtf<T>(__ldg(g + lane)) - (g0 ? cvtf<T>(__ldg(g0 + lane)) : T(0)) : T(0), 0);
            } else {
                for (int y0 = 0; y0 < rr; y0 += 8) {
                    // all loads of a piece go out before the first is used
                    const int y = y0 + (lane & 7), x0 = lane >> 3;
                    const int e = x0 * rr + y;
                    T v[8], v0[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const bool live = 4 * k + x0 < rl && y < rr;
                        v[k] = live ? cvtf<T>(__ldg(g + e + 4 * k * rr)) : T(0);
                        v0[k] = live && g0 ? cvtf<T>(__ldg(g0 + e + 4 * k * rr)) : T(0);
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k) stage[(4 * k + x0) * SP + (lane & 7)] = v[k] - v0[k];
                    __syncwarp();
                    const T *sr = stage + lane * SP;  // (rows from rl on are zero)
                    if (rr - y0 >= 8) {
#pragma unroll
                        for (int k = 0; k < 8; ++k) add(sr[k], y0 + k);
                    } else {
                        for (int k = 0; k < rr - y0; ++k) add(sr[k], y0 + k);
                    }
                    __syncwarp();
                }
            }
        };
        auto contract = [&](int f, const float *g, const float *g0) {
            if (jb == 1) contract_n(std::integral_constant<int, 1>(), f, g, g0);
            else if (JB == 4 || jb <= 4) contract_n(std::integral_constant<int, 4>(), f, g, g0);
            else contract_n(std::integral_constant<int, JB>(), f, g, g0);
        };
        // chunk reference row (FP32, stencil along the fiber): G(i0) . R
        if (!F64 && role == 1) {
            for (int f = warp; f < 5; f += NWARP) {
                contract(f, s_core[f] + (long long)i0 * rl * rr, nullptr);
#pragma unroll
                for (int q = 0; q < JB1; ++q)
                    if (lane < cl4 && q < jb) Cref[(f * JB1 + q) * CS + lane] = acc[q];
            }
            __syncthreads();
        }
        // contracted rows, zero-padded to a multiple of 4 entries; column = (row or point,
        // fixed index), the one that neighbouring threads below take varying fastest
        // (their float4 reads of rows CS apart then hit distinct banks)
        const int np = role == 1 ? cn + 6 : cn;
        const int cs_p = role == 1 ? 1 : jb, cs_q = role == 1 ? np : 1;
        // a first mode's rows have one entry: a thread per entry (a warp per row left 31
        // lanes idle, and fd = 0 fibers of the first mode took 663 us of 4127)
        if (rl == 1 && role != 2) {
            for (int u = threadIdx.x; u < 5 * np * jb; u += XT) {
                const int f = u / (np * jb), r = u - f * np * jb, pp = r / jb, q = r - pp * jb;
                bool flip = false;
                const int c = role == 1 ? ghost_source(i0 - 3 + pp, n_fd, bc_lo, bc_hi, flip) : i0 + pp;
                const float *g = s_core[f] + (long long)c * rr, *g0 = s_core[f] + (long long)i0 * rr;
                const T *fv = fixv + f * VP * JB + q;
                T acc1 = T(0);
                if (!F64 && role == 1)
                    for (int y = 0; y < rr; ++y) acc1 = fma(__ldg(g + y) - __ldg(g0 + y), fv[y * JB], acc1);
                else
                    for (int y = 0; y < rr; ++y) acc1 = fma(cvtf<T>(__ldg(g + y)), fv[y * JB], acc1);
                if (flip && f == 1 + fd) acc1 = F64 ? -acc1 : -acc1 - T(2) * Cref[(f * JB1 + (q & (JB1 - 1))) * CS];
                T *row = C + (f * cap + pp * cs_p + q * cs_q) * cs;
                row[0] = acc1;
                for (int x = 1; x < cl4; ++x) row[x] = T(0);
            }
        } else
        for (int u = warp; u < 5 * np; u += NWARP) {
            const int f = u / np, pp = u - f * np;
            bool flip = false;
            int c = role == 1 ? i0 - 3 + pp : i0 + pp;
            if (role == 1) c = ghost_source(c, n_fd, bc_lo, bc_hi, flip);
            const float *g = s_core[f];
            contract(f, g + (long long)c * rl * rr, !F64 && role == 1 ? g + (long long)i0 * rl * rr : nullptr);
            flip = flip && f == 1 + fd;
            if (lane < cl4) {
                T *row = C + (f * cap + pp * cs_p) * cs + lane;
#pragma unroll
                for (int q = 0; q < JB; ++q) {
                    if (q < jb) {
                        if (flip) acc[q] = F64 ? -acc[q] : -acc[q] - T(2) * Cref[(f * JB1 + (q & (JB1 - 1))) * CS + lane];
                        row[q * cs_q * cs] = acc[q];
                    }
                }
            }
        }
        __syncthreads();

        if (role == 1) {
            // The stencil moves along the fiber: neighbouring samples of one varying
            // index share six of their seven points and one of their two faces, so
            // each point's split flux and each face's WENO5(+/-) is formed once per
            // block of vb lines (varying index, fixed index), as many as make each
            // phase one pass.
            const int vb = XT / np;
            const long long nline = nvar * jn;
            for (long long l0 = 0; l0 < nline; l0 += vb) {
                const int nv = nline - l0 < vb ? (int)(nline - l0) : vb;
                const long long vbase = l0 / jn;
                const int qbase = (int)(l0 - vbase * jn);
                // line vl of the block: varying index vbase + dv, fixed index j0 + q
                auto line = [&](int vl, int &dv, int &q) {
                    q = qbase + vl;
                    dv = q / jn;
                    q -= dv * jn;
                };
                if constexpr (!F64) {  // reference values (row i0) of the block's lines
                    for (int u = threadIdx.x; u < nv * 5; u += XT) {
                        const int vl = u / 5, f = u - 5 * vl;
                        int dv, q;
                        line(vl, dv, q);
                        CT[u] = row_dot(var + (vbase + dv) * nsv * 5 * VP + f * VP, Cref + (f * JB1 + q) * CS, clen, cl4);
                    }
                    __syncthreads();
                }
                for (int u = threadIdx.x; u < nv * np; u += XT) {  // split fluxes of every chunk point
                    const int vl = u / np, pp = u - vl * np;
                    int dv, jq;
                    line(vl, dv, jq);
                    const int col = jq * np + pp;
                    const T *lv = var + (vbase + dv) * nsv * 5 * VP;
                    T q[5], a5[5], b5[5];
#pragma unroll
                    for (int f = 0; f < 5; ++f) q[f] = row_dot(lv + f * VP, C + (f * cap + col) * cs, clen, cl4);
                    RefState<3> rs;
                    if constexpr (!F64) cross_ref(CT + vl * 5, (float)gm1, rs);
                    cross_flux(fd, q, rs, alpha, gm1, a5, b5);
                    T *fl = FL + u * FLS;
#pragma unroll
                    for (int f = 0; f < 5; ++f) { fl[f] = a5[f]; fl[5 + f] = b5[f]; }
                }
                __syncthreads();
                // face fluxes (face k lies before sample k), one work item per face and field
                for (int u = threadIdx.x; u < 5 * nv * (cn + 1); u += XT) {
                    const int f = u / (nv * (cn + 1)), r = u - f * (nv * (cn + 1));
                    const int vl = r / (cn + 1), k = r - vl * (cn + 1);
                    const T *fl = FL + (vl * np + k) * FLS + f;
                    FF[f * XT + r] = cross_face(fl, fl + 5, FLS, eps, E);
                }
                __syncthreads();
                for (int u = threadIdx.x; u < nv * cn; u += XT) {
                    const int vl = u / cn, ii = u - vl * cn;
                    int dv, q;
                    line(vl, dv, q);
                    const long long o = (j0 + q) * outstride_j + (vbase + dv) * outstride_v + (long long)(i0 + ii) * S.n_right;
#pragma unroll
                    for (int f = 0; f < 5; ++f) {
                        const T *F = FF + f * XT + vl * (cn + 1) + ii;
                        out[f * plane + o] = -(F[1] - F[0]) * ih;
                    }
                }
                // (the next block's first writes go to CT and FL, which no thread reads
                // after the barrier above)
            }
            continue;
        }
        // samples (v, column): 7 stencil values per field, split fluxes, two interfaces
        const int ncol = cn * jn;
        if constexpr (!F64) {
            // A block of varying indices at a time, nv x ncol <= XT samples: the 35
            // values of every sample go through shared memory, formed in register tiles
            // of 7 shifts x NC columns (a thread per sample kept all 35 and the 70 split
            // fluxes in registers, and loaded 7 vectors for each column).
            T *Q = base + SM::q7;
            const int G = (ncol + NC - 1) / NC, nvb = XT / ncol;
            const float ih6 = (float)(1.0 / (6.0 * in.h[fd]));
            for (long long v0 = 0; v0 < nvar; v0 += nvb) {
                const int nv = nvar - v0 < nvb ? (int)(nvar - v0) : nvb;
                for (int u = threadIdx.x; u < nv * 5 * G; u += XT) {
                    const int vf = u / G, g = u - vf * G, vl = vf / 5, f = vf - vl * 5;
                    const T *vv = var + (v0 + vl) * 35 * VP + f * VP;
                    const T *cr[NC];
                    float2 a2[7][NC];
#pragma unroll
                    for (int j = 0; j < NC; ++j) {
                        const int cu = min(g + j * G, ncol - 1), ii = cu / jn;
                        cr[j] = C + (f * cap + ii * jb + (cu - ii * jn)) * cs;
#pragma unroll
                        for (int k = 0; k < 7; ++k) a2[k][j] = bc2(0.0f);
                    }
                    for (int x = 0; x < cl4; x += 4) {
                        float4 c4[NC];
#pragma unroll
                        for (int j = 0; j < NC; ++j) c4[j] = *reinterpret_cast<const float4 *>(cr[j] + x);
#pragma unroll
                        for (int k = 0; k < 7; ++k) {
                            const float4 w4 = __ldg(reinterpret_cast<const float4 *>(vv + k * 5 * VP + x));
#pragma unroll
                            for (int j = 0; j < NC; ++j)
                                a2[k][j] = fma2(make_float2(w4.z, w4.w), make_float2(c4[j].z, c4[j].w),
                                                fma2(make_float2(w4.x, w4.y), make_float2(c4[j].x, c4[j].y), a2[k][j]));
                        }
                    }
#pragma unroll
                    for (int j = 0; j < NC; ++j) {
                        if (g + j * G >= ncol) continue;
                        T *o = Q + f * 7 * XT + vl * ncol + g + j * G;
#pragma unroll
                        for (int k = 0; k < 7; ++k) o[k * XT] = a2[k][j].x + a2[k][j].y;
                    }
                }
                __syncthreads();
                for (int u = threadIdx.x; u < nv * ncol; u += XT) {
                    const int vl = u / ncol, cu = u - vl * ncol, ii = cu / jn, jj = cu - ii * jn;
                    // out[f][l][i][r]: role 0 varies l and fixes r, role 2 the other way round
                    const long long o = (j0 + jj) * outstride_j + (v0 + vl) * outstride_v + (long long)(i0 + ii) * S.n_right;
                    cross_sample(Q + u, XT, fd, alpha, (float)gm1, eps,
                                 [&](int f, float r) { out[f * plane + o] = r * ih6; });
                }
                __syncthreads();
            }
        } else {
            for (long long u = threadIdx.x; u < nvar * ncol; u += XT) {
                const long long v = (unsigned long long)u < (1ull << 32) ? (long long)((unsigned)u / (unsigned)ncol) : u / ncol;
                const int cu = (int)(u - v * ncol), ii = cu / jn, jj = cu - ii * jn, col = ii * jb + jj;
                T q7[5][7];
#pragma unroll
                for (int f = 0; f < 5; ++f) {  // the 7 shifted vectors against the column's row
                    T acc[7];
                    const T *vv = var + (v * 7) * 5 * VP + f * VP;
                    const T *crow = C + (f * cap + col) * cs;
#pragma unroll
                    for (int k = 0; k < 7; ++k) acc[k] = T(0);
                    for (int x = 0; x < clen; ++x) {
                        const T cx = crow[x];
#pragma unroll
                        for (int k = 0; k < 7; ++k) acc[k] += vv[k * 5 * VP + x] * cx;
                    }
#pragma unroll
                    for (int k = 0; k < 7; ++k) q7[f][k] = acc[k];
                }
                T fp7[5][7], fm7[5][7];
                RefState<3> rs;
#pragma unroll
                for (int k = 0; k < 7; ++k) {
                    T q[5], a5[5], b5[5];
#pragma unroll
                    for (int f = 0; f < 5; ++f) q[f] = q7[f][k];
                    cross_flux(fd, q, rs, alpha, gm1, a5, b5);
#pragma unroll
                    for (int f = 0; f < 5; ++f) { fp7[f][k] = a5[f]; fm7[f][k] = b5[f]; }
                }
                // out[f][l][i][r]: role 0 varies l and fixes r, role 2 the other way round
                const long long o = (j0 + jj) * outstride_j + v * outstride_v + (long long)(i0 + ii) * S.n_right;
#pragma unroll
                for (int f = 0; f < 5; ++f) {
                    const T Flo = cross_face(fp7[f], fm7[f], 1, eps, E), Fhi = cross_face(fp7[f] + 1, fm7[f] + 1, 1, eps, E);
                    out[f * plane + o] = -(Fhi - Flo) * ih;
                }
            }
        }
    }
}

template <bool F64, int XT, int CH> static constexpr size_t cross_dyn_bytes()
{
    return (F64 ? sizeof(double) : sizeof(float)) * (size_t)CrossSmem<F64, XT, CH>::total;
}

int cross_vec_len() { return VP; }
int cross_num_variants() { return kNumCrossVariants; }
void cross_default(bool fp64, int *variant, int *ctas_per_sm)
{
    *variant = fp64 ? 1 : 7;
    *ctas_per_sm = 2;
}

// Work items of a set for the chunk length of a variant: jb fixed indices and
// `rows` rows each.  Several fixed indices share a core row's loads and the
// varying vectors; where there are few fixed indices the columns are rows.  With
// fd = m several fixed indices pay for the larger share of halo rows only where a
// row's matrix is large (64 entries).  With fewer than a few items per resident
// CTA the rows are halved.
long long cross_items(const CrossSet &S, int rows)
{
    return (long long)S.njb * ((S.n_mode + rows - 1) / rows);
}
long long cross_plan(CrossSet *sets, int n_sets, bool fp64, int variant)
{
    const int chunk = variant_chunk(fp64, variant), threads = kCrossVariants[variant].threads;
    long long total = 0;
    for (int k = 0; k < n_sets; ++k) {
        CrossSet &S = sets[k];
        const long long nfix = S.fd > S.mode ? S.n_left : S.n_right;
        const int most = S.fd != S.mode ? cross_jb(fp64) : fp64 || S.r_mode < 64 ? 1 : JB1;
        S.jb = (int)((nfix + (nfix + most - 1) / most - 1) / ((nfix + most - 1) / most));  // blocks of equal size
        S.njb = (int)((nfix + S.jb - 1) / S.jb);
        if (fp64) {
            S.rows = S.fd != S.mode ? chunk / S.jb : chunk;
        } else {
            const int cap = std::min(threads, (chunk + 6) * CS / cross_cs(false, S.r_row));
            if (S.fd == S.mode) S.rows = cap / S.jb - 6;
            else S.rows = threads / ((threads + cap - 1) / cap) / S.jb;  // blocks of threads samples: an equal part of one
        }
        total += cross_items(S, S.rows);
    }
    for (int cut = 0; cut < 3 && total < 6ll * sm_count(); ++cut) {
        total = 0;
        for (int k = 0; k < n_sets; ++k) {
            CrossSet &S = sets[k];
            const int least = S.fd == S.mode ? (S.jb == 1 ? 16 : 8) : 4;
            if (S.rows / 2 >= least) S.rows /= 2;
            total += cross_items(S, S.rows);
        }
    }
    total = 0;
    for (int k = 0; k < n_sets; ++k) {
        sets[k].work_begin = total;
        total += cross_items(sets[k], sets[k].rows);
    }
    return total;
}
void cross_variant(int v, int *threads, int *chunk)
{
    *threads = kCrossVariants[v].threads;
    *chunk = kCrossVariants[v].chunk;
}

template <bool F64, int V>
static cudaError_t set_attr()
{
    constexpr int XT_ = kCrossVariants[V].threads, CH_ = variant_chunk(F64, V), MB_ = kCrossVariants[V].minb;
    return cudaFuncSetAttribute(k_cross<F64, XT_, CH_, MB_>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)cross_dyn_bytes<F64, XT_, CH_>());
}

// Shared-memory limits of every variant, set once before any launch (and so
// never inside a stream capture).
cudaError_t cross_set_attributes()
{
    static bool done = false;
    if (done) return cudaSuccess;
    cudaError_t e = cudaSuccess, r;
#define X(V) \
    if ((r = set_attr<false, V>()) != cudaSuccess) e = r; \
    if ((r = set_attr<true, V>()) != cudaSuccess) e = r;
    X(0) X(1) X(2) X(3) X(4) X(5) X(6) X(7)
#undef X
    if (e == cudaSuccess) done = true;
    return e;
}

template <bool F64, int V>
static cudaError_t launch_main(const CrossArgs &a, long long blocks, cudaStream_t s)
{
    constexpr int XT_ = kCrossVariants[V].threads, CH_ = variant_chunk(F64, V), MB_ = kCrossVariants[V].minb;
    k_cross<F64, XT_, CH_, MB_><<<(unsigned)blocks, XT_, cross_dyn_bytes<F64, XT_, CH_>(), s>>>(a);
    return cudaGetLastError();
}

// variant: index into kCrossVariants; ctas_per_sm: persistent grid = SM count x that
// (capped by the number of work items).
cudaError_t launch_cross(const CrossArgs &a, int variant, int ctas_per_sm, cudaStream_t s)
{
    if (variant < 0 || variant >= kNumCrossVariants || ctas_per_sm < 1) return cudaErrorInvalidValue;
    cudaError_t ea = cross_set_attributes();
    if (ea != cudaSuccess) return ea;
    // enough CTAs per set that the largest sets' do not outlast the rest (576 sets: with 4
    // each the SMs stood idle half of the 138 us, with 16 it takes 107)
    const int per_set = (int)std::min(64ll, std::max(16ll, (32ll * sm_count() + a.n_sets - 1) / a.n_sets));
    if (a.fp64) k_cross_vecs<true><<<dim3(a.n_sets, per_set), XT, 0, s>>>(a);
    else k_cross_vecs<false><<<dim3(a.n_sets, per_set), XT, 0, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    long long blocks = (long long)sm_count() * ctas_per_sm;
    if (blocks > a.n_work) blocks = a.n_work;
    if (blocks < 1) blocks = 1;
#define X(V)                                                                             \
    if (variant == V) return a.fp64 ? launch_main<true, V>(a, blocks, s) : launch_main<false, V>(a, blocks, s);
    X(0) X(1) X(2) X(3) X(4) X(5) X(6) X(7)
#undef X
    return cudaErrorInvalidValue;
}

int cross_max_rank() { return VP; }

}  // namespace wg
