// weno_dev.cuh -- device building blocks of the GB300 WENO5-JS residual:
// FP64 <-> FP32 conversions on the integer pipe, ghost-index mapping,
// WENO5-JS reconstruction, point fluxes with Lax-Friedrichs splitting, and the
// device control block.
//
// On GB300 the FP64 pipe (DFMA/DADD) and the FP32<->FP64 conversion
// instructions both issue at about 1.7 per clock per SM, against about 86
// FFMA per clock per SM, so the FP32-bulk path never converts with cvt and
// keeps FP64 arithmetic to one DADD per field per stage.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace wg {

enum { BC_PERIODIC = 0, BC_TRANSMISSIVE = 1, BC_REFLECTIVE = 2, BC_INFLOW = 3 };
enum { ST_NONPHYSICAL = 1, ST_TIMEOUT = 2, ST_BADINDEX = 4 };

// Device control block of one handle: time, step size and the stage alphas.
// alpha[s] holds the bit pattern of a non-negative double so that atomicMax
// on the 64-bit integer is a max on the value (order-independent, so the
// result is bitwise deterministic).  Slot 0: alpha(U^n); slots 1..3: alpha of
// the states written by stages 1..3.
struct Ctl {
    double t;              // current time
    double t_next;         // time after the current step
    double dt;             // dt of the current step (0: the step is a no-op)
    double t_end;
    double dt_req;         // > 0: fixed dt; otherwise CFL
    double cfl_h;          // cfl * min_d h_d
    unsigned long long alpha[4];
    unsigned long long alpha_dir[4][3];  // per-direction max(|u_d| + a), same slots (per-direction mode)
    long long steps;       // steps taken since the last set_time
    long long max_steps;   // steps bound of the current run call
    int status;            // ST_* bits, latched
    unsigned ticket;       // blocks of k_alpha that are done (0 between launches)
    float2 bdt[3];         // b_k dt of stage k (1, 1/4, 2/3) as FP32 pairs hi + lo, set with dt
    unsigned long long alpha_new[4];  // k_alpha's maxima, all and per direction (0 between launches)
};

// ----------------------------------------------------------------- conversions

// Splits a finite FP64 x into FP32 hi + lo: hi is x truncated to 24 significant
// bits, lo approximates x - hi (the next 23 bits), on the integer pipe plus one
// FSUB.  hi: a funnel shift lines the exponent and mantissa up with the FP32
// fields and one add rebiases the exponent by 1023 - 127.  lo: the low 29
// mantissa bits m29 are worth m29 * 2^(e-1075); 2^E (1 + (m29 >> 6) / 2^23) with
// E = e - 1046, minus 2^E, gives that value (exact, up to the 6 dropped bits).
// |x| < 2^-103 (and zero) gives hi = lo = +-0; |x| >= 2^128 is not representable
// (states that large are non-physical).
__device__ __forceinline__ void split_f64(double x, float &hi, float &lo)
{
    const unsigned xh = (unsigned)__double2hiint(x);
    const unsigned xl = (unsigned)__double2loint(x);
    const unsigned sgn = xh & 0x80000000u;
    const unsigned fs = __funnelshift_l(xl, xh, 3) + 0x40000000u;  // [e - 896 : 8][mantissa : 23]
    const unsigned hb = (fs & 0x7FFFFFFFu) | sgn;
    const unsigned eb = (fs - 0x0B800000u) & 0x7F800000u;          // exponent field of 2^(e - 1046)
    const float l = __uint_as_float(eb | ((xl >> 6) & 0x7FFFFFu)) - __uint_as_float(eb);
    const bool ok = ((xh >> 20) & 0x7FFu) >= 920u;
    hi = __uint_as_float(ok ? hb : sgn);
    lo = __uint_as_float(ok ? (__float_as_uint(l) | sgn) : sgn);
}

// FP32 -> FP64, exact for normal numbers (subnormals flush to +-0).
__device__ __forceinline__ double f32_to_f64(float f)
{
    const unsigned b = __float_as_uint(f);
    const unsigned e = (b >> 23) & 0xFFu;
    const unsigned sgn = b & 0x80000000u;
    unsigned hi = sgn | ((e + 896u) << 20) | ((b >> 3) & 0xFFFFFu);
    unsigned lo = b << 29;
    if (e == 0u) { hi = sgn; lo = 0u; }
    if (e == 255u) { hi = sgn | 0x7FF00000u | ((b >> 3) & 0xFFFFFu); }
    return __hiloint2double((int)hi, (int)lo);
}

// FP64 -> FP32 by truncation (hi part of split_f64), integer pipe only.
__device__ __forceinline__ float f64_to_f32(double x)
{
    float hi, lo;
    split_f64(x, hi, lo);
    return hi + lo;
}

// An FP64 coefficient as an unevaluated FP32 pair hi + lo (to about 2^-48
// relative): multiplying by hi alone would bias every use the same way by up
// to 2^-24, which over many time steps is a systematic error.
__device__ __forceinline__ float2 f64_to_f32x2(double x)
{
    const float hi = f64_to_f32(x);
    return make_float2(hi, f64_to_f32(x - f32_to_f64(hi)));
}

__device__ __forceinline__ float fast_rcp(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ------------------------------------------------------------------ ghosts

// Interior source index of a (possibly ghost) index c in [-3, n+2] along a
// direction with n >= 3 cells (Sec. 4.5): periodic wraps, transmissive clamps,
// reflective mirrors (and the caller negates the normal momentum).
__device__ __forceinline__ int ghost_source(int c, int n, int bclo, int bchi, bool &flip)
{
    flip = false;
    if (c < 0) {
        if (bclo == BC_PERIODIC) return c + n;
        if (bclo == BC_TRANSMISSIVE) return 0;
        flip = true;
        return -1 - c;
    }
    if (c >= n) {
        if (bchi == BC_PERIODIC) return c - n;
        if (bchi == BC_TRANSMISSIVE) return n - 1;
        flip = true;
        return 2 * n - 1 - c;
    }
    return c;
}

// Full-grid ghost mapping: as ghost_source, plus inflow sides, whose ghosts
// hold a given state: *inflow is set to the side (0 low, 1 high) and a valid
// interior index is returned (the caller replaces the value); -1 otherwise.
__device__ __forceinline__ int ghost_map(int c, int n, int bclo, int bchi, bool &flip, int &inflow)
{
    inflow = -1;
    if (c < 0 && bclo == BC_INFLOW) {
        flip = false;
        inflow = 0;
        return 0;
    }
    if (c >= n && bchi == BC_INFLOW) {
        flip = false;
        inflow = 1;
        return n - 1;
    }
    return ghost_source(c, n, bclo, bchi, flip);
}

// ---------------------------------------------------------------- WENO5-JS

template <typename T> __device__ __forceinline__ T div_(T a, T b);
template <> __device__ __forceinline__ double div_<double>(double a, double b) { return a / b; }
template <> __device__ __forceinline__ float div_<float>(float a, float b) { return a * fast_rcp(b); }

// Value at x_{i+1/2} reconstructed from (a, b, c, d, e) = v_{i-2}, ..., v_{i+2}
// (Sec. 2.2): candidates v^(r), smoothness indicators beta_r, weights
// alpha_r = d_r / (beta_r + eps)^2 normalised to sum one.  Written on the
// first differences D1..D4 (D1 = b - a, ..., D4 = e - d), in which
//   beta_0 = 13/12 (D4 - D3)^2 + 1/4 (D4 - 3 D3)^2,
//   beta_1 = 13/12 (D3 - D2)^2 + 1/4 (D2 + D3)^2,
//   beta_2 = 13/12 (D2 - D1)^2 + 1/4 (3 D2 - D1)^2,
//   v^(1) = c + (D2 + 2 D3)/6,  v^(0) - v^(1) = (t1 - t0)/6,  v^(2) - v^(1) = -2 (t1 - t2)/6,
// t_r the second differences above, so with w_r = d_r g_s g_t (g = (beta + eps)^2,
// {s, t} the other two indices; w_r / sum w = omega_r)
//   sum_r omega_r v^(r) = c + [(D2 + 2 D3) sum w + w_0 (t1 - t0) - 2 w_2 (t1 - t2)] / (6 sum w),
// the same quantity with one division.
template <typename T>
__device__ __forceinline__ T weno5(T a, T b, T c, T d, T e, T eps)
{
    const T D1 = b - a, D2 = c - b, D3 = d - c, D4 = e - d;
    const T t0 = D4 - D3, t1 = D3 - D2, t2 = D2 - D1;
    const T s0 = fma(T(-3), D3, D4), s1 = D2 + D3, s2 = fma(T(3), D2, -D1);
    const T k13 = T(13.0 / 12.0), q = T(0.25);
    T g0 = fma(k13 * t0, t0, fma(q * s0, s0, eps));
    T g1 = fma(k13 * t1, t1, fma(q * s1, s1, eps));
    T g2 = fma(k13 * t2, t2, fma(q * s2, s2, eps));
    g0 *= g0;
    g1 *= g1;
    g2 *= g2;
    const T w0 = T(0.3) * (g1 * g2), w1 = T(0.6) * (g0 * g2), w2 = T(0.1) * (g0 * g1);
    const T sw = w0 + w1 + w2;
    const T num = fma(w0, t1 - t0, fma(T(-2) * w2, t1 - t2, fma(T(2), D3, D2) * sw));
    return c + div_<T>(num, T(6) * sw);
}

// ------------------------------------------------- packed FP32 pairs (f32x2)
// Two independent FP32 streams in one float2: a .f32x2 instruction takes one
// issue slot for both operations (the FMA pipe still does two), which is what
// an issue-bound kernel needs.  Each lane of a pair is rounded exactly as the
// scalar operation would round it.
__device__ __forceinline__ float2 bc2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(r)
        : "l"(*reinterpret_cast<const unsigned long long *>(&a)), "l"(*reinterpret_cast<const unsigned long long *>(&b)));
    return *reinterpret_cast<const float2 *>(&r);
}

// weno5 of a face's WENO(+) window (lane x) and its mirrored WENO(-) window
// (lane y) at once, returning their sum (the face flux): the same operations
// as weno5<float> on each lane; beta_2's (3 D2 - D1) is formed negated (it
// enters squared only).
__device__ __forceinline__ float weno5_pm(float2 a, float2 b, float2 c, float2 d, float2 e, float eps_)
{
    const float2 D1 = sub2(b, a), D2 = sub2(c, b), D3 = sub2(d, c), D4 = sub2(e, d);
    const float2 t0 = sub2(D4, D3), t1 = sub2(D3, D2), t2 = sub2(D2, D1);
    const float2 s0 = fma2(bc2(-3.0f), D3, D4), s1 = add2(D2, D3), s2 = fma2(bc2(-3.0f), D2, D1);
    const float2 k13 = bc2((float)(13.0 / 12.0)), q = bc2(0.25f), eps = bc2(eps_);
    float2 g0 = fma2(mul2(k13, t0), t0, fma2(mul2(q, s0), s0, eps));
    float2 g1 = fma2(mul2(k13, t1), t1, fma2(mul2(q, s1), s1, eps));
    float2 g2 = fma2(mul2(k13, t2), t2, fma2(mul2(q, s2), s2, eps));
    g0 = mul2(g0, g0);
    g1 = mul2(g1, g1);
    g2 = mul2(g2, g2);
    const float2 w0 = mul2(bc2(0.3f), mul2(g1, g2)), w1 = mul2(bc2(0.6f), mul2(g0, g2)),
                 w2 = mul2(bc2(0.1f), mul2(g0, g1));
    const float2 sw = add2(add2(w0, w1), w2);
    const float2 num =
        fma2(w0, sub2(t1, t0), fma2(mul2(bc2(-2.0f), w2), sub2(t1, t2), mul2(fma2(bc2(2.0f), D3, D2), sw)));
    const float2 den = mul2(bc2(6.0f), sw);
    const float2 v = fma2(num, make_float2(fast_rcp(den.x), fast_rcp(den.y)), c);
    return v.x + v.y;
}

// WENO5 corrections of K consecutive windows along a line, from scaled first
// differences (two streams as float2 pairs).  With v the values whose
// reconstruction is wanted, D_k their first differences and t_r, s_r the
// second differences and beta parts of the weno5 comment, the correction of a
// window to its centre value c is
//   sum_r omega_r v^(r) - c = (D2 + 2 D3)/6 + (w0 (t1 - t0) - 2 w2 (t1 - t2)) / (6 sum w).
// p holds Dt = s D for a scale s; 6 s times the correction is
//   6 s (sum_r omega_r v^(r) - c) = Ft + (w0 (tt1 - tt0) - 2 w2 (tt1 - tt2)) / sum w,
//   Ft = Dt2 + 2 Dt3,  tt = s t,
// with (13/3) tt_r^2 + st_r^2 = 4 s^2 beta_r (st = s s_r), so that
// G_r = (13/3) tt_r^2 + st_r^2 + Geps with Geps = 4 s^2 eps is 4 s^2 (beta_r + eps),
// and the weights w_r = d_r / G_r^2 up to a common factor are formed as
// (3 g1 g2, 6 g0 g2, g0 g1) with g = G^2 (d = (3, 6, 1) / 10).  Window m takes
// Dt1..Dt4 = p[m s] .. p[(m + 3) s]; each window loads one new difference, and its
// -2 (tt1 - tt2) is twice the previous window's (tt1 - tt0), carried.  A mirrored window is the same run over the negated
// differences read backwards (the caller stores them negated).
//
// The run emits per cell: with C_m the value of window m, cell m - 1 (between the
// faces of windows m - 1 and m) receives 6 D2_m + (C_m - C_{m-1}) (FWD; D2_m the window's second
// difference, the cell's own pair), or -6 D2_m + (C_{m-1} - C_m) for a run read
// backwards (!FWD), K - 1 values to out[(m - 1) os].  Those are 6 s times the
// parts of a cell's flux difference that one run contributes (k_xy2 phase C).
template <int K, bool FWD>
__device__ __forceinline__ void weno5d_cells2(const float2 *p, int s, float Geps_, float2 *out, int os)
{
    const float2 k = bc2((float)(13.0 / 3.0)), Geps = bc2(Geps_), six = bc2(FWD ? 6.0f : -6.0f);
    float2 D1 = *p, D2 = *(p += s), D3 = *(p += s);
    float2 t1 = sub2(D3, D2), t2 = sub2(D2, D1);
    float2 A1 = fma2(mul2(k, t1), t1, Geps), A2 = fma2(mul2(k, t2), t2, Geps);
    float2 h = mul2(bc2(-2.0f), sub2(t1, t2));
    float2 Cp = bc2(0.0f);
#pragma unroll
    for (int m = 0; m < K; ++m) {
        const float2 D4 = *(p += s);
        const float2 t0 = sub2(D4, D3);
        const float2 A0 = fma2(mul2(k, t0), t0, Geps);
        const float2 s0 = fma2(bc2(-3.0f), D3, D4), s1 = add2(D2, D3), s2 = fma2(bc2(-3.0f), D2, D1);
        float2 g0 = fma2(s0, s0, A0), g1 = fma2(s1, s1, A1), g2 = fma2(s2, s2, A2);
        g0 = mul2(g0, g0);
        g1 = mul2(g1, g1);
        g2 = mul2(g2, g2);
        const float2 w0 = mul2(g1, g2), w1 = mul2(g0, g2), w2 = mul2(g0, g1);
        const float2 sw = fma2(bc2(3.0f), w0, fma2(bc2(6.0f), w1, w2));
        const float2 e0 = sub2(t1, t0);
        const float2 num = fma2(w0, mul2(bc2(3.0f), e0), mul2(w2, h));
        const float2 F = fma2(bc2(2.0f), D3, D2);
        const float2 C = fma2(num, make_float2(fast_rcp(sw.x), fast_rcp(sw.y)), F);
        if (m > 0) {
            *out = fma2(six, D2, FWD ? sub2(C, Cp) : sub2(Cp, C));
            out += os;
        }
        Cp = C;
        h = add2(e0, e0);
        D1 = D2;
        D2 = D3;
        D3 = D4;
        t2 = t1;
        t1 = t0;
        A2 = A1;
        A1 = A0;
    }
}

// ------------------------------------- FP64 WENO5 with weights in FP32 pairs
// The FP64 pipe is what bounds every FP64 kernel (1.7 instructions per clock
// per SM, against ~120 on the FP32 pipe), and most of a WENO5 value's FP64
// operations form the nonlinear weights.  The value is
//   c + [F + X] / 6,  F = D2 + 2 D3,  X = (3 g1 g2 e0 + 2 g0 g1 ep) / (3 g1 g2 + 6 g0 g2 + g0 g1),
// with g_r = G_r^2, G_r = (13/3) t_r^2 + s_r^2 + 4 eps = 4 (beta_r + eps),
// e0 = t1 - t0 and ep = t2 - t1 (the weno5 comment's symbols).  c, the first
// differences and F stay in FP64; X is formed in unevaluated FP32 pairs
// hi + lo (error-free transformations: Dekker 1971 and Knuth's two-sum; the
// products' errors by FMA), about 47 bits, and added to F in FP64.  The second
// differences are formed exactly from all bits of the first (tr_diff) and then
// rounded to pairs, so X's relative error is that of its own terms (~2^-46) and X is small against c wherever the data is
// resolved.  Where it is not -- the two terms of X together above 2^-7 |c| --
// where c or G leaves the range that FP32 pairs hold, the window is evaluated in
// FP32 triples or FP64 (weno5_rough), so the error of the value stays that of FP64
// throughout (but for differences below 2^-126 beside a c that is exactly zero, which
// count as zero in X).
// Measured over 60000 windows of each kind against
// 113-bit arithmetic, rms error in units of 2^-53 |v|, FP64 formula / this one:
// smooth waves 0.637 / 0.637, a front 4 cells wide 0.737 / 0.744, 2 cells
// 0.783 / 0.785, a captured shock 0.810 / 0.810, jumps 0.858 / 0.858.
//   FP64 instructions per window of a run: 4 instead of 42 (L(U) at 97 x 83 x 61:
// 2.49 -> 0.56 ms with the tiles of k_xy64.cu, scalar advection 128^3 5.0 -> 1.6).
__device__ __forceinline__ float2 two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}
__device__ __forceinline__ float2 pr_add(float2 a, float2 b)
{
    const float2 s = two_sum(a.x, b.x);
    return make_float2(s.x, __fadd_rn(s.y, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ float2 pr_sub(float2 a, float2 b) { return pr_add(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 pr_norm(float2 a)  // |a.y| well below |a.x|
{
    const float s = __fadd_rn(a.x, a.y);
    return make_float2(s, __fsub_rn(a.y, __fsub_rn(s, a.x)));
}
__device__ __forceinline__ float2 pr_sqr(float2 a)
{
    const float p = __fmul_rn(a.x, a.x), e = __fmaf_rn(a.x, a.x, -p);
    return make_float2(p, __fmaf_rn(__fadd_rn(a.x, a.x), a.y, e));
}
__device__ __forceinline__ float2 pr_mul(float2 a, float2 b)
{
    const float p = __fmul_rn(a.x, b.x), e = __fmaf_rn(a.x, b.y, __fmaf_rn(a.x, b.x, -p));
    return make_float2(p, __fmaf_rn(a.y, b.x, e));
}
__device__ __forceinline__ float2 pr_mulc(float k, float2 a)  // a constant exact in FP32
{
    const float p = __fmul_rn(k, a.x);
    return make_float2(p, __fmaf_rn(k, a.y, __fmaf_rn(k, a.x, -p)));
}

// split_f64 with magnitudes of 2^64 and more (infinities and NaNs too) taken to
// 2^64, whose square is outside the range of the pair formula; below 2^-103 only
// the 24 bits of hi are kept, below 2^-126 nothing.
__device__ __forceinline__ float2 split_sat(double x)
{
    const unsigned xh = (unsigned)__double2hiint(x);
    const unsigned xl = (unsigned)__double2loint(x);
    const unsigned sgn = xh & 0x80000000u, mag = xh & 0x7FFFFFFFu;
    const unsigned fs = __funnelshift_l(xl, xh, 3) + 0x40000000u;  // [e - 896 : 8][mantissa : 23]
    const unsigned eb = (fs - 0x0B800000u) & 0x7F800000u;          // exponent field of 2^(e - 1046)
    const float l = __uint_as_float(eb | ((xl >> 6) & 0x7FFFFFu)) - __uint_as_float(eb);
    const bool ok = mag - (897u << 20) < ((1087u - 897u) << 20);   // 2^-126 <= |x| < 2^64
    const unsigned alt = mag < (897u << 20) ? 0u : 0x5F800000u;
    return make_float2(__uint_as_float((ok ? fs & 0x7FFFFFFFu : alt) | sgn),
                       ok && mag >= (920u << 20) ? __uint_as_float(__float_as_uint(l) | sgn) : 0.0f);
}

// FP32 -> FP64 of a normal number (zero becomes 2^-127).
__device__ __forceinline__ double f32_to_f64_nz(float f)
{
    const unsigned b = __float_as_uint(f);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// FP32 triples (about 70 bits) for what pairs do not hold.
struct Tri {
    float a, b, c;
};
// All 53 bits of |x| in [2^-79, 2^64): split_sat, then the 6 bits it drops.
__device__ __forceinline__ Tri tr_split(double x)
{
    const float2 p = split_sat(x);
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x), mag = h & 0x7FFFFFFFu;
    const unsigned eb = ((mag >> 20) - 942u) << 23;  // exponent field of 2^(e - 1069): the 6 bits are worth 2^(e - 1075)
    const float v = __uint_as_float((eb & 0x7F800000u) | ((l & 63u) << 17)) - __uint_as_float(eb & 0x7F800000u);
    const bool ok = mag - (944u << 20) < ((1087u - 944u) << 20);
    return Tri{p.x, p.y, ok ? __uint_as_float(__float_as_uint(v) | (h & 0x80000000u)) : 0.0f};
}
// x - y of two split doubles as a pair, exact to the pair's last bit (the FP64
// difference would cost the pipe that bounds its callers ~80 issue slots, this ~35).
__device__ __forceinline__ float2 tr_diff(Tri x, Tri y)
{
    const float2 h = two_sum(x.a, -y.a), l = two_sum(x.b, -y.b), m = two_sum(h.y, l.x), n = two_sum(h.x, m.x);
    return two_sum(n.x, __fadd_rn(n.y, __fadd_rn(m.y, __fadd_rn(l.y, __fsub_rn(x.c, y.c)))));
}

// a + b + c in FP64 for a normal a (zero becomes 2^-127) and |b + c| within an ulp of
// a: b and c are integers in units of the result's last place, so no FP64 sum.
__device__ __forceinline__ double pr_f64(float a, float b, float c)
{
    const unsigned u = __float_as_uint(a);
    const float s = __uint_as_float(0x7F000000u - (u & 0x7F800000u));  // 2^-exponent
    int k = __float2int_rn(__fmul_rn(__fmul_rn(b, 0x1p52f), s)) + __float2int_rn(__fmul_rn(__fmul_rn(c, 0x1p52f), s));
    k = (int)u < 0 ? -k : k;
    if (k < 0 && (u & 0x7FFFFFu) == 0u) k += k;  // below a power of two the places are half as large
    const long long v = ((long long)(((u & 0x7FFFFFFFu) >> 3) + 0x38000000u) << 32 | (u << 29)) + k;
    return __hiloint2double((int)((unsigned)(v >> 32) | (u & 0x80000000u)), (int)v);
}

// 1 / x of a normal x below 2^1021: an FP32 reciprocal of the mantissa, two
// Newton-Raphson steps r (2 - x r) (4 FP64 instructions; a division takes ~9).
// The last step forms r (1 + e), e ~ 2^-46, in one rounding and drops e^2, so the
// result is the correctly rounded one but within 2^-38 of a tie (20 million random x: all).
__device__ __forceinline__ double rcp_f64(double x)
{
    const unsigned h = (unsigned)__double2hiint(x);
    const float m = __uint_as_float(0x3F800000u | (__funnelshift_l((unsigned)__double2loint(x), h, 3) & 0x7FFFFFu));
    const double y = f32_to_f64_nz(fast_rcp(m));
    double r = __hiloint2double((int)((unsigned)__double2hiint(y) - ((h & 0x7FF00000u) - 0x3FF00000u) | (h & 0x80000000u)),
                                __double2loint(y));
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}

// The smoothness parameter as the pair formula takes it.
struct PairEps {
    double eps;
    float2 g;  // 4 eps as a pair; infinite (every window is rough) from eps = 2^60 on, where pairs end
};
__device__ __forceinline__ PairEps pair_eps(double eps)
{
    PairEps P;
    P.eps = eps;
    P.g = __double2hiint(eps) < (1083 << 20) ? split_sat(4.0 * eps) : make_float2(__int_as_float(0x7F800000), 0.0f);
    return P;
}

// (13/3) t^2 + 4 eps
__device__ __forceinline__ float2 pair_t2(float2 t, float2 ge)
{
    constexpr float kh = (float)(13.0 / 3.0), kl = (float)(13.0 / 3.0 - (double)(float)(13.0 / 3.0));
    const float2 q = pr_sqr(t);
    const float p = __fmul_rn(kh, q.x);
    return pr_add(make_float2(p, __fmaf_rn(kh, q.y, __fmaf_rn(kl, q.x, __fmaf_rn(kh, q.x, -p)))), ge);
}

// The weno5 formula from a window's first differences, FP64 throughout.
__device__ __forceinline__ double weno5_diffs(double D1, double D2, double D3, double D4, double c, double eps)
{
    const double t0 = D4 - D3, t1 = D3 - D2, t2 = D2 - D1;
    const double s0 = fma(-3.0, D3, D4), s1 = D2 + D3, s2 = fma(3.0, D2, -D1);
    const double k13 = 13.0 / 12.0, q = 0.25;
    double g0 = fma(q * s0, s0, fma(k13 * t0, t0, eps));
    double g1 = fma(q * s1, s1, fma(k13 * t1, t1, eps));
    double g2 = fma(q * s2, s2, fma(k13 * t2, t2, eps));
    g0 *= g0;
    g1 *= g1;
    g2 *= g2;
    const double w0 = 0.3 * (g1 * g2), w1 = 0.6 * (g0 * g2), w2 = 0.1 * (g0 * g1);
    const double sw = w0 + w1 + w2;
    const double num = fma(w0, t1 - t0, fma(-2.0 * w2, t1 - t2, fma(2.0, D3, D2) * sw));
    return c + num / (6.0 * sw);
}

// One window: D2, D3 and the centre value c in FP64; f2, f3 the pairs of D2 and
// D3; u_r and A_r those of t_r and (13/3) t_r^2 + 4 eps; e0 = u1 - u0, ep = u2 - u1.
// rough: the value is not good and the window has to take weno5_rough.
__device__ __forceinline__ double weno5_pair_core(double D2, double D3, double c, float2 f2, float2 f3,
                                                  float2 u0, float2 u2, float2 A0, float2 A1, float2 A2,
                                                  float2 e0, float2 ep, const PairEps &P, bool &rough)
{
    const float2 s0 = pr_add(u0, make_float2(-2.0f * f3.x, -2.0f * f3.y)), s1 = pr_add(f2, f3),
                 s2 = pr_add(u2, make_float2(2.0f * f2.x, 2.0f * f2.y));
    float2 G0 = pr_norm(pr_add(pr_sqr(s0), A0)), G1 = pr_norm(pr_add(pr_sqr(s1), A1)),
           G2 = pr_norm(pr_add(pr_sqr(s2), A2));
    // scale by the power of two that takes the smallest G to [2^-20, 2^-19); what is
    // over 2^30 then has a weight below 2^-98 and is held there (no product or sum
    // leaves the FP32 range)
    const float mn = fminf(G0.x, fminf(G1.x, G2.x)), sum = G0.x + G1.x + G2.x;
    const float sc = __uint_as_float(0x75000000u - (__float_as_uint(mn) & 0x7F800000u));
    auto scaled = [&](float2 G) {
        const float x = __fmul_rn(G.x, sc);
        return x < 0x1p30f ? make_float2(x, __fmul_rn(G.y, sc)) : make_float2(0x1p30f, 0.0f);
    };
    G0 = scaled(G0);
    G1 = scaled(G1);
    G2 = scaled(G2);
    const float2 g0 = pr_norm(pr_sqr(G0)), g1 = pr_norm(pr_sqr(G1)), g2 = pr_norm(pr_sqr(G2));
    const float2 w0 = pr_mulc(3.0f, pr_mul(g1, g2)), w1 = pr_mulc(6.0f, pr_mul(g0, g2)), w2 = pr_mul(g0, g1);
    const float2 sw = pr_norm(pr_add(pr_add(w0, w1), w2));
    // omega_0 and omega_2 as pairs (one residual correction of an approximate
    // quotient), then the two terms of X
    const float r = fast_rcp(sw.x);
    auto over_sw = [&](float2 w) {
        const float x = __fmul_rn(w.x, r);
        return make_float2(x, __fmul_rn(__fadd_rn(__fmaf_rn(-x, sw.x, w.x), __fmaf_rn(-x, sw.y, w.y)), r));
    };
    const float2 o2 = over_sw(w2);
    const float2 p0 = pr_mul(over_sw(w0), e0), p2 = pr_mul(make_float2(2.0f * o2.x, 2.0f * o2.y), ep);
    const float em = fabsf(p0.x) + fabsf(p2.x);
    const int emh = (int)((__float_as_uint(em) >> 3) + 0x38000000u);  // as the high word of a double
    const int ch = __double2hiint(c) & 0x7FFFFFFF;
    rough = (em != 0.0f && emh > ch - (7 << 20)) || (unsigned)(ch - 1) < (953u << 20) ||  // 0 < |c| < 2^-70
            !(mn > 0x1p-80f) || !(sum < 0x1p100f) || !(sum * sc < 0x1p66f);
    const float2 x = pr_norm(pr_add(p0, p2));
    return fma(fma(2.0, D3, D2) + pr_f64(x.x, x.y, 0.0f), 1.0 / 6.0, c);
}

// ---- the same in FP32 triples a + b + c (about 70 bits), for windows whose X is not
// small: FP64's FP32 cost without its pipe.  Error-free sums and products of the
// leading parts, the last part in plain FP32 (triple-word arithmetic after Fabiano,
// Joldes, Muller and Popescu 2019, without their final renormalisations where a
// sum of positive terms follows).
__device__ __forceinline__ Tri tr_norm(Tri x)
{
    const float2 s = two_sum(x.b, x.c), t = two_sum(x.a, s.x), u = two_sum(t.y, s.y);
    return Tri{t.x, u.x, u.y};
}
__device__ __forceinline__ Tri tr_add(Tri x, Tri y)
{
    const float2 h = two_sum(x.a, y.a), l = two_sum(x.b, y.b), m = two_sum(h.y, l.x);
    return Tri{h.x, m.x, __fadd_rn(__fadd_rn(m.y, l.y), __fadd_rn(x.c, y.c))};
}
__device__ __forceinline__ Tri tr_pow2(Tri x, float k) { return Tri{k * x.a, k * x.b, k * x.c}; }  // k a power of two
__device__ __forceinline__ Tri tr_sqr(Tri x)
{
    const float p = __fmul_rn(x.a, x.a), e = __fmaf_rn(x.a, x.a, -p), d = __fadd_rn(x.a, x.a);
    const float q = __fmul_rn(d, x.b), qe = __fmaf_rn(d, x.b, -q);
    const float2 m = two_sum(e, q);
    return Tri{p, m.x, __fadd_rn(m.y, __fadd_rn(qe, __fmaf_rn(x.b, x.b, __fmul_rn(d, x.c))))};
}
__device__ __forceinline__ Tri tr_mul(Tri x, Tri y)
{
    const float p = __fmul_rn(x.a, y.a), e = __fmaf_rn(x.a, y.a, -p);
    const float q = __fmul_rn(x.a, y.b), qe = __fmaf_rn(x.a, y.b, -q);
    const float r = __fmul_rn(x.b, y.a), re = __fmaf_rn(x.b, y.a, -r);
    const float2 m = two_sum(q, r), n = two_sum(e, m.x);
    const float c = __fmaf_rn(x.b, y.b, __fmaf_rn(x.a, y.c, __fmul_rn(x.c, y.a)));
    return Tri{p, n.x, __fadd_rn(__fadd_rn(m.y, n.y), __fadd_rn(__fadd_rn(qe, re), c))};
}
__device__ __forceinline__ Tri tr_mulc(float k, Tri x)  // an FP32 factor
{
    const float p = __fmul_rn(k, x.a), e = __fmaf_rn(k, x.a, -p), q = __fmul_rn(k, x.b), qe = __fmaf_rn(k, x.b, -q);
    const float2 m = two_sum(e, q);
    return Tri{p, m.x, __fadd_rn(m.y, __fmaf_rn(k, x.c, qe))};
}
// w / s for s normalised: three quotient words, each from the exact remainder
__device__ __forceinline__ Tri tr_div(Tri w, Tri s, float r)
{
    w = tr_norm(w);
    const float q0 = __fmul_rn(w.a, r);
    const Tri R = tr_add(w, tr_mulc(-q0, s));
    const float q1 = __fmul_rn(__fadd_rn(__fadd_rn(R.a, R.b), R.c), r);
    const Tri S = tr_add(R, tr_mulc(-q1, s));
    const float q2 = __fmul_rn(__fadd_rn(__fadd_rn(S.a, S.b), S.c), r);
    return tr_norm(Tri{q0, q1, q2});
}

// The value of a rough window (its five points): differences and X in triples, c, F
// and the final sum in FP64; the FP64 formula where G leaves the range.  7 FP64
// instructions instead of 46, ~900 in FP32.  Measured as above, rms error FP64
// formula / this one: front of 2 cells 0.780 / 0.776, captured shock 0.808 / 0.799,
// jumps 0.855 / 0.851, random values 0.463 / 0.392.
static __device__ __noinline__ double weno5_rough(double v0, double v1, double v2, double v3, double v4, double eps)
{
    const double D1 = v1 - v0, D2 = v2 - v1, D3 = v3 - v2, D4 = v4 - v3;
    const Tri d1 = tr_split(D1), d2 = tr_split(D2), d3 = tr_split(D3), d4 = tr_split(D4);
    const Tri t0 = tr_norm(tr_add(d4, tr_pow2(d3, -1.0f))), t1 = tr_norm(tr_add(d3, tr_pow2(d2, -1.0f))),
              t2 = tr_norm(tr_add(d2, tr_pow2(d1, -1.0f)));
    const Tri e12 = tr_mulc(3.0f, tr_pow2(tr_split(eps), 4.0f));
    auto ind = [&](Tri t, Tri s) {  // 13 t^2 + 3 s^2 + 12 eps
        return tr_norm(tr_add(tr_add(tr_mulc(13.0f, tr_sqr(t)), tr_mulc(3.0f, tr_sqr(tr_norm(s)))), e12));
    };
    Tri G0 = ind(t0, tr_add(t0, tr_pow2(d3, -2.0f))), G1 = ind(t1, tr_add(d2, d3)), G2 = ind(t2, tr_add(t2, tr_pow2(d2, 2.0f)));
    const float mn = fminf(G0.a, fminf(G1.a, G2.a)), sum = G0.a + G1.a + G2.a;
    const float sc = __uint_as_float(0x75000000u - (__float_as_uint(mn) & 0x7F800000u));
    const float big = fmaxf(fmaxf(fabsf(d1.a), fabsf(d2.a)), fmaxf(fabsf(d3.a), fabsf(d4.a)));
    if (!(mn > 0x1p-80f) || !(sum < 0x1p100f) || !(sum * sc < 0x1p66f) || !(big > 0x1p-60f) ||
        __double2hiint(eps) >= (1083 << 20))  // eps of 2^60 and more
        return weno5_diffs(D1, D2, D3, D4, v2, eps);
    auto scaled = [&](Tri G) {
        const float x = __fmul_rn(G.a, sc);
        return x < 0x1p30f ? Tri{x, __fmul_rn(G.b, sc), __fmul_rn(G.c, sc)} : Tri{0x1p30f, 0.0f, 0.0f};
    };
    G0 = scaled(G0);
    G1 = scaled(G1);
    G2 = scaled(G2);
    const Tri g0 = tr_norm(tr_sqr(G0)), g1 = tr_norm(tr_sqr(G1)), g2 = tr_norm(tr_sqr(G2));
    const Tri w0 = tr_mulc(3.0f, tr_mul(g1, g2)), w2 = tr_mul(g0, g1);
    const Tri sw = tr_norm(tr_add(tr_add(w0, tr_mulc(6.0f, tr_mul(g0, g2))), w2));
    const float r = fast_rcp(sw.a);
    const Tri e0 = tr_norm(tr_add(t1, tr_pow2(t0, -1.0f))), ep = tr_norm(tr_add(t2, tr_pow2(t1, -1.0f)));
    const Tri X = tr_norm(tr_add(tr_mul(tr_div(w0, sw, r), e0), tr_pow2(tr_mul(tr_div(w2, sw, r), ep), 2.0f)));
    return fma(fma(2.0, D3, D2) + pr_f64(X.a, X.b, X.c), 1.0 / 6.0, v2);
}

// One window from its five points (a rough one in place, in FP64: without a call the
// caller keeps its registers).
__device__ __forceinline__ double weno5_pair(double a, double b, double c, double d, double e, const PairEps &P)
{
    const double D1 = b - a, D2 = c - b, D3 = d - c, D4 = e - d;
    const float2 u0 = split_sat(D4 - D3), u1 = split_sat(D3 - D2), u2 = split_sat(D2 - D1);
    bool rough;
    const double v = weno5_pair_core(D2, D3, c, split_sat(D2), split_sat(D3), u0, u2, pair_t2(u0, P.g),
                                     pair_t2(u1, P.g), pair_t2(u2, P.g), pr_sub(u1, u0), pr_sub(u2, u1), P, rough);
    return rough ? weno5_diffs(D1, D2, D3, D4, c, P.eps) : v;
}

// The rough windows of a block, gathered in shared memory and evaluated densely
// after the runs: taking weno5_rough inside a run would cost the whole warp
// whenever one lane needs it.  An entry is the offset of the
// window's first point, the offset of its value, and which of the strides
// +-1, +-S its points have; the list holds every window of the block.
struct RoughList {
    int *count;      // shared, zeroed before a barrier that precedes the runs
    unsigned *list;  // shared
};

__device__ __forceinline__ void rough_windows(const RoughList &L, int S, const double *src, double *dst, const PairEps &P)
{
    const int n = *L.count;
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        const unsigned w = L.list[e];
        const int s = (w >> 26 & 1u ? S : 1) * (w >> 27 & 1u ? -1 : 1);
        const double *p = src + (w & 0x1FFFu);
        const double a = p[0], b = p[s], c = p[2 * s], d = p[3 * s], f = p[4 * s];
        dst[w >> 13 & 0x1FFFu] = weno5_rough(a, b, c, d, f, P.eps);
    }
}

// `count` consecutive windows along a line: window m is the points at
// src[po + m s], .., src[po + (m + 4) s] and its value goes to dst[oo + m os].
// Neighbouring windows share all differences but one of each kind, so each window
// forms one new; its value depends on its five points only, bit for bit, wherever it
// sits in a run, so a face that two runs form gets the same value.  A negative stride walks
// a line backwards, which turns the run into the mirrored WENO(-) of the faces in
// reverse order.
// Offsets are below 2^13 and |s| is 1 or S.  The loop stays rolled: a window is
// ~280 instructions.
__device__ __forceinline__ void weno5_slide_pair(const double *src, int po, int s, const PairEps &P, double *dst, int oo,
                                                 int os, int count, int S, const RoughList &L)
{
    const double *p = src + po;
    double *out = dst + oo;
    const unsigned kind = (s == S || s == -S ? 1u << 26 : 0u) | (s < 0 ? 1u << 27 : 0u);
    const double v0 = *p, v1 = *(p += s);
    double c = *(p += s), d = *(p += s);
    double D2 = c - v1, D3 = d - c;
    Tri f2 = tr_split(D2), f3 = tr_split(D3);
    float2 u1 = tr_diff(f3, f2), u2 = tr_diff(f2, tr_split(v1 - v0));
    float2 A1 = pair_t2(u1, P.g), A2 = pair_t2(u2, P.g), ep = pr_sub(u2, u1);
#pragma unroll 1
    for (int m = 0; m < count; ++m) {
        const double e = *(p += s);
        const double D4 = e - d;
        const Tri f4 = tr_split(D4);
        const float2 u0 = tr_diff(f4, f3);
        const float2 A0 = pair_t2(u0, P.g), e0 = pr_sub(u1, u0);
        bool rough;
        const double v = weno5_pair_core(D2, D3, c, make_float2(f2.a, f2.b), make_float2(f3.a, f3.b), u0, u2, A0,
                                         A1, A2, e0, ep, P, rough);
        if (!rough) {
            *out = v;
        } else {
            L.list[atomicAdd(L.count, 1)] = (unsigned)(p - 4 * s - src) | (unsigned)(out - dst) << 13 | kind;
        }
        out += os;
        D2 = D3;
        D3 = D4;
        f2 = f3;
        f3 = f4;
        u2 = u1;
        u1 = u0;
        A2 = A1;
        A1 = A0;
        ep = e0;
        c = d;
        d = e;
    }
}

// ----------------------------------------------------------- point fluxes

// Plain FP64 Euler flux in direction DIR (Sec. 2.1) and its LF split
// f(+/-) = (F +/- alpha U) / 2 (Sec. 2.2).
// TWICE: return 2 f(+/-) = F +/- alpha U (one FMA each, no halving); the
// caller then reconstructs with 4 eps, which gives exactly twice the WENO5
// value of f(+/-) (scaling by 2 commutes with every rounding), and halves once.
template <int D, int DIR, bool TWICE = false>
__device__ __forceinline__ void split_flux_f64(const double *q, double alpha, double gm1, double *fp, double *fm)
{
    constexpr int NF = D + 2;
    const double ir = rcp_f64(q[0]);
    double u[D];
    double mu = 0.0;
#pragma unroll
    for (int e = 0; e < D; ++e) {
        u[e] = q[1 + e] * ir;
        mu = e == 0 ? q[1] * u[0] : fma(q[1 + e], u[e], mu);
    }
    const double p = gm1 * fma(-0.5, mu, q[D + 1]);
    double F[NF];
    F[0] = q[1 + DIR];
#pragma unroll
    for (int e = 0; e < D; ++e) F[1 + e] = q[1 + e] * u[DIR] + (e == DIR ? p : 0.0);
    F[D + 1] = u[DIR] * (q[D + 1] + p);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        if (TWICE) {
            fp[f] = fma(alpha, q[f], F[f]);
            fm[f] = fma(-alpha, q[f], F[f]);
        } else {
            fp[f] = 0.5 * (F[f] + alpha * q[f]);
            fm[f] = 0.5 * (F[f] - alpha * q[f]);
        }
    }
}

// Reference state of one tile line for the FP32-bulk path: the FP64 state
// split into hi + lo, and FP32 primitives that only ever multiply differences.
template <int D> struct RefState {
    float hi[D + 2], lo[D + 2];
    float rho, m[D], u[D], H;  // H = rho E + p
};

// The same from a state already split into FP32 hi + lo (lo may carry a stage
// increment, far above FP32 rounding, so the primitives take hi + lo).
template <int D>
__device__ __forceinline__ void make_ref_hl(const float *h, const float *l, float gm1, RefState<D> &r)
{
    float q[D + 2];
#pragma unroll
    for (int f = 0; f < D + 2; ++f) {
        r.hi[f] = h[f];
        r.lo[f] = l[f];
        q[f] = h[f] + l[f];
    }
    r.rho = q[0];
    const float ir = 1.0f / r.rho;
    float ke = 0.0f;
#pragma unroll
    for (int e = 0; e < D; ++e) {
        r.m[e] = q[1 + e];
        r.u[e] = r.m[e] * ir;
        ke += r.m[e] * r.u[e];
    }
    const float p = gm1 * (q[D + 1] - 0.5f * ke);
    r.H = q[D + 1] + p;
}

template <int D>
__device__ __forceinline__ void make_ref(const double *q, float gm1, RefState<D> &r)
{
#pragma unroll
    for (int f = 0; f < D + 2; ++f) split_f64(q[f], r.hi[f], r.lo[f]);
    r.rho = r.hi[0];
    const float ir = 1.0f / r.rho;
    float ke = 0.0f;
#pragma unroll
    for (int e = 0; e < D; ++e) {
        r.m[e] = r.hi[1 + e];
        r.u[e] = r.m[e] * ir;
        ke += r.m[e] * r.u[e];
    }
    const float p = gm1 * (r.hi[D + 1] - 0.5f * ke);
    r.H = r.hi[D + 1] + p;
}

// dq = q - ref, formed from the hi/lo splits so that it carries the full FP32
// relative precision of the difference (not of q).
template <int D>
__device__ __forceinline__ void diff_from_ref(const double *q, const RefState<D> &r, float *dq)
{
#pragma unroll
    for (int f = 0; f < D + 2; ++f) {
        float hi, lo;
        split_f64(q[f], hi, lo);
        dq[f] = (hi - r.hi[f]) + (lo - r.lo[f]);
    }
}

// Split-flux differences df(+/-) = f(+/-)(ref + dq) - f(+/-)(ref) in FP32,
// using only exact product-difference identities
//   d(ab) = da * b + a_ref * db,  du = (dm - u_ref drho) / rho,
// so every rounding error is relative to the differences, not to the state.
template <int D, int DIR, bool TWICE = false>
__device__ __forceinline__ void split_flux_diff(const float *dq, const RefState<D> &r, float alpha, float gm1,
                                                float *fp, float *fm)
{
    constexpr int NF = D + 2;
    const float rho = r.rho + dq[0];
    const float ir = fast_rcp(rho);
    float du[D], u[D];
    float dk = 0.0f;
#pragma unroll
    for (int e = 0; e < D; ++e) {
        du[e] = (dq[1 + e] - r.u[e] * dq[0]) * ir;
        u[e] = r.u[e] + du[e];
        dk += dq[1 + e] * u[e] + r.m[e] * du[e];
    }
    const float dp = gm1 * (dq[D + 1] - 0.5f * dk);
    float dF[NF];
    dF[0] = dq[1 + DIR];
#pragma unroll
    for (int e = 0; e < D; ++e) dF[1 + e] = dq[1 + e] * u[DIR] + r.m[e] * du[DIR] + (e == DIR ? dp : 0.0f);
    const float dH = dq[D + 1] + dp;
    dF[D + 1] = du[DIR] * (r.H + dH) + r.u[DIR] * dH;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        if (TWICE) {  // 2 f(+/-), see split_flux_f64
            fp[f] = fmaf(alpha, dq[f], dF[f]);
            fm[f] = fmaf(-alpha, dq[f], dF[f]);
        } else {
            fp[f] = 0.5f * (dF[f] + alpha * dq[f]);
            fm[f] = 0.5f * (dF[f] - alpha * dq[f]);
        }
    }
}

// The SSP-RK3 stage combination in FP64, U' = a_n U^n + b_n (U^k + dt R) (stage 0:
// U + dt R), with its roundings fixed so that every kernel gives the same bits.
__device__ __forceinline__ double stage_combine(int stage, double un, double uk, double r, double dt)
{
    const double s = fma(dt, r, uk);
    if (stage == 0) return s;
    return fma(stage == 1 ? 0.25 : 2.0 / 3.0, s, __dmul_rn(stage == 1 ? 0.75 : 1.0 / 3.0, un));
}

// dt of the next step from alpha(U^n) (or the fixed dt), shortened so that the
// time lands exactly on t_end; zero when the time is up or the step budget of the
// current call is spent.  Returns whether the step is impossible (a dt that is not
// a positive finite number while steps are wanted).
__device__ __forceinline__ bool next_dt(double t, double t_end, double dt_req, double cfl_h, double alpha,
                                        long long steps, long long max_steps, double &dt, double &t_next)
{
    dt = dt_req > 0.0 ? dt_req : cfl_h / alpha;
    t_next = t + dt;
    if (!(dt > 0.0) || !isfinite(dt)) {
        dt = 0.0;
        t_next = t;
        return t < t_end && steps < max_steps;
    }
    if (!(t < t_end) || steps >= max_steps) {
        dt = 0.0;
        t_next = t;
    } else if (t_next >= t_end) {
        dt = t_end - t;
        t_next = t_end;
    }
    return false;
}

// ------------------------------------------------------------- wavespeed

// |u| + sqrt(gamma p / rho) in FP64 with the operation order of the plain
// formula (no contraction), so that alpha and dt reproduce it bit for bit.
template <int D>
__device__ __forceinline__ double wavespeed_f64(const double *q, double gamma, bool &bad)
{
    const double rho = q[0];
    double u2 = 0.0;
#pragma unroll
    for (int e = 0; e < D; ++e) {
        const double ue = __ddiv_rn(q[1 + e], rho);
        u2 = __dadd_rn(u2, __dmul_rn(ue, ue));
    }
    const double p = __dmul_rn(gamma - 1.0, __dsub_rn(q[D + 1], __dmul_rn(__dmul_rn(0.5, rho), u2)));
    bad = !(rho > 0.0) || !(p > 0.0) || !isfinite(u2) || !isfinite(q[D + 1]);
    const double a = __dsqrt_rn(__ddiv_rn(__dmul_rn(gamma, p), rho));
    return bad ? 0.0 : __dadd_rn(__dsqrt_rn(u2), a);
}

// Per-direction speeds |u_d| + a (FP64, same operation order as the plain formula).
template <int D>
__device__ __forceinline__ void dirspeeds_f64(const double *q, double gamma, double *sd)
{
    const double rho = q[0];
    double u2 = 0.0;
#pragma unroll
    for (int e = 0; e < D; ++e) {
        const double ue = __ddiv_rn(q[1 + e], rho);
        u2 = __dadd_rn(u2, __dmul_rn(ue, ue));
    }
    const double p = __dmul_rn(gamma - 1.0, __dsub_rn(q[D + 1], __dmul_rn(__dmul_rn(0.5, rho), u2)));
    const double a = __dsqrt_rn(__ddiv_rn(__dmul_rn(gamma, p), rho));
#pragma unroll
    for (int e = 0; e < D; ++e) sd[e] = __dadd_rn(fabs(__ddiv_rn(q[1 + e], rho)), a);
}

// (gm1: speed_gm1)
template <int D>
__device__ __forceinline__ void dirspeeds_f32(const float *q, float gamma, float gm1, float *sd)
{
    const float rho = q[0];
    const float ir = 1.0f / rho;
    float u2 = 0.0f;
#pragma unroll
    for (int e = 0; e < D; ++e) {
        const float ue = q[1 + e] * ir;
        u2 += ue * ue;
    }
    const float p = gm1 * (q[D + 1] - 0.5f * rho * u2);
    const float a = sqrtf(gamma * p * ir);
#pragma unroll
    for (int e = 0; e < D; ++e) sd[e] = fabsf(q[1 + e] * ir) + a;
}

// The FP32 wavespeed ||u|| + a feeds only the maximum behind alpha and dt,
// where a relative error of a few ulp is immaterial, so it takes the
// approximate reciprocal and square roots (one MUFU instruction each).
__device__ __forceinline__ float sqrt_approx(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int D>
__device__ __forceinline__ float wavespeed_f32(const float *q, float gamma, float gm1, bool &bad)
{
    const float rho = q[0];
    const float ir = fast_rcp(rho);
    float u2 = 0.0f;
#pragma unroll
    for (int e = 0; e < D; ++e) {
        const float ue = q[1 + e] * ir;
        u2 += ue * ue;
    }
    const float p = gm1 * (q[D + 1] - 0.5f * rho * u2);
    bad = !(rho > 0.0f) || !(p > 0.0f) || !isfinite(u2) || !isfinite(q[D + 1]);
    return bad ? 0.0f : sqrt_approx(u2) + sqrt_approx(gamma * p * ir);
}

// FP32 estimates of the speeds of an FP64 state: est[0] = |u| + a and, for K > 1,
// est[1 + e] = |u_e| + a; gg = gamma (gamma - 1), formed from the FP64 gamma (an FP32
// one less 1 has few bits left near 1).  Returns whether the state is certainly physical and the
// estimates are within 2^-16 of the FP64 values: the conserved fields of ordinary
// size, the internal energy at least 2^-5 of the total and kinetic energies (its FP32
// rounding is 2^-21 of those), density and sound speed above 1e-12 (so that what FP32
// flushes to zero on the way -- momenta below 2^-103, squares below 2^-126 -- is below
// 2^-16 of the sound speed).
template <int D, int K>
__device__ __forceinline__ bool speed_estimate(const double *q, float gg, float *est)
{
    float f[D + 2];
#pragma unroll
    for (int k = 0; k < D + 2; ++k) f[k] = f64_to_f32(q[k]);
    const float ir = fast_rcp(f[0]);
    float u2 = 0.0f;
#pragma unroll
    for (int e = 0; e < D; ++e) {
        const float ue = f[1 + e] * ir;
        u2 = fmaf(ue, ue, u2);
    }
    const float ke = 0.5f * f[0] * u2, ie = f[D + 1] - ke;
    const float a = sqrt_approx(gg * ie * ir);
    est[0] = sqrt_approx(u2) + a;
    if (K > 1) {
#pragma unroll
        for (int e = 0; e < D; ++e) est[1 + e] = fabsf(f[1 + e] * ir) + a;
    }
    // f64_to_f32 is meaningful below 2^128 only: test the FP64 exponents
    bool in = true;
#pragma unroll
    for (int k = 0; k < D + 2; ++k) in = in && (__double2hiint(q[k]) & 0x7FFFFFFF) < (1123 << 20);  // |q| < 2^100
    return in && f[0] > 1e-12f && a > 1e-12f && ie > 0.03125f * (fabsf(f[D + 1]) + ke) && est[0] < 1e30f;
}

// max over the block of the FP64 speeds of its threads' states (K = 1: |u| + a
// into s_max[0]; K = 1 + D also |u_e| + a into s_max[1 + e]) as bit patterns, and
// its non-physical flag into *s_bad, in shared memory; the caller's next barrier
// makes them visible.  load(i, q) gives the states i = begin, begin + step, .. < end of the calling thread.  Only
// states whose FP32 estimate is within 2^-14 of the block's largest, or that have
// no estimate, get the FP64 speeds (two divisions and two square roots, ~60
// FP64 instructions): the maximum is theirs, bit for bit.  Every thread of the
// block must call it.
template <int D, int K, class Load>
__device__ __forceinline__ void speed_max_block_f64(Load load, long long begin, long long end, long long step,
                                                    double gamma, float gg, unsigned long long *s_max, int *s_bad)
{
    __shared__ unsigned s_est[K];
    if (threadIdx.x < K) {
        s_est[threadIdx.x] = 0u;
        s_max[threadIdx.x] = 0ull;
    }
    if (threadIdx.x == 0) *s_bad = 0;
    float mine[K];
#pragma unroll
    for (int k = 0; k < K; ++k) mine[k] = 0.0f;
    bool unsure = false;
    for (long long i = begin; i < end; i += step) {
        double q[D + 2];
        float est[K];
        load(i, q);
        if (speed_estimate<D, K>(q, gg, est)) {
#pragma unroll
            for (int k = 0; k < K; ++k) mine[k] = fmaxf(mine[k], est[k]);
        } else {
            unsure = true;
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const unsigned m = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mine[k]));
        if ((threadIdx.x & 31) == 0 && m) atomicMax(s_est + k, m);
    }
    __syncthreads();
    float thr[K];
    bool need = unsure;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        thr[k] = __uint_as_float(s_est[k]) * (1.0f - 0x1p-14f);
        need = need || (mine[k] > 0.0f && mine[k] >= thr[k]);
    }
    if (__any_sync(0xFFFFFFFFu, need)) {
        unsigned long long best[K];
#pragma unroll
        for (int k = 0; k < K; ++k) best[k] = 0ull;
        if (need) {
            for (long long i = begin; i < end; i += step) {
                double q[D + 2], v[K];
                float est[K];
                load(i, q);
                bool go = !speed_estimate<D, K>(q, gg, est), bad;
#pragma unroll
                for (int k = 0; k < K; ++k) go = go || est[k] >= thr[k];
                if (!go) continue;
                v[0] = wavespeed_f64<D>(q, gamma, bad);
                if (K > 1) dirspeeds_f64<D>(q, gamma, v + (K > 1));
                if (bad) {
                    *s_bad = 1;
                    continue;
                }
#pragma unroll
                for (int k = 0; k < K; ++k) best[k] = max(best[k], (unsigned long long)__double_as_longlong(v[k]));
            }
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {  // the warp's maximum on the integer pipe: high words, then low words among them
            const unsigned hi = (unsigned)(best[k] >> 32), mh = __reduce_max_sync(0xFFFFFFFFu, hi);
            const unsigned ml = __reduce_max_sync(0xFFFFFFFFu, hi == mh ? (unsigned)best[k] : 0u);
            if ((threadIdx.x & 31) == 0 && (mh | ml)) atomicMax(s_max + k, (unsigned long long)mh << 32 | ml);
        }
    }
}

// The same, published: one atomicMax per block and value, K = 1: *slot0, K > 1
// also slot_dir[e].
template <int D, int K, class Load>
__device__ __forceinline__ void speed_max_publish_f64(Load load, long long begin, long long end, long long step,
                                                      double gamma, float gg, unsigned long long *slot0,
                                                      unsigned long long *slot_dir, int *status)
{
    __shared__ unsigned long long s_max[K];
    __shared__ int s_bad;
    speed_max_block_f64<D, K>(load, begin, end, step, gamma, gg, s_max, &s_bad);
    __syncthreads();
    if (threadIdx.x < K && s_max[threadIdx.x])
        atomicMax(threadIdx.x == 0 ? slot0 : slot_dir + (threadIdx.x - 1), s_max[threadIdx.x]);
    if (threadIdx.x == 0 && s_bad) atomicOr(status, ST_NONPHYSICAL);
}

// FP32 variant for the FP32-bulk kernels: the max runs on the bit patterns of
// the non-negative floats with the single-instruction warp reduction, and only
// the block's result is widened to FP64 (on the integer pipe).
__device__ __forceinline__ void block_max_publish_f32(float v, bool bad, unsigned long long *slot, int *status)
{
    __shared__ unsigned warp_max[32];
    __shared__ int any_bad;
    if (threadIdx.x == 0) any_bad = 0;
    const unsigned m = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(v));
    __syncthreads();
    if (bad) any_bad = 1;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) warp_max[wid] = m;
    __syncthreads();
    if (wid == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        const unsigned mm = __reduce_max_sync(0xFFFFFFFFu, lane < nw ? warp_max[lane] : 0u);
        if (lane == 0) {
            if (mm > 0u) atomicMax(slot, (unsigned long long)__double_as_longlong(f32_to_f64(__uint_as_float(mm))));
            if (any_bad) atomicOr(status, ST_NONPHYSICAL);
        }
    }
}

// The same with one barrier: K values, each reduced per warp with the
// single-instruction reduction and combined with a shared-memory atomicMax
// into s_max[K] (with the non-physical flag into *s_bad); the caller zeroes
// s_max and *s_bad before a barrier that precedes this call.  Value 0 goes to
// *slot0, value k > 0 to slot_dir[k - 1].  Every thread of the block must call it.
template <int K>
__device__ __forceinline__ void block_max_publish_f32_1b(const float *v, bool bad, unsigned *s_max, int *s_bad,
                                                         unsigned long long *slot0, unsigned long long *slot_dir,
                                                         int *status)
{
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const unsigned m = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(v[k]));
        if ((threadIdx.x & 31) == 0 && m > 0u) atomicMax(s_max + k, m);
    }
    if (bad) *s_bad = 1;
    __syncthreads();
    if (threadIdx.x < K) {
        const unsigned mm = s_max[threadIdx.x];
        unsigned long long *sl = threadIdx.x == 0 ? slot0 : slot_dir + (threadIdx.x - 1);
        if (mm > 0u) atomicMax(sl, (unsigned long long)__double_as_longlong(f32_to_f64(__uint_as_float(mm))));
    }
    if (threadIdx.x == 0 && *s_bad) atomicOr(status, ST_NONPHYSICAL);
}

// Block-wide max of a non-negative value, then one atomicMax per block on the
// 64-bit pattern of the double.  Also ORs the block's non-physical flag into
// the status word.  Every thread of the block must call it.
__device__ __forceinline__ void block_max_publish(double v, bool bad, unsigned long long *slot, int *status)
{
    __shared__ double warp_max[32];
    __shared__ int any_bad;
    if (threadIdx.x == 0) any_bad = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    __syncthreads();
    if (bad) any_bad = 1;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) warp_max[wid] = v;
    __syncthreads();
    if (wid == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        double m = lane < nw ? warp_max[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
        if (lane == 0) {
            if (m > 0.0) atomicMax(slot, (unsigned long long)__double_as_longlong(m));
            if (any_bad) atomicOr(status, ST_NONPHYSICAL);
        }
    }
}

}  // namespace wg
