// k_sweep.cu -- the fused per-direction residual kernel of the WENO5-JS scheme.
//
// One launch handles one direction d of one stage.  A CTA owns a tile of W
// grid lines along d, S cells each (fitted to the grid, sweep_tile), and runs three
// phases through shared memory:
//   A. every stencil point of the tile (S + 6 per line: three ghost layers per
//      side, Sec. 4.5) is loaded once, its ghost index mapped by the boundary
//      rule, and its Lax-Friedrichs split flux f(+/-) (Sec. 2.2) computed once;
//   B. every interface flux F^_{i+1/2} = WENO(+)(f+) + WENO(-)(f-) of the tile
//      (S + 1 per line and component) is computed once, as one work item per
//      (interface, component);
//   C. every cell forms -(F^_{i+1/2} - F^_{i-1/2}) / h_d (Sec. 4.1) and the
//      epilogue stores it, adds it to the accumulator of earlier directions,
//      writes L(U), or -- for the last direction of a stage -- applies the
//      SSP-RK3 stage combination (Eq. tt-ssprk3 without rounding) and
//      publishes the wavespeed max of the new state for the next stage's alpha.
//
// FP64 mode computes everything in FP64 but the WENO weights (FP32 pairs and triples at
// FP64's accuracy, weno5_slide_pair).  FP32-bulk mode computes phases A-C
// in FP32 on differences from a per-line reference state (exact to FP32
// relative precision of the differences), and only the final state update
// U^(k+1) = U^(k) + D is an FP64 add.
//
// The model M selects the conservation law: the Euler equations (M = 0, the
// only one with an FP32-bulk form), or one scalar field u under linear
// advection with unit velocity in every direction (M = 1, f_d(u) = u, Sec. 5.1)
// or Burgers' equation (M = 2, f_d(u) = u^2 / 2, Sec. 5.2).  The scalar laws
// run through every direction of 1D, 2D and 3D grids with this kernel.
#include <type_traits>

#include "weno_dev.cuh"
#include "weno_internal.h"

namespace wg {

constexpr int NT = 256;

// Bounds of a tile: lines, points (lines x (cells + 6 halo points)).  The launch
// picks the tile within them for the grid (sweep_tile).
template <int M, int DIR> struct Tile { static constexpr int W = 32, S = 26, P = W * (S + 6); };  // y, z: 32 x-lines, 26 cells
template <int M> struct Tile<M, 0> {  // x: rows; a scalar's runs need 1024 points to fill the warps
    static constexpr int W = 32, S = 250, P = M == MODEL_EULER ? NT : 1024;
};
// FP32-bulk: a row's points lie within 124 cells of its reference, the middle cell (the
// rounding errors of L(U) grow with that distance: 250 cells with the reference in the
// first have twice the error of 243 cells at 200000 cells).
constexpr int BULK_S = 243;

constexpr size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

template <int M> constexpr int nfields(int D) { return M == MODEL_EULER ? D + 2 : 1; }

template <int M, int D, int DIR, bool BULK> struct Layout {
    using T = typename std::conditional<BULK, float, double>::type;
    // (interfaces per line and component: cells + 1, fewer than points)
    static constexpr int NF = nfields<M>(D), MP = Tile<M, DIR>::P, MI = DIR == 0 ? MP : Tile<M, DIR>::W * (Tile<M, DIR>::S + 1);
    static constexpr size_t fp_off = 0;
    static constexpr size_t fm_off = fp_off + sizeof(T) * NF * MP;
    static constexpr size_t F_off = fm_off + sizeof(T) * NF * MP;
    static constexpr int NS = BULK ? 1 : 2;   // face-flux copies: FP64 keeps WENO(+) and WENO(-) apart
    static constexpr int RF = 9;              // faces per FP64 sliding run
    static constexpr size_t ref_off = align16(F_off + sizeof(T) * NS * NF * MI);
    // FP32-bulk: the lines' reference states; FP64: the rough windows' list (every window)
    static constexpr size_t bytes = ref_off + (BULK ? sizeof(RefState<D>) * Tile<M, DIR>::W : sizeof(unsigned) * 2 * NF * MI);
    static_assert(2 * NF * MP <= 8192 && 2 * NF * MI <= 8192, "offsets of a RoughList entry");
};

// Split fluxes f(+/-) = (f(u) +/- alpha u) / 2 of a scalar law (Eq. lax-friedrichs).
template <int M>
__device__ __forceinline__ void split_flux_scalar(double u, double alpha, double &fp, double &fm)
{
    const double f = M == MODEL_ADVECT ? u : 0.5 * u * u;
    fp = 0.5 * (f + alpha * u);
    fm = 0.5 * (f - alpha * u);
}

template <int M, int D, int DIR, bool BULK, int EPI>
__global__ void __launch_bounds__(NT, 4) k_sweep(const SweepArgs a)
{
    static_assert(M == MODEL_EULER || !BULK, "the FP32-bulk form exists for the Euler equations only");
    using L = Layout<M, D, DIR, BULK>;
    using T = typename L::T;
    constexpr int NF = L::NF, MP = L::MP, MI = L::MI;
    const int W = a.tile_w, S = a.tile_s, NP = S + 6, NI = S + 1;
    extern __shared__ __align__(16) unsigned char smem[];
    T *sfp = reinterpret_cast<T *>(smem + L::fp_off);
    T *sfm = reinterpret_cast<T *>(smem + L::fm_off);
    T *sF = reinterpret_cast<T *>(smem + L::F_off);
    RefState<D> *sref = reinterpret_cast<RefState<D> *>(smem + L::ref_off);
    __shared__ int s_rough;
    const RoughList rough{&s_rough, reinterpret_cast<unsigned *>(smem + L::ref_off)};
    if (!BULK && threadIdx.x == 0) s_rough = 0;

    const long long dtbits = __double_as_longlong(a.ctl->dt);
    if (a.check_dt && dtbits == 0) return;  // the step is a no-op (time reached t_end)
    const double dt = __longlong_as_double(dtbits);

    const long long N = a.N;
    const int n = a.n[DIR];
    const long long st = a.stride[DIR];
    int seg, lg, other;
    if (DIR == 0) { seg = blockIdx.x; lg = blockIdx.y; other = blockIdx.z; }
    else if (DIR == 1) { lg = blockIdx.x; seg = blockIdx.y; other = blockIdx.z; }
    else { lg = blockIdx.x; other = blockIdx.y; seg = blockIdx.z; }
    const int c0 = seg * S;
    // Base offset of line w of the tile; false if the line lies outside the grid.
    auto line = [&](int w, long long &base) -> bool {
        if (DIR == 0) {
            const int y = lg * W + w;
            base = (long long)other * a.stride[2] + (long long)y * a.stride[1];
            return y < a.n[1];
        }
        const int x = lg * W + w;
        base = (long long)other * (DIR == 1 ? a.stride[2] : a.stride[1]) + x;
        return x < a.n[0];
    };

    const double alpha = a.per_dir ? __longlong_as_double((long long)a.ctl->alpha_dir[a.slot_in][DIR])
                                   : __longlong_as_double((long long)a.ctl->alpha[a.slot_in]);
    const float alpha_f = BULK ? f64_to_f32(alpha) : 0.0f;  // integer pipe: cvt issues at FP64 rate
    const double gm1 = a.gamma - 1.0;
    const T eps = BULK ? (T)a.eps_f : (T)a.eps;

    // ---- phase 0 (FP32-bulk): reference state of every line, its middle cell's
    if constexpr (BULK) {
        for (int w = threadIdx.x; w < W; w += NT) {
            long long base;
            const bool ok = line(w, base);
            double q[NF];
            const int cr = c0 + S / 2 < n ? c0 + S / 2 : n - 1;
#pragma unroll
            for (int f = 0; f < NF; ++f)
                q[f] = ok ? a.U[f * N + base + (long long)cr * st] : (f == 0 || f == NF - 1 ? 1.0 : 0.0);
            make_ref<D>(q, a.gm1_f, sref[w]);
        }
        __syncthreads();
    }

    // ---- phase A: split point fluxes of the S + 6 stencil points of every line
    for (int u = threadIdx.x; u < W * NP; u += NT) {
        int w, p;
        if (DIR == 0) { w = u / NP; p = u - w * NP; }
        else { p = u / W; w = u - p * W; }
        long long base;
        T fpv[NF], fmv[NF];
        if (line(w, base)) {
            int c = c0 - 3 + p;
            c = c < n + 2 ? c : n + 2;
            bool flip;
            int inflow;
            const int cm = ghost_map(c, n, a.bc[DIR][0], a.bc[DIR][1], flip, inflow);
            const double *src = a.U + base + (long long)cm * st;
            double q[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) q[f] = inflow >= 0 ? a.bc_state[DIR][inflow][f] : __ldg(src + f * N);
            if (M == MODEL_EULER && flip) q[1 + DIR] = -q[1 + DIR];
            if constexpr (M != MODEL_EULER) {
                split_flux_scalar<M>(q[0], alpha, fpv[0], fmv[0]);
            } else if constexpr (BULK) {
                float dq[NF];
                diff_from_ref<D>(q, sref[w], dq);
                split_flux_diff<D, DIR>(dq, sref[w], alpha_f, a.gm1_f, fpv, fmv);
            } else {
                split_flux_f64<D, DIR>(q, alpha, gm1, fpv, fmv);
            }
        } else {
#pragma unroll
            for (int f = 0; f < NF; ++f) fpv[f] = fmv[f] = T(0);
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            sfp[f * MP + u] = fpv[f];
            sfm[f * MP + u] = fmv[f];
        }
    }
    __syncthreads();

    // ---- phase B: interface fluxes.  FP64: a sliding run of RF faces per work item
    // (line, segment, component, sign), WENO(+) and WENO(-) kept apart; FP32-bulk:
    // one work item per (interface, component)
    const int nfaces = n - c0 + 1 < NI ? n - c0 + 1 : NI;  // none right of the last cell's right face
    if constexpr (!BULK) {
        const PairEps P = pair_eps(eps);
        const int nseg = (nfaces + L::RF - 1) / L::RF;
        const int pst = DIR == 0 ? 1 : W;
        for (int u = threadIdx.x; u < 2 * NF * W * nseg; u += NT) {
            // neighbouring lanes: segments of a row (x), columns (y, z) -- distinct banks
            const int q = DIR == 0 ? nseg : W, r = u / q, lo = u - r * q, hi = r % (DIR == 0 ? W : nseg);
            const int w = DIR == 0 ? hi : lo, seg_ = DIR == 0 ? lo : hi, fs = u / (W * nseg);
            const int j0 = seg_ * L::RF, cnt = nfaces - j0 < L::RF ? nfaces - j0 : L::RF;
            long long base;
            if (!line(w, base)) continue;
            const bool minus = fs >= NF;
            // face j: f+ at points j..j+4, f- mirrored at j+5..j+1 (sfm follows sfp)
            const int jp = minus ? j0 + cnt + 4 : j0, jo = minus ? j0 + cnt - 1 : j0, st_ = minus ? -pst : pst;
            const int po = fs * MP + (DIR == 0 ? w * NP : w) + jp * pst;
            const int oo = fs * MI + (DIR == 0 ? w * NI : w) + jo * pst;
            weno5_slide_pair(sfp, po, st_, P, sF, oo, st_, cnt, pst, rough);
        }
        __syncthreads();
        rough_windows(rough, pst, sfp, sF, P);
    } else {
        for (int u = threadIdx.x; u < NF * W * NI; u += NT) {
            const int f = u / (W * NI);
            const int r = u - f * (W * NI);
            int w, j;
            if (DIR == 0) { w = r / NI; j = r - w * NI; }
            else { j = r / W; w = r - j * W; }
            if (j >= nfaces) continue;
            const T *P = sfp + f * MP;
            const T *M = sfm + f * MP;
            const int pw = DIR == 0 ? w * NP : w;
            const int ps = DIR == 0 ? 1 : W;
            // interface between local cells j-1 and j: f+ at points j..j+4, f- mirrored at j+5..j+1
            const T Fh = weno5<T>(P[pw + j * ps], P[pw + (j + 1) * ps], P[pw + (j + 2) * ps], P[pw + (j + 3) * ps],
                                  P[pw + (j + 4) * ps], eps) +
                         weno5<T>(M[pw + (j + 5) * ps], M[pw + (j + 4) * ps], M[pw + (j + 3) * ps],
                                  M[pw + (j + 2) * ps], M[pw + (j + 1) * ps], eps);
            sF[f * MI + (DIR == 0 ? w * NI + j : j * W + w)] = Fh;
        }
    }
    __syncthreads();

    // ---- phase C: flux difference and epilogue
    const T ih = BULK ? (T)a.inv_h_f[DIR] : (T)a.inv_h[DIR];
    double cmax = 0.0;
    float cmaxf = 0.0f;
    bool bad = false;
    // FP32-bulk: the stage combination U' = a_n U^n + b_n (U^k + dt R) (Eq. tt-ssprk3) with a_n and b_n dt as hi + lo pairs (no systematic coefficient rounding)
    const float anf = a.stage == 0 ? 0.0f : (a.stage == 1 ? 0.75f : (float)(1.0 / 3.0));
    const float anf_lo = a.stage == 2 ? (float)(1.0 / 3.0 - (double)(float)(1.0 / 3.0)) : 0.0f;
    const double bn = a.stage == 0 ? 1.0 : (a.stage == 1 ? 0.25 : 2.0 / 3.0);
    const float2 bdtf = BULK ? f64_to_f32x2(bn * dt) : make_float2(0.0f, 0.0f);
    double qout[NF];
    bool has = false;
    for (int u = threadIdx.x; u < W * S; u += NT) {
        int w, i;
        if (DIR == 0) { w = u / S; i = u - w * S; }
        else { i = u / W; w = u - i * W; }
        long long base;
        if (!line(w, base) || c0 + i >= n) continue;
        const long long cell = base + (long long)(c0 + i) * st;
        const int jl = DIR == 0 ? w * NI + i : i * W + w;
        const int jr = DIR == 0 ? jl + 1 : jl + W;
        T rd[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            if constexpr (BULK) {
                rd[f] = -(sF[f * MI + jr] - sF[f * MI + jl]) * ih;
            } else {
                const T *Fp = sF + f * MI, *Fm = Fp + NF * MI;
                rd[f] = -((Fp[jr] + Fm[jr]) - (Fp[jl] + Fm[jl])) * ih;
            }
        }
        T *acc = reinterpret_cast<T *>(a.acc);
        if (EPI == EPI_STORE) {
#pragma unroll
            for (int f = 0; f < NF; ++f) acc[f * N + cell] = rd[f];
        } else if (EPI == EPI_ADD) {
#pragma unroll
            for (int f = 0; f < NF; ++f) acc[f * N + cell] += rd[f];
        } else {
            T r[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) r[f] = (D == 1) ? rd[f] : acc[f * N + cell] + rd[f];
            if (EPI == EPI_RHS) {
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    if constexpr (BULK) a.Rout[f * N + cell] = f32_to_f64(r[f]);
                    else a.Rout[f * N + cell] = r[f];
                }
            } else {  // EPI_STAGE
                double out[NF];
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    const double uk = a.U[f * N + cell];
                    if constexpr (BULK) {
                        float hk, lk;
                        split_f64(uk, hk, lk);
                        float dlt = fmaf(bdtf.x, r[f], bdtf.y * r[f]);
                        if (a.stage > 0) {
                            float hn, ln;
                            split_f64(a.Un[f * N + cell], hn, ln);
                            const float x = (hn - hk) + (ln - lk);
                            dlt = fmaf(anf, x, fmaf(anf_lo, x, dlt));
                        }
                        out[f] = uk + f32_to_f64(dlt);
                    } else {
                        out[f] = stage_combine(a.stage, a.stage == 0 ? 0.0 : a.Un[f * N + cell], uk, r[f], dt);
                    }
                    a.Uout[f * N + cell] = out[f];
                }
                bool b;
                if constexpr (M != MODEL_EULER) {  // |f'(u)|: 1 for advection, |u| for Burgers
                    b = !isfinite(out[0]);
                    cmax = fmax(cmax, M == MODEL_ADVECT ? 1.0 : fabs(out[0]));
                } else if constexpr (BULK) {
                    float qf[NF];
#pragma unroll
                    for (int f = 0; f < NF; ++f) qf[f] = f64_to_f32(out[f]);
                    cmaxf = fmaxf(cmaxf, wavespeed_f32<D>(qf, a.gamma_f, a.gms_f, b));
                } else {  // (one cell per thread: its speed is formed below)
                    static_assert(M != MODEL_EULER || MP <= NT, "one cell per thread");
#pragma unroll
                    for (int f = 0; f < NF; ++f) qout[f] = out[f];
                    has = true;
                    b = false;
                }
                bad |= b;
            }
        }
    }
    if constexpr (EPI == EPI_STAGE && M == MODEL_EULER && !BULK) {
        // 1D: |u_x| + a is the x slot's
        const int K = a.per_dir ? 2 : 1;
        auto load = [&](long long, double *q) {
#pragma unroll
            for (int f = 0; f < NF; ++f) q[f] = qout[f];
        };
        if (K == 2)
            speed_max_publish_f64<D, 2>(load, 0, has ? 1 : 0, 1, a.gamma, a.gg_f, &a.ctl->alpha[a.slot_out],
                                        a.ctl->alpha_dir[a.slot_out], &a.ctl->status);
        else
            speed_max_publish_f64<D, 1>(load, 0, has ? 1 : 0, 1, a.gamma, a.gg_f, &a.ctl->alpha[a.slot_out],
                                        a.ctl->alpha_dir[a.slot_out], &a.ctl->status);
    } else if (EPI == EPI_STAGE) {
        if (BULK) cmax = (double)cmaxf;
        block_max_publish(cmax, bad, &a.ctl->alpha[a.slot_out], &a.ctl->status);
        // 1D: |u_x| + a equals |u| + a, so the x slot takes the same maximum
        if (M == MODEL_EULER && D == 1 && a.per_dir) block_max_publish(cmax, false, &a.ctl->alpha_dir[a.slot_out][0], &a.ctl->status);
    }
}

static inline unsigned cdiv(long long a, long long b) { return (unsigned)((a + b - 1) / b); }

// The tile for a grid: segments of equal length (a 150-cell row is 2 x 75, not
// 122 + 28), columns likewise; rows as many as the points allow while there are two
// tiles for every SM, and on small grids shorter segments for the same reason (a row
// costs 6 halo points per segment, so not below 20 cells).  Advection at 128^3, x:
// 7 rows of 128 cells (210 runs, the warps full); 3 rows of 64 (48 runs) took 164 us.
// In 1D a tile is 250 cells (FP32-bulk: 243), a point per thread.
template <int M, int DIR, bool BULK> static void sweep_tile(SweepArgs &a)
{
    const int n = a.n[DIR];
    if (DIR == 0) {
        const long long rows = (long long)a.n[1] * a.n[2];
        const long long want = rows == 1 ? sm_count() : 4ll * sm_count();  // (a 1D tile is one row: a CTA per SM fills its warps best)
        long long most = (n * rows + want - 1) / want;
        constexpr int longest = BULK ? BULK_S : Tile<M, 0>::S;
        most = most < 20 ? 20 : most > longest ? longest : most;
        a.tile_s = (int)cdiv(n, cdiv(n, most));
        long long w = Tile<M, 0>::P / (a.tile_s + 6), share = rows * cdiv(n, a.tile_s) / (2ll * sm_count());
        share = share < 2 ? 2 : share;  // (2 rows keep the grid's y extent in range)
        w = w > Tile<M, 0>::W ? Tile<M, 0>::W : w;
        w = w > share ? share : w;
        a.tile_w = fit_extent(a.n[1], (int)w);
    } else {
        a.tile_s = (int)cdiv(n, cdiv(n, Tile<M, DIR>::S));
        a.tile_w = (int)cdiv(a.n[0], cdiv(a.n[0], Tile<M, DIR>::W));
    }
}

template <int M, int D, int DIR, bool BULK, int EPI>
static cudaError_t launch_t(SweepArgs a, cudaStream_t s)
{
    using L = Layout<M, D, DIR, BULK>;
    sweep_tile<M, DIR, BULK>(a);
    dim3 grid;
    if (DIR == 0) grid = dim3(cdiv(a.n[0], a.tile_s), cdiv(a.n[1], a.tile_w), (unsigned)a.n[2]);
    else if (DIR == 1) grid = dim3(cdiv(a.n[0], a.tile_w), cdiv(a.n[1], a.tile_s), (unsigned)a.n[2]);
    else grid = dim3(cdiv(a.n[0], a.tile_w), (unsigned)a.n[1], cdiv(a.n[2], a.tile_s));
    k_sweep<M, D, DIR, BULK, EPI><<<grid, NT, L::bytes, s>>>(a);
    return cudaGetLastError();
}

template <int M, int D, int DIR, bool BULK, int EPI>
static cudaError_t attr_t()
{
    using L = Layout<M, D, DIR, BULK>;
    return cudaFuncSetAttribute(k_sweep<M, D, DIR, BULK, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)L::bytes);
}

// Euler: 1D grids only (2D and 3D grids run in the fused k_xy* and k_z* kernels).
// Scalar laws (FP64): every direction; the first stores, the middle one of 3D
// adds, the last runs the residual or stage epilogue.
#define WG_SWEEP_TABLE(X)                                                                       \
    X(MODEL_EULER, 1, 0, false, EPI_RHS) X(MODEL_EULER, 1, 0, false, EPI_STAGE)                  \
    X(MODEL_EULER, 1, 0, true, EPI_RHS) X(MODEL_EULER, 1, 0, true, EPI_STAGE)                    \
    WG_SCALAR_ROWS(X, MODEL_ADVECT) WG_SCALAR_ROWS(X, MODEL_BURGERS)
#define WG_SCALAR_ROWS(X, M)                                                                     \
    X(M, 1, 0, false, EPI_RHS) X(M, 1, 0, false, EPI_STAGE)                                      \
    X(M, 2, 0, false, EPI_STORE) X(M, 2, 1, false, EPI_RHS) X(M, 2, 1, false, EPI_STAGE)         \
    X(M, 3, 0, false, EPI_STORE) X(M, 3, 1, false, EPI_ADD) X(M, 3, 2, false, EPI_RHS)           \
    X(M, 3, 2, false, EPI_STAGE)

cudaError_t sweep_set_attributes()
{
    cudaError_t e = cudaSuccess, r;
#define X(M, D, DIR, B, E) \
    if ((r = attr_t<M, D, DIR, B, E>()) != cudaSuccess) e = r;
    WG_SWEEP_TABLE(X)
#undef X
    return e;
}

cudaError_t launch_sweep(int model, int dim, int dir, bool bulk, int epi, const SweepArgs &a, cudaStream_t s)
{
#define X(M, D, DIR, B, E) \
    if (model == M && dim == D && dir == DIR && bulk == B && epi == E) return launch_t<M, D, DIR, B, E>(a, s);
    WG_SWEEP_TABLE(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace wg
