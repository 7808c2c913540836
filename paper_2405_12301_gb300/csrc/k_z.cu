// k_z.cu -- z direction of the FP64 WENO5-JS residual for 3D grids, ending the
// residual of a stage (the x and y directions run in k_xy.cu; FP32-bulk's z
// direction is k_z2.cu).
#include "weno_dev.cuh"
#include "weno_internal.h"

namespace wg {

// A CTA owns 32 x-cells x TZ = 8 z-cells of one y-row, one cell per thread, plus
// the 3 + 3 halo z-planes of its 32 columns.  Phases: split fluxes of every point
// (own and one halo point per thread), sliding WENO runs along the columns (one
// run of 9 faces per column, component and sign), then each cell's flux
// difference is added to the x+y part left in the accumulator by
// k_xy<3, ..., EPI_STORE>, and the epilogue writes L(U) or applies the SSP-RK3
// stage combination and publishes the wavespeed max.
namespace zs {
constexpr int NT = 256;
constexpr int TX = 32, TZ = 8;
constexpr int BZ = TZ + 6;                  // column extent with halo
constexpr int NZP = TX * BZ;                // z-flux points: 32 x 14
constexpr int NZI = TX * (TZ + 1);          // z interfaces: 32 x 9
constexpr int NHALO = 6 * TX;               // 192 halo points
constexpr int NF = 5;
constexpr size_t fz_off = sizeof(double) * 2 * NF * NZI;
constexpr size_t rough_off = fz_off + sizeof(double) * 2 * NF * NZP;
constexpr size_t bytes = rough_off + sizeof(unsigned) * 2 * NF * NZI;  // (every window)
}  // namespace zs

template <int EPI, bool PD>
__global__ void __launch_bounds__(zs::NT, 3) k_z(const SweepArgs a)
{
    using namespace zs;
    extern __shared__ __align__(16) unsigned char smem[];
    double *Fz = reinterpret_cast<double *>(smem);           // [2][NF][TZ+1][TX]
    double *fz = reinterpret_cast<double *>(smem + fz_off);  // [2][NF][BZ][TX]
    __shared__ int s_rough;
    const RoughList rough{&s_rough, reinterpret_cast<unsigned *>(smem + rough_off)};
    if (threadIdx.x == 0) s_rough = 0;

    const double dt = a.ctl->dt;
    if (a.check_dt && __double_as_longlong(dt) == 0) return;
    const double alpha = PD ? __longlong_as_double((long long)a.ctl->alpha_dir[a.slot_in][2])
                            : __longlong_as_double((long long)a.ctl->alpha[a.slot_in]);

    const int nx = a.n[0], nz = a.n[2];
    const long long N = a.N, sz = a.stride[2];
    // z-tiles are the fastest grid index, so that tiles sharing halo planes run
    // close together and find those planes in L2
    const int x0 = blockIdx.y * TX, z0 = blockIdx.x * TZ;
    const long long yoff = (long long)blockIdx.z * a.stride[1];
    const int tx = threadIdx.x & 31, tz = threadIdx.x >> 5;
    const int gx = x0 + tx, gz = z0 + tz;
    const bool own = gx < nx && gz < nz;
    const long long cell = yoff + (long long)(gz < nz ? gz : nz - 1) * sz + (gx < nx ? gx : nx - 1);

    double un[NF];
    if (EPI == EPI_STAGE && a.stage > 0) {
#pragma unroll
        for (int f = 0; f < NF; ++f) un[f] = __ldg(a.Un + f * N + cell);
    }
    const double gm1 = a.gamma - 1.0;
    const bool interior = z0 >= 3 && z0 + TZ + 3 <= nz && x0 + TX <= nx;

    auto load_point = [&](int lx, int lz, double *q) {
        int cx = x0 + lx, cz = z0 + lz;
        bool fz_ = false;
        if (!interior) {
            int inz;
            cx = cx < nx ? cx : nx - 1;  // columns beyond the grid only feed cells that are not written
            cz = cz < nz + 2 ? cz : nz + 2;
            cz = ghost_map(cz, nz, a.bc[2][0], a.bc[2][1], fz_, inz);
            if (inz >= 0) {  // a ghost of an inflow side holds the given state
#pragma unroll
                for (int f = 0; f < NF; ++f) q[f] = a.bc_state[2][inz][f];
                return;
            }
        }
        const double *src = a.U + yoff + (long long)cz * sz + cx;
#pragma unroll
        for (int f = 0; f < NF; ++f) q[f] = __ldg(src + f * N);
        if (fz_) q[3] = -q[3];
    };
    auto flux_store = [&](const double *q, int lx, int lz) {
        double fp[NF], fm[NF];
        split_flux_f64<3, 2, true>(q, alpha, gm1, fp, fm);
        const int o = (lz + 3) * TX + lx;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            fz[f * NZP + o] = fp[f];
            fz[(NF + f) * NZP + o] = fm[f];
        }
    };

    double uk[NF], qd[NF];
    load_point(tx, tz, uk);
    const bool halo = threadIdx.x < NHALO;
    const int hx = threadIdx.x & 31, hz = (threadIdx.x >> 5) < 3 ? (threadIdx.x >> 5) - 3 : TZ + (threadIdx.x >> 5) - 3;
    if (halo) load_point(hx, hz, qd);
    flux_store(uk, tx, tz);
    if (halo) flux_store(qd, hx, hz);
    __syncthreads();

    {
        // the shared arrays hold 2 f(+/-): reconstruct with 4 eps (twice the WENO5 value)
        const PairEps P = pair_eps(4.0 * a.eps);
#pragma unroll 1
        for (int run = threadIdx.x; run < 2 * NF * TX; run += NT) {
            const int fs = run >> 5, lx = run & 31;
            int po = fs * NZP + lx, oo = fs * NZI + lx, st = TX;
            if (fs >= NF) {  // WENO(-): the same run read backwards from the far end
                po += (TZ + 5) * TX;
                oo += TZ * TX;
                st = -TX;
            }
            weno5_slide_pair<0>(fz, po, st, P, Fz, oo, st, TZ + 1, TX, rough);
        }
        __syncthreads();
        rough_windows<0>(rough, TX, fz, Fz, P);
    }
    __syncthreads();

    const double ihz = 0.5 * a.inv_h[2];  // face fluxes are twice F^
    const double *acc = reinterpret_cast<const double *>(a.acc);
    const double *FzM = Fz + NF * NZI;
    double r[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const int o = f * NZI + tz * TX + tx;
        const double dz = (Fz[o + TX] + FzM[o + TX]) - (Fz[o] + FzM[o]);
        r[f] = acc[f * N + cell] + (-dz * ihz);
    }
    if (EPI == EPI_RHS) {
        if (own) {
#pragma unroll
            for (int f = 0; f < NF; ++f) a.Rout[f * N + cell] = r[f];
        }
        return;
    }
    double out[NF];
    if (own) {
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            out[f] = stage_combine(a.stage, un[f], uk[f], r[f], dt);
            a.Uout[f * N + cell] = out[f];
        }
    }
    speed_max_publish_f64<3, PD ? 4 : 1>(
        [&](long long, double *q) {
#pragma unroll
            for (int f = 0; f < NF; ++f) q[f] = out[f];
        },
        0, own ? 1 : 0, 1, a.gamma, &a.ctl->alpha[a.slot_out], a.ctl->alpha_dir[a.slot_out], &a.ctl->status);
}

template <int EPI, bool PD>
static cudaError_t launch_z_t(const SweepArgs &a, cudaStream_t s)
{
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_z<EPI, PD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)zs::bytes);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    dim3 grid((unsigned)((a.n[2] + zs::TZ - 1) / zs::TZ), (unsigned)((a.n[0] + zs::TX - 1) / zs::TX), (unsigned)a.n[1]);
    k_z<EPI, PD><<<grid, zs::NT, zs::bytes, s>>>(a);
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
