// weno_internal.h -- interface between the C ABI layer and the kernels.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace wg {

struct Ctl;

// Epilogue of a sweep kernel (what it does with the direction's residual).
enum Epi { EPI_STORE = 0, EPI_ADD = 1, EPI_RHS = 2, EPI_STAGE = 3 };
// Conservation law: Euler (nf = dim + 2), scalar advection or Burgers (nf = 1).
enum Model { MODEL_EULER = 0, MODEL_ADVECT = 1, MODEL_BURGERS = 2 };

// A tile of the FP64 2D and 3D kernels: w x s cells, nseg x-runs of at most len
// faces per row (k_xy64), nt threads (0: no tile planned), its shared memory.
struct Tile64 {
    int w, s, nseg, len, nt;
    unsigned smem;
};

struct SweepArgs {
    const double *U;     // stencil state U^(k) (device, FP64 SoA)
    const double *Un;    // U^n, read by the stage-2/3 combination
    double *Uout;        // U^(k+1)
    void *acc;           // residual accumulator: float (FP32-bulk) or double (FP64)
    double *Rout;        // output of EPI_RHS
    // 2D FP32-bulk stage state (k_xy2): the FP32 hi/lo split of U^n, written
    // by stage 1, and the FP32 increments Delta_k = U^(k) - U^n
    // 2D: planes H, L of float4 [N] each; 3D: planes H4, L4 (float4 [N]: rho, m_x,
    // m_y, m_z) then H1, L1 (float [N]: E)
    float2 *hl;
    const float *din;    // Delta_k read by stages 2 and 3 (3D: the float4 [N] plane of the first four fields)
    float *dout;         // Delta_{k+1} written by stages 1 and 2 (3D: as din)
    const float *din1;   // 3D: Delta_k of E (float [N])
    float *dout1;        // 3D: Delta_{k+1} of E
    Ctl *ctl;
    long long N;         // cells per field (field stride)
    int n[3];
    long long stride[3]; // 1, nx, nx * ny
    int bc[3][2];
    double bc_state[3][2][5];  // conserved state held by the ghosts of an inflow side
    const double *bcs;   // the same in device memory ([3][2][5]), for out-of-line boundary loads
    double inv_h[3];
    double gamma;
    double eps;
    float gamma_f, gm1_f, eps_f;  // the same constants in FP32, rounded on the host
    float gg_f;          // gamma (gamma - 1) in FP32
    float gms_f;         // gamma - 1 of the FP32 wavespeeds (speed_gm1)
    float inv_h_f[3];
    float2 ih23[3];      // -(2/3) / h_d as FP32 pairs hi + lo (the 2D FP32-bulk residual factor)
    int stage;           // 0, 1, 2
    int slot_in;         // alpha slot used for the splitting
    int slot_out;        // alpha slot the EPI_STAGE epilogue publishes to
    int check_dt;        // skip all work when ctl->dt == 0
    int tile_w, tile_s;  // k_sweep: lines and cells per line of a tile, chosen at the launch
    Tile64 txy, tz;      // k_xy64, k_z: the handle's tiles
    int per_dir;         // LF alpha per direction (alpha_dir slots) instead of one global alpha
};

// gamma - 1 of the FP32 wavespeeds: the FP32 gamma less 1, good to 2^-21 from 1.25 up
// (alpha and dt keep their bits there), and the rounded FP64 difference below, where the
// FP32 one loses its bits (none left at 1 + 1e-8).
inline float speed_gm1(double gamma) { return gamma < 1.25 ? (float)(gamma - 1.0) : (float)gamma - 1.0f; }

// Launches the sweep of direction dir for a dim-dimensional grid.
cudaError_t launch_sweep(int model, int dim, int dir, bool bulk, int epi, const SweepArgs &a, cudaStream_t s);
cudaError_t sweep_set_attributes();
// nsteps whole SSP-RK3 steps of a small 1D FP64 Euler grid on U in place; alpha(U)
// must be in slot 0 (k_run1d.cu).
bool run1d_takes(long long n);
cudaError_t launch_run1d(const SweepArgs &a, double *U, int nsteps, cudaStream_t s);
// Fused FP64 x+y residual of a 2D grid (EPI_RHS / EPI_STAGE) or of the z-planes of a 3D grid (EPI_STORE).
cudaError_t launch_xy64(int dim, int epi, const SweepArgs &a, cudaStream_t s);
// Fused FP32-bulk x+y residual of the z-planes of a 3D grid, left in the accumulator.
cudaError_t launch_xy(const SweepArgs &a, cudaStream_t s);
// 2D FP32-bulk residual / stage in pair-difference form (EPI_RHS / EPI_STAGE).
cudaError_t launch_xy2(int epi, const SweepArgs &a, cudaStream_t s);
// z direction of a 3D FP64 grid, adding the accumulator and ending the residual (EPI_RHS / EPI_STAGE).
cudaError_t launch_z(int epi, const SweepArgs &a, cudaStream_t s);
// z direction of a 3D FP32-bulk grid in pair-difference form (EPI_RHS / EPI_STAGE).
cudaError_t launch_z2(int epi, const SweepArgs &a, cudaStream_t s);

// What k_alpha's last block does with alpha(U) besides storing it in slot 0.
struct AlphaThen {
    double *out;           // not null: alpha goes there too
    int set_run, begin;    // set t_end .. max_steps of a run; begin its first step
    double t_end, dt_req, cfl_h;
    long long max_steps;
};
cudaError_t launch_alpha(int model, int dim, bool bulk, const double *U, long long N, double gamma, Ctl *ctl,
                         int per_dir, const AlphaThen &then, cudaStream_t s);
// Ends a step and, if `begin`, begins the next.
cudaError_t launch_step_end(Ctl *ctl, bool begin, cudaStream_t s);
cudaError_t launch_sums(const double *U, int nf, long long N, double *partials, int nblocks, double *out,
                        cudaStream_t s);
int sums_blocks(long long N);
// Number of SMs of the current device (queried once per device; persistent and
// grid-stride launches are sized from it).
int sm_count();

// Tiles of equal extent along n cells: the smallest extent that needs no more tiles
// than `most` does (97 cells in tiles of at most 32: 4 x 25, not 3 x 32 + 1).
inline int fit_extent(long long n, int most)
{
    const long long t = (n + most - 1) / most;
    return (int)((n + t - 1) / t);
}

// Cycles of the fullest SM of a launch over Tile64 t: FP64 warp instructions at 20
// cycles each -- `cell` for 32 cells' fluxes and update, ~22 for 32 halo points' flux,
// ~7 for a round of windows, a phase's warps filling all four sub-partitions -- but no
// less than the chains of windows (~1000 cycles each) that its rounds of CTAs wait for,
// more where few CTAs or warps share the SM, and part of one chain that nothing hides.
double tile64_cycles(long long tiles, const Tile64 &t, int regs, int cells, double cell, int halo, int runs, int longest);
Tile64 plan_xy64(int dim, const long long n[3]);
Tile64 plan_z(const long long n[3]);

}  // namespace wg
