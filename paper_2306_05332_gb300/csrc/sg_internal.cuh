// Internal declarations shared by the CUDA kernels and the host orchestration.
// Nothing here is part of the C ABI (include/sg.h is).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <cstdint>
#include <cstddef>

namespace sg {

// Geometry and boundary description of one multigrid level.  Arrays are dense
// [nz][ny][nx] (x fastest) without ghost cells; the ghost values of Sec. 2.3 are
// produced on the fly by the kernels:
//   periodic axis           -> the cell on the opposite side (Eq. periodic)
//   Dirichlet with faces    -> 2 * face - active              (Eq. solution_ghost)
//   Dirichlet without faces -> -active                        (Eq. error_ghost)
struct LevelGeom {
    int nx, ny, nz;
    double ihx2, ihy2, ihz2;          // 1 / h_d^2
    float ihx2f, ihy2f, ihz2f;        // the same in FP32: FP32 kernels must never convert from FP64
                                      // (GB300 issues FP64 and its conversions at 1/64 of the FP32 rate)
    int per[3];                       // periodic flag per axis (x, y, z)
    const double* face[6];            // -x,+x,-y,+y,-z,+z or all nullptr (homogeneous)
    int twod;                         // a two-dimensional level (Sec. 2.2): nz = 1, z periodic, 1 / h_z^2 = 0,
                                      // so the seven-point kernels compute the five-point operator exactly;
                                      // restriction averages 4 cells, prolongation weighs 9/3/3/1
};

// 1 / h^2 per axis in the kernel's precision.
template <typename T> __host__ __device__ __forceinline__ T ih2x(const LevelGeom& g);
template <> __host__ __device__ __forceinline__ float ih2x<float>(const LevelGeom& g) { return g.ihx2f; }
template <> __host__ __device__ __forceinline__ double ih2x<double>(const LevelGeom& g) { return g.ihx2; }
template <typename T> __host__ __device__ __forceinline__ T ih2y(const LevelGeom& g);
template <> __host__ __device__ __forceinline__ float ih2y<float>(const LevelGeom& g) { return g.ihy2f; }
template <> __host__ __device__ __forceinline__ double ih2y<double>(const LevelGeom& g) { return g.ihy2; }
template <typename T> __host__ __device__ __forceinline__ T ih2z(const LevelGeom& g);
template <> __host__ __device__ __forceinline__ float ih2z<float>(const LevelGeom& g) { return g.ihz2f; }
template <> __host__ __device__ __forceinline__ double ih2z<double>(const LevelGeom& g) { return g.ihz2; }

// Per-stage coefficients of one RKL stage (App. A, Eq. RKL_intermediate_source).
//   first stage : z = tau (L Y0 - f);  Y1 = Y0 + mut1 * z;   (RKL2 stores z as Z0)
//   later stages: Yj = mu Y_{j-1} + nu Y_{j-2} + mut_tau (L Y_{j-1} - f)
//                      [RKL2: + c0 Y0 + gt Z0]
// (FP64 stages store Z0 without its factor tau and apply it with gt.)
struct StageCoef {
    double tau;
    double mut1;      // first stage only: mu~_1
    double mu, nu;
    double mut_tau;   // mu~_j * tau
    double c0;        // 1 - mu_j - nu_j (RKL2)
    double gt;        // gamma~_j (RKL2; multiplies Z0 = tau (M Y0 - f))
};

// Deterministic two-pass reductions: kernels write one Partial per block, a
// single-block kernel folds them in a fixed order into a Reduced.
struct Partial {
    double sumsq;     // sum of r^2
    double maxabs;    // max |r|
    double sum;       // sum of a secondary field (coarse rhs for the periodic mean)
    double pad;
};
struct Reduced {
    double sumsq, maxabs, sum, count;
};

constexpr int kRedThreads = 256;

// ---- launchers (kernels_stencil.cu) ----------------------------------------
// Number of blocks (= Partial slots) a residual / residual-restrict launch uses.
long long residual_blocks(const LevelGeom& g);
long long residual_zero_blocks(const LevelGeom& g);   // launch_residual_zero, both passes
long long restrict_blocks(const LevelGeom& g);
constexpr long long kSumBlocks = 152LL * 8;     // grid of the 1D reduction kernels

template <typename T>
cudaError_t launch_stage(const LevelGeom& g, int order, bool first, const StageCoef& c,
                         const T* ym1, const T* ym2, const T* y0, const T* z0, const T* rhs,
                         T* out, T* z0_out, cudaStream_t st);

// One colour (0: (i + j + k) even, 1: odd) of a red-black Gauss-Seidel / SOR
// sweep of L u = rhs, in place (periodic extents must be even).
template <typename T>
cudaError_t launch_gsrb(const LevelGeom& g, int colour, double omega, T* u, const T* rhs, cudaStream_t st);

// r = rhs - L u (TI), optionally stored as TO (r_out) and in full precision
// (r_full), block partials of sum r^2 / max|r|.
template <typename TI, typename TO>
cudaError_t launch_residual(const LevelGeom& g, const TI* u, const TI* rhs, TO* r_out,
                            Partial* partials, int* nblocks_out, cudaStream_t st, TI* r_full = nullptr);
// The same for u = 0 (FP64 rhs): r = rhs - L 0, the face terms only
// (*nkernels: the kernels it launched, one or two).
template <typename TO>
cudaError_t launch_residual_zero(const LevelGeom& g, const double* rhs, TO* r_out, Partial* partials,
                                 int* nblocks_out, cudaStream_t st, double* r_full = nullptr,
                                 int* nkernels = nullptr);

// Fused residual + 8-cell restriction.  `want`: the block partials it writes besides
// (the norms of r and the sum of the coarse values; the sum alone; nothing: a
// V-cycle reads the sum only where every axis is periodic, and the norms cost an FP64
// level two operations a cell).
constexpr int kWantNothing = 0, kWantSum = 1, kWantNorms = 2;
template <typename T>
cudaError_t launch_residual_restrict(const LevelGeom& fine, const T* u, const T* rhs,
                                     T* coarse_out, Partial* partials, int* nblocks_out,
                                     cudaStream_t st, int want = kWantNorms);

// fine += P(coarse) with coarse ghosts by the homogeneous/periodic rule.
template <typename T>
cudaError_t launch_prolong_correct(const LevelGeom& fine, const T* coarse, T* fine_u,
                                   cudaStream_t st);

cudaError_t launch_finalize(const Partial* partials, int n, Reduced* out, cudaStream_t st);

// The FP64 residual r = rhs - A u (r into r_full, its FP32 copy into r_out,
// the norms of the copy into partials) with the neighbour sum in exact 64-bit
// fixed point: a pre-pass writes the scale into *scratch (one word on the
// device), then the residual (*nkernels: the kernels launched, two; one, the
// FP64 residual, for levels that are not strips of four cells).
cudaError_t launch_residual_exact(const LevelGeom& g, const double* u, const double* rhs, float* r_out,
                                  double* r_full, Partial* partials, unsigned* scratch, int* nblocks_out,
                                  int* nkernels, cudaStream_t st);
// phi += e (FP64) and r64 -= A_0 e (FP64 residual by recurrence, A_0 e summed
// error-free in FP32), r32 = r64 rounded, block partials of |r32|.
cudaError_t launch_update_residual(const LevelGeom& g, double* phi, const float* e, double* r64, float* r32,
                                  Partial* partials, int* nblocks_out, cudaStream_t st);

template <typename T>
cudaError_t launch_subtract_mean(T* x, long long n, const Reduced* red, cudaStream_t st);

cudaError_t launch_scale_copy(const double* src, double* dst, double scale, long long n,
                              cudaStream_t st);
// dst = scale src (or a plain copy when !scaled) where src or dst is pinned
// host memory mapped into the device address space.
cudaError_t launch_link_copy(const double* src, double* dst, double scale, bool scaled, long long n,
                             cudaStream_t st);
cudaError_t launch_add_f32_to_f64(double* phi, const float* e, long long n, cudaStream_t st);
cudaError_t launch_sub_mean_f64(double* x, long long n, const Reduced* red, cudaStream_t st);
cudaError_t launch_sum_partials_f64(const double* x, long long n, Partial* partials,
                                    int* nblocks_out, cudaStream_t st);

// ---- FP64 throughput probe (kernels_probe.cu) -------------------------------
// TFLOP/s of FP64 FMA chains on every SM of the current device (2 flops per FMA).
cudaError_t probe_fp64_rate(double* tflops, double* ms);

// ---- the convergence loop on the device (kernels_loop.cu) -------------------
constexpr int kLoopHistory = 256;          // entries of the residual history kept (SG_MAX_HISTORY)
constexpr int kLoopRunning = 0, kLoopDone = 1, kLoopNotConverged = 2, kLoopNonFinite = 3;
// State of one solve's cycle loop in device memory: set by the host before
// the solve graph is launched, read back once when it has finished.
struct LoopState {
    double rden;            // ||L 0 - f|| (1 if zero)
    double nn;              // cells of level 0
    double tol;             // relative L2 tolerance
    double mtol;            // > 0: stop on max |r| <= mtol instead
    int limit;              // cycle cap (or the fixed count)
    int fixed;              // run exactly `limit` cycles
    int confirm;            // mixed precision: confirm a met recurrence residual in FP64
    int m;                  // cycles run
    int status;             // kLoop*
    int pending;            // the inner loop ended for a confirmation
    int sched_len;          // entries of the coarse schedule
    int confirms;           // times the inner loop ended (the confirmation step ran)
    long long coarse_cells; // cells of the coarsest level
    long long coarse_stage_cells;   // sum over cycles of coarse cells x stages
    double rel, maxabs;     // the last recorded residual
};
struct DeviceLoop : LoopState {
    double history[kLoopHistory];
    int coarse_ss[kLoopHistory];
};
// has_inner false: the inner loop is no WHILE node (the resident solve runs it in one launch)
cudaError_t launch_loop_init(const DeviceLoop* d, cudaGraphConditionalHandle outer, cudaGraphConditionalHandle inner,
                             bool has_inner, cudaStream_t st);
// partials, nb: the residual's block partials, folded into *red first (confirm: none where nb = 0)
cudaError_t launch_loop_step(DeviceLoop* d, const Partial* partials, int nb, Reduced* red, const int* ss_done,
                             const int* sched, cudaGraphConditionalHandle inner, cudaStream_t st);
cudaError_t launch_loop_confirm(DeviceLoop* d, const Partial* partials, int nb, Reduced* red,
                                cudaGraphConditionalHandle outer, cudaGraphConditionalHandle inner, bool has_inner,
                                cudaStream_t st);
__host__ __device__ __forceinline__ bool loop_met(const LoopState& d, double rel, double maxabs) {
    return d.mtol > 0.0 ? maxabs <= d.mtol : rel <= d.tol;
}
__host__ __device__ __forceinline__ double loop_rel(const LoopState& d, const Reduced& r) {
    return sqrt(r.sumsq / d.nn) / d.rden;
}
// The decision after a cycle with relative residual rel and largest residual maxabs, on
// the counters of d: true to run another.  *record: the residual goes into the history.
__host__ __device__ __forceinline__ bool loop_decide(LoopState& d, double rel, double maxabs, bool* record) {
    d.m += 1;
    const bool finite = isfinite(rel);
    const bool met = loop_met(d, rel, maxabs);
    *record = true;
    if (!d.fixed && finite && met && d.confirm) {
        d.pending = 1;                      // the true residual decides (k_loop_confirm)
        *record = false;
        return false;
    }
    d.rel = rel;
    d.maxabs = maxabs;
    if (!finite) d.status = kLoopNonFinite;
    else if (!d.fixed && met) d.status = kLoopDone;
    else if (d.m >= d.limit) d.status = d.fixed ? kLoopDone : kLoopNotConverged;
    else return true;
    return false;
}
// The decision after the inner loop, red: the residual f - A phi (mixed precision), else that
// of the last cycle; true to resume the cycles.  A residual that is not finite ends the
// solve as such also where nothing waits for the confirmation (a fixed cycle count, the
// cycle cap): a launch that gave up a wait leaves its NaN in phi after its last decision.
__host__ __device__ __forceinline__ bool loop_confirm(DeviceLoop& d, const Reduced& red) {
    d.confirms += 1;
    const double rel = loop_rel(d, red);
    const bool finite = isfinite(rel);
    if (!d.pending && finite) return false;
    d.pending = 0;
    if (d.m < kLoopHistory) d.history[d.m] = rel;
    d.rel = rel;
    d.maxabs = red.maxabs;
    if (!finite) d.status = kLoopNonFinite;
    else if (loop_met(d, rel, red.maxabs)) d.status = kLoopDone;
    else if (d.m >= d.limit) d.status = kLoopNotConverged;
    else return true;
    return false;
}

// ---- fused super-step, FP32 (kernels_fused.cu) -----------------------------
constexpr int kFusedMaxS = 6;
struct FusedCoef {
    float tau, mut1;                        // first stage
    float mu[kFusedMaxS + 1], nu[kFusedMaxS + 1], mut_tau[kFusedMaxS + 1];
    float c0[kFusedMaxS + 1], gt[kFusedMaxS + 1];
};
// True if the fused kernel handles (order, s): 2 <= s <= kFusedMaxS.
bool fused_supported(int order, int s);
cudaError_t fused_configure();
// out = Y_s of one super-step from y0 (nullptr: Y0 = 0) with homogeneous or
// periodic ghosts; out must not alias y0.
// s = 2, 3: tile_rows 0 without tma takes the kernel with one column per thread;
// 14 or 16 the one with one stage per thread and tiles of so many rows, tma the
// same with planes staged by tensor-map box copies where the level allows it.
cudaError_t launch_superstep_fused(const LevelGeom& g, int order, int s, bool zero_y0, const FusedCoef& cf,
                                   const float* y0, const float* f, float* out, cudaStream_t st,
                                   int tile_rows = 0, bool tma = false);
// s = 2, 3: stage-balanced variant with reflected halos (kernels_superstep.cu).
cudaError_t lean_configure();
cudaError_t launch_superstep_lean(const LevelGeom& g, int order, int s, bool zero_y0, const FusedCoef& cf,
                                  const float* y0, const float* f, float* out, cudaStream_t st, int tile_rows,
                                  bool tma);
// s = 2, 3: one thread per column (kernels_columns.cu).
cudaError_t columns_configure();
bool columns_configured();              // columns_configure has run in the current device's context
cudaError_t launch_superstep_columns(const LevelGeom& g, int order, int s, bool zero_y0, const FusedCoef& cf,
                                     const float* y0, const float* f, float* out, cudaStream_t st);
// Launches of the TMA path that gave up a bounded wait (or found their shared
// memory misaligned) since the library was loaded; each wrote a NaN into its
// output, so the solve that ran it reports a non-finite residual.
unsigned lean_wait_failures();

// ---- coarsest-level solver (kernels_coarse.cu) -----------------------------
struct CoarseParams {
    LevelGeom g;          // homogeneous
    const void* rhs;      // level rhs (T)
    void* u_out;          // result (T)
    const int* sched;     // s per super-step
    int max_ss;
    double tol;           // relative residual stop, 0 = fixed count
    double tau_unit;      // tau_frac * 2 / lambda_max (mu~_j tau = mu_j * tau_unit)
    int* ss_done;         // device int
};
template <typename T>
size_t coarse_smem_bytes(long long n);
template <typename T>
bool coarse_fits(long long n);
template <typename T>
cudaError_t launch_coarse_solve(const CoarseParams& p, cudaStream_t st);
// Raise the dynamic shared-memory limit of the coarse kernels (once per process).
cudaError_t coarse_configure();

// ---- the coarse end of the V-cycle in one cluster launch (kernels_cluster.cu) --
constexpr int kTailMaxS = 32;            // smoothing stages the coefficient table holds
constexpr int kTailMaxLevels = 12;
// Cells up to which every CTA holds a level whole (FP32: four a thread, all that fit).  Solves
// with the line at 64, 512, 1024 and 2560: 24^3 814, 695, 695, 684 us, 32^3 1050, 941, 941, 941,
// 256^2 1847, 1786, 1741, 1738.
constexpr long long kTailWhole = 2560;
// The same in FP64, whose arithmetic is worth splitting over more SMs: at 64, 512 and 2048 16^3
// 2816, 2717, 2722 us, 24^3 2762, 2636, 3801, 256^2 5970, 5602, 5605.
constexpr long long kTailWhole64 = 512;
// FP64: cells of the first level up to which 16 SMs beat a launch per stage on all of them.
// With 4096 cells on the cluster and not: 32^3 3518 and 3852 us; with 8000: 40^3 4517 and 3679,
// 80^3 9930 and 8938; with 13824: 48^3 6327 and 4272, 96^3 13609 and 11524.
constexpr long long kTailCells64 = 4096;
// FP64, the coarsest level alone, whose other way is one SM: on the cluster and not, 22^3 cells
// 5446 and 10216 us, 24^3 6.2 and 10.7 ms.  (28^3 and 32^3 would gain too: 10.5 -> 8.1 ms.)
constexpr long long kTailCoarse64 = 16384;
template <typename T>
constexpr int tail_threads() {           // largest block, by the registers of a thread's cells
    return sizeof(T) == 8 ? 512 : 640;
}
template <typename T>
struct TailLevel {
    int nx, ny, nz;                      // two-dimensional levels: nx x 1 x ny
    int n_pre, n_post;
    T hx, hy, hz, md;                    // 1 / h^2, -2 (hx + hy + hz)
    double tau;
    T omega, inv_cells;
    int split;                           // cut into z slabs over the cluster
    int group;                           // threads that work on it: 0 the whole CTA, 1 four warps, 2 one warp
    int row, fld, buf, f;                // row stride, size of a buffer, offsets of the two buffers and of f
    int scaled;                          // offset of mu~_j tau, gamma~_j tau (j = 1 .. s)
    float inv_nq, inv_ny, inv_pairs;     // 1 / (nx / 2), 1 / ny (two-dimensional: 1), 1 / (nz / 2)
    short first[17];                     // first plane pair of each CTA (split levels)
};
template <typename T>
struct TailParams {
    int nl;                              // levels, finest first
    int per[3];
    int order, s, gsrb;
    T mu[kTailMaxS + 1], nu[kTailMaxS + 1], c0[kTailMaxS + 1];
    double mut[kTailMaxS + 1], gt[kTailMaxS + 1];
    int remove_mean;                     // every axis periodic: f -= mean(f) below the first level
    const int* sched;                    // coarse solve: s per super-step (device)
    int max_ss;
    T tol, tau_unit;                     // relative residual stop (0 = fixed count); mu~_j tau = mu_j tau_unit
    const T* rhs;                        // f of the first level (device)
    T* u_out;                            // its e (device)
    int* ss_done;                        // coarse super-steps done (device int)
    TailLevel<T> lv[kTailMaxLevels];
    // The whole inner loop of a mixed solve in this launch (FP32, the first level is
    // level 0): the loop's state (nullptr: one V-cycle), phi and the carried FP64
    // residual r = f - A phi of level 0, 1 / h^2 in FP64.
    DeviceLoop* loop;
    double* phi;
    double* r64;
    double ihx2, ihy2, ihz2;
    int resident_off;                    // words to the copies of phi and r in shared memory
};
struct TailLaunch {
    int nc, threads;
    size_t bytes;
};
cudaError_t tail_configure();
// Launches of it with a bounded wait that gave up since the library was loaded; each wrote a NaN into its output.
unsigned tail_wait_failures();
// Fills the layout of p.lv (sizes and nl set) and the launch shape; false where
// the levels (and, when p.loop is set, phi and r of the first one) do not fit one
// cluster.
template <typename T>
bool tail_plan(TailParams<T>& p, bool twod, TailLaunch* t);
template <typename T>
cudaError_t launch_tail(const TailParams<T>& p, bool twod, const TailLaunch& t, cudaStream_t st);

}  // namespace sg
