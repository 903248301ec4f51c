// lks_internal.h -- host-side declarations shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "lks_device.cuh"

namespace lks {

template <typename C>
inline StepParams<C> convert_params(const StepParams<double>& d) {
    static_assert(sizeof(C) == 4, "FP64 steps take the FP64 parameters as they are");
    StepParams<C> o;
    o.nx = d.nx;
    o.ny = d.ny;
    o.N = d.N;
    o.omega_f = (C)d.omega_f;
    o.omega_m = (C)d.omega_m;
    o.src_coef = (C)d.src_coef;
    o.Fx = (C)d.Fx;
    o.B0 = (C)d.B0;
    o.om1f = (C)d.om1f;
    o.om1m = (C)d.om1m;
    o.owf0 = (C)d.owf0;
    o.owf1 = (C)d.owf1;
    o.owf5 = (C)d.owf5;
    o.owm0 = (C)d.owm0;
    o.owm1 = (C)d.owm1;
    o.sw0 = (C)d.sw0;
    o.sw1 = (C)d.sw1;
    o.sw5 = (C)d.sw5;
    o.src3 = (C)d.src3;
    o.coupling = d.coupling;
    const WallCoef<double>* src[2] = {&d.bot, &d.top};
    WallCoef<C>* dst[2] = {&o.bot, &o.top};
    for (int k = 0; k < 2; ++k) {
        dst[k]->r = (C)src[k]->r;
        dst[k]->bc = (C)src[k]->bc;
        dst[k]->kx = (C)src[k]->kx;
        dst[k]->du = (C)src[k]->du;
        dst[k]->U = (C)src[k]->U;
    }
    return o;
}

// Step parameters (relaxation rates, force, field and both walls' closure coefficients) of a
// channel; c = INFINITY selects each closure's perfectly conducting limit.
StepParams<double> make_step_params(int nx, int ny, int closure, double tau_f, double tau_m, double B0, double Fx,
                                    double c_bot, double c_top, double u_bot, double u_top, int coupling = 0);

// Threads per block of the FP64 step kernels.  An FP64 warp instruction holds its SM sub-partition's
// FP64 unit for 64 clocks, so warps that share a sub-partition add up: a 4 x 65 channel took 9.8 us of
// FP64 work a step as 2 blocks of 256 (4 warps deep on 2 SMs).  Blocks of 64 put one or two warps on
// an SM as long as every SM gets one block at most; blocks of 128 have one warp per sub-partition.  With
// them and the shorter collision: 4 x 65 channel 12.7 -> 5.2 us a step, 128 x 128 duct 28.7 -> 14.3;
// large lattices take the same time with blocks of 64, 128 and 256.
inline unsigned block_f64(int64_t N) { return N <= 152 * 64 ? 64 : 128; }

// Threads per block of the FP32 and 16-bit step kernels, for `items` (nodes, or words of two nodes) a row with a
// grid row to each, or for `items` in one flat row.  256 for large lattices; smaller blocks where they pad a row
// less, or where 256 would leave SMs without a block (us a step, 256 / 128 / 64 threads: FP16 280 x 447 4.15 / 4.33 /
// 3.69, 300 x 1200 8.93 / 8.88 / 7.08, BF16 85 x 798 3.75 / 2.63 / 2.82, 126 x 287 2.54 / 2.20 / 2.25, FP32
// 360 x 360 3.56 / 3.29 / 3.19, 1000 x 513 8.18 / 8.16 / 8.26).
inline unsigned block_f32(int64_t items, int64_t rows) {
    auto padded = [&](int64_t b) { return (items + b - 1) / b * b; };
    const int64_t best = padded(64);
    if (rows * items >= (int64_t)1 << 21 && padded(256) * 16 <= best * 17) return 256;
    return padded(128) * 16 > best * 17 || rows * padded(128) / 128 < 4 * 152 ? 64 : 128;
}

// Do the FP32 and 16-bit step kernels take a grid row to each row of `items` (nodes, or words of two nodes), or the
// flattened index?  The latter costs a division but no idle lanes, and its own-node loads and its stores stay
// aligned where rows do not start on a 32-byte sector (us a step, grid rows / flat: FP32 132 x 2800 8.6 / 7.3,
// 270 x 900 5.9 / 5.4, 777 x 555 9.3 / 8.8, in place 1001 x 800 14.8 / 13.5, BF16 270 x 1200 7.7 / 6.3; where they do:
// FP32 96 x 3000 5.7 / 6.1, 520 x 700 7.1 / 7.3).  Large lattices keep grid rows (BF16 in place 1001 x 3000 44.5 /
// 55.2, FP16 1500 x 1500 27.5 / 29.4), and so do wide rows, few of which end with the moment closure's long wall row
// (FP32 2500 x 75 4.97 / 5.35, 3001 x 60 5.20 / 5.39).
inline bool rows2d(int items, int ny, int64_t N) {
    return items >= 64 && ny <= 65535 && (items % 8 == 0 || items >= 1024 || N >= (int64_t)1 << 21);
}

// Bytes per stored population for each lks_storage value.
inline size_t storage_bytes(int storage) { return storage == 0 ? 8 : (storage == 1 ? 4 : 2); }

// Storage order of a single lattice's populations: an in-place handle with 16-bit storage and even
// nx keeps every row interleaved for its two-nodes-per-thread kernels (32-bit word w holds nodes
// x = w and x = w + nx/2, so a shift by one node is a shift by one word); the value is the row
// length the readout kernels need (0: plain node order, all other handles).
inline int interleave_row(int storage, int nx, int inplace) {
    return (inplace && storage >= 2 && (nx % 2) == 0) ? nx : 0;
}

// The staged 16-bit steps (lks_step_staged.cu): rows staged through shared memory by bulk copies.
// They apply to 16-bit storage with nx a multiple of 8 and nx >= 1024: the whole step of a
// two-buffer handle, phase 0 of an in-place handle's pair of steps.  err is a device word set when
// one of their bounded waits runs out, grid the number of resident blocks.
struct StagedStep {
    int* err;
    unsigned grid;
};
bool staged_step_applies(int storage, int nx, int inplace);
// Opt the storage type's staged kernels (two-buffer or in-place) into their shared memory (before any
// graph capture) and return the grid that keeps one wave of blocks resident.
cudaError_t prepare_staged_step(int storage, int inplace, unsigned* grid);
// One warp that waits at most limit_ns on an mbarrier nothing completes, then sets *err (self-test of
// the bounded waits of the staged kernels).
cudaError_t launch_wait_timeout_probe(int* err, uint64_t limit_ns, cudaStream_t st);

cudaError_t launch_step_staged(int storage, int closure, const void* fin, const void* gin, void* fout, void* gout,
                               const StepParams<float>& p, const StagedStep& ss, cudaStream_t st);
cudaError_t launch_step_aa_staged(int storage, int closure, void* f, void* g, const StepParams<float>& p,
                                  const StagedStep& ss, cudaStream_t st);

// One fused step: (fin, gin) -> (fout, gout) on stream st; with ss, 16-bit storage takes the staged
// kernel where it applies.
cudaError_t launch_step(int storage, int closure, const void* fin, const void* gin, void* fout, void* gout,
                        const StepParams<double>& p, cudaStream_t st, const StagedStep* ss = nullptr);
// In-place (one-buffer) step, phase 0 or 1 of a pair (lks_aa.cuh); f, g are the single buffers.
cudaError_t launch_step_aa(int storage, int closure, int phase, void* f, void* g, const StepParams<double>& pd,
                           cudaStream_t st, const StagedStep* ss = nullptr);

// kRowSteps fused steps per pass over memory (lks_step_rows.cu): FP32 and 16-bit storage.  kRowSteps is odd,
// so that a fused pass of a two-buffer handle moves the state to the other buffer as that many single steps do.
// strip: columns per block (words of two nodes for 16-bit storage), 0 where the kernel does not apply; chunk: rows
// per block; edge: rows of the blocks at the bottom wall (at the top wall: what is left).
constexpr int kRowSteps = 3;
struct RowsPlan {
    int strip, chunk, edge;
};
cudaError_t plan_rows(int storage, int closure, const StepParams<double>& p, int inplace, RowsPlan* rp);
// In place (fin = fout; FP32): `work` holds rows_workspace() bytes; null for two buffers.
size_t rows_workspace(int nx, int ny, const RowsPlan& rp);
cudaError_t launch_rows(int storage, int closure, const void* fin, const void* gin, void* fout, void* gout,
                        const StepParams<double>& pd, const RowsPlan& rp, void* work, cudaStream_t st);

// Small lattices held in one cluster's shared memory for all steps of a call (lks_resident.cu).  ctas: 0
// where it does not apply.  fin / fout: the buffers before and after `steps` steps (they may be the same);
// ilv as interleave_row.
constexpr int kResidentThreads = 1024;  // FP64: half
// Most nodes: above these single steps on all SMs are faster (us a step, resident against single: FP32 64 x 120
// 1.17 / 1.41, 64 x 190 1.44 / 1.40; BF16 96 x 96 1.41 / 2.2).  For FP64 also most nodes of a CTA, which with fewer
// rows than 16 are more than a 16th of the lattice: from 129 on two warps share a sub-partition (link closure: 8 x 256,
// 128 a CTA, 4.73 / 4.98, 128 x 16 5.02 / 4.96; 7 x 289, 133, 6.44 / 5.28, 200 x 8, 200, 8.13 / 5.05, 160 x 3, 320,
// 11.2 / 4.9).  FP32 and 16-bit CTAs of few wide rows meet the shared-memory limit first (250 x 8 1.17 / 1.70).
constexpr int64_t kResidentNodesF64 = 2048, kResidentNodesF32 = 10240, kResidentNodes16 = 12288;
constexpr int kResidentCtaNodesF64 = 128;
constexpr int kResidentQuads = 2;  // groups of 32 nodes a CTA, four warps each (FP64, Maxwell coupling)
struct ResidentPlan {
    int ctas, threads, rows_max, quads, least;
    size_t smem;
};
// Fewest steps of a call that are taken in the cluster: starting it, loading the bands and storing them takes 12 us
// and more, and a step there saves less over one on all SMs the more nodes there are.  us a call, resident / single
// steps (in brackets: the least):
//   FP32 4 x 65 (12) 8 steps 20.6 / 16.5, 12 steps 22.7 / 26.7; 16 x 128 (16) 16 steps 28.8 / 26.7, 20 steps 30.9 /
//   35.0; 64 x 64 (28) 20 steps 35.0 / 32.9, 32 steps 45.3 / 47.2; 64 x 128 (79) 64 steps 92.3 / 90.3, 96 steps 129 /
//   137; 16-bit 64 x 128 (28) 16 steps 39.1 / 34.9, 20 steps 43.2 / 45.2; 110 x 110 (48) 32 steps 80.0 / 73.5, 48 steps
//   109 / 111; FP64 4 x 65 (4) 2 steps 18.6 / 12.5, 4 steps 22.7 / 22.7; 4 x 257 (14) 8 steps 46.3 / 43.1, 12 steps
//   62.7 / 67.7; 8 x 256 (45) 32 steps 168 / 162, 48 steps 243 / 244.
inline int resident_least(int storage, int64_t N) {
    const int64_t n2 = N * N;
    return (int)(storage == 0 ? 4 + n2 / 100000 : 12 + n2 / (storage == 1 ? 1000000 : 4000000));
}
cudaError_t plan_resident(int storage, int closure, int coupling, int nx, int ny, ResidentPlan* rp);
cudaError_t launch_resident(int storage, int closure, const void* fin, const void* gin, void* fout, void* gout,
                            const StepParams<double>& pd, const ResidentPlan& rp, int ilv, int steps, cudaStream_t st);

// Initial equilibrium state (deviation form) with the counter-based perturbation.
cudaError_t launch_init(int storage, void* f, void* g, int nx, int ny, double B0, uint64_t seed, double amp,
                        cudaStream_t st, int ilv = 0);

// Moments of a stored state: out[m*N + n] (what = 0) or x-averaged profiles out[m*ny + j] (what = 1).
// coupling / tau_m: the moment model of the state (0: Maxwell stress; 1: Lorentz force, which needs tau_m).
cudaError_t launch_moments(int storage, const void* f, const void* g, int nx, int ny, double B0, double Fx,
                           int what, double* out, cudaStream_t st, int coupling = 0, double tau_m = 1.0,
                           int ilv = 0);

// The device address of the host array at p if conversion kernels may access it directly (page-locked
// memory, LKS_HOST_STAGING unset or "0"); nullptr otherwise.
void* host_direct_ptr(const void* p);

// Per-node moments of the M nodes n0 .. n0+M-1 of an N-node state: out[m*M + i] for node n0 + i.
cudaError_t launch_node_moments(int storage, const void* f, const void* g, int64_t N, int64_t n0, int64_t M,
                                double B0, double Fx, double* out, cudaStream_t st, int coupling = 0,
                                double tau_m = 1.0, int ilv = 0);

// Residual partial sums: nblk blocks write partial[4*blk + k] = (sum du^2, sum u^2, sum db^2, sum b^2)
// and refresh the snapshot snap[0..N) = u_x, snap[N..2N) = B_x; then one block reduces in fixed order
// into out[0..4), device or page-locked host memory.  residual_blocks(N) never exceeds kResidualMaxBlocks
// (8 blocks per SM on 152 SMs).
constexpr int kResidualMaxBlocks = 1216;
int residual_blocks(int64_t N);

// Steady-state bookkeeping shared by lks_run_to_steady, lks3_run_to_steady and the batch engine.
// A run is STALLED when its residual has not reached a new minimum for kStallChecks checks in a row
// while already below the rounding floor of the storage type (1e-12 FP64, 1e-4 FP32, 1e-2 16-bit);
// the long window keeps slowly converging runs (residual falling by well under 1 % per check and
// jittering) from being stopped early.
constexpr int kStallChecks = 1000;
inline double stall_floor(int storage) { return storage == 0 ? 1e-12 : (storage == 1 ? 1e-4 : 1e-2); }
// A residual of exactly 0 means that u_x and B_x did not change by one bit over a whole check
// interval.  On a channel driven by a body force or a moving wall, with FP32 or 16-bit storage, that
// is the state stagnating because the per-step increments fell below the resolution of the stored
// deviations -- not convergence: the profile can be far from the steady solution.  It is reported as
// a stall.  (FP64's resolution is far below any tolerance a caller can ask for, and an undriven
// channel has no increment to lose.)
inline bool zero_residual_is_stall(int storage, double Fx, double u_bot, double u_top) {
    return storage != 0 && (Fx != 0.0 || u_bot != 0.0 || u_top != 0.0);
}
cudaError_t launch_residual(int storage, const void* f, const void* g, int nx, int ny, double B0, double Fx,
                            double* snap, double* partial, double* out, cudaStream_t st, int coupling = 0,
                            double tau_m = 1.0, int ilv = 0);
cudaError_t launch_snapshot(int storage, const void* f, const void* g, int nx, int ny, double B0, double Fx,
                            double* snap, cudaStream_t st, int coupling = 0, double tau_m = 1.0, int ilv = 0);

// FP64 absolute populations <-> stored deviations, for the nodes n0 .. n0 + M - 1 of an N-node lattice;
// fabs / gabs hold those nodes in planes of stride M (9 and 10 planes).
cudaError_t launch_to_abs(int storage, const void* f, const void* g, int64_t N, int64_t n0, int64_t M, double B0,
                          double* fabs, double* gabs, cudaStream_t st, int coupling = 0, int ilv = 0);
cudaError_t launch_from_abs(int storage, const double* fabs, const double* gabs, int64_t N, int64_t n0, int64_t M,
                            double B0, void* f, void* g, cudaStream_t st, int coupling = 0, int ilv = 0);

}  // namespace lks
