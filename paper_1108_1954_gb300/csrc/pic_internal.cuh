// pic_internal.cuh -- kernel argument blocks and launcher declarations shared
// by the translation units of libpic (not part of the public ABI).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include <nvtx3/nvToolsExt.h>

#include "../../include/pic.h"

namespace pic {

// A named NVTX range over a call of the C ABI, so that a timeline tool shows
// each stage (push, solve, sort, step_n, pool advance, host copies) with its
// kernels and copies; without a tool attached the calls do nothing.
struct TraceRange {
    explicit TraceRange(const char *name) { nvtxRangePushA(name); }
    ~TraceRange() { nvtxRangePop(); }
    TraceRange(const TraceRange &) = delete;
    TraceRange &operator=(const TraceRange &) = delete;
};

constexpr unsigned kFull = 0xffffffffu;   // all lanes of a warp

// Fixed-point deposit: each particle adds exactly 2^24 to the density sum.
constexpr int kFixBits = 24;
constexpr uint32_t kFixOne = 1u << kFixBits;

// Bits of the device error word.
enum : uint32_t {
    kErrPosition = 1u,   // a position outside [0, L) or not finite
    kErrSortKey = 4u,    // a sort key outside the grid
    kErrInput = 8u,      // an uploaded position outside [0, L) (pic_init, pic_set_state)
    kErrWait = 16u,      // a wait ran out (the grid barrier of steps.cu, the CG's sums)
};

// Float32 constants of the push, formed once on the host.  In the float32
// modes a position is kept as its cell coordinate u = x NG / L in [0, NG)
// (cell units: node g sits at u = g + 1/2), so the box end is the exact
// float NG and locating a particle needs no scale factor.
struct PushConsts {
    int ng;          // NG
    float ngf;       // (float)NG, exact: the box length in cell units
    float kdrift;    // (float)(dt NG / L): u advances by v kdrift per step
    float qmdt;      // (float)(qm * dt)
};

// Fused push + fixed-point deposit (or deposit alone when push == false).
struct PushArgs {
    float *x, *v;                 // N each (x: cell coordinates), 16-byte aligned
    long long n;                  // N
    const float *E32;             // field at the nodes, float32 [NG]
    unsigned long long *rho_q;    // fixed-point density accumulator [NG]
    double *partials;             // per-block [sum v_old v_new, sum v_new]
    unsigned int *err;            // device error word
    bool wide;                    // a block may take 2^20 particles or more
    PushConsts c;
};

// Float64 push (PIC_FP64) and float32 push with float32 atomic deposit.
struct PushArgs64 {
    double *x, *v;                // 32-byte aligned
    long long n;
    const double *E64;
    unsigned long long *rho_w;    // density sums in 2^-53: [NG][2], the low 40
                                  // bits of the blocks' sums and the rest
    double *partials;
    unsigned int *err;
    int ng;
    double inv_dx, length, qmdt, dt;
};

struct PushArgsF32Atomic {
    float *x, *v;                 // 16-byte aligned
    long long n;
    const float *E32;
    float *rho_acc;               // sum of float32 weights per node [NG]
    double *partials;
    unsigned int *err;
    int copies;                   // sums per node of a block's tile (set by the launcher)
    PushConsts c;
};

// Per-block share of the step diagnostics.
enum { kDiagFE = 0, kDiagCharge, kDiagModes,
       kDiagFields = kDiagModes + 2 * PIC_NMODES };

// Field solve (one cluster of up to 16 blocks).
struct SolveArgs {
    int mode;                     // PIC_FP32_FIXED / PIC_FP32_ATOMIC / PIC_FP64
    unsigned long long *rho_q;    // FIXED: accumulator (read, then zeroed)
    unsigned long long *rho_q_last; // FIXED: copy of the consumed sums
    float *rho_f32;               // FP32_ATOMIC accumulator
    unsigned long long *rho_w;    // FP64 accumulator, [NG][2]
    double *rho, *phi, *E64;      // outputs [NG]
    float *E32;                   // output copy for the gather [NG]
    const double *partials;       // per-block sums of the push that ran
    int npartials;                // 0: no push ran since the last solve
    pic_diag_row *hist;           // history ring
    int hist_len;
    long long *dstep;             // device step counter
    int ng;
    long long npart_total;        // N
    double k_rho;                 // rho_ion / (N 2^B)
    double k_e;                   // (dx/2) k_rho / NG
    double k_phi;                 // -dx^2 k_rho / NG
    double k_mode;                // 2 / NG: mode amplitude of the mode sums
    double dx;
    double mass;                  // particle mass m = Q0/qm
    unsigned *err;                // device error word (the CG's waits)
    unsigned wait_limit;          // CG: tries of a wait ...
    unsigned wait_missing;        // ... and values it expects beyond those sent (0; tests)
    int solver;                   // PIC_SOLVER_EXACT / PIC_SOLVER_CG
    int cg_maxit;                 // CG: iterations per solve
};

// B by precision mode: a density sum counts 2^-B of a particle.
__host__ __device__ constexpr int density_bits(int mode) {
    return mode == PIC_FP32_FIXED ? kFixBits : mode == PIC_FP32_ATOMIC ? 30 : 53;
}

// The most particles of a density tile whose carries share the counts' words
// (particle_ops.cuh).
constexpr int kCountBits = 20;
constexpr long long kPackedCount = (1ll << kCountBits) - 1;

// Many steps of a fixed-point run in one cooperative launch (steps.cu).
struct StepsArgs {
    float *x, *v;                 // N each, 16-byte aligned
    long long n;
    float *E32;                   // field of the first step in, of the last one out
    double *E64, *phi, *rho;      // of the last step, out
    unsigned long long *rho_q_last; // idem
    unsigned long long *acc;      // [kStepsSlots][NG] density sums ([NG][2] in float64, as rho_w),
                                  // 0 between launches
    double *partials;             // [kStepsSlots][kStepsMaxGrid][2]: per-block push sums (float32
                                  // runs: as pairs of float32, sum and rest)
    unsigned *err;
    unsigned *sync;               // [4], 16-byte aligned: arrivals of the workers, steps
                                  // done by each diagnostics block; never reset ...
    unsigned base[3];             // ... their values before this launch
    unsigned wait_limit;          // polls of a wait
    int diag_blocks;              // 1 or 2: the last of the run's blocks, without particles
    int first_block, blocks;      // the run's part of a pool's grid
    int log_copies;               // copies of a block's tile (set by the launcher)
    pic_diag_row *hist;
    int hist_len;
    long long step0;              // steps taken before this launch
    long long *dstep;             // device step counter
    int steps;
    PushConsts c;
    PushArgs64 d;                 // float64 runs: x, v and the push's constants
    long long weight_total;       // N 2^24 (fixed point)
    double k_rho, k_e, k_phi, k_mode, dx, mass;   // as SolveArgs
};
// Limits of the waits (some seconds, and about one) when the caller sets none.
constexpr unsigned kStepsWaitLimit = 1u << 23, kCgWaitLimit = 1u << 20;
constexpr int kStepsMaxGrid = 256;
constexpr int kStepsSlots = 6;     // accumulators in turn
constexpr int kStepsDiag = 2;      // blocks of a single run's grid without particles, at most
// Two of them write the rows of steps up to kStepsSlots - 1 apart in no fixed
// order, each step its own row and the one before: up to kStepsSlots rows, where
// those can be one slot of the ring, a run has one (us a step with one and two: 2e4
// particles on 64 cells 3.9, 2.8; 1e6 on 1024 7.7, 8.0; 1e6 on 4096 17.7, 12.3).
constexpr int steps_diag_blocks(int hist_len) { return hist_len > kStepsSlots ? kStepsDiag : 1; }
constexpr int kStepsPoolBlock = 1024;
constexpr int kStepsMaxCells = 4096;
// largest runs: up to 2048 cells, and beyond
constexpr int64_t kStepsMaxParticles = 24000000, kStepsMaxParticlesWide = 12500000;
constexpr int64_t kSteps64MaxParticles = 1000000;
cudaError_t steps_prepare(int variant, int ng, int block, bool small, int *per_sm);
cudaError_t launch_steps(StepsArgs a, int variant, int grid, int block, bool small, cudaStream_t s);
cudaError_t steps64_prepare(int ng, int block, int *per_sm);
cudaError_t launch_steps64(const StepsArgs &a, int grid, int block, cudaStream_t s);
cudaError_t steps_pool_prepare(int *per_sm);
int steps_pool_copies();
cudaError_t launch_steps_pool(const StepsArgs *runs, int nrun, int grid, int ng_max, cudaStream_t s);

// Counting sort by cell.
template <typename T>
struct SortArgs {
    const T *x, *v;               // source
    T *x_out, *v_out;             // destination
    long long n;
    int ng;
    T inv_dx;                     // NG / L in the particle precision
    int nchunk;                   // blocks of the count/scatter passes
    long long chunk;              // particles per block
    int nseg;                     // chunk segments of the column scan
    int seg_len;                  // chunks per segment
    unsigned int *hist;           // [nchunk][NG] counts, then offsets
    unsigned int *segtot;         // [nseg][NG] segment totals, then offsets
    unsigned int *base;           // [NG] first slot of each cell
    unsigned int *err;
};

// One run of a batched ensemble (device descriptor; host-built).
struct BatchRun {
    float *x, *v;                 // particles (cell coordinates u), 16-byte aligned
    float *xa, *va;               // the sort's destination (sort_interval > 0)
    int sort_interval;            // S: sort by cell before steps n % S == 0, n > 0
    long long n;                  // N
    PushConsts pc;                // ng, c = NG/L, L, qm dt, dt (float32)
    float *E32;                   // [NG] field of the current step (state)
    double *E64, *phi, *rho;      // [NG] written at the end of a launch
    unsigned long long *rho_q_last;  // [NG] idem
    pic_diag_row *hist;           // history ring of the run
    int hist_len;
    int steps;                    // steps to advance in this launch (0: idle)
    long long *step;              // device step counter of the run
    long long weight_total;       // N 2^24
    double k_rho, k_e, k_phi, dx, mass;
    double k_mode;                // 2 / NG: mode amplitude of the mode sums
};

struct BatchArgs {
    BatchRun *runs;
    const int *order;             // runs to process, largest first
    int nrun;                     // entries of order
    unsigned *next;               // work-queue ticket (0 at launch)
    unsigned *err;                // device error word
    int push;                     // 1: advance `steps`; 0: deposit + solve only
    int ng_max;                   // largest NG of the launch (tile size)
};

// Device-side initial loading (load.cu).
struct LoadArgs {
    float *x, *v;
    long long n;
    double length;
    float lengthf;
    float v0, vth;
    unsigned long long seed;
    int nmodes;
    float k[PIC_LOAD_MAX_MODES], amp[PIC_LOAD_MAX_MODES], phase[PIC_LOAD_MAX_MODES];
};
cudaError_t launch_load(const LoadArgs &a, int sms, cudaStream_t s);
int make_load_args(const pic_loading *ld, long long n, double length, float *x, float *v,
                   LoadArgs *out);

// Internal kernel choice of the fused push for the nearest-grid-point shape
// (not a public deposit variant: PIC_SHAPE_NGP selects it).
constexpr int kDepositNgp = 15;
// The single run's kernels' form of PIC_DEPOSIT_ATOMIC (cell tiles).
constexpr int kDepositCells = 14;

// Phase-space histogram (phase.cu).
constexpr int kPhaseMaxBins = 16384;
template <typename T>
struct PhaseArgs {
    const T *x, *v;
    long long n;
    int nx, nv;
    float sx;             // nx / L
    float vmin, sv;       // nv / (vmax - vmin)
    unsigned *counts;     // [nv][nx]
};
template <typename T>
cudaError_t launch_phase(const PhaseArgs<T> &a, int sms, cudaStream_t s);

// Range check of uploaded positions: sets kErrInput unless every x is in
// [0, L) (phase.cu).
template <typename T>
cudaError_t launch_check_positions(const T *x, long long n, T length, unsigned *err, int sms,
                                   cudaStream_t s);

// Unit conversions of float32 positions (phase.cu), both rounded once from a
// float64 product:
//   to cells     u = (float)((double)x (NG/L)), a u that rounds to NG is 0;
//                sets kErrInput unless x is in [0, (float)L); in place.
//   to physical  x = (float)((double)u (L/NG)), at most the largest float
//                below (float)L.
// The host forms the same two products in pool_to_physical (ensemble.cu).
cudaError_t launch_to_cells(float *x, long long n, double to_cells, float ngf, float length32,
                            unsigned *err, int sms, cudaStream_t s);
cudaError_t launch_to_physical(const float *u, float *x, long long n, double to_phys,
                               float length32, int sms, cudaStream_t s);
// Cell coordinates read back from a caller: every u must lie in [0, NG).
cudaError_t launch_check_cells(const float *u, long long n, float ngf, unsigned *err, int sms,
                               cudaStream_t s);
float below(float v);            // the largest float below v (v > 0)

// Parameter checks shared by the single-run and the pool entry points.
int validate_params(const pic_params *p);

// Launchers (each returns the launch's cudaError_t).
cudaError_t launch_push_fixed(const PushArgs &a, int grid, int block,
                              int variant, int unroll, bool push, cudaStream_t s);
cudaError_t launch_push_f32_atomic(PushArgsF32Atomic a, int grid, int block, bool push,
                                   cudaStream_t s);
cudaError_t launch_push_f64(const PushArgs64 &a, int grid, int block,
                            bool push, cudaStream_t s);
size_t push_smem_bytes(int mode, int ng, bool wide, int block);
bool push_wide_tile(long long n, int sms);
cudaError_t push_prepare_attributes(int mode);
int push_max_blocks_per_sm(int mode, int variant, int unroll, int block, int ng, bool wide);

cudaError_t launch_solve(const SolveArgs &a, cudaStream_t s);
cudaError_t solve_prepare_attributes();

cudaError_t launch_sort_f32(const SortArgs<float> &a, cudaStream_t s);
cudaError_t launch_sort_f64(const SortArgs<double> &a, cudaStream_t s);
cudaError_t sort_prepare_attributes(int ng);
constexpr int kSortThreads = 256;

cudaError_t launch_batch(const BatchArgs &a, int variant, int cluster, int block,
                         int nclusters, cudaStream_t s);
size_t batch_smem_bytes(int ng_max, int cluster, int block);
int batch_max_clusters(int variant, int cluster, int block, int ng_max);
cudaError_t batch_prepare_attributes();

// A launch whose blocks may come up while the kernel ahead of it in the stream
// still runs (programmatic serialisation): the kernel waits where it first reads
// or writes what that one, or any before it, works on
// (cudaGridDependencySynchronize; all before it too, as each such kernel waits
// itself before it ends).  A kernel lets the next one's blocks come up with
// cudaTriggerProgrammaticLaunchCompletion.  The solve does not: a push that comes up
// while the solve's blocks still hold some SMs is spread unevenly where its own
// shape leaves room (2^25 particles, one block of 512 per SM: 166 us a step, 121
// without).  So a push follows as the solve's blocks end, a solve as the push's
// do.  us a step, plain launches and these: from a graph, 2e4 particles on 64 cells
// 12.3, 12.0, 1e6 on 1024 21.6, 20.5; launched one by one, 2e6 on 1024 26.6, 22.3;
// float32 atomic, 2^24 on 1024 68.2, 63.
template <class... P>
cudaError_t launch_after(void (*k)(P...), dim3 grid, int block, size_t smem, cudaStream_t s, int cluster,
                         const P &...args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 0 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

}  // namespace pic
