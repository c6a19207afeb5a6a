// ade_internal.h -- types shared by the host entry points and the kernels of libade_sph.so.
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include "../../include/ade_sph.h"
#include "pool.h"

struct ade_ctx;

namespace ade {

constexpr int kMaxSubdiv = 6;                                   // cells per support radius
constexpr int kMaxRows = (2 * kMaxSubdiv + 1) * (2 * kMaxSubdiv + 1);
constexpr int kRateThreads = 128;                              // direct variant
constexpr int kTileThreads = 256;                              // tiled variant
constexpr int kMaxCellBits = 24;                                // ncells <= 2^24
constexpr int kScanTileCells = 2048;                            // cells per scan block (cells.cu)
constexpr int kGraphSteps = 32;                                 // steps captured in ade_run's long graph

// Programmatic dependent launch (griddepcontrol, sm_90 and later).  A kernel launched by
// launch_pdl may have its CTAs scheduled while the kernel before it on the stream is still
// running; it calls pdl_wait() before its first access to memory that earlier work on the stream
// writes or reads (the wait returns once those grids have completed and their writes are visible;
// without a programmatic predecessor it returns at once), then pdl_trigger(), which lets the next
// kernel's CTAs be scheduled once every CTA of this grid has started.  The cell-build kernels and
// the statistics fold start with both calls, so each launch gap overlaps the tail of the previous
// kernel and no data dependency changes.  The rate kernels only wait: when their grid fits in one
// wave an early trigger would park the next launch's CTAs, waiting, beside them for the whole
// launch (measured up to 15 us slower per step at 512^2); the implicit trigger at completion
// still hides the launch gap.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, unsigned block, size_t smem, cudaStream_t s,
                       Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Origin of the cell grid of a build, in fixed-point words.  Steps of a uniform flow build their
// cells in a frame that moves with the particles (origin = steps taken x the drift per step), so a
// particle stays in its cell, and a run gives the same bits wherever it is split into calls and
// whether the list is rebuilt or kept for a call's next steps.  words[0..2]: the next build's
// origin; words[4..6]: the last build's.  A build moves words[0..2] to words[4..6] and advances
// words[0..2] by adv.  words NULL: origin `add` (0: the absolute grid).  A batch holds kFrameWords
// words per plume, advanced by `steps` times the plume's drift per step (corr[p].inc).
struct RateParams;
struct CellFrame {
    uint32_t *words = nullptr;
    uint32_t adv[3] = {0u, 0u, 0u};
    uint32_t add[3] = {0u, 0u, 0u};
    const RateParams *corr = nullptr;
    int plumes = 0;
    uint32_t steps = 0u;
};
constexpr int kFrameWords = 8;

// One row of the neighbour-cell stencil: cells (cx - w .. cx + w, cy + dy, cz + dz).
struct StencilRow {
    signed char dy, dz, w, pad;
};

// Everything the interaction kernel needs, passed by value (kernel parameter space).
// Lengths are in fixed-point units of the x axis (L_x / 2^32).
struct RateParams {
    int n;
    int ncx, ncy, ncz;
    int nrows;
    StencilRow rows[kMaxRows];
    float H2;        // support radius squared
    float Hg2;       // squared radius the cell grid is built for (velocity-field mode: H + skin)
    float invH;      // 1 / support radius
    float sy, sz;    // L_y / L_x, L_z / L_x (1 for a cubic box)
    // Pair factor of Eq. 5 for the uniform tensor of Eq. 3 (K = 2D): Dcal = a (vhat . e)^2 + b with
    // e = x_ab / r, a = 2 Gamma (alpha_L - alpha_T)|v|, b = 2 (Gamma - dim) d_T - 2 (alpha_L - alpha_T)|v|,
    // d_T = alpha_T |v| + D_m.  The walks evaluate t = (uw . x_ab) / r with uw = sqrt(|a|) vhat and
    // Dcal' = t^2 + ub, ub = sign(a) b, so Dcal = sign(a) Dcal'; the sign is folded into upf.
    float uw[3];
    float ub;
    float upf;       // sign(a) * pf
    float pf;        // 1/2 (m / rho) * kernel prefactor of W'(r)/r
    float dt;        // step length used by the epilogue
    uint32_t inc[3]; // fixed-point position increment used by the epilogue
    uint32_t back[3];// evaluation position minus cell-build position (0, or the half-step drift)
    int variant;     // 0 = direct walk (branch-free), 1 = shared-memory tiles, 2 = direct walk
                     // branching on the support test, 3 / 4 = 0 / 2 with per-particle trimmed rows,
                     // 5 / 6 / 7 / 8 = 0 / 3 / 2 / 4 with two targets per thread (packed FP32x2)
    int k;           // halo width in cells (cells per support radius)
    int tx, ty, tz;  // target cells per tile
    int ntx, nty, ntz;  // tiles per axis
    int cap;         // staged-particle capacity of a tile
    double u[3];     // FP64 length of one fixed-point unit per axis (L_i / 2^32)
    double H2d;      // FP64 support radius squared (pair counting decides support in FP64)
    unsigned fz_base, fz_stride, fz_regions;   // weight table: first line, lines of a chunk's region (0: no
                     // table) and chunks that have one (FrozenTab)
    int goff;        // batched plumes: first particle (caller and sorted order) of this plume
    int coff;        // batched plumes: first cell of this plume in the global cell table
    int m1;               // -1: the multiplier of the walks' separations (see sep in rate_common.cuh)
    const uint32_t *frame;   // cell frame of the last build (CellFrame words; NULL: the absolute grid)
    const uint4 *pencil;  // trimmed walks: per pencil (cy, cz) the transverse bounding box
                          // {min y, max y, min z, max z} of its particles at the cell build
};

// Velocity-field mode: per-particle velocities (Eq. 1) and tensors (Eq. 3).
struct FieldParams {
    double aL, aT, Dm;       // Eq. 3 coefficients (the per-particle D is formed in FP64)
    float gamma;             // Gamma of Eq. 5
    float pconv;             // (m / rho) kc L_x / 2^32: convective prefactor (x_ab in x-axis units)
    double vscale[3];        // dt / L_i * 2^32: fixed-point drift per unit velocity over one step
};

// Per-particle field records of velocity-field mode (workspace).  v is constant in time, so the
// records are formed once per field (or dispersivity change) in the caller's order and only
// permuted into the cell-sorted order after each cell build:
//   2D: V = {vx, vy, 0, 0},          DA = {Dxx, Dxy, Dyy, lo(Dxy)}
//   3D: V = {vx, vy, vz, lo(Dxz)},   DA = {Dxx, Dxy, Dxz, lo(Dxy)}, DB = {Dyy, Dyz, Dzz, lo(Dyz)}
//   Inc = {hx, hy, hz, c}: fixed-point half-step drift h_i = round(v_i dt/2 / L_i 2^32) and the
//   full-step drift round(v_i dt / L_i 2^32) = 2 h_i + c_i, c_i in {-1, 0, 1} packed as 2-bit
//   fields (c_i + 1) << 2i.
struct FieldWork {
    float4 *Vc, *DAc, *DBc;  // [n] caller order (DBc: 3D only)
    uint4 *IncC;             // [n] caller order
    float4 *V, *DA, *DB;     // [n] cell-sorted order
    uint4 *Inc;              // [n] cell-sorted order
    unsigned *vmax_bits;     // max |v_a| as FP32 bits (ade_set_velocity_field)
};

// Parameter sweep (sweep.cu): one group of up to kSweepGroup parameter sets per launch.
constexpr int kSweepGroup = 8;
constexpr int kSweepMax = 64;     // parameter sets per sweep
struct SweepParams {
    float vh[3];                  // unit vector of the uniform velocity (x axis when v = 0)
    float g2, bT;                 // 2 Gamma, 2 (Gamma - d) + 2
    int g0;                       // first set of the group
    int nt;                       // sets in the group: 1, 2, 4 or 8
    float dL[kSweepGroup];        // alpha_L |v| + D_m and alpha_T |v| + D_m per set (0 beyond nt)
    float dT[kSweepGroup];
};

struct SweepOut {
    float *rate;                  // single evaluation: [P][n] caller order (may be NULL)
    float *Cout;                  // on-the-fly predictor: sorted half-step concentrations
    float *C;                     // final state: caller concentrations [P][n]
    uint32_t *xq;                 // final state: caller positions
    int *status;                  // set to 1 on a non-finite C
    unsigned long long *pairs;    // pair counter (counting launch)
};

// Weight table of the evaluations over one cell list (rate_frozen.cu), in lines of 32 words: a region of
// RateParams::fz_stride lines for each of the first fz_regions chunks from RateParams::fz_base on, and from line `pool` on `cap` lines
// that an atomic cursor hands out to chunks that outgrow theirs; slots: two words of 16 bytes per chunk
// number (put_chunk in frozen_table.cuh).
constexpr int kFrozenThreads = 128;
// Numbers given to the chunks of n particles in np pencils (find_chunk in frozen_table.cuh), and from how many
// on they are counted (launch_chunk_numbers).  Without the count one number per pencil may belong to no chunk,
// and the warps that get them idle in their block: on a chip that is full (a wave: 152 SMs of 48 warps) they
// cost what their share of the warps is (per step: 128^3, four chunks and a gap per pencil, 989 us against
// 955; 57^3 190 against 160), on less they cost nothing and the launch would (2 us a call).
__host__ __device__ inline int chunk_numbers(int n, int np) { return (n >> 5) + np; }
constexpr int kCountChunksFrom = 152 * 48;
struct FrozenTab {
    float *words;
    uint4 *slots;
    unsigned long long *cursor;
    unsigned pool, cap;
    uint32_t *dense;       // chunks before each pencil (launch_chunk_numbers; NULL: numbers with gaps)
    float *low;            // plane of low parts, half as many lines (the adjoint's table)
};
// Lines that a set's chunks need, counted by size: two bins per octave.
struct ChunkBin {
    unsigned count, most;
    unsigned long long sum;
};
constexpr int kChunkBins = 64;
// How a table is divided: `lines` hold every chunk, `regions` of them `stride` lines each and the others in the pool.
struct TablePlan {
    unsigned stride, regions;
    size_t lines;
};
// Concentrations (and Eq. 14's flux) of such a run in sorted order: C at level l, Ch at l + 1/2, each
// pencil's twice back to back ([2n] words).
struct FrozenState {
    float *C, *Ch;
    float *Q;             // Eq. 14: caller order (read by the build, written by the finish); NULL: Eq. 1
    float *Qs, *Qh;       // sorted, at l and l + 1/2
    float tau_inv;
};

// Batched plumes: chunk number `chunk` of one plume; its slot is the item's index.
struct FrozenItem {
    int plume, chunk;
};

// Steps of one sweep call: sorted positions, cell table, weight table, concentrations (planes of
// four sets, doubled per pencil) at levels l and l + 1/2, and the constants of the table's weights.
struct SweepRun {
    const uint4 *P;
    const uint32_t *cs, *perm;
    FrozenTab tab;
    float *C, *Ch;
    float g2, bT;                 // as in SweepParams
};

// One work item of the batched rate kernel: `count` sorted particles of plume `plume` starting
// at plume-local sorted index `start`.
struct BatchTile {
    int plume, start, count, pad;
};

// Outputs of the fused epilogues.
struct EpiOut {
    float *rate;              // EPI_RATE: dC/dt in caller order
    uint4 *Pout;              // EPI_PREDICT: sorted half-step state
    uint32_t *xq;             // EPI_CORRECT: caller state, updated in place
    float *C;                 // EPI_CORRECT
    float4 *wpart;            // EPI_CORRECT: per-warp {sum C as FP32 hi + lo, min C, max C}
    int *status;              // EPI_CORRECT: set to 1 on a non-finite C
    unsigned long long *pairs; // optional in-support pair counter
    float *Q;                 // Eq. 14 (NULL: Eq. 1): flux dC/dt in caller order, updated by the corrector
    float *Qh;                // Eq. 14: sorted half-step flux (predictor writes, corrector reads)
    float tau_inv;            // Eq. 14: 1 / tau
};

enum Epilogue { EPI_RATE = 0, EPI_PREDICT = 1, EPI_CORRECT = 2 };

// Device buffers carved out of the caller's workspace.
struct Work {
    uint32_t *keys;        // [n] cell key per caller particle
    uint32_t *rank;        // [n] provisional rank inside the cell
    uint32_t *count;       // [ncells] particles per cell
    uint32_t *block_sums;  // [scan blocks]
    uint32_t *perm_tmp;    // [n] provisional cell-sorted permutation
    uint32_t *perm;        // [n] caller index at each sorted position
    uint32_t *cell_start;  // [ncells + 1]
    uint4 *P0;             // [n] sorted {x, y, z, C} at level l
    uint4 *P1;             // [n] sorted state at level l + 1/2
    uint4 *pencil = nullptr;  // [ncy * ncz] transverse bounding boxes of the pencils (NULL: not built)
    uint32_t *frame = nullptr;                 // CellFrame words of the steps (NULL: absolute grid)
    uint32_t *tile_sums = nullptr;             // [tiles of 4096 cells, 128 B apart] totals for the one-pass scan
                                               // (k_count adds, k_place clears; null: multi-launch scan)
    double *partials;      // per-block reduction partials (state statistics)
    float4 *wpart;         // per-warp partials of the corrector (EpiOut::wpart)
    double *stats;         // {sum C, min C, max C, -, closed-form slots}
    double *cf_partials;   // closed-form error partials
    int *status;           // non-finite flag
    unsigned long long *pairs;
};

// NVTX range for the duration of a host call (visible in Nsight timelines; no cost without a tool).
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// Records msg as the calling thread's last error (read by ade_last_error) and returns code.
int report_error(int code, const char *msg);

// The interaction walks' form of Eq. 5's pair factor for the tensor of Eq. 3 (RateParams uw, ub, upf;
// pf must be set first).
void rate_pair_consts(int dim, double gamma, const double *v, double alpha_L, double alpha_T, double D_m,
                      RateParams *rp);

// Launchers (cells.cu, rate.cu, reduce.cu).  All return cudaGetLastError() of the launches.
int scan_blocks(int m);
// Kernel launches of one launch_build_cells (the scan takes one launch with look-back flags, else
// two, or three on large grids).
int tile_blocks(int m);          // tiles of the one-pass scan
size_t tile_sums_bytes(int m);   // their totals (one 128-byte line each)
int cell_build_launches(int n, int ncells, bool onepass);
// count_zero: w.count[0, ncells) is known to be zero (every build leaves it zero), so the memset
// that otherwise starts the build is skipped.
cudaError_t launch_build_cells(int dim, const uint32_t *xq, const float *C, int n, const int *nc,
                               int ncells, const Work &w, cudaStream_t s, bool count_zero = false,
                               const CellFrame &frame = CellFrame());
// Positions of the last build (its sorted records), in the caller's order and moved by add, into xq [dim][n].
cudaError_t launch_build_positions(const uint4 *P, const uint32_t *perm, int n, int dim, const uint32_t *add, uint32_t *xq,
                                   cudaStream_t s);
// Writes a CellFrame's words: the next build's origin, and the last build's.
cudaError_t launch_set_frame(uint32_t *words, const uint32_t *origin, cudaStream_t s);
// Batched plumes: keys are coff_p + local key; plume_of[i] gives the plume of caller particle i.
cudaError_t launch_build_cells_batch(int dim, const uint32_t *xq, const float *C, int n, int ncells,
                                     const RateParams *descs, const uint16_t *plume_of,
                                     const Work &w, cudaStream_t s, const CellFrame &frame);
// paired: the persistent kernel's threads take two adjacent sorted particles (the paired walk).
cudaError_t launch_rate_batch(int dim, int kernel, int epi, const uint4 *Pe, const uint32_t *cell_start,
                              const uint32_t *perm, const RateParams *descs, const BatchTile *tiles,
                              int ntiles, unsigned *queue, int grid, const EpiOut &out, cudaStream_t s,
                              bool paired = false);
cudaError_t launch_batch_stats(const float *C, const int *offsets, int nplumes, double *stats,
                               cudaStream_t s);
cudaError_t launch_rate(int dim, int kernel, bool iso, int epi, const uint4 *Pe, const uint4 *Pc,
                        const uint32_t *cell_start, const uint32_t *perm, const RateParams &prm,
                        const EpiOut &out, cudaStream_t s);
// Fixed-order fold of the corrector's m per-warp partials into stats[0..2] = {sum C (FP64),
// min C, max C}: one thread-block cluster of up to kFoldMaxCtas CTAs (reduce.cu).
constexpr int kFoldMaxCtas = 8;
cudaError_t launch_fold_warp_partials(const float4 *wpart, int m, double *stats, cudaStream_t s);
cudaError_t launch_closed_form_error(int dim, const uint32_t *xq, const float *C, int n,
                                     const double *box, const double *center, const double *Sinv,
                                     double amp, double C0, double vol, int nimg,
                                     double *partials, int nblocks, double *out, cudaStream_t s);

cudaError_t launch_state_stats(const float *C, int n, double *partials, double *stats, cudaStream_t s);

// Velocity-field mode (rate_field.cu).
// Caller-order records from v [dim][n] (vx, vy, vz into Vc; v_dev may be NULL to re-form the
// tensors from the velocities already in Vc), and max |v| into fw.vmax_bits when v_dev is given.
cudaError_t launch_field_records(int dim, const float *v_dev, int n, const FieldParams &fp, const FieldWork &fw,
                                 cudaStream_t s);
// Sorted records: V[i] = Vc[perm[i]] (and DA, DB).
cudaError_t launch_field_permute(int dim, const uint32_t *perm, int n, const FieldWork &fw, cudaStream_t s);
// Paired walks (variants 5-8; rate_pair.cu), called by launch_rate.
cudaError_t launch_rate_pair(int dim, int kernel, int epi, bool iso, const uint4 *Pe, const uint4 *Pc,
                             const uint32_t *cs, const uint32_t *perm, const RateParams &prm, const EpiOut &out,
                             cudaStream_t s);
// Partials the velocity-field corrector writes.
int field_partials(int dim, const RateParams &prm);
cudaError_t launch_rate_field(int dim, int kernel, int epi, const uint4 *Pe, const uint32_t *cell_start,
                              const uint32_t *perm, const FieldWork &fw, const RateParams &prm,
                              const FieldParams &fp, const EpiOut &out, cudaStream_t s);

// Blocks of the table's kernels (kFrozenThreads threads): a warp per chunk number.
unsigned frozen_blocks(const RateParams &prm);
// dense[p] = chunks of the pencils before p, p = 0..np (nothing where dense is NULL).
cudaError_t launch_chunk_numbers(const uint32_t *cs, const RateParams &prm, uint32_t *dense, cudaStream_t s);
// Slots of a table, enough for every grid the context may switch to.
size_t table_slots(const ade_ctx *c);
// The plan of a table with `val` words per pair (`lines` 0: above the limit; then `stride` is that of the whole table
// all the same): counted for the current positions (waits for the stream; the limit is kTableMaxBytes), or the
// estimate for an even set (host only; kEstimateMaxBytes).
int plan_context_table(ade_ctx *c, int val, bool counted, TablePlan *plan, cudaStream_t s);
constexpr double kTableMaxBytes = 16e9, kEstimateMaxBytes = 4e9;
// Division of `lines` lines (fz_base, fz_stride, fz_regions, pool, cap).
void divide_table(const TablePlan &plan, size_t lines, RateParams *rp, FrozenTab *tab);
// Cell build of the current positions in the steps' moving frame.
int framed_cells(ade_ctx *c, cudaStream_t s);
// Adds the lines that every chunk needs to bins[kChunkBins]; batch: items [first, last), bins of the plumes from
// that of the first item on.
cudaError_t launch_chunk_need(int dim, bool iso, const uint4 *P, const uint32_t *cs, const RateParams &prm, int val,
                              ChunkBin *bins, cudaStream_t s);
cudaError_t launch_chunk_need_batch(int dim, const uint4 *P, const uint32_t *cs, const RateParams *descs, const FrozenItem *items,
                                    int first, int last, ChunkBin *bins, cudaStream_t s);
// Evaluations over one cell list with stored weights (rate_frozen.cu): the table, one predictor or
// corrector (prm.dt), and the final state in the caller's order (prm.inc: the drift of all steps).
cudaError_t launch_frozen_build(int dim, int kernel, bool iso, const uint4 *P, const uint32_t *cs, const uint32_t *perm,
                                const RateParams &prm, const FrozenTab &tab, const FrozenState &st, cudaStream_t s);
cudaError_t launch_frozen_rate(int dim, int kernel, bool iso, int epi, const uint4 *P, const uint32_t *cs,
                               const RateParams &prm, const FrozenTab &tab, const FrozenState &st, cudaStream_t s);
cudaError_t launch_frozen_finish(int dim, const uint4 *P, const uint32_t *cs, const uint32_t *perm, const RateParams &prm,
                                 const FrozenTab &tab, const FrozenState &st, const EpiOut &out, cudaStream_t s);

// The same for a batch: the table and the first predictor (build), or one evaluation.
cudaError_t launch_frozen_batch(int dim, int kernel, int epi, bool build, const uint4 *P, const uint32_t *cs,
                                const RateParams *descs, const FrozenItem *items, int nitems, const FrozenTab &tab,
                                const FrozenState &st, cudaStream_t s);
cudaError_t launch_frozen_finish_batch(int dim, const uint4 *P, const uint32_t *cs, const uint32_t *perm, int n,
                                       const RateParams *descs, const uint16_t *plume_of, uint32_t steps,
                                       const FrozenTab &tab, const FrozenState &st, const EpiOut &out, cudaStream_t s);

// Parameter sweep (sweep.cu): the table and the sorted concentrations (doubled pencils), one predictor or
// corrector of a group (prm.dt; out.C set: the call's last corrector, prm.inc the drift of all steps); and
// for short calls the gather and one evaluation with the geometry on the fly.
cudaError_t launch_sweep_table(int dim, int kernel, bool iso, const SweepRun &r, const RateParams &prm, const float *C,
                               int sets, int P4, cudaStream_t s);
cudaError_t launch_sweep_pass(int dim, int kernel, bool iso, int epi, const SweepRun &r, const SweepParams &sp,
                              const RateParams &prm, const SweepOut &out, cudaStream_t s);
cudaError_t launch_sweep_gather(const uint32_t *perm, const float *C, int n, int P, int P4, float *Cs, cudaStream_t s);
cudaError_t launch_rate_sweep(int dim, int kernel, int epi, bool count, const uint4 *Pe, const float *Ce,
                              const uint32_t *cell_start, const uint32_t *perm, const RateParams &prm,
                              const SweepParams &sp, const SweepOut &out, cudaStream_t s);

int rate_blocks(int n);
int rate_launch_blocks(int dim, const RateParams &prm, bool iso);
// Warps of one uniform-velocity rate launch (= per-warp partials its corrector writes).
int rate_launch_warps(int dim, const RateParams &prm, bool iso);
size_t tiled_smem_bytes(int dim, const RateParams &prm);
int closed_form_blocks(int n);

// Captured steps of a context's run calls, three at most: kGraphSteps steps, one step, and the remainder
// that the last calls had in common (run_graphs in api.cu).
struct StepGraphs {
    cudaGraph_t graph[3];
    cudaGraphExec_t exec[3];
    int rest;                // steps of the last remainder
    cudaStream_t stream;     // captured on
};

}  // namespace ade

struct ade_ctx {
    ade_params p;
    int n;
    int dim;
    int nc[3];
    int ncells;
    int subdiv;
    int ncells_cap;       // workspace capacity in cells (every grid the autotuner may pick)
    int partials_cap;     // workspace capacity in reduction partials
    int wpart_cap;        // workspace capacity in per-warp corrector partials
    bool count_clean;     // w.count[0, ncells_cap) is zero (cleared once; every cell build leaves it so)
    uint32_t *xq;
    float *C;
    void *ws;
    size_t ws_bytes;
    ade::Work w;
    double H;
    double dt;
    double pf;            // RateParams::pf in FP64
    double D[9];
    ade::RateParams rp;   // rate constants (dt/inc set per use)
    uint32_t inc[3];
    uint32_t inc_half[3];
    bool iso;
    double t;
    long long step;
    long long pairs;
    ade::StepGraphs graphs;   // of ade_run
    bool status_cleared;
    cudaEvent_t ev[5];    // per-phase timing events (created on first timed step)
    bool ev_ready;
    bool frame_set;       // w.frame holds the frame of the current step
    bool cells_framed;    // the last build was in the moving frame; the last step that used it started from its
    uint32_t cells_add[3];   // positions moved by cells_add
    // weight table of multi-step calls (ade_set_weights), in the caller's buffer
    bool frozen;          // there is one for the grid in use
    bool cursor_clean;    // its pool's counter has been cleared
    ade::FrozenTab frozen_tab;
    size_t frozen_lines;  // lines of the table
    float *frozen_C;      // [2][2n] concentrations of such a call (FrozenState)
    ade::TablePlan plan, adj_plan;   // as last asked for (stride 0: not since the last change of grid)
    // velocity-field mode (p.vmax > 0)
    bool field;
    bool field_set;       // a valid field has been copied in
    bool field_dirty;     // tensors must be re-formed (dispersivities changed)
    // Cattaneo form (Eq. 14, p.tau > 0)
    bool catt;
    bool flux_set;        // Q holds a flux (ade_set_flux)
    float *Q;             // [n] caller order
    float *Qh;            // [n] sorted half-step flux
    double Hgrid;         // radius the cell grid is built for: H, or H + skin in field mode
    double skin;
    ade::FieldParams fp;  // constants (scales set per use)
    ade::FieldWork fw;
};
