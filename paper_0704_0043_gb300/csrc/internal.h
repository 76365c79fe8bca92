// internal.h -- shared declarations of the liblbm translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/lbm.h"

namespace lbm {

// Device layout of a population field: plane-major, rows padded.  Element
// (k, y, x) lives at k * plane + y * pitch + kLead + x.  The kLead elements in
// front of every row and the kTail (at least) after it are zero and never
// written, so a warp may read a window of columns around its strip a few
// elements past either edge of the lattice (the fused kernel's 16-byte
// copies reach up to 68 columns past the last column).
constexpr int kLead = 32;
constexpr int kTail = 96;
__host__ __device__ inline int row_pitch(int nx) { return ((nx + 31) / 32) * 32 + kLead + kTail; }

// Boundary kinds (LBM_BC_*): which directions wrap, and whether the outer
// ring of nodes lies on the walls.
__host__ __device__ inline bool bc_wrap_x(int b) { return b == 1 || b == 2; }
__host__ __device__ inline bool bc_wrap_y(int b) { return b == 1; }
__host__ __device__ inline bool bc_node_walls(int b) { return b == 3 || b == 4; }

// Ensemble-dependent limiter bits (LBM_LIM_SMOOTH | LBM_LIM_THRESHOLD |
// LBM_LIM_ENTTHRESH): a pass with any of them first reduces dS over the lattice.
constexpr unsigned kLimEnsemble = 8u | 16u | 32u;

// State of the device solve of Eq. EntThresh (entthresh.cu): a radix descent
// over the bit patterns of the pass's dS field, 8 bits a level, keeping
// prefix (the determined high bits of the bin that holds dS_0), and the count
// and sum of the values above that bin.
struct EntState {
    double rhs;                  // delta_0 (1 - (2 beta - 1)^2) sum dS
    double s_above;              // sum of the values above the current bin
    unsigned long long m_above;  // their count
    unsigned long long prefix;   // determined high bits (in place)
    double t;                    // result: dS_t = max(dS_0, threshold_delta)
    int done;                    // the solve ended early (no value, rhs <= 0, or dS_0 = 0)
    unsigned ticket;             // FP32 fields: blocks of the level that are done
    unsigned long long cnt[256];  // histogram of the current level: counts
    double sum[256];              // and sums (FP32 fields: 64-bit integers in the bin's unit)
};

// Sticky device status bits.
enum : unsigned { kStatNonfinite = 1u, kStatTimeout = 2u, kStatCandOverflow = 4u };

// Block rows of the tiled kernel are summed in chunks of kChunkRows by the
// last block of each chunk to finish (fixed order within the chunk); the tail
// kernel reduces the chunk rows.
constexpr int kChunkRows = 256;
__host__ __device__ inline int chunks_for(int blocks) { return (blocks + kChunkRows - 1) / kChunkRows; }

// Per-block partial sums written by the step kernels, reduced in a fixed
// order by the finalise kernel.
enum { P_MASS = 0, P_SUM_DS, P_SUM_IN, P_DS_LIM, P_NPOS, P_NMED, P_NBAD, P_NSTAT };

// The fused kernel hands out its work items dynamically, so which warp sums
// which sites varies from run to run.  To keep the step statistics the same
// bit for bit, it sums them exactly: each work item's FP32 sums (a fixed
// evaluation order within the item) are converted to 128-bit two's-complement
// fixed point in units of 2^-64 and added as integers, whose sum does not
// depend on the order.  A fixed-point partial row holds kFxWords words:
// FX_SUM + 2 s (low word) and FX_SUM + 2 s + 1 (high word) for the FP
// statistic s = P_MASS (sum of rho - rho_ref) .. P_DS_LIM; the site and
// limiter counts; and a bit per FP statistic that met a nonfinite or
// out-of-range (>= 2^63) item sum.
// Each block of the fused kernel adds its row atomically into accumulator row
// (block % kFxRows) of its lattice's partials; the tail kernel sums the
// kFxRows rows and clears them.
constexpr int kFxWords = 16;
constexpr int kFxRows = 8;
enum { FX_SUM = 0, FX_SITES = 8, FX_NPOS, FX_NMED, FX_NBAD, FX_BAD };

// Ehrenfests' candidate: FP64 key dS(f') (NaN: not keyed yet), phi of the
// limiter pass, site index, and dS(f') in FP32 (the key rounded, or the FP32
// value the candidate was recorded on; within 1/64 of the key where select.cuh's kSureDelta
// and kSureFlow say so).
struct Cand {
    double key;
    double phi;
    int32_t site;
    float ds32;
};

// Device-wide preselection of Ehrenfests' candidates: when a pass records
// more candidates than the tail's block holds in shared memory, the tail runs
// as a grid of one block per SM.  The grid finds, by two 12-bit radix levels
// over the FP32 dS bit patterns of the candidates certainly above delta, a
// lower bound T of the k-th largest; keys in FP64 the candidates with FP32 dS
// of at least T (1 - 1/32) and those near delta; counts the valid candidates;
// and hands block 0 the short list of valid candidates at or above the bound,
// which holds every candidate the exact top-k can take.
constexpr int kSelBins = 4096;   // bins of one radix level
// Lattices of at least this many sites get the grid tail.  Its launch costs
// one to two microseconds per step, a tenth of a smaller lattice's step; on
// those, one block keys and selects the candidates, about 0.1 us per
// candidate without a key (a tenth of a second when every site of a 2^20-site
// lattice is one).
constexpr long long kSelMinSites = 1ll << 20;
constexpr int kSelList = 65536;  // the longest list block 0 is handed
struct SelState {
    unsigned hist1[kSelBins];  // level 1: bits 30..19 of the FP32 dS pattern
    unsigned hist2[kSelBins];  // level 2: bits 18..7 within level 1's bin
    unsigned bar;              // grid barrier: arrivals so far (block 0 resets it)
    unsigned count;            // list entries (more than kSelList: overflow)
    unsigned n_valid;          // candidates with dS above delta
    unsigned pad;
    int list[kSelList];        // candidate indices
};

struct DevStats {  // mirrors lbm_step_stats
    long long step;
    double mass, sum_dS, dS_lbgk, dS_lim;
    long long n_pos, n_med, n_ehr, n_cand, n_bad;
    int status;
    int reserved;
};

// Fixed-point form of a site's moments (site_moments): FP32 / 16-bit storage.
struct MomentFx {
    long long rest;  // sum of rho_ref W_k in units
    float scale;     // 2^(27 - exponent of rho_ref)
    float lim;       // deviations below it fit (0: never)
    int exp;         // the unit is 2^exp
};

struct StepParams {
    MomentFx mfx;
    int nx, ny, pitch;
    long long plane;           // elements per population plane
    int boundary;              // LBM_BC_*
    unsigned limiters;
    int median_mode;
    int collide;               // 1: free flight + collision; 0: limiter pass on stored state
    int eq;                    // 0: polynomial f*, quadratic dS; 1: entropic f*, exact dS (FP64 storage)
    double a;                  // 2 beta - 1
    double delta_m, delta_e;
    double u_lid;              // lid x-velocity (wall rule of LBM_BC_DIFFUSIVE)
    double beta;               // LBGK / ELBM relaxation parameter (Eq. elbm)
    int coll;                  // LBM_COLL_* (ELBM: FP64 entropic path)
    int phi_rule;              // LBM_PHI_* (LBM_PHI_ENTROPY: FP64 entropic path)
    double lid[9];             // ((6 W_k) rho_wall) (c_kx u_lid), added on links through the lid
    // the same term for FP32 arithmetic as an unevaluated sum hi + lo: adding
    // both parts keeps the rounding of the constant out of every wall step
    // (a single FP32 constant would bias the lid momentum by ~1e-9 per step)
    float lidf[9], lidlo[9];
    float rho_ref;             // FP32 storage holds g_k = f_k - rho_ref W_k
    double rw[9];              // rho_ref W_k in FP64 (absolute value of FP32 storage: (double) g + rw)
    float rwf[9];              // rho_ref W_k in FP32
    // scratch (library-owned)
    Cand *cand;
    int *cand_count;
    int cand_cap;
    double *partials;          // tiled kernel: [blocks][P_NSTAT] doubles
    double *partials2;         // tiled kernel: [chunks][P_NSTAT] sums of kChunkRows block rows each
    unsigned long long *fx_rows;  // fused kernel: [kFxRows][kFxWords] fixed-point accumulators (own region)
    unsigned *chunk_cnt;       // tiled kernel: blocks of each chunk done this launch (reset by its last block)
    unsigned *status;
    int *work;                 // fused kernel: counter of work items handed out (nullptr: one item per warp)
    double *ds_out;            // optional FP64 dS(f') field (nx * ny) or nullptr
    // ensemble-dependent limiters (LBM_LIM_SMOOTH / LBM_LIM_THRESHOLD)
    double smooth_delta, smooth_k, threshold_c, threshold_delta;
    const double *ens;         // {E(dS), smooth_delta / E^smooth_k, sum dS, count} of this pass (the ensemble reduction)
    void *ent_field;           // LBM_LIM_ENTTHRESH: dS of every site (compute type; 0 where excluded)
    EntState *ent;             // LBM_LIM_ENTTHRESH: the solve's state; ent->t is the pass's dS_t
};

struct FinalParams {
    MomentFx mfx;
    int nblocks;               // partial rows to reduce
    int fixed;                 // the rows are fixed-point rows of the fused kernel
    int *work;                 // work-item counter to clear for the next step, or nullptr
    double one_minus_a2;       // 1 - (2 beta - 1)^2
    long long k_max;
    int ehrenfest;             // apply Ehrenfests' step
    int collide;
    int eq;                    // as StepParams::eq
    int nx, ny, pitch;
    long long plane;
    double *partials;          // fused kernel: the accumulator rows, cleared once read
    Cand *cand;
    int *cand_count;
    int cand_cap;
    int *sel;                  // selected sites out
    int sel_cap;
    int *sel_count;
    unsigned *status;
    DevStats *stats_ring;
    int ring_len;
    long long *counters;       // [0] steps taken (incremented when collide), [1] records written
    // pre-step populations of the pass (FP32 / BF16 / FP16 storage): the
    // Ehrenfests' step evaluates f*(m) from them, with the same FP32 free
    // flight as the step kernel, so the stored result is rounded once
    const void *src;
    int boundary;
    double a, delta_e;
    double lid[9];
    float lidf[9], lidlo[9];
    float rho_ref;
    double rw[9];
    // control-point record (Sec. 4.4.2): after each step, rho, u_x, u_y of site
    // probe_site into probe[3 ((step - 1) mod probe_cap) ...]; probe == nullptr: off
    double *probe;
    long long probe_cap;
    int probe_site;
    // dense candidates: the grid's shared selection state (launches of more
    // than one block only; nullptr otherwise; FinalParams{} zeroes it)
    SelState *sel_state;
};

// Arguments of one fused-kernel instance (a lattice, its buffers and its
// strip / segment decomposition).
struct FusedArgs {
    StepParams p;
    const void *src;  // float, __nv_bfloat16 or __half deviations
    void *dst;
    int strips, segs, seg_rows, items, blocks;  // work items: strips of 62 finished columns x row segments
    float a, b2, delta_m, thr_e, rho_ref;  // b2 = 2 beta
    float lid4, lid7, lid8;  // FP32 moving-wall terms of the links through the lid (hi + lo)
    float lo4, lo7, lo8;
};

// One tiled-kernel instance (batched launches) and one tail instance.
struct TiledArgs {
    StepParams p;
    const void *src;
    void *dst;
    int gx, blocks;  // blocks along x, blocks in total
};
struct FinalArgs {
    FinalParams p;
    void *f;
};
// One tube-kernel instance of a batched launch (FP32 D1Q3 lattices).
struct TubeArgs {
    StepParams p;
    const void *src;
    void *dst;
};

// Many steps of a small lattice in one cooperative launch (step_resident.cu).
constexpr int kResRows = 4;        // steps whose block rows are kept: the tail may lag this far behind
// Arrival words, a step each in turn.  A word is used again kResSlots steps later.
// Its readers have then read it: a worker reads step s before it arrives at s + 1,
// and a worker arrives at step s only when the tail has recorded step
// s - kResRows - 1 (the row wait of step s - 1), so kResRows + 1 words do.
constexpr int kResSlots = 8;
static_assert(kResSlots > kResRows, "an arrival word's readers are done before it is used again");
constexpr int kResMaxBlocks = 160;
constexpr int kResMaxSteps = 1024;  // steps of one launch
// Lattices up to these sizes take the resident kernel.  Measured us per step, resident
// against launch by launch (square cavities with the median filter / with all
// limiters; tubes with Ehrenfests' steps):
//   D2Q9 FP32 (16-bit alike): 256^2 6.2 / 12.9 against 13.7 / 27.2, 384^2 8.1 / 15.2
//   against 15.2 / 29.5, 480^2 10.3 / 17.4 against 16.2 / 29.8.  The limit was set with
//   lower tiles than round_cost now gives (512^2 14.9 / 23.2 against 14.5 / 26.7): above it
//   the fused kernel evaluates two sites a lane and reads each plane once;
//   D2Q9 FP64: 512^2 151 / 156 against 224 / 234, 700^2 261 / 267 against 384 / 396;
//   D1Q3 FP32: 2e5 9.1 against 15.8, 1e6 15.4 against 20.7;
//   D1Q3 FP64: 800 9.5 against 13.5, 5e5 100 against 125.
constexpr long long kResMaxSites = 240000;      // D2Q9, FP32 and 16-bit storage
constexpr long long kResMaxSites64 = 1ll << 19;  // FP64 storage
constexpr long long kResMaxSites3 = 1ll << 20;   // D1Q3, FP32 storage
struct ResRow {
    double v[4];  // P_MASS .. P_DS_LIM of a worker block's sites
    int c[4];     // positivity, median, flagged sites
};
struct ResState {
    // low word: worker arrivals, high word: candidates recorded, both of all the
    // steps of this slot since the launch.  A word per step, because a reader may
    // be late: a worker by one step, the tail by kResRows.  In one word for all
    // steps, the candidates of workers that are ahead would count as the step's.
    unsigned long long arrived[kResSlots];
    unsigned done;               // steps whose candidates are finished
    unsigned stats_done;         // steps whose record is written
    unsigned rows_in[kResRows];  // worker rows written, steps of each slot
    unsigned keyed;              // workers that keyed their share of a dense step's candidates
    ResRow rows[kResRows][kResMaxBlocks];
};
struct ResArgs {
    StepParams p;
    FinalParams f;
    void *buf[2];
    int cur, nsteps;
    int aw, gx, tiles, blocks;  // see ResGrid
    double rest;        // rest_mass
    ResState *rs;
};
double rest_mass(const StepParams &p);
bool resident_applies(const lbm_config &c);
// The grid of a resident launch: warps that carry sites, tiles along x, tiles, blocks, and
// the most steps a launch takes (it holds its SMs for all of them: kResLaunchUs).
struct ResGrid {
    int aw, gx, tiles, blocks, most_steps;
};
// False: the lattice is stepped launch by launch.  A resident block fills its SM, so grids
// that do not fit beside one another run one after the other, and what waits for the tail
// or the barrier in one of them is lost to the others.  With lattices on several streams
// the grid takes at most its share of the SMs, one round of tiles, or there is none.
// us for a step of all of 1 / 2 / 4 / 8 lattices on their own streams (Ehrenfests' steps
// and median): 300^2 FP32 resident on all SMs 15 / 30 / 60 / 120, launch by launch 27 / 29 /
// 33 / 39; 100^2 FP32 on all SMs 12 / 23 / 46 / 93, on its share 12 / 12 / 13 and, where it
// does not fit, launch by launch 34; 200^2 FP64 launch by launch 71 / 126 / 243 for 2 / 4 / 8.
bool resident_grid(const lbm_config &c, int streams, ResGrid *g);
constexpr double kResLaunchUs = 8000.0;  // about the longest launch
// The smallest FP32 D2Q9 lattices without Ehrenfests' steps: one thread-block
// cluster, populations in shared memory (step_cluster.cu).  us per step against
// the resident kernel, median filter, boundary nodes: 32^2 3.4 / 6.0, 64^2 3.4 / 6.2,
// 100^2 3.8 / 6.3, 128^2 5.3 / 6.3; 150^2 7.1 / 4.9 (16 SMs against 95: tiles of eight rows
// fill the resident grid there, of four below).
constexpr long long kCluMaxSites = 128 * 128;
constexpr size_t kCluMaxBytes = 200 * 1024;  // dynamic shared memory of a block
bool cluster_applies(const lbm_config &c);
cudaError_t launch_cluster(ResArgs a, cudaStream_t s);
// Takes a.nsteps steps from a.buf[a.cur]; a.f as for the tail of a step.
template <typename S>
cudaError_t launch_resident(int q, ResArgs a, cudaStream_t s);

// Launchers (stream-ordered, no synchronisation).  Return cudaGetLastError().
template <typename T>
cudaError_t launch_tiled(int q, const StepParams &p, const T *src, T *dst, int *nblocks,
                         cudaStream_t s);
// The tail: one block, or (grid > 1, p.sel_state set) a cooperative grid of
// `grid` blocks that preselects dense candidates; the launch returns the
// launch error without a fallback.
template <typename T>
cudaError_t launch_finalize(int q, const FinalParams &p, T *f, cudaStream_t s, int grid = 1);
// Blocks of the tail's cooperative grid on this device: one per SM (0 when a
// block does not fit or the device has no cooperative launch).
template <typename T>
int finalize_grid(int q);
// Field kernels take the StepParams of the context for the layout (nx, ny,
// pitch, plane) and the FP32 storage offsets (rw).
template <typename T>
cudaError_t launch_init(int q, const StepParams &p, const double *rho, const double *ux, const double *uy, T *f,
                        cudaStream_t s);
template <typename T>
cudaError_t launch_moments(int q, const StepParams &p, const T *f, double *rho, double *ux, double *uy,
                           cudaStream_t s);
template <typename T>
cudaError_t launch_get(int q, const StepParams &p, const T *f, double *out, cudaStream_t s);
template <typename T>
cudaError_t launch_set(int q, const StepParams &p, const double *in, T *f, cudaStream_t s);
template <typename T>
cudaError_t launch_delta_s(int q, const StepParams &p, const T *f, double *out, cudaStream_t s);
// E(dS) of the pass p is about to run and the smooth limiter's alpha, into
// ens[2 kEnsBlocks], ens[2 kEnsBlocks + 1] (ens[0 .. 2 kEnsBlocks) is scratch).
constexpr int kEnsBlocks = 608;
// Behind them (in doubles from the start of the E(dS) scratch): {E, alpha, sum,
// count}, then kFxRows fixed-point rows of the fused E(dS) pass and its
// work-item counter (launch_fused_epass).
constexpr int kEnsFxOffset = 2 * kEnsBlocks + 4;
constexpr int kEnsDoubles = kEnsFxOffset + 8 * 16 + 2;
template <typename S>
cudaError_t launch_fused_epass(const StepParams &p, const S *src, cudaStream_t s);
template <typename T>
cudaError_t launch_ens_mean(int q, const StepParams &p, const T *src, double *ens, cudaStream_t s);
// Eq. EntThresh on the field p.ent_field (filled by the ensemble reduction):
// p.ent->t = max(dS_0, threshold_delta).  T is the compute type of the field.
template <typename T>
cudaError_t launch_entthresh(const StepParams &p, double delta0, long long n, cudaStream_t s);
// launches of one EntThresh solve (for the launch count)
int entthresh_launches(bool fp64);

// Sets the calling thread's error message (read by lbm_last_error(NULL)); returns s.
int set_thread_error_impl(int s, const char *msg);
#define set_thread_error(s, msg) ((lbm_status)::lbm::set_thread_error_impl((int)(s), (msg)))

// Fused D2Q9 step for LBM_BC_WALLS (row-streaming kernel; FP32, BF16 or FP16
// storage).
template <typename S>
cudaError_t launch_fused_d2q9(const StepParams &p, const S *src, S *dst, int *nblocks, cudaStream_t s);
int fused_d2q9_blocks(int nx, int ny);  // most blocks (partial-sum rows) any launch of the lattice uses
int fused_slots(int elem_bytes, bool batched);  // resident work items (warps) of one wave
// Fills the instance arguments: row segments of `seg_rows` rows (0: about
// `slots` work items); returns the block count.
int fused_make_args(const StepParams &p, const void *src, void *dst, int seg_rows, int slots, FusedArgs *out);
// Batched launches.  Fused: `items` work items over all instances, item i
// being item map[i].y of instance map[i].x, handed out dynamically through
// the counter *work (cleared by the tail after the launch).  Tiled: `blocks`
// blocks, block b running instance map[b].x as its block map[b].y.
// med / pos: the lattices' median / positivity code is needed (a smaller kernel otherwise).
cudaError_t launch_fused_batched(const FusedArgs *table, const int2 *map, int items, int *work, bool med, bool pos,
                                 cudaStream_t s);
cudaError_t launch_tiled_batched_f32(int q, const TiledArgs *table, const int2 *map, int blocks, cudaStream_t s);
cudaError_t launch_finalize_batched_f32(int q, const FinalArgs *table, int n, cudaStream_t s);
// D1Q3 streaming step (FP32 / FP64 storage): *chunked is false when the grid
// fits one chunk of the tail's reduction, whose rows the tail then reads itself.
template <typename S>
cudaError_t launch_tube(const StepParams &p, const S *src, S *dst, int *nblocks, bool *chunked, cudaStream_t s);
bool tube_applies(const lbm_config &c, unsigned limiters);  // the pass runs on the tube kernel
// Batched FP32 tubes: `items` work items (groups of chunks, item i = group
// map[i].y of tube map[i].x) handed out through *work; each item writes its
// tube's partial row of its group (the tail reads tube_groups(nx) rows).
cudaError_t launch_tube_batched(const TubeArgs *table, const int2 *map, int items, int *work, cudaStream_t s);
int tube_groups(int nx);
int tube_blocks(bool fp64, int nx);                          // blocks (partial rows) of one launch
int sm_count();
int tiled_grid_x(int q, int nx);
int tiled_blocks_for(int q, int nx, int ny);
bool fused_d2q9_fits(long long plane);  // 32-bit plane offsets inside the kernel

}  // namespace lbm

// Library-owned state of one lattice (opaque to callers, see include/lbm.h).
struct lbm_ctx {
    lbm_config cfg{};
    cudaStream_t stream = nullptr;
    int device = 0;
    int q = 9;
    int pitch = 0;
    long long plane = 0;
    size_t elem = 4;
    size_t field_bytes = 0;
    void *arena = nullptr;  // the one allocation behind the arrays below (but stage and probe)
    void *buf[2] = {nullptr, nullptr};
    int cur = 0;
    lbm::Cand *cand = nullptr;
    int cand_cap = 0;
    lbm::SelState *sel_state = nullptr;  // Ehrenfests' limiter: the cooperative tail's selection state
    int fin_grid = 0;                     // blocks of the cooperative tail (0: one-block tail only)
    bool capturing = false;               // a graph capture is in progress (one-block tail)
    bool cluster = false;                 // the resident steps run as one cluster
    bool listed = false;                  // the stream is in the list of live contexts' streams
    lbm::ResState *res = nullptr;         // resident steps: counters and rows (nullptr: stepped launch by launch)
    double *ens = nullptr;  // [kEnsBlocks][2] partial sums and counts of dS, then E(dS), alpha, sum, count
    void *ent_field = nullptr;   // LBM_LIM_ENTTHRESH: the pass's dS field
    lbm::EntState *ent = nullptr;  // LBM_LIM_ENTTHRESH: solve state
    int *counts = nullptr;  // [0] candidate count, [1] chosen count, [2] fused work items handed out, [3] unused
    int *sel = nullptr;
    int sel_cap = 0;
    double *partials = nullptr;
    int partial_rows = 0;
    unsigned *chunk_cnt = nullptr;  // tiled kernel: per-chunk block counters
    unsigned *status = nullptr;
    lbm::DevStats *ring = nullptr;
    int ring_len = 1;
    long long *counters = nullptr;  // [0] steps, [1] records
    double *stage = nullptr;
    size_t stage_bytes = 0;
    bool ready = false;
    bool timing = false;
    bool timing_now = false;    // the current pass records its events
    int timing_every = 1;       // record one pass in this many
    long long timing_pass = 0;  // passes since timing was enabled
    std::vector<cudaEvent_t> events;  // three per timed step
    size_t events_used = 0;
    long long launches = 0;
    int64_t device_bytes = 0;
    // CUDA-graph replay of runs of graph_steps steps (0: off): one graph per
    // starting buffer, captured on gstream (the context's own stream may be
    // the legacy default stream, which cannot be captured)
    int graph_steps = 0;
    cudaStream_t gstream = nullptr;
    cudaEvent_t gev = nullptr;
    cudaGraphExec_t gexec[2] = {nullptr, nullptr};
    long long graph_launches = 0;  // kernel launches one replay performs
    // control-point record (lbm_probe)
    double *probe = nullptr;
    long long probe_cap = 0, probe_alloc = 0, probe_step0 = 0;
    int probe_site = -1;
    std::string err;
};

namespace lbm {
// Geometry and physics of a step for configuration g, stored with row pitch
// `pitch` and `plane` elements per population plane; every scratch pointer is
// left null for the caller to fill.
StepParams cfg_step_params(const lbm_config &g, int q, int pitch, long long plane, int collide, unsigned limiters);
// The tail's parameters that follow from g and from the step's p (scratch
// pointers null).
FinalParams cfg_final_params(const lbm_config &g, const StepParams &p, int collide, unsigned limiters, int nblocks);
// Per-step parameters of a context (collide = 0 for a limiter pass).
StepParams ctx_step_params(lbm_ctx *c, int collide, unsigned limiters);
// The fused kernel's accumulator rows of a context (the tail's partials when fixed = 1).
double *ctx_fx_rows(lbm_ctx *c);
FinalParams ctx_final_params(lbm_ctx *c, int collide, unsigned limiters, int nblocks);
// lbm_create; `batched`: without what only lone lattices use.
lbm_status create_ctx(const lbm_config *cfg, void *cuda_stream, bool batched, lbm_ctx **out);
bool ctx_uses_fused(const lbm_ctx *c);
}  // namespace lbm
