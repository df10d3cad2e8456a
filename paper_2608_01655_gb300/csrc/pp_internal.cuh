// Internal declarations of libprefixplace (not installed, not part of the ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <string>
#include <vector>

#include "pp_reduce_shape.h"
#include "prefixplace.h"

namespace pp {

// ---------------------------------------------------------------------------
// DP row metadata.  Rows are preorder positions, swept from n-1 down to 0.
// The skip branch of Eq. 9 reads row next(i):
//   kSkipCur   next(i) == i + 1: the row just computed (kept in registers)
//   kSkipZero  next(i) == n: the boundary row D[n][.] = 0
//   level >= 0 a row saved earlier on the skip-row stack at that level
// A row is pushed only when a position q < r - 1 reads it (next(q) == r),
// so the stack holds one row per pending subtree continuation and its depth
// is bounded by the tree depth.
// Packed in one int32: low 16 bits skip code + 2, high 16 bits push level + 1.
// ---------------------------------------------------------------------------
constexpr int kSkipZero = -2;
constexpr int kSkipCur = -1;
constexpr int kMaxStackLevels = 65533;

__host__ __device__ inline int meta_skip(int32_t m) { return (m & 0xFFFF) - 2; }
__host__ __device__ inline int meta_push(int32_t m) { return ((m >> 16) & 0xFFFF) - 1; }
inline int32_t meta_pack(int skip, int push)
{
    return (int32_t)(((uint32_t)(push + 1) << 16) | (uint32_t)(skip + 2));
}

// Row metadata of the wavefront DP kernel: the skip-row stack top is kept in
// registers (every stack read is of the top, and the zero row D[n][.] is the
// top of the empty stack), so a row needs only: its weight, whether its skip
// row is the row just computed (next(i) = i + 1) or the top, and whether it
// pushes (store the new row at `level`; it becomes the top) or pops (reload
// the new top from `level`, or reset it to the zero row when the stack empties).
// bits 0-2 weight-1 (weights <= 8), 3-4 kind, 5 reload, 6 push, 7 zero top,
// 16-31 level.
constexpr int kWaveCur = 0, kWaveTop = 2;
constexpr int kWaveReload = 1 << 5, kWavePush = 1 << 6, kWaveZeroTop = 1 << 7;
__host__ __device__ inline int32_t wave_pack(int w, int kind, int flags, int level)
{
    return (int32_t)((uint32_t)(w - 1) | ((uint32_t)kind << 3) | (uint32_t)flags | ((uint32_t)level << 16));
}

// Column geometry of one DP launch: thread t of the chain owns columns
// t*C + c + 1 (c = 0..C-1); column 0 is the boundary D[.][0] = 0.  Decision
// bits of row i are kpad/32 words; word (t/32)*C + c holds bit (t%32) for the
// column t*C + c + 1, i.e. one __ballot_sync per (warp, c).
struct DpGeom {
    int C = 1;        // columns per thread
    int T = 32;       // threads per chain (all CTAs)
    int kpad = 32;    // T * C columns
    int words = 1;    // decision words per row (kpad / 32)
    int P = 1;        // warps per chain
    int wave = 0;     // 1: wavefront kernel (cluster of CL CTAs x WPC warps)
    int CL = 1;       // CTAs per chain (thread-block cluster)
    int WPC = 1;      // warps per CTA
    int WMAX = 1;     // largest chunk weight the wavefront kernel is built for
    int L_smem = 0;   // skip-row stack levels held in shared memory
    size_t smem = 0;  // dynamic shared memory per CTA
    // Split launch (wavefront kernel, batch just above what clusters of CL
    // CTAs hold at one CTA per SM): the `split` items with the most kept rows
    // run as clusters of CL, the rest concurrently as clusters of CL2 = CL / 2
    // CTAs x WPC2 = 2 * WPC warps on the SMs left over (same P, C and bit
    // layout).  Both launches reserve more than half an SM's shared memory so
    // that no SM hosts two CTAs.  split = 0: one launch.
    int split = 0;
    size_t smem_x = 0;                       // the wide launch's shared memory when split
    int CL2 = 0, WPC2 = 0, L_smem2 = 0;
    size_t smem2 = 0;
};
// Decision bits of every DP kernel, packed by each thread over blocks of 32
// rows in sweep order (row r = n - 1 - i, block r / 32, bit r % 32): for chain
// warp g, lane and column offset c, the word
//   (((item * P + g) * nblk + r / 32) * C + c) * 32 + lane
// holds the take decisions of column (g * 32 + lane) * C + c + 1, with
// nblk = ceil(n / 32).

// Workspace of one batched DP launch (pp_dp_bits_size bytes, carved in this
// order): decision bits, then the pruned sweep (rows kept in sweep order, the
// inverse map position -> kept index or -1, prefix counts of positive
// profits, kept-row counts).  A row is dropped when every strict descendant
// of its parent has a non-positive profit: such a parent's interior is never
// taken and leaves D[parent+1] = D[next(parent)], so dropping those rows
// changes no value and no bit of a kept row (see pp_prune.cuh).  Then the exact
// reduction's: states, sets as bitmaps, scratch.
// For the traceback, per kept row t (kept index, sweep order): skip[t] = kept
// index of next(row t), -1 when next(row t) = n; wsuf[t] = sum of the
// weights of kept rows t..nkept-1.
struct DpWork {
    uint32_t *bits = nullptr;      // [batch][P][nblk][C][32]
    int32_t *rowlist = nullptr;    // [batch][n]
    int32_t *kidx = nullptr;       // [batch][n]
    int32_t *cnt = nullptr;        // [batch][n + 1]
    int32_t *nkept = nullptr;      // [batch]
    int32_t *skip = nullptr;       // [batch][n]
    int32_t *wsuf = nullptr;       // [batch][n + 1]
    int64_t *rowp = nullptr;       // [batch][n] profit of each kept row, sweep order
    int32_t *rowm = nullptr;       // [batch][n] wave-kernel metadata of each kept row
    // exact reduction (pp_reduce.cu), null when the tree has none.
    // red[item] = 1: solved, the optimal set is `taken` and nkept[item] the
    // number of rows that were undecided; the pruned sweep's kernels leave
    // it alone.  2: those kernels sweep only the rows in `undecided`, with the
    // budget left[item]; base[item] is the value of the decided rows, which
    // are in `taken`.  0: they sweep all rows.  A launch without the reduction
    // writes 0 too, so what reads the workspace later does not depend on the
    // switches then.
    int32_t *red = nullptr;        // [batch]
    int32_t *left = nullptr;       // [batch]
    int64_t *base = nullptr;       // [batch]
    uint32_t *taken = nullptr;     // [batch][ceil(n / 32)] by preorder position
    uint32_t *undecided = nullptr; // [batch][ceil(n / 32)]
    char *red_scratch = nullptr;   // [batch][reduce_item_bytes]
    bool reduce = false;           // launches on this workspace try the reduction
    int items = 0;                 // items in flight together with this launch's (0: only those)
    int64_t *clear = nullptr;      // [batch] or null: zeroed by the reduction (the planner's next held sums)
};
size_t dp_work_bytes(const pp_instance *inst, int batch, int words);
DpWork dp_work_split(const pp_instance *inst, void *base, int batch, int words);
// the same workspace seen as a batch of one: item `item` of `w`
DpWork dp_work_item(const pp_instance *inst, const DpWork &w, int item, int words);

// Status word values written by kernels (same numbering as pp_status).
constexpr int32_t kDevOk = PP_OK;

// Layout of the exact reduction (pp_reduce.cu): host tables while an instance
// is built (their sizes: pp_reduce_shape.h).
constexpr int32_t kReduceMinRows = 128;     // below, the sweep is as short (501 rows: 79 us swept, 40 reduced)
struct ReduceTables {
    struct Info {
        int32_t x, y;
    };
    struct Stream {
        int32_t tile, tiles;
    };
    struct Cluster {
        int cl, acc;                // CTAs of an item; accumulators of a CTA, at most
        int path;                   // tiles in sequence: over the levels, the most of one warp
    };
    int bins = 0, max_kids = 0;
    std::vector<Info> info;
    std::vector<int32_t> pos;
    std::vector<uint8_t> form;
    std::vector<Cluster> cluster;   // largest first
    std::vector<Stream> stream;
    std::vector<int32_t> lev, binlev, binslot, nacc;
};

struct Scratch {
    void *ptr = nullptr;
    size_t bytes = 0;
};

}  // namespace pp

struct pp_instance {
    int32_t n = 0;
    int32_t W = 0;
    int32_t mode = 0;
    int device = 0;
    int sm_count = 0;
    int32_t stack_depth = 0;            // skip-row stack levels needed by the DP
    int64_t total_weight = 0;           // sum of chunk weights
    int32_t max_weight = 1;             // largest chunk weight
    int32_t trace_skips = 1;            // skips the traceback speculates per step beyond the first
    // DP launch-shape overrides of this instance (pp_tune_dp; 0 = automatic)
    int32_t tune_cl = 0, tune_c = 0, tune_flat = 0, tune_noprune = 0;
    std::vector<int32_t> h_order, h_next, h_par, h_budget, h_wpre;
    // device tables, preorder-indexed unless noted
    int32_t *d_order = nullptr;         // [n] position -> node id
    int32_t *d_next = nullptr;          // [n]
    int32_t *d_wpre = nullptr;          // [n] chunk weight
    int2 *d_pspan = nullptr;            // [n] parent x's strict-descendant range (x+1, next(x)); roots -1
    int32_t *d_budget = nullptr;        // [W]
    int64_t *d_a = nullptr;             // mode 0: [W][n] a_m(b)       (Eq. 2)
    int64_t *d_delta = nullptr;         // mode 0: [n]    Delta(b)     (Eq. 3)
    int64_t *d_own = nullptr;           // mode 0: [W][n] Lambda_m(b) [w_m(b) - f_m(b)]_+ (own first-copy gain)
    int64_t *d_pop = nullptr;           // mode 0: [W][n] Lambda_m(b)
    int64_t *d_rec = nullptr;           // [W][n] w_m(b) by node id
    int64_t *d_tr = nullptr;            // by node id: mode 0 [W][n] f_m(b), mode 1 [W][W][n] f_{m<-h}(b)
    int64_t *d_g = nullptr;             // mode 1: [W][W][n] Lambda_m(b) q_{m<-h}(b) at [h][m][i] (Eq. 5)
    int32_t *d_status = nullptr;        // device status word
    pp::ReduceShape red;                // exact reduction's layout (pp_reduce.cu); no bins: none
    void *d_red = nullptr;              // its tables
    pp::Scratch stack;                  // skip-row stack spill of pp_tree_dp
    pp::Scratch plan;                   // pp_plan_run working set
    pp::Scratch plan_bits;              // pp_plan_run decision bits
    pp::Scratch sg;                     // safeguard candidates' working set
    pp::Scratch rp;                     // epoch update working set
    pp::Scratch top2;                   // top-2 holder tables of the planner
    // split DP launches: the two launches run on these streams (higher and
    // lower priority), forked from and joined back to the caller's stream
    cudaStream_t split_hi = nullptr, split_lo = nullptr;
    cudaEvent_t split_fork = nullptr, split_join_hi = nullptr, split_join_lo = nullptr;
    // pp_plan_run without lock step: a stream per start or group (up to kPlanStreams),
    // forked from and joined back to the caller's stream
    std::vector<cudaStream_t> plan_streams;
    std::vector<cudaEvent_t> plan_join;
    cudaEvent_t plan_fork = nullptr;
    int32_t *sweep_flags = nullptr;          // pinned host memory: starts that go on
    int sweep_flags_count = 0;
    std::vector<cudaEvent_t> sweep_events;
    cudaStream_t sg_stream = nullptr;        // safeguard candidates beside a plan
    cudaEvent_t sg_fork = nullptr, sg_join = nullptr;
    std::vector<cudaEvent_t> phase_events;      // timing events of pp_plan_run, reused across calls
};

namespace pp {

// Kernels of one update follow each other on a stream within microseconds:
// each is launched while the one before still runs (programmatic dependent
// launch), waits for it to be complete with chain_wait() before it touches
// memory, and lets the next one be launched with chain_release().
#ifdef __CUDACC__
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// error reporting (thread-local message)
pp_status fail(pp_status s, const std::string &msg);
pp_status cuda_fail(cudaError_t e, const char *what);
#define PP_CUDA(call)                                                   \
    do {                                                                \
        cudaError_t e_ = (call);                                        \
        if (e_ != cudaSuccess) return ::pp::cuda_fail(e_, #call);       \
    } while (0)

pp_status ensure_scratch(Scratch &s, size_t bytes);
void free_scratch(Scratch &s);

// DP launch geometry for a given largest budget (after clamping to the
// instance's total weight).  Returns false when the budget is too large.
bool dp_geometry(const pp_instance *inst, int32_t max_budget, DpGeom *g, int batch = 1);

// Launchers used by both the ABI calls and the planner.
//   prof_by_node: profits indexed by node id (ABI) instead of preorder
//   item_budget:  [batch] budgets; item_active: [batch] or null (0 = skip item)
// stack_item: the launch's items use skip-row stack scratch from item slot
// stack_item on (launches of disjoint slots may run concurrently)
pp_status launch_tree_dp(pp_instance *inst, int batch, const int64_t *profit, bool prof_by_node,
                         const int32_t *item_budget, const int32_t *item_active,
                         const DpGeom &g, int64_t *best, const DpWork &work, cudaStream_t st,
                         int32_t max_budget, unsigned long long *rows_kept = nullptr, int stack_item = 0);
// The exact reduction (pp_reduce.cu).  `par` is the parent's position (-1: root).
bool build_reduce_tables(int32_t n, const std::vector<int32_t> &par, const std::vector<int32_t> &next,
                         const std::vector<int32_t> &wpre, int64_t total_weight, int32_t max_weight,
                         ReduceTables *out);
size_t reduce_tables_bytes(const ReduceTables &R);
void reduce_tables_pack(const ReduceTables &R, char *dst);
ReduceShape reduce_shape(const ReduceTables &R, int32_t n, int32_t max_weight);
pp_status reduce_device(ReduceShape *r);
size_t reduce_item_bytes(const pp_instance *inst);
// whether launches of this instance try the reduction first (not without
// pruning, and not while pp_test_inject makes a warp of the sweep silent)
bool reduce_on(const pp_instance *inst);
pp_status launch_reduce(pp_instance *inst, int batch, const int64_t *profit, bool by_node,
                        const int32_t *item_budget, const int32_t *item_active, int64_t *best, const DpWork &work,
                        cudaStream_t st, int32_t max_budget, unsigned long long *rows_kept);
// levels of the stack of skipped rows that do not fit in shared memory
int dp_global_levels(const pp_instance *inst, const DpGeom &g);
// scratch for the skip-row stack of `items` item slots of geometry g
pp_status ensure_dp_stack(pp_instance *inst, const DpGeom &g, int items);

pp_status launch_marginals(pp_instance *inst, int batch, const int32_t *worker,
                           const uint32_t *mask, bool by_node, const int32_t *item_active,
                           int64_t *profit, int64_t *oldsum, cudaStream_t st);

pp_status launch_objective(pp_instance *inst, int batch, const uint32_t *mask,
                           const uint8_t *chosen, int64_t *obj, cudaStream_t st);

// Top-2 holder tables of the source-dependent marginals, per start (batch
// item), for the holder masks `seen`; every worker's marginals, and which of
// them are stale (bit per worker).
struct Top2 {
    int64_t *v1 = nullptr;       // [batch][W][n]
    int64_t *v2 = nullptr;       // [batch][W][n]
    int64_t *marg = nullptr;     // [batch][W][n]
    uint32_t *seen = nullptr;    // [batch][n]
    uint32_t *stale = nullptr;   // [batch][n]
    int8_t *l1 = nullptr;        // [batch][W][n]
};
pp_status launch_marginals_top2(pp_instance *inst, int batch, const int32_t *worker,
                                const uint32_t *mask, const int32_t *item_active, const Top2 &t2,
                                int64_t *profit, int64_t *oldsum, cudaStream_t st);


// Traceback of pp_tree_dp's bits.  With mask == nullptr it writes chosen[]
// bytes by node id (ABI); otherwise it is the planner's accept-and-update
// step (see pp_plan.cu) and writes holder-mask bits in preorder.
struct AcceptArgs {
    const int32_t *worker = nullptr;    // [batch] h per item
    const int64_t *best = nullptr;      // [batch] D[0][k]
    const int64_t *oldsum = nullptr;    // [batch] sum of p_h over the current T_h
    int32_t *active = nullptr;          // [batch] start still refining
    int32_t *improved = nullptr;        // [batch] set on an accepted update
    int32_t *accepted = nullptr;        // [batch] accepted-update counter
    uint32_t *mask = nullptr;           // [batch][n] holder masks (preorder)
    int greedy = 0;                     // 1: always accept (WorkerGreedy pass)
    // optional [batch]: item b walks the decision bits (and pruned-sweep data)
    // of DP item bits_item[b] of the workspace instead of item b
    const int32_t *bits_item = nullptr;
};
pp_status launch_traceback(pp_instance *inst, int batch, const DpWork &work, const DpGeom &g,
                           const int32_t *item_budget, uint8_t *chosen, const AcceptArgs *acc,
                           cudaStream_t st);

pp_status plan_impl(pp_instance *inst, int32_t S, const int32_t *orders, int32_t R, uint8_t *placement,
                    int64_t *objective, pp_plan_stats *stats, cudaStream_t st, bool orders_only = false);

// Safeguard candidates (requester-side): Independent, Popularity, LocalDedup
// holder masks in preorder (in inst->sg, valid until the next call), their
// objectives, and what they cost.
struct SafeguardRun {
    const uint32_t *masks = nullptr;     // [3][n], device
    const int64_t *obj = nullptr;        // [3], device
    int launches = 0, dp_launches = 0;
    int64_t cells = 0;
    bool enqueued = false;
};
// `beside`: other work of the instance runs meanwhile, so enqueue nothing if the
// DP's stack of skipped rows, which that work may use, would be needed
pp_status safeguards_enqueue(pp_instance *inst, cudaStream_t st, SafeguardRun *run, bool beside);
pp_status safeguards_read(const SafeguardRun &run, cudaStream_t st, int64_t *obj);

}  // namespace pp
