// Internal declarations shared by the translation units of libpp (host launchers + device view).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "pp.h"

namespace pp {

// Device view of one problem.  Ranks are an order-preserving recoding of the gamma doubles:
// 0 stands for +0.0, the all-ones value of the element type for +inf, 1..N for the gamma
// values in increasing order (equal doubles share a rank).  min/max/compare on ranks give the
// same selections as on the doubles (the sweep never does arithmetic on values).
struct Dev {
    int L, k, Lpad;            // Lpad: row stride in elements (32-byte multiple)
    int U;                     // number of distinct non-zero off-diagonal bandwidth values
    int elem;                  // bytes per state element: 2 or 4
    const uint64_t *bits;      // [L]
    const uint64_t *M;         // [L+1] prefix sums of layer memory
    const uint64_t *cap;       // [k]
    const uint32_t *bw;        // [k*k]
    const int16_t *lo;         // [k*L] lo[w*L+c'] = first c >= 0 whose successor segment c+1..c' fits w
                               //        (= c' when even the single layer c' does not fit)
    const int16_t *pair_u;     // [k*k] index into ubw of the pair's bandwidth, -1 if unusable
    const uint32_t *ubw;       // [U] distinct bandwidth values
    const uint32_t *masks;     // [2^k - 1] all non-empty masks by popcount, each level in revolving-door
                               //        order (neighbours differ by one node swapped for another)
    const uint32_t *level_off; // [k+2] masks of popcount j are masks[level_off[j] .. level_off[j+1])
    int16_t *pos;              // [L] position of layer c in the ascending order of bits
    int16_t *order;            // [L] layer at each position
    double *gu;                // [U*L] gu[u*L+i] = bits[order[i]] / ubw[u]  (ascending in i)
    uint32_t *cnt;             // [U*L] number of quotients below gu[u*L+i] (accumulated by the rank build)
    uint32_t *rk;              // [U*L] rank of gu[u*L+i] = 1 + cnt
    uint32_t *inv;             // [U*L+2] inv[r] = some entry e with rk[e] == r (equal ranks hold equal doubles)
    void *rank;                // [k*k*Lpad] rank[(w*k+v)*Lpad + c] of gamma[c][v][w], element type
    void *table;               // [2^k * k * Lpad] state rows, row (S, v) at (S*k+v)*Lpad
    uint64_t table_elems;      // elements of the state table / of the rank table: what an index
    uint64_t rank_elems;       //        may reach (checked only in the bounds-checking build)
    unsigned long long *best;  // packed (rank, popcount, mask, v) of the best final state
    int32_t *err;              // device error word (0 = fine, kErrBacktrack)
    const void *fast_meta;     // per-node window constants of the register-tiled sweep, or null
    const uint32_t *gen_meta;  // [k*Lpad] per-(node, position) lookup words of its general-window step, or null
    int gen_levels;            // levels of that step's sparse table (1 + floor(log2(longest window)))
    const void *pair_meta;     // per-node window constants of the two-mask sweep, or null
};

// Lets a kernel be launched with any amount of dynamic shared memory a block can have beside `own` bytes (or more) of its
// own.  The limit belongs to the kernel, not to a launch: set to what one call needs, it is lowered by another thread's
// smaller call between the two steps of this one, whose launch then fails.
constexpr size_t kBlockShared = (size_t)227 << 10;
template <typename... Params>
inline cudaError_t allow_shared(void (*kernel)(Params...), size_t own = 0)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kBlockShared - own));
}

static constexpr unsigned long long kNoBest = ~0ull;
static constexpr int32_t kErrBacktrack = 1;  // the backtrack found no predecessor (inconsistent table)
static constexpr int32_t kErrBounds = 3;     // bounds-checking build: an index left its table

// Bounds-checking build (-DPP_DEBUG_BOUNDS, libpp_dbg.so): every access to a table of the searches (states and
// ranks, the bounded search's rows, keys, maps and lists, the placement stage's table of bottlenecks) and every
// look of the scoring kernels into their tables goes through PP_IN_BOUNDS, which counts it, records kErrBounds
// in an error word and makes the caller skip the access when the index is outside the table.
// Nothing traps; the solve then reports PP_ERR_CUDA, a scoring kernel the status 255 for the plans of the
// block.  In the normal build the check is `true`.
struct Bounds {
    int32_t *err;
};
#ifdef PP_DEBUG_BOUNDS
static __device__ unsigned long long pp_checks;  // made by the kernels of this source
__device__ __forceinline__ bool pp_check(int32_t *err, bool ok)
{
    atomicAdd(&pp_checks, 1ull);
    if (!ok) atomicCAS(err, 0, kErrBounds);
    return ok;
}
#define PP_IN_BOUNDS(d, index, limit) pp::pp_check((d).err, (uint64_t)(index) < (uint64_t)(limit))
// an error word of the block; the block synchronises before the first check
#define PP_BLOCK_BOUNDS(name)          \
    __shared__ int32_t name##_word;    \
    const Bounds name{&name##_word};   \
    if (threadIdx.x == 0) name##_word = 0
#define PP_RESET(name) *(name).err = 0
#define PP_BROKEN(name) (*reinterpret_cast<volatile int32_t *>((name).err) != 0)
#define PP_CHECKS_OF(name)                                              \
    unsigned long long name##_checks()                                  \
    {                                                                   \
        unsigned long long n = 0, zero = 0;                             \
        if (cudaMemcpyFromSymbol(&n, pp_checks, sizeof n) != cudaSuccess || cudaMemcpyToSymbol(pp_checks, &zero, sizeof n) != cudaSuccess) return 0; \
        return n;                                                       \
    }
#else
#define PP_IN_BOUNDS(d, index, limit) true
#define PP_BLOCK_BOUNDS(name) [[maybe_unused]] const Bounds name{nullptr}
#define PP_RESET(name) (void)0
#define PP_BROKEN(name) false
#define PP_CHECKS_OF(name) unsigned long long name##_checks() { return 0; }
#endif
// Checks made by the kernels of one source since the last call (pp_debug_bounds_checks); synchronises.
unsigned long long prune_checks();
unsigned long long batch_checks();
unsigned long long match_checks();
unsigned long long eval_checks();
unsigned long long random_checks();

// final-state key: smaller is better; rank in the high bits, then popcount, mask, node
__host__ __device__ inline unsigned long long pack_best(uint32_t rank, int popc, uint32_t mask, int v)
{
    return ((unsigned long long)rank << 30) | ((unsigned long long)popc << 25) |
           ((unsigned long long)mask << 5) | (unsigned long long)v;
}

cudaError_t launch_rank_base(const Dev &d, cudaStream_t s, int *launches);
cudaError_t launch_sweep_generic(const Dev &d, int level, cudaStream_t s);
size_t fast_meta_bytes();
bool fast_meta_build(int L, int k, const int16_t *lo, void *out);
int gen_meta_build(int L, int k, int Lpad, const int16_t *lo, uint32_t *out);
bool fast_sweep_supported(const Dev &d);
// first_level: the kernel follows the rank build directly and must wait for it before reading anything
cudaError_t launch_sweep_fast(const Dev &d, int level, cudaStream_t s, bool first_level);
size_t pair_meta_bytes();
bool pair_meta_build(int L, int k, const int16_t *lo, void *out);
bool pair_sweep_takes(const Dev &d, int level, bool whenever_possible);
cudaError_t launch_sweep_pair(const Dev &d, int level, cudaStream_t s, bool first_level);
cudaError_t launch_finalize(const Dev &d, pp_solution *out, cudaStream_t s, bool dependent);
// What the evaluator and the random plans look up, laid out with the inputs of a problem as their
// kernels stage it in shared memory: output bits of the layers, bandwidths with a row and a column of
// zeros for "no such node", forward windows fwd[w * L + first] = layers from `first` on that fit node w
// (a row of zeros for no such node, one entry more for a segment that would start behind the chain).
struct PlanTables {
    size_t bits, bw, fwd, total;
};
__host__ __device__ inline PlanTables plan_tables(int L, int k)
{
    PlanTables t;
    t.bits = 0;
    t.bw = ((size_t)L * 8 + 15) & ~(size_t)15;
    t.fwd = t.bw + (((size_t)(k + 1) * (k + 1) * 4 + 15) & ~(size_t)15);
    t.total = t.fwd + ((((size_t)(k + 1) * L + 1) * 2 + 15) & ~(size_t)15);
    return t;
}
// early: the launch may start before the one in front of it on the stream has ended, and reads the tables at once.
// Not where the copy of the tables may still be under way.
cudaError_t launch_eval(const Dev &d, const unsigned char *tables, int64_t B, const uint8_t *nseg, const int32_t *ends,
                        const int32_t *nodes, double *beta, uint8_t *status, bool early, cudaStream_t s);
cudaError_t launch_eval_packed(const Dev &d, const unsigned char *tables, int64_t B, int64_t total, const uint8_t *nseg, const uint32_t *off,
                               const uint16_t *ends, const uint8_t *nodes, double *beta, uint8_t *status,
                               bool early, cudaStream_t s);
size_t batch_smem_bytes(int L, int k);
int batch_block_threads(bool narrow);
int batch_blocks_per_sm(int L, int k, bool narrow);
bool batch_narrow(int64_t B, int L, int k, int sms);
// Row numbering of the batched search, per (device, k): rows ordered by (popcount, mask, node), the masks
// listed by (popcount, value) with the first of each popcount, source mask | target node << 16 of every row
// with the first row of each popcount.
struct LaneTables {
    const uint32_t *rowoff = nullptr, *mlist = nullptr, *moff = nullptr, *rows = nullptr, *first = nullptr;
};
// narrow: blocks of few threads (batch_narrow).  early: may start beside the launch in front of it on the stream, which is a
// piece of the same batch.
cudaError_t launch_batch(int64_t B, bool narrow, int L, int k, const LaneTables &lt, int sms, const uint64_t *bits, const uint64_t *mem,
                         const uint64_t *cap, const uint32_t *bw, double *beta, int32_t *m,
                         int32_t *cuts, int32_t *placement, int8_t *status, bool early, cudaStream_t s);
// Many-instance search with one instance per lane (pp_batch_lanes.cu): tables of a chunk of
// instances in global memory, instance-minor in pieces of two words, so that the 32 lanes of a warp read
// 256 neighbouring bytes.  Group g holds instances 32 g .. 32 g + 31 of the chunk.
struct BatchLanes {
    uint32_t *table;          // [group][compact row][LH / 2][32][2]: states, two cut positions per word
    uint32_t *rank;           // [group][v * k + w][LH / 2][32][2]: gamma ranks, same packing
    uint32_t *len;            // [group][w][LH / 2][32][2]: window lengths c' - lo_w(c'), same packing
    uint32_t *win;            // [group][w][LH][32][2]: per cut position the two sparse-table cells whose minimum
                              // is the window minimum, as byte offsets into a warp's table (see pp_batch_lanes.cu)
    unsigned long long *key;  // [group][32]: smallest final state so far (value, popcount, mask, node)
    int8_t *flag;             // [group][32]: 1 = an input beyond the limits
    int32_t *err;             // device error word (bounds-checking build: kErrBounds when an index left its table)
    size_t table_words, rank_words, len_words, win_words;  // sizes of the four tables in 32-bit words
    const uint32_t *rowoff;   // [2^k]: compact row of (S, lowest node of S), rows ordered by (popcount, mask, node)
    const uint32_t *mlist;    // masks by (popcount, value)
    const uint32_t *moff;     // [k + 2]: first entry of each popcount in mlist
    uint32_t rows;            // k * 2^(k-1)
    int LH;                   // words per row in these tables: 4, 8, 12 or 16
};
// Instances whose tables share its scratch memory at a time.
constexpr int64_t kBatchLanesChunk = 4096;
// Nodes up to which chains of up to eight layers (four words a row) go an instance to a lane; with more they go to a warp,
// whatever the size of the batch, and the levels of more nodes are not there.
constexpr int kLanesShortK = 7;
bool batch_lanes_takes(int64_t B, int L, int k, int sms);
int batch_lanes_words(int L);
// test hook: n quotients as the preparing kernel ranks them, and by CUDA's division
cudaError_t launch_quotients(int64_t n, const uint64_t *bits, const uint32_t *kbps, double *by_reciprocal, double *divided,
                             cudaStream_t s);
// prep: one block per instance ranks gamma and writes the instance's column of the tables
cudaError_t launch_batch_prep(int64_t B, int L, int k, const uint64_t *bits, const uint64_t *mem,
                              const uint64_t *cap, const uint32_t *bw, const BatchLanes &t, cudaStream_t s);
// the levels and the backtrack over a prepared chunk; *launches counts the kernels queued
cudaError_t launch_batch_lanes(int64_t B, int L, int k, const uint64_t *bits, const uint32_t *bw,
                               const BatchLanes &t, double *beta, int32_t *m, int32_t *cuts,
                               int32_t *placement, int8_t *status, cudaStream_t s);
// The same with an instance to a warp (pp_batch_warps.cu).  others: the tables of k - 1 nodes
bool batch_warps_takes(int64_t B, int L, int k);
cudaError_t launch_batch_warps(int64_t B, int L, int k, const LaneTables &others, int sms, const uint64_t *bits, const uint64_t *mem,
                               const uint64_t *cap, const uint32_t *bw, double *beta, int32_t *m, int32_t *cuts,
                               int32_t *placement, int8_t *status, cudaStream_t s);
// The search as a bounded sparse frontier (pp_prune.cu), one launch per solve.
struct PruneCtl {              // device; the kernel leaves it as it found it
    unsigned long long best;   // best final state of the levels done: pack_best of its key
    unsigned long long count[64];  // node sets appended to the frontier by the level of that many nodes (a second
                               // search over the class of the optimum counts from 32); in the upper half the
                               // blocks that have arrived at the level's end
    uint32_t left;             // blocks that have left
    uint32_t failed;           // a barrier ran out of polls: the other blocks need not wait any longer
    int32_t err;               // bounds-checking build: kErrBounds when an index left its table
};
struct PruneNote {             // what the host learns about a launch
    long long ns;              // duration on the device
    int32_t dense;             // 1 = the frontier outgrew its rows, or is too large to resolve a class in
    int32_t thresholds;        // 1 = the result is that of the search by thresholds, 2 = it left the search to the frontier; 0: not asked
};
struct PruneDev {
    int L, k, Lp;              // Lp: row stride in keys
    int clustered;             // the blocks are one cluster (set by the launch)
    uint32_t arrivals;         // blocks a barrier in global memory waits for, and polls before it gives up (set by
    int polls;                 // the launch)
    uint32_t late;             // bounds-checking build: number + 1 of the block that pp_debug_late holds up, or 0
    int key_shift;             // keys: 1 + (bits of the double - key_base) >> key_shift
    unsigned long long key_base, key_top;  // bits of the smallest and of the largest positive term
    unsigned long long key_floor;  // bits of a value that no plan is below
    uint32_t fallback;         // 1 = the caller has another search (note->dense asks for it)
    uint32_t whole;            // nodes that hold the whole chain
    uint32_t tight_levels;     // bit j: some rest of the chain may not fit the nodes that j used ones leave
    const int16_t *lo;         // [k*L] window starts (see Dev), or null: the kernel works them out
    uint32_t *live;            // [2^k] nodes v whose row (S, v) is kept
    unsigned long long *rowmap;  // [2^k * k] (S, v): smallest key << 32 | row
    uint32_t *list;            // [2^k] node sets of the frontier, level after level
    uint32_t *gam;             // [k*k*Lp] key of gamma[c][v][w] at (w*k + v)*Lp + c
    uint32_t *gmin;            // [k*k] its minimum over the cut positions
    uint32_t *rows;            // [row_cap * Lp]
    unsigned long long row_cap;
    uint32_t *seg;             // Eq. 1: [k*L*Lp] keys of the compute times of every run of layers; null for Eq. 2
    PruneCtl *ctl;
    pp_solution *out;          // device or mapped host memory
    PruneNote *note;           // device or mapped host memory
};
// Test hook (pp_debug_starve): polls of the next launch whose blocks meet, which then waits for one block
// more than it has; 0 = an ordinary launch.  Asking for it uses it up.
int starved_polls();
// Test hook (pp_debug_late): polls of the next search by thresholds, in which block *block comes late; 0 = an ordinary one.
int late_polls(int *block);
void prune_key_range(double lo, double hi, PruneDev *d);
void prune_node_bounds(const uint64_t *cap, uint64_t total, PruneDev *d);
int prune_row_pad(int L, int k);
void prune_ctl_init(PruneCtl *c);
// Tables of the bounded search, in scratch memory or in a block's shared memory; the rows come last.
struct SparseLayout {
    size_t live, rowmap, list, gam, gmin, rows;
};
__host__ __device__ inline SparseLayout sparse_layout(int k, int Lp)
{
    SparseLayout w;
    size_t o = 0;
    auto take = [&o](size_t bytes) { size_t at = o; o = (o + bytes + 255) & ~(size_t)255; return at; };
    w.live = take((size_t)4 << k);
    w.rowmap = take((size_t)k * 8 << k);
    w.list = take((size_t)4 << k);
    w.gam = take((size_t)k * k * Lp * 4);
    w.gmin = take((size_t)k * k * 4);
    w.rows = o;
    return w;
}
struct PruneHost {             // host arrays, read before launch_prune returns
    const uint64_t *bits, *M, *cap;  // [L], [L+1] memory prefix sums, [k]
    const uint32_t *bw;        // [k*k]
    const uint64_t *Wp;        // Eq. 1 only: [L+1] prefix sums of the layers' work, [k] speeds
    const uint32_t *speed;
};
// whether the search of such a problem needs no scratch in global memory; compute: the bounded one of Eq. 1
bool prune_in_shared(int L, int k, bool compute);
bool prune_in_shared(const PruneDev &d, const PruneHost &h);  // Eq. 1, by thresholds first or not
cudaError_t launch_prune(const PruneDev &d, const PruneHost &h, int sms, cudaStream_t s);
// Random comparison baseline (Section 4): P plans of problem d from 2 k draws each.
cudaError_t launch_random_plans(const Dev &d, const unsigned char *tables, int64_t P, const uint32_t *draws, uint8_t *nseg,
                                int32_t *ends, int32_t *nodes, bool early, cudaStream_t s);
// Greedy comparison baseline (Section 4), one warp per instance.
cudaError_t launch_greedy(int64_t B, int L, int k, const uint64_t *bits, const uint64_t *mem,
                          const uint64_t *cap, const uint32_t *bw, double *beta, int32_t *m, int32_t *cuts,
                          int32_t *place, int8_t *status, cudaStream_t s);

// Partition stage of the paper's heuristic (Algorithm 1), one warp per chain.
size_t partition_smem_bytes(int L);
cudaError_t launch_partition_minsum(int64_t B, int L, int cap_seg, const uint64_t *weight, const uint64_t *mem,
                                    const uint64_t *kappa, uint64_t *cost, int32_t *m, int32_t *cuts,
                                    uint64_t *sizes, int8_t *status, cudaStream_t s);
// The same for a few chains in host arrays that travel as kernel parameters (partition_as_params says which);
// the outputs are device or page-locked memory.
bool partition_as_params(int64_t B, int L);
cudaError_t launch_partition_params(int64_t B, int L, int cap_seg, const uint64_t *weight, const uint64_t *mem,
                                    const uint64_t *kappa, uint64_t *cost, int32_t *m, int32_t *cuts, uint64_t *sizes,
                                    int8_t *status, cudaStream_t s);
// Colour-coding k-path search of the placement stage (Algorithm 2's K-PATH), one block per query.
size_t kpath_smem_bytes(int kk);
cudaError_t launch_kpath(int n, int kk, int64_t Q, const uint32_t *bw, const uint32_t *threshold, const int32_t *start,
                         const int32_t *end, const unsigned long long *alive, const uint8_t *colours, uint8_t *found,
                         int32_t *path, cudaStream_t s);
// Placement stage in one launch (pp_match.cu).
struct MatchRun {
    int32_t first, cuts;       // a run of cuts of one class, in serving order
};
struct MatchOut {
    int32_t bounds;            // bounds-checking build: 1 when an index left the table
    int32_t status, nodes[64];
    uint32_t threshold[64];
};
struct MatchDev {
    int n, n_cuts, n_runs, trials, kk;  // kk: vertices of the longest path
    const uint32_t *bw, *draws;
    const MatchRun *runs;
    unsigned long long *records;  // [2][2][stride][4]: by `half`, by the parity of the run, by block; this half is
    int half, stride;             // zero before the launch and the launch zeroes the other; stride: blocks at most
    int posts, polls;             // records a run waits for, and polls before it gives up (set by the launch)
    MatchOut *out;             // mapped host memory
};
size_t match_smem_bytes(int n, int kk);
// The inputs one after another: bandwidths, draws, at an even word the runs.
__host__ __device__ inline size_t match_runs_at(int n, int trials) { return ((size_t)n * n + (size_t)trials * n + 1) & ~(size_t)1; }
bool match_as_params(size_t words);
size_t match_record_bytes(int sms);
// d.bw null: the inputs go with the launch, from host memory.
cudaError_t launch_match(const MatchDev &d, const uint32_t *in, size_t words, cudaStream_t s);
// Issue-rate probe (pp_probe.cu): `blocks` blocks of 1024 threads, cycles[b] = SM clocks block b took.
cudaError_t launch_probe(int op, int iters, int blocks, long long *cycles, uint32_t *sink, cudaStream_t s);
double probe_instr_per_block(int iters);

}  // namespace pp
