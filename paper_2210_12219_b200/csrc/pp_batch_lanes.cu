// Many-instance exact search, one instance per lane.
//
// The block-per-instance kernel (pp_batch.cu) spends most of its instructions on addressing: a
// thread owns one word of one row and has to find out which.  Here a warp owns one source mask P of
// 32 instances at once, lane <-> instance.  Every lane then walks the same masks, nodes and cut
// positions, so all of that is uniform and unrolled, and the only per-lane data are the states, the
// gamma ranks and the window lengths.  Those live in global memory, instance-minor: the 32 lanes of a
// warp read 32 neighbouring pieces of two words.  Batches whose tables are larger than L2 (4096 x (k = 8, L = 24): 219 MB
// against 126) go an instance to a warp (batch_warps_takes).
//
// Per chunk of instances:
//   1. k_lanes_prep, one block per instance: staging, windows, the ranking of gamma (Eq. 3); writes
//      the instance's column of the rank table, the window lengths, the base frontier and the best
//      single-node plan;
//   2. one launch per popcount level, k_lanes_level<NV, LH>: a warp takes (group of 32 instances,
//      source mask P of NV nodes), keeps the NV rows of P in registers (two cut positions per 32-bit
//      word, LH words per row), and for every node w outside P forms
//      g[c] = min_v max(dp[P][v][c], rank[v][w][c]) with packed 16-bit min/max, takes the window
//      minimum over [lo_w(c'), c'-1] from a sparse table of g in the lane's own column of shared
//      memory (the one place where a lane needs an index of its own), stores the row of (P + w, w), and keeps the smallest final state
//      (value, popcount, mask, node), merged into the instance's key with one atomic per lane;
//   3. k_lanes_back, one warp per instance: the backtrack by the
//      threshold rule, lanes over the candidates.
// Same recurrence, final choice and backtrack rule as the single-instance path (pp_sweep.cu).
#include <algorithm>

#include "pp_blocks.cuh"

namespace pp {

namespace {

constexpr int kLevelWarps = 4;
constexpr int kLevelFourBlocks = 5;  // source masks of up to this many nodes: registers capped for four blocks per SM
// Registers for twelve blocks an SM; shared memory leaves room for 11 at k = 8, L = 24 (19 KB a block) and for nine at
// L = 32 (23 KB), the widest shape.
constexpr int kPrepThreads = 128, kPrepBlocks = 12;
constexpr int kFlagLimit = 1;     // BatchLanes::flag: an input beyond the limits
constexpr int kBackWarps = 8;
constexpr int kLanesMaxK = 8;   // NV <= 7 rows of a source mask in registers
constexpr int kLanesMaxL = 32;  // LH <= 16 words per row

// Sparse table of one row g in a warp's shared memory: level s holds T_s[c] = min g[c - 2^s + 1 .. c],
// two positions per 32-bit word like the rows, word (s, wd) of lane l at byte ((s LH + wd) 32 + l) 4:
// every lane reads and writes its own bank.  Word kWinLevels * LH holds +inf.  A cell is named by
// its byte offset without the lane's part, which fits 16 bits.
constexpr int kWinLevels = 5;  // windows of up to 31 positions
__host__ __device__ inline uint32_t win_cell(int s, int pos, int LH)
{
    return (uint32_t)((s * LH + (pos >> 1)) * 128 + (pos & 1) * 2);
}
__host__ __device__ inline size_t win_bytes_per_warp(int LH) { return (size_t)(kWinLevels * LH + 1) * 128; }

// Checked access to one of the tables of BatchLanes: in the bounds-checking build an address outside
// [base, base + words) is recorded in the error word and the access skipped (a load gives +inf); in
// the normal build PP_IN_BOUNDS is `true` and these are plain loads and stores.
__device__ __forceinline__ uint32_t ld_table(const BatchLanes &t, const uint32_t *p, const uint32_t *base, size_t words)
{
    return PP_IN_BOUNDS(t, (size_t)(p - base), words) ? *p : 0xFFFFFFFFu;
}
__device__ __forceinline__ void st_table(const BatchLanes &t, uint32_t *p, const uint32_t *base, size_t words, uint32_t v)
{
    if (PP_IN_BOUNDS(t, (size_t)(p - base), words)) *p = v;
}

// Word e of an instance's column (rows of LH words one after another): the 32 instances of a group lie
// side by side in pieces of kPiece words, so that a lane moves a piece at a time.
constexpr int kPiece = 2;   // 4096 x (k = 8, L = 24), us a call: 1 word 261, 2 words 235, 4 words 245 (spills in the level kernels)
struct alignas(4 * kPiece) Piece {
    uint32_t w[kPiece];
};
__host__ __device__ inline size_t word_at(size_t e) { return e / kPiece * (32 * kPiece) + e % kPiece; }
__device__ __forceinline__ Piece ld_piece(const BatchLanes &t, const uint32_t *p, const uint32_t *base, size_t words)
{
    Piece x;
    if (PP_IN_BOUNDS(t, (size_t)(p - base), words)) {
        x = *reinterpret_cast<const Piece *>(p);
    } else {
        for (int i = 0; i < kPiece; ++i) x.w[i] = 0xFFFFFFFFu;
    }
    return x;
}
__device__ __forceinline__ void st_piece(const BatchLanes &t, uint32_t *p, const uint32_t *base, size_t words, const Piece &v)
{
    if (PP_IN_BOUNDS(t, (size_t)(p - base), words)) *reinterpret_cast<Piece *>(p) = v;
}

// Test hook: the quotients of n pairs, and the same by CUDA's division.
__global__ void k_quotients(const int64_t n, const uint64_t *__restrict__ bits, const uint32_t *__restrict__ kbps,
                            double *__restrict__ by_reciprocal, double *__restrict__ divided)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double x = (double)bits[i], b = (double)kbps[i];
        by_reciprocal[i] = quotient(x, b, __drcp_rn(b));
        divided[i] = __ddiv_rn(x, b);
    }
}

// Shared memory of an instance in the preparing kernel (byte offsets; every part 16-byte aligned).
// Distinct sizes, distinct bandwidths and their reciprocals: where val[] goes later, which is the larger one from 288
// quotients on (k = 4, L = 9 has 108: 720 bytes more a block).
constexpr size_t kDoubles = 32 + 2 * 56;
struct PrepLayout {
    size_t val, key, rk, M, bits, dbits, cap, bw, ubw, hist, pair_u, cls, total;
};

__host__ __device__ inline PrepLayout prep_layout(int L, int k)
{
    PrepLayout p;
    const size_t n = (size_t)k * (k - 1) * L;  // quotients
    size_t o = 0;
    auto take = [&o](size_t bytes) { size_t at = o; o = (o + bytes + 15) & ~(size_t)15; return at; };
    p.val = take(n * 4 > kDoubles * 8 ? n * 4 : kDoubles * 8);
    p.key = take(n * 4);
    p.rk = take(n * 2);
    p.M = take(33 * 8);
    p.bits = take(32 * 8);
    p.dbits = take(32 * 8);
    p.cap = take(8 * 8);
    p.bw = take(64 * 4);
    p.ubw = take(64 * 4);
    p.hist = take((size_t)kRankBuckets * 4);
    p.pair_u = take(64);
    p.cls = take(32);
    p.total = o;
    return p;
}

// One block of four warps per instance (L <= 32 layers, k * k <= 64 node pairs): staging, the windows, the
// ranking of gamma (Eq. 3), and the instance's column of the tables of BatchLanes.
//   * distinct usable bandwidths and distinct transfer sizes listed in order of first appearance;
//   * window start lo_w(c2) by a branch-free binary search over the memory prefix sums;
//   * ranks by rank_quotients, the quotients of its first pass by the reciprocals of the distinct bandwidths, three fp64
//     instructions each where a division and two conversions take some thirty (4096 x (k = 8, L = 24) 219.2 -> 217.0 us a
//     call, L = 32 296.6 -> 294.2, L = 9 150.7 -> 149.6; 2048 x (8, 24) 137.2 -> 136.3; 4096 x (5, 24) 63.1 -> 62.6, (4, 12)
//     42.1 -> 41.6; the runs of one side lie within 0.3 % of their median).
// What is left is a chain of short dependent phases, a third as long with four warps to an instance as with
// one; the SM's other instances hide it.
__global__ void __launch_bounds__(kPrepThreads, kPrepBlocks)
k_lanes_prep(const BatchLanes t, const int64_t B, const int L, const int k, const uint64_t *__restrict__ g_bits,
             const uint64_t *__restrict__ g_mem, const uint64_t *__restrict__ g_cap,
             const uint32_t *__restrict__ g_bw)
{
    extern __shared__ __align__(16) unsigned char smem_prep[];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const PrepLayout lay = prep_layout(L, k);
    uint32_t *s_val = reinterpret_cast<uint32_t *>(smem_prep + lay.val);
    double *s_size = reinterpret_cast<double *>(smem_prep + lay.val), *s_link = s_size + 32, *s_recip = s_link + 56;
    unsigned long long *M = reinterpret_cast<unsigned long long *>(smem_prep + lay.M);
    unsigned long long *s_bits = reinterpret_cast<unsigned long long *>(smem_prep + lay.bits);
    unsigned long long *s_cap = reinterpret_cast<unsigned long long *>(smem_prep + lay.cap);
    uint32_t *s_bw = reinterpret_cast<uint32_t *>(smem_prep + lay.bw);
    uint32_t *ubw = reinterpret_cast<uint32_t *>(smem_prep + lay.ubw);
    uint32_t *hist = reinterpret_cast<uint32_t *>(smem_prep + lay.hist);
    uint32_t *s_key = reinterpret_cast<uint32_t *>(smem_prep + lay.key);
    uint16_t *rk = reinterpret_cast<uint16_t *>(smem_prep + lay.rk);
    unsigned long long *dbits = reinterpret_cast<unsigned long long *>(smem_prep + lay.dbits);
    int8_t *pair_u = reinterpret_cast<int8_t *>(smem_prep + lay.pair_u);
    uint8_t *cls = smem_prep + lay.cls;
    __shared__ uint32_t s_first[3], s_sum[kPrepThreads / 32];
    const int LH = t.LH, kk = k * k;
    const uint32_t FULL = 0xFFFFFFFFu;
    // floor(x / k) for x < 64, floor(x / LH) for x < k k LH <= 1024
    const uint32_t recip_k = (65536u + (uint32_t)k - 1u) / (uint32_t)k;
    const uint32_t recip_LH = (65536u + (uint32_t)LH - 1u) / (uint32_t)LH;
    for (int64_t inst = blockIdx.x; inst < B; inst += gridDim.x) {
        __syncthreads();
        // ---- staging, prefix sums of the memory ----
        bool bad = false;
        if (wid == 0) {
            const unsigned long long b = lane < L ? g_bits[inst * L + lane] : 0ull;
            unsigned long long x = lane < L ? g_mem[inst * L + lane] : 0ull;
            bad = b >= PP_MAX_BITS;
            s_bits[lane] = b;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(FULL, x, o);
                if (lane >= o) {
                    if (y > ~0ull - x) bad = true;  // the 64-bit sum would wrap: PP_ERR_LIMIT
                    x += y;
                }
            }
            if (lane == 0) M[0] = 0ull;
            M[lane + 1] = x;  // beyond L: the total, never read
        } else if (wid < 3) {
            const int p = tid - 32, v = (int)(((uint32_t)p * recip_k) >> 16);
            const uint32_t x = p < kk ? g_bw[inst * kk + p] : 0u;
            bad = x >= PP_MAX_KBPS;
            s_bw[p] = p < kk && v != p - v * k ? x : 0u;  // 0: no usable link
        } else if (lane < k) {
            s_cap[lane] = g_cap[inst * k + lane];
        }
        bad = __syncthreads_or(bad);
        // ---- distinct usable bandwidths, distinct sizes, in order of first appearance ----
        uint32_t x = 0;
        int f = 0;
        if (wid < 2) {
            x = s_bw[tid];
#pragma unroll 4
            for (int p4 = 60; p4 >= 0; p4 -= 4) {  // descending: the first appearance stays
                const uint4 q = *reinterpret_cast<const uint4 *>(s_bw + p4);
                f = q.w == x ? p4 + 3 : f;
                f = q.z == x ? p4 + 2 : f;
                f = q.y == x ? p4 + 1 : f;
                f = q.x == x ? p4 : f;
            }
            const uint32_t firsts = __ballot_sync(FULL, x != 0u && f == tid);
            if (lane == 0) s_first[wid] = firsts;
        } else if (wid == 3) {
            const unsigned long long mine = s_bits[lane];
#pragma unroll 4
            for (int i = 30; i >= 0; i -= 2) {
                const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(s_bits + i);
                f = q.y == mine ? i + 1 : f;
                f = q.x == mine ? i : f;
            }
            const uint32_t firsts = __ballot_sync(FULL, lane < L && f == lane);
            const int c = __popc(firsts & ((1u << f) - 1u));
            cls[lane] = (uint8_t)c;
            if (lane < L && f == lane) {
                dbits[c] = mine;
                s_size[c] = (double)mine;
            }
            if (lane == 0) s_first[2] = firsts;
        }
        // ---- windows, base frontier ----
        {
            uint32_t *lT = t.len + (size_t)(inst >> 5) * (size_t)(k * LH) * 32 + (inst & 31) * kPiece;
            uint32_t *tT = t.table + (size_t)(inst >> 5) * (size_t)t.rows * LH * 32 + (inst & 31) * kPiece;
            uint32_t *wT = t.win + (size_t)(inst >> 5) * (size_t)(k * 2 * LH) * 32 + (inst & 31) * kPiece;
            const unsigned long long Mc = M[lane + 1];  // memory of layers 0..lane
            for (int w = 3 - wid; w < k; w += kPrepThreads / 32) {
                const unsigned long long capw = s_cap[w];
                // c* = number of prefix sums M[0..lane+1] below M[lane+1] - cap: the first start layer
                // from which the segment ending at this layer fits; window start = max(c* - 1, 0)
                const unsigned long long thr = Mc > capw ? Mc - capw : 0ull;
                int cs = 0;
#pragma unroll
                for (int step = 32; step; step >>= 1)
                    if (cs + step <= lane + 2 && M[cs + step - 1] < thr) cs += step;
                const int lo = cs > 0 ? cs - 1 : 0;
                const uint32_t len = lane < L ? (uint32_t)(lane - lo) : 0u;
                const uint32_t inf = (lane < L && Mc <= capw) ? 0u : 0xFFFFu;
                const uint32_t len0 = __shfl_sync(FULL, len, 2 * lane), len1 = __shfl_sync(FULL, len, 2 * lane + 1);
                const uint32_t inf0 = __shfl_sync(FULL, inf, 2 * lane), inf1 = __shfl_sync(FULL, inf, 2 * lane + 1);
                // window [lo, lane - 1] of length len >= 1 = union of the two runs of 2^s positions
                // that end at lane - 1 and that start at lo, s = floor(log2 len): their sparse-table
                // cells; an empty window reads the cell that holds +inf
                uint32_t code = win_cell(kWinLevels, 0, LH) * 0x00010001u;
                if (len != 0u) {
                    const int sl = 31 - __clz((int)len);
                    code = win_cell(sl, lane - 1, LH) | (win_cell(sl, lo + (1 << sl) - 1, LH) << 16);
                }
                // position 0 has no window: its entry carries the highest level this node's windows read
                const uint32_t longest = __reduce_max_sync(FULL, len);
                if (lane == 0) code = longest > 1u ? (uint32_t)(31 - __clz((int)longest)) : 0u;
                if (lane < 2 * LH) st_table(t, wT + word_at(w * 2 * LH + lane), t.win, t.win_words, code);
                if (lane < LH) {
                    st_table(t, lT + word_at(w * LH + lane), t.len, t.len_words, lane < 16 ? len0 | (len1 << 16) : 0u);
                    st_table(t, tT + word_at((size_t)t.rowoff[1u << w] * LH + lane), t.table, t.table_words,
                             lane < 16 ? inf0 | (inf1 << 16) : 0xFFFFFFFFu);
                }
            }
        }
        __syncthreads();
        const uint32_t m0 = s_first[0], m1 = s_first[1];
        const int n0 = __popc(m0), U = n0 + __popc(m1);
        if (wid < 2) {
            const int u = x == 0u ? -1 : f < 32 ? __popc(m0 & ((1u << f) - 1u)) : n0 + __popc(m1 & ((1u << (f - 32)) - 1u));
            pair_u[tid] = (int8_t)u;
            if (x != 0u && f == tid) {
                ubw[u] = x;
                s_link[u] = (double)x;
                s_recip[u] = __drcp_rn((double)x);
            }
        }
        if (tid == kPrepThreads - 1) {
            unsigned long long best = kNoBest;
            for (int v = k - 1; v >= 0; --v)
                if (M[L] <= s_cap[v]) best = pack_best(0u, 1, 1u << v, v);
            t.key[inst] = best;
            t.flag[inst] = (int8_t)(bad ? kFlagLimit : 0);
        }
        // ---- ranks of the quotients ----
        {
            const unsigned long long b = s_bits[lane];
            const uint32_t p0 = s_bw[lane], p1 = s_bw[lane + 32];
            const uint32_t least = __reduce_min_sync(FULL, lane < L && b ? __float_as_uint(__ull2float_rd(b)) : 0x7F800000u);
            const uint32_t most = __reduce_max_sync(FULL, lane < L ? __float_as_uint(__ull2float_ru(b)) : 0u);
            const uint32_t fast = __reduce_max_sync(FULL, max(p0, p1));
            const uint32_t slow = __reduce_min_sync(FULL, min(p0 ? p0 : FULL, p1 ? p1 : FULL));
            rank_quotients<kPrepThreads, uint32_t, 11>(dbits, ubw, U, __popc(s_first[2]),
                                                       [&](int u, int d) { return quotient(s_size[d], s_link[u], s_recip[u]); },
                                                       __ddiv_rd((double)__uint_as_float(least), (double)fast),
                                                       __ddiv_ru((double)__uint_as_float(most), (double)slow), s_key, s_val,
                                                       hist, rk, s_sum);
        }
        // ---- rank table, two positions per word: rank[v][w][c] = rank of (bandwidth of v -> w, layer c) ----
        {
            const int D = __popc(s_first[2]);
            uint32_t *rT = t.rank + (size_t)(inst >> 5) * (size_t)(kk * LH) * 32 + (inst & 31) * kPiece;
            for (int e = tid; e < kk * LH; e += kPrepThreads) {
                const int pr = (int)(((uint32_t)e * recip_LH) >> 16), c0 = 2 * (e - pr * LH);
                const int u = pair_u[pr];
                const uint32_t a = u >= 0 && c0 < L ? rk[u * D + cls[c0]] : 0xFFFFu;
                const uint32_t c = u >= 0 && c0 + 1 < L ? rk[u * D + cls[c0 + 1]] : 0xFFFFu;
                st_table(t, rT + word_at(e), t.rank, t.rank_words, a | (c << 16));
            }
        }
    }
}

__device__ __forceinline__ void st_shared_u32(uint32_t addr, uint32_t v)
{
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_shared_u16(uint32_t addr)
{
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
    return v;
}

template <int NV, int LH>
__global__ void __launch_bounds__(kLevelWarps * 32, NV <= kLevelFourBlocks ? 4 : 3)
k_lanes_level(const BatchLanes t, const int64_t B, const int k, const int L, const int split)
{
    // Launched as a programmatic dependent of the kernel before it: nothing is read before that
    // kernel is complete, and the next one may be scheduled as soon as this one's blocks retire.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const int lane = threadIdx.x & 31;
    extern __shared__ __align__(16) unsigned char smem_level[];
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem_level) +
                           (uint32_t)((threadIdx.x >> 5) * win_bytes_per_warp(LH)) + (uint32_t)lane * 4u;
    // A state of j segments ends at layer j - 1 at the earliest: rows of this level's sources (NV
    // nodes) are +inf before position NV - 1 and the rows written here before position NV.  Words
    // that hold only such positions are neither read, computed nor written, here and in the next
    // level alike; their cells of the sparse table are set to +inf once.
    constexpr int W0 = (NV - 1) / 2;  // first word of a source row that can hold a state
    constexpr int C0 = NV;            // first position of a target row that can
    constexpr int O0 = NV / 2;        // its word: the first one stored (the next level's W0)
    st_shared_u32(sbase + win_cell(kWinLevels, 0, LH), 0xFFFFFFFFu);
#pragma unroll
    for (int sl = 0; sl < kWinLevels; ++sl)
#pragma unroll
        for (int wd = 0; wd < W0; ++wd) st_shared_u32(sbase + win_cell(sl, 2 * wd, LH), 0xFFFFFFFFu);
    const uint32_t nmasks = t.moff[NV + 1] - t.moff[NV];
    const int64_t G = (B + 31) >> 5;
    // a level with few source masks gives the targets of one mask to `split` warps
    const int64_t items = G * nmasks * split;
    const uint32_t full = (1u << k) - 1u;
    const int wfin = (L - 1) >> 1, sfin = ((L - 1) & 1) * 16;
    for (int64_t item = (int64_t)blockIdx.x * kLevelWarps + (threadIdx.x >> 5); item < items;
         item += (int64_t)gridDim.x * kLevelWarps) {
        const int64_t g = item / (nmasks * split);
        const uint32_t within = (uint32_t)(item - g * (nmasks * split));
        const uint32_t P = t.mlist[t.moff[NV] + within / (uint32_t)split];
        const int part = (int)(within % (uint32_t)split);
        // lanes past the end of the batch read the last instance's column and store to their own
        const int64_t left = B - g * 32;
        const int valid = left < 32 ? (int)left : 32;
        const int col = lane < valid ? lane : valid - 1;
        const uint32_t *tab = t.table + (size_t)g * t.rows * (LH * 32) + col * kPiece;
        uint32_t *tabw = t.table + (size_t)g * t.rows * (LH * 32) + lane * kPiece;
        const uint32_t *rk = t.rank + (size_t)g * (size_t)(k * k) * (LH * 32) + col * kPiece;
        const uint32_t *wn = t.win + (size_t)g * (size_t)(k * 2) * (LH * 32) + col * kPiece;
        uint32_t d[NV][LH];
        int vs[NV];
        {
            const uint32_t row0 = t.rowoff[P];
            uint32_t rem = P;
#pragma unroll
            for (int vi = 0; vi < NV; ++vi) {
                vs[vi] = __ffs(rem) - 1;
                rem &= rem - 1;
#pragma unroll
                for (int q = W0 / kPiece; q < LH / kPiece; ++q) {
                    const Piece x = ld_piece(t, tab + word_at((size_t)(row0 + vi) * LH + kPiece * q), t.table, t.table_words);
#pragma unroll
                    for (int i = 0; i < kPiece; ++i) d[vi][kPiece * q + i] = x.w[i];
                }
            }
        }
        unsigned long long key = kNoBest;
        int turn = part;
        for (uint32_t wrem = full & ~P; wrem; wrem &= wrem - 1) {
            if (turn-- != 0) continue;  // another warp's target
            turn = split - 1;
            const int w = __ffs(wrem) - 1;
            // the window cells of this node, asked for before anything else; position 0 has no window
            // and its entry carries the highest level of the sparse table this (instance, node) reads
            uint32_t cw[2 * LH];
#pragma unroll
            for (int q = C0 / kPiece; q < 2 * LH / kPiece; ++q) {
                const Piece x = ld_piece(t, wn + word_at((size_t)(w * 2 * LH) + kPiece * q), t.win, t.win_words);
#pragma unroll
                for (int i = 0; i < kPiece; ++i) cw[kPiece * q + i] = x.w[i];
            }
            const uint32_t lvl = C0 < kPiece ? cw[0] : ld_table(t, wn + word_at((size_t)(w * 2 * LH)), t.win, t.win_words);
            uint32_t gg[LH];
            auto rank_row = [&](int vi, int q) {
                return ld_piece(t, rk + word_at((size_t)((vs[vi] * k + w) * LH) + kPiece * q), t.rank, t.rank_words);
            };
#pragma unroll
            for (int q = W0 / kPiece; q < LH / kPiece; ++q) {
                const Piece a = rank_row(0, q);
#pragma unroll
                for (int i = 0; i < kPiece; ++i) gg[kPiece * q + i] = __vmaxu2(d[0][kPiece * q + i], a.w[i]);
            }
#pragma unroll
            for (int vi = 1; vi + 1 < NV; vi += 2) {
#pragma unroll
                for (int q = W0 / kPiece; q < LH / kPiece; ++q) {
                    const Piece a = rank_row(vi, q), b = rank_row(vi + 1, q);
#pragma unroll
                    for (int i = 0; i < kPiece; ++i) {
                        const int wd = kPiece * q + i;
                        gg[wd] = __vimin3_u16x2(gg[wd], __vmaxu2(d[vi][wd], a.w[i]), __vmaxu2(d[vi + 1][wd], b.w[i]));
                    }
                }
            }
            if (!(NV & 1)) {
#pragma unroll
                for (int q = W0 / kPiece; q < LH / kPiece; ++q) {
                    const Piece a = rank_row(NV - 1, q);
#pragma unroll
                    for (int i = 0; i < kPiece; ++i)
                        gg[kPiece * q + i] = __vminu2(gg[kPiece * q + i], __vmaxu2(d[NV - 1][kPiece * q + i], a.w[i]));
                }
            }
            // Window minimum over [lo_w(c2), c2 - 1] for every c2: the sparse table of g goes to the
            // lane's column of shared memory, level s from level s - 1 by one packed minimum per word
            // (level 1 needs the row shifted by one position), up to the highest level a lane of this
            // warp reads; every cut position then reads the two cells the preparing kernel named for it.
            {
                const int top = (int)__reduce_max_sync(0xFFFFFFFFu, lvl);
                uint32_t cur[LH];
#pragma unroll
                for (int wd = W0; wd < LH; ++wd) {
                    st_shared_u32(sbase + win_cell(0, 2 * wd, LH), gg[wd]);
                    const uint32_t prev = wd > W0 ? gg[wd - 1] : 0xFFFFFFFFu;
                    cur[wd] = __vminu2(gg[wd], __byte_perm(prev, gg[wd], 0x5432));  // positions 2wd-1, 2wd
                    st_shared_u32(sbase + win_cell(1, 2 * wd, LH), cur[wd]);
                }
#pragma unroll
                for (int sl = 2; sl < kWinLevels; ++sl) {
                    if (sl > top) break;
                    const int shift = 1 << (sl - 2);  // words
#pragma unroll
                    for (int wd = LH - 1; wd >= W0; --wd) {  // downwards: cur[wd - shift] is still the level below
                        if (wd - shift >= W0) cur[wd] = __vminu2(cur[wd], cur[wd - shift]);
                        st_shared_u32(sbase + win_cell(sl, 2 * wd, LH), cur[wd]);
                    }
                }
            }
            uint32_t ob[2 * LH];
#pragma unroll
            for (int c2 = 2 * O0; c2 < 2 * LH; ++c2) {
                ob[c2] = 0xFFFFu;
                if (c2 >= C0) {
                    // (bounds-checking build: a cell outside the warp's table reads the +inf cell instead)
                    const uint32_t o1 = PP_IN_BOUNDS(t, cw[c2] & 0xFFFFu, win_bytes_per_warp(LH) - 126) ? cw[c2] & 0xFFFFu
                                                                                                       : win_cell(kWinLevels, 0, LH);
                    const uint32_t o2 = PP_IN_BOUNDS(t, cw[c2] >> 16, win_bytes_per_warp(LH) - 126) ? cw[c2] >> 16
                                                                                                 : win_cell(kWinLevels, 0, LH);
                    const uint32_t a = ld_shared_u16(sbase + o1), b2 = ld_shared_u16(sbase + o2);
                    ob[c2] = min(a, b2);
                }
            }
            const uint32_t S2 = P | (1u << w);
            const uint32_t row = t.rowoff[S2] + (uint32_t)__popc(S2 & ((1u << w) - 1u));
            uint32_t xw = 0xFFFFFFFFu;
#pragma unroll
            for (int q = O0 / kPiece; q < LH / kPiece; ++q) {
                Piece o;
#pragma unroll
                for (int i = 0; i < kPiece; ++i) {
                    const int wd = kPiece * q + i;
                    o.w[i] = wd >= O0 ? ob[2 * wd] | (ob[2 * wd + 1] << 16) : 0xFFFFFFFFu;
                    if (wd == wfin) xw = o.w[i];
                }
                st_piece(t, tabw + word_at((size_t)row * LH + kPiece * q), t.table, t.table_words, o);
            }
            const uint32_t x = (xw >> sfin) & 0xFFFFu;
            if (x != 0xFFFFu) {
                const unsigned long long cand = pack_best(x, NV + 1, S2, w);
                key = cand < key ? cand : key;
            }
        }
        if (key != kNoBest && lane < valid) atomicMin(&t.key[g * 32 + lane], key);
    }
}

// state or rank of one (row, position) of one instance's column
__device__ __forceinline__ uint32_t lanes_elem(const BatchLanes &t, const uint32_t *col, const uint32_t *base, size_t words,
                                               size_t row, int LH, int c)
{
    return (ld_table(t, col + word_at(row * LH + (size_t)(c >> 1)), base, words) >> ((c & 1) * 16)) & 0xFFFFu;
}

__global__ void __launch_bounds__(kBackWarps * 32)
k_lanes_back(const BatchLanes t, const int64_t B, const int L, const int k, const uint64_t *__restrict__ g_bits,
             const uint32_t *__restrict__ g_bw, double *__restrict__ o_beta, int32_t *__restrict__ o_m,
             int32_t *__restrict__ o_cuts, int32_t *__restrict__ o_place, int8_t *__restrict__ o_status)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31;
    const int LH = t.LH;
    const double kInf = __longlong_as_double(0x7FF0000000000000ll);
    __shared__ uint32_t s_len[kBackWarps][kLanesMaxK * 16];  // the instance's window lengths: one load fewer per step
    uint32_t *mylen = s_len[threadIdx.x >> 5];
    for (int64_t inst = (int64_t)blockIdx.x * kBackWarps + (threadIdx.x >> 5); inst < B;
         inst += (int64_t)gridDim.x * kBackWarps) {
        const size_t g = (size_t)(inst >> 5);
        const int col = (int)(inst & 31);
        const uint32_t *tab = t.table + g * t.rows * (size_t)(LH * 32) + col * kPiece;
        const uint32_t *rk = t.rank + g * (size_t)(k * k) * (size_t)(LH * 32) + col * kPiece;
        const uint32_t *ln = t.len + g * (size_t)k * (size_t)(LH * 32) + col * kPiece;
        const unsigned long long key = t.key[inst];
        const int bad = t.flag[inst] & kFlagLimit;
        int32_t *cuts = o_cuts ? o_cuts + inst * (k - 1) : nullptr;
        int32_t *place = o_place + inst * k;
        if (lane < k) place[lane] = -1;
        if (cuts && lane < k - 1) cuts[lane] = -1;
        __syncwarp();
        for (int e = lane; e < k * LH; e += 32) mylen[e] = ld_table(t, ln + word_at(e), t.len, t.len_words);
        __syncwarp();
        if (bad || key == kNoBest) {
            if (lane == 0) {
                o_beta[inst] = kInf;
                o_m[inst] = 0;
                o_status[inst] = bad ? (int8_t)PP_ERR_LIMIT : (int8_t)PP_INFEASIBLE;
            }
            continue;
        }
        const uint32_t rstar = (uint32_t)(key >> 30);
        const int m = (int)((key >> 25) & 31);
        uint32_t S = (uint32_t)((key >> 5) & 0xFFFFF);
        int w = (int)(key & 31), c2 = L - 1;
        int my_cut = 0, my_node = 0;  // lane j: cut and node of segment j
        if (lane == 0) {
            o_m[inst] = m;
            o_status[inst] = (int8_t)PP_OK;
#ifdef PP_DEBUG_BOUNDS
            if (*t.err != 0) o_status[inst] = (int8_t)PP_ERR_CUDA;  // an index left its table somewhere in this piece
#endif
        }
        for (int j = m - 1; j >= 0; --j) {
            if (lane == j) {
                my_node = w;
                my_cut = c2;
                place[j] = w;
                if (j < m - 1) cuts[j] = c2;
            }
            if (j == 0) break;
            const uint32_t P = S & ~(1u << w);
            const int l0 = c2 - (int)((mylen[w * LH + (c2 >> 1)] >> ((c2 & 1) * 16)) & 0xFFFFu);
            const uint32_t prow = t.rowoff[P];
            const int np = __popc(P), total = (c2 - l0) * np;
            // candidates (position, node of P), lanes over all of them at once: the loads of a step are
            // independent, the smallest (position, node) that meets the threshold wins
            const uint32_t recip = (65536u + (uint32_t)np - 1u) / (uint32_t)np;  // floor(x / np) for x <= 31 * 7
            uint32_t nodes = 0;  // the nodes of P, four bits each
            int n = 0;
            for (uint32_t rem = P; rem; rem &= rem - 1, n += 4) nodes |= (uint32_t)(__ffs(rem) - 1) << n;
            unsigned int pick = 0xFFFFFFFFu;
#pragma unroll 1
            for (int it = lane; it < total; it += 32) {
                const int ci = (int)(((uint32_t)it * recip) >> 16), vi = it - ci * np;
                const int c = l0 + ci, v = (int)((nodes >> (4 * vi)) & 15u);
                // a state of np segments ends at layer np - 1 at the earliest; earlier positions were never written
                const uint32_t a = c >= np - 1 ? lanes_elem(t, tab, t.table, t.table_words, (size_t)prow + vi, LH, c) : 0xFFFFu;
                const uint32_t b = lanes_elem(t, rk, t.rank, t.rank_words, (size_t)(v * k + w), LH, c);
                if (max(a, b) <= rstar) pick = min(pick, ((unsigned)c << 5) | (unsigned)v);
            }
            pick = __reduce_min_sync(0xFFFFFFFFu, pick);
            if (pick == 0xFFFFFFFFu) {  // inconsistent table: flag the instance, keep going
                if (lane == 0) o_status[inst] = (int8_t)PP_ERR_CUDA;
                break;
            }
            S = P;
            w = (int)(pick & 31u);
            c2 = (int)(pick >> 5);
        }
        // beta* is the bottleneck of the plan: no link of it ranks above the optimum, and no plan is better
        const int next_node = __shfl_down_sync(0xFFFFFFFFu, my_node, 1);
        unsigned long long worst = 0ull;  // non-negative doubles order like their bits
        if (lane < m - 1)
            worst = (unsigned long long)__double_as_longlong(
                __ddiv_rn((double)g_bits[inst * L + my_cut], (double)g_bw[inst * k * k + my_node * k + next_node]));
#pragma unroll
        for (int o = 4; o; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(0xFFFFFFFFu, worst, o);
            worst = other > worst ? other : worst;
        }
        if (lane == 0) o_beta[inst] = __longlong_as_double((long long)worst);
    }
}

template <typename... Args, typename... Params>
cudaError_t launch_dependent(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                             Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <int LH>
cudaError_t launch_level(int nv, const BatchLanes &t, int64_t B, int k, int L, int split, unsigned grid, cudaStream_t s)
{
    switch (nv) {
#define PP_CASE(N)                                                                                                     \
    case N:                                                                                                            \
        if constexpr (LH != 4 || N < kLanesShortK) { /* nodes in front: one less than the problem has */               \
            const size_t sm = win_bytes_per_warp(LH) * kLevelWarps;                                                    \
            cudaError_t e = cudaFuncSetAttribute(k_lanes_level<N, LH>, cudaFuncAttributeMaxDynamicSharedMemorySize,    \
                                                 (int)sm);                                                             \
            if (e != cudaSuccess) return e;                                                                            \
            return launch_dependent(k_lanes_level<N, LH>, grid, kLevelWarps * 32, sm, s, t, B, k, L, split);           \
        }                                                                                                              \
        break;
        PP_CASE(1) PP_CASE(2) PP_CASE(3) PP_CASE(4) PP_CASE(5) PP_CASE(6) PP_CASE(7)
#undef PP_CASE
        default: break;
    }
    return cudaErrorInvalidValue;
}

}  // namespace

// A batch that fits the GPU at once goes an instance to a block (pp_batch.cu), which then takes the time of one
// instance; here every level is a launch, however few warps it has.  us a call, here and there: 64 x (k = 4, L = 24)
// 21.9, 12.5, 444 of them 23.8, 14.5; 300 x (k = 6, L = 24) 35.0, 20.7; 148 x (k = 8, L = 24) 50.5, 35.0, 444 of
// them 62.1, 53.5; in narrow blocks 888 x (k = 6, L = 24) 41.8, 30.9.  From there on blocks cost by the wave, lanes by the
// instance (three seeds; the runs of one side lie within 1 %).  A second wave is the faster one
//   for k = 4, 5                 1000 x (4, 17) 26.4, 22.8, 1776 30.1, 27.2; (5, 32) 37.3, 30.8 and 45.3, 39.2
//   for k = 6, 7 up to 16 layers 1776 x (6, 16) 47.4, 43.3; 460 x (7, 16) 41.2, 36.8, 888 49.2, 45.3
//       and from 25 on           1776 x (6, 25) 59.7, 57.6, (6, 32) 62.1, 59.7; 888 x (7, 25) 63.9, 60.6, (7, 32) 66.8, 61.7
//   for k = 8 up to 16           460 x (8, 16) 54.5, 51.8, 888 67.9, 67.9; (8, 9) 51.5, 47.5 and 64.6, 63.8.
// From 17 to 24 positions a block's rows are 32 long, the ones here 24.  With k = 6 the lines then cross in the middle of
// that wave: 1000 x (6, 17) 41.3, 41.5, 1330 47.2, 45.8, 1500 49.5, 51.3, 1776 52.0, 55.6; (6, 24) 43.3, 43.2, 49.1, 47.4, 51.5,
// 51.7, 54.5, 57.3; k = 7 hardly gains anywhere (460, 600, 888 x (7, 24) 46.1, 45.8, 49.6, 51.5, 56.1, 59.7) and k = 8 loses
// (460 x (8, 24) 64.1, 74.1), with longer rows too (888 x (8, 28) 99.6, 104.8; two blocks to an SM from 29 on: 600 x (8, 32)
// 84.4, 106.7).  A third wave loses (2200 x (6, 24) 60.2, 70.1, (4, 17) 32.6, 35.1) or gains 3 to 5 % ((5, 32) 50.5, 48.2).
// These lines know blocks and lanes; a warp is asked for only beyond them (batch_warps_takes), although it is faster already in front
// of some for uniform sizes and links (888 x (8, 9) 63.8 in blocks, 889 in warps 40.7; identical blocks 79).
bool batch_lanes_takes(int64_t B, int L, int k, int sms)
{
    if (k < 2 || k > kLanesMaxK || L > kLanesMaxL) return false;
    const int64_t wave = (int64_t)sms * batch_blocks_per_sm(L, k, batch_narrow(B, L, k, sms));
    if (B <= wave) return false;
    const bool second = k >= 4 && (k <= 6 || L <= 16 || (k == 7 && L > 24));
    const int64_t most = k == 6 && L > 16 && L <= 24 ? wave + wave / 2 : 2 * wave;
    return !(second && B <= most);
}

cudaError_t launch_quotients(int64_t n, const uint64_t *bits, const uint32_t *kbps, double *by_reciprocal, double *divided,
                             cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    k_quotients<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, s>>>(n, bits, kbps, by_reciprocal, divided);
    return cudaGetLastError();
}

int batch_lanes_words(int L)
{
    const int Lh = (L + 1) / 2;
    return Lh <= 4 ? 4 : Lh <= 8 ? 8 : Lh <= 12 ? 12 : 16;
}

cudaError_t launch_batch_prep(int64_t B, int L, int k, const uint64_t *bits, const uint64_t *mem,
                              const uint64_t *cap, const uint32_t *bw, const BatchLanes &t, cudaStream_t s)
{
    if (B <= 0) return cudaSuccess;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t blocks = B < (int64_t)sms * 64 ? B : (int64_t)sms * 64;
    k_lanes_prep<<<(unsigned)blocks, kPrepThreads, prep_layout(L, k).total, s>>>(t, B, L, k, bits, mem, cap, bw);
    return cudaGetLastError();
}

cudaError_t launch_batch_lanes(int64_t B, int L, int k, const uint64_t *bits, const uint32_t *bw,
                               const BatchLanes &t, double *beta, int32_t *m, int32_t *cuts,
                               int32_t *placement, int8_t *status, cudaStream_t s)
{
    if (B <= 0) return cudaSuccess;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t G = (B + 31) >> 5;
    const int jmax = k < L ? k : L;
    uint64_t binom = (uint64_t)k;  // C(k, j - 1), the source masks of level j
    const int64_t slots = (int64_t)sms * 16;  // warps the GPU holds at a time, roughly
    for (int j = 2; j <= jmax; ++j) {
        int split = 1;  // warps per source mask: a level with few masks spreads the k - j + 1 targets
        while (split < k - j + 1 && G * (int64_t)binom * split < 3 * slots) ++split;
        const int64_t items = G * (int64_t)binom * split;
        int64_t blocks = (items + kLevelWarps - 1) / kLevelWarps;
        const int64_t cap = (int64_t)sms * 32;
        if (blocks > cap) blocks = cap;
        cudaError_t e;
        switch (t.LH) {
            case 4: e = launch_level<4>(j - 1, t, B, k, L, split, (unsigned)blocks, s); break;
            case 8: e = launch_level<8>(j - 1, t, B, k, L, split, (unsigned)blocks, s); break;
            case 12: e = launch_level<12>(j - 1, t, B, k, L, split, (unsigned)blocks, s); break;
            case 16: e = launch_level<16>(j - 1, t, B, k, L, split, (unsigned)blocks, s); break;
            default: e = cudaErrorInvalidValue;
        }
        if (e != cudaSuccess) return e;
        binom = binom * (uint64_t)(k - j + 1) / (uint64_t)j;
    }
    int64_t blocks = (B + kBackWarps - 1) / kBackWarps;
    if (blocks > (int64_t)sms * 8) blocks = (int64_t)sms * 8;
    return launch_dependent(k_lanes_back, (unsigned)blocks, kBackWarps * 32, 0, s, t, B, L, k, bits, bw, beta, m, cuts,
                            placement, status);
}

}  // namespace pp
