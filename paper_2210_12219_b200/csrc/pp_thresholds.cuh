// The exact search by thresholds: a block answers whether some plan has no term above t, and the blocks of a grid ask it
// for different t.
//
// Under a threshold the recurrence of the search is one about sets of cut positions: with the positions that a (node set,
// last node) reaches as the bits of a few words,
//   reach[S + w][w] = { c' : some c in [lo_w(c'), c' - 1] is in G },  G = OR over v in S of reach[S][v] & under_t[v][w],
// where under_t[v][w] are the layers whose output the link moves within t.  With the layers in the order of their size
// that is one of L prefixes, so that a link's share of a threshold is a number.  Under Eq. 1 a threshold also shortens the
// windows.  Near the optimum few rows are anything but empty (tens to some hundreds, see pp_prune.cu), and those few fit a
// block's shared memory, where a level costs a barrier of the block, 1500 cycles with its rows, and not one of the grid that
// hands rows on, 8000.
//
// The optimum is one of the terms (a quotient of Eq. 3, under Eq. 1 also a compute time).  In the first round the blocks take
// thresholds spread over the range of the terms on the scale of the doubles' bits; what is left between the largest one
// without a plan and the next is a few dozen terms, which the blocks take in the second round.  The block of the smallest
// one with a plan then has in its table what the backtrack's threshold rule asks for.  A block that runs out of rows says
// so; where that leaves the optimum open the caller has the bounded search.
//
// On the device, us a solve back to back, the bounded search / this: Eq. 1 on geometric graphs, 50 layers on 12 nodes, four instances
// 23.8, 31.3, 37.0, 22.7 / 18.6, 20.7, 22.7, 18.0, on blocks 63.7, 58.8, 57.8, 56.6 / 47.4, 43.1, 39.1, 45.3.
#pragma once
#include "pp_blocks.cuh"

namespace pp {

constexpr int kThresholdK = 12;   // nodes, and words of a row, of the largest problems that are searched so
constexpr int kThresholdW = 2;
// Node sets that a block works through; the bounded search takes over where the optimum needs more of them.
constexpr size_t kThresholdSets = 640;
constexpr int kCandidates = 512;  // terms that are ranked at a time
constexpr int kThresholdRounds = 4;
constexpr int kThresholdWords = 56;  // PruneCtl::count from here on: the votes of the rounds
constexpr int kLatePolls = 1 << 20;  // test hook (pp_debug_late): after so many the late block comes in any case

// Shared memory of the search.  W: words of a row.
struct ThresholdLayout {
    size_t raw, sorted, order, under, end, count, code, cand, place, head, list, rows, total;
    int set_cap;
};
__host__ __device__ inline ThresholdLayout threshold_layout(int L, int k, int W, bool compute, size_t from, size_t budget)
{
    ThresholdLayout p{};
    if (k > kThresholdK || W > kThresholdW) return p;
    size_t o = from;
    auto take = [&o](size_t bytes) { size_t at = o; o = (o + bytes + 15) & ~(size_t)15; return at; };
    p.raw = take((size_t)W * 32 * 8);
    p.sorted = take((size_t)W * 32 * 8);
    p.order = take((size_t)L * 2);
    p.under = take((size_t)L * W * 4);
    p.end = take((size_t)k * (L + 1) * 2 * (compute ? 2 : 1));
    p.count = take((size_t)k * k * 2);
    p.code = take((size_t)kCandidates * 4);
    p.cand = take((size_t)kCandidates * 16);
    p.place = take((size_t)kCandidates * 8);
    p.head = take((size_t)4 << k);
    // every set has room for a row to each node (that of its successor with the node, as it happens)
    p.list = take((size_t)4 << k);
    size_t sets = (budget > o + 64 ? budget - o - 64 : 0) / ((size_t)k * (W + 1) * 4);
    if (sets > (size_t)1 << k) sets = (size_t)1 << k;
    if (sets > kThresholdSets) sets = kThresholdSets;
    p.set_cap = (int)sets;
    p.rows = take(sets * k * (W + 1) * 4);
    p.total = o;
    return p;
}

// What the search has of a problem, in shared memory.
struct ThresholdIn {
    int L, k;
    const unsigned long long *raw;      // [L] size << 10 | layer
    const unsigned long long *M, *cap;  // [L + 1], [k]
    const uint32_t *bw;                 // [k * k]
    const unsigned long long *Wp;       // Eq. 1: [L + 1] prefix sums of the work, [k] speeds
    const uint32_t *speed;
};
enum ThresholdOutcome { kThresholdOpen, kThresholdSolved, kThresholdNoPlan, kThresholdGaveUp };

// The votes of a round: every block adds one arrival, whether its threshold is not known to be too small, and whether it
// ran out of rows on it.  Nothing but this word passes between the blocks, so that it needs no fence (1100 cycles; the barrier
// of the bounded search, which hands rows on, 3500).  False when a wait ran out, and then for all blocks: one that gives up
// marks the word in the same step in which it sees that arrivals are missing, and a block that comes after it reads the mark.
constexpr unsigned long long kVoteLeft = 1ull << 63;
__device__ __forceinline__ bool threshold_vote(const PruneDev &d, unsigned long long *word, uint32_t open, uint32_t over, [[maybe_unused]] bool terms, uint32_t *opens,
                                               uint32_t *overs)
{
    __shared__ unsigned long long s_seen;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long seen;
        auto waiting = [&] { return !(seen & kVoteLeft) && (uint32_t)(seen >> 40) < d.arrivals; };
        auto look = [&] { asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(seen) : "l"(word) : "memory"); };
#ifdef PP_DEBUG_BOUNDS
        if (terms && d.late == blockIdx.x + 1) {  // test hook: behind a block that gave up
            int i = 0;
            do look();
            while (!(seen & kVoteLeft) && ++i < kLatePolls);
        }
#endif
        asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(word), "l"((1ull << 40) | ((unsigned long long)open << 20) | over) : "memory");
        int spins = 0;
        do look();
        while (waiting() && ++spins < d.polls);
        while (waiting()) {  // as often as other blocks change the word, at most
            const unsigned long long now = atomicCAS(word, seen, seen | kVoteLeft);
            seen = now == seen ? seen | kVoteLeft : now;
        }
        s_seen = seen;
    }
    __syncthreads();
    const unsigned long long seen = s_seen;
    *opens = (uint32_t)(seen >> 20) & 0xFFFFFu;
    *overs = (uint32_t)seen & 0xFFFFFu;
    return !(seen & kVoteLeft);
}

// W: words of a row; NT: threads of the block.  Ends with the block in step.  Solved: *winner is the block that has the
// plan in s_node and s_cut (-1 beyond it), *m_out and *beta_out are set there.
// What bounds it is the length of its chain of instructions (half of the stalls of a warp are waits for the next
// instruction): short code is worth more than clever code here.
template <int W, bool CT, int NT>
__device__ __forceinline__ int threshold_search(const PruneDev &d, const ThresholdIn in, const ThresholdLayout lay, unsigned char *smem, const Bounds chk,
                                                int *s_cut, int *s_node, int *winner, int *m_out, double *beta_out)
{
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    constexpr int kStride = W + 1, kWarps = NT / 32, kWide = W * 32, kParts = NT / kWide / 2;
    static_assert(kParts >= 1, "a layer's place is counted by a thread at least");
    // Links are the business of the first threads, windows of the others.
    constexpr int kLinks = (kThresholdK * kThresholdK + 31) / 32 * 32;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, L = in.L, k = in.k, cuts = L - 1;
    const int nblk = (int)gridDim.x, words = (L + 31) / 32;
    unsigned long long *sorted = reinterpret_cast<unsigned long long *>(smem + lay.sorted);
    uint16_t *order = reinterpret_cast<uint16_t *>(smem + lay.order);
    uint32_t *under = reinterpret_cast<uint32_t *>(smem + lay.under);
    uint16_t *fit = reinterpret_cast<uint16_t *>(smem + lay.end), *end = CT ? fit + k * (L + 1) : fit;
    uint16_t *count = reinterpret_cast<uint16_t *>(smem + lay.count);
    uint32_t *code = reinterpret_cast<uint32_t *>(smem + lay.code), *place = reinterpret_cast<uint32_t *>(smem + lay.place), *near = place + kCandidates;
    unsigned long long *cand = reinterpret_cast<unsigned long long *>(smem + lay.cand), *ranked = cand + kCandidates;
    uint32_t *list = reinterpret_cast<uint32_t *>(smem + lay.list);
    uint32_t *head = reinterpret_cast<uint32_t *>(smem + lay.head), *rows = reinterpret_cast<uint32_t *>(smem + lay.rows);
    const uint32_t set_cap = (uint32_t)lay.set_cap;
    [[maybe_unused]] const uint32_t full = (1u << k) - 1u;
    const uint32_t recip_k = 0xFFFFFFFFu / (uint32_t)k + 1u;  // it / k by a multiplication
    // by level, so that no thread reads what another one writes for the next
    __shared__ uint32_t s_added[kThresholdK + 2], s_final[kThresholdK + 2], s_n;
    [[maybe_unused]] const size_t n_under = (size_t)L * W, n_rows = (size_t)set_cap * k * kStride;
    const unsigned long long top_key = d.key_top;
    const double per_block = 1.0 / (double)(nblk > 1 ? nblk - 1 : 1);

    // ---- the layers in the order of their size, the prefixes of that order, the ends of the windows ----
    for (int i = tid; i < 1 << k; i += NT) head[i] = 0u;
    uint32_t n_sets = (uint32_t)k;  // sets in the table
    // A layer's place is the number of smaller ones, counted in parts by as many threads as there are.
    if (tid < kWide) place[tid] = 0u;
    __syncthreads();
    const int n_end = k * (L + 1), run = (n_end + NT - kLinks - 1) / (NT - kLinks), e_first = tid < kLinks ? n_end : min((tid - kLinks) * run, n_end),
              e_last = min(e_first + run, n_end), w_first = e_first / (L + 1), i_first = e_first - w_first * (L + 1);
    if (tid < NT / 2) {
        const int c = tid % kWide, part = tid / kWide, each = (cuts + kParts - 1) / kParts, o1 = min((part + 1) * each, cuts);
        if (c < cuts && part < kParts) {
            const unsigned long long mine = in.raw[c];
            uint32_t below = 0u;
#pragma unroll 4
            for (int o = part * each; o < o1; ++o) below += in.raw[o] < mine ? 1u : 0u;
            if (below) atomicAdd(&place[c], below);
        }
    }
    // fit: one behind the last layer of a segment of w that starts at layer i; i itself: none fits.  Neighbouring starts by
    // stepping on.
    if (tid >= NT / 2) {
        const int per = (n_end + NT / 2 - 1) / (NT / 2), e1 = min((tid - NT / 2 + 1) * per, n_end);
        int e = min((tid - NT / 2) * per, n_end), w = e / (L + 1), i = e - w * (L + 1), at = -1;
        for (; e < e1; ++e) {
            const unsigned long long from = in.M[i], most = from + in.cap[w] < from ? ~0ull : from + in.cap[w];
            if (at < i) {
                at = i;
#pragma unroll 1
                for (int step = W * 16; step; step >>= 1)
                    if (at + step <= L && in.M[at + step] <= most) at += step;
            }
            while (at < L && in.M[at + 1] <= most) ++at;
            fit[e] = (uint16_t)at;
            if (++i > L) {
                i = 0;
                ++w;
                at = -1;
            }
        }
    }
    __syncthreads();
    // one node: layers 0 .. c, a row for every node, first in the list and never cleared
    auto first_row = [&](int v, int upto) {
#pragma unroll
        for (int j = 0; j < W; ++j) rows[v * kStride + j] = upto >= 32 * j + 32 ? kAll : upto > 32 * j ? (1u << (upto - 32 * j)) - 1u : 0u;
    };
    if (tid >= NT - 32 && tid - (NT - 32) < k) {
        const int v = tid - (NT - 32);
        first_row(v, (int)fit[v * (L + 1)]);
        rows[v * kStride + W] = (uint32_t)v;
        head[1u << v] = (uint32_t)(v * kStride) + 1u;
        list[v] = 1u << v;
    }
    if (tid < cuts) {
        const uint32_t at = place[tid];
        sorted[at] = in.raw[tid] >> 10;
        order[at] = (uint16_t)tid;
    }
    __syncthreads();
    // under[n]: the positions of the n smallest layers, in pieces of 32 places for a word each
    auto piece_of = [&](int p, int j) -> uint32_t {  // this lane's layer of piece p, as a bit of word j
        const int n = p * 32 + lane;
        const uint32_t c = n > 0 && n < L ? order[n - 1] : 0xFFFFu;
        return (int)(c >> 5) == j ? 1u << (c & 31u) : 0u;
    };
    for (int e = wid; e < words * words; e += kWarps) {
        const int p = e / words, j = e - p * words, n = p * 32 + lane;
        uint32_t before = 0u, x = piece_of(p, j);
        for (int o = 0; o < p; ++o) before |= piece_of(o, j);
        before = __reduce_or_sync(kAll, before);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kAll, x, o);
            if (lane >= o) x |= y;
        }
        if (n < L && PP_IN_BOUNDS(chk, n * W + j, n_under)) under[n * W + j] = x | before;
    }
    __syncthreads();

    // the largest size that a link of bandwidth b moves within t
    auto size_within = [&](double t, double b) -> unsigned long long {
        const SizeBracket fits = sizes_within(t, b);
        if (!(fits.most < 1099511627776.0)) return 1ull << 40;
        const unsigned long long most = (unsigned long long)fits.most;
        return (double)most > fits.sure && __ddiv_rn((double)most, b) > t ? most - 1ull : most;  // a size of 0 is within any t
    };
    auto places_within = [&](unsigned long long most) -> int {
        int c = 0;
#pragma unroll 1
        for (int step = W * 16; step; step >>= 1)
            if (c + step <= cuts && sorted[c + step - 1] <= most) c += step;
        return c;
    };
    // largest amount of work that a node of speed b does within t; amounts are below 2^48
    auto work_within = [&](double t, uint32_t b) -> unsigned long long {
        const double p = __dmul_rd(t, (double)b), edge = __dadd_rn(p, 0.125);
        if (!(edge < 562949953421312.0)) return 1ull << 49;
        const unsigned long long n = (unsigned long long)edge;
        return n > 0 && (double)n > p && __ddiv_rn((double)n, (double)b) > t ? n - 1 : n;
    };
    // the rows of `level` nodes from the sets list[beg .. to - 1], which have one fewer
    auto make_level = [&](int level, uint32_t beg, uint32_t to) {
        const uint32_t items = (to - beg) * (uint32_t)k;
        for (uint32_t it = (uint32_t)tid; it < items; it += NT) {
            const uint32_t li = __umulhi(it, recip_k), S = list[beg + li];
            const int w = (int)(it - li * (uint32_t)k);
            if (S >> w & 1u) continue;
            uint32_t g[W], any = 0u;
#pragma unroll
            for (int j = 0; j < W; ++j) g[j] = 0u;
            for (uint32_t at = head[S]; at != 0u;) {
                if (!PP_IN_BOUNDS(chk, at - 1u + W, n_rows)) break;
                const uint32_t *row = rows + (at - 1u), info = row[W];
                const uint32_t *in_t = under + count[(info & 0xFFu) * k + w];
#pragma unroll
                for (int j = 0; j < W; ++j)
                    if (j < words) {
                        g[j] |= row[j] & in_t[j];
                        any |= g[j];
                    }
                at = info >> 8;
            }
            if (any == 0u) continue;
            const uint32_t S2 = S | (1u << w);
            // behind a cut at c the segment of w ends anywhere up to stop[c] - 1
            const uint16_t *stop = end + w * (L + 1) + 1;
            uint32_t more = 0u;
            int over = 0;  // one behind what earlier words reach, from the start of this one
            bool final = false;
            auto below = [](int n) -> uint32_t { return n >= 32 ? 0xFFFFFFFFu : n > 0 ? (1u << n) - 1u : 0u; };
#pragma unroll
            for (int j = 0; j < W; ++j) {
                uint32_t cov = below(over), x = g[j];
                while (x != 0u) {
                    const int c = __ffs(x) - 1, h = (int)stop[32 * j + c] - 32 * j;
                    const uint32_t reached = below(h) & ~((2u << c) - 1u);
                    cov |= reached;
                    over = over > h ? over : h;
                    const uint32_t inside = x & reached;  // later cuts within this segment: the last one goes on from here
                    x = inside ? x & ~((1u << (31 - __clz(inside))) - 1u) : x & (x - 1u);
                }
                over -= 32;
                if (j == (L - 1) >> 5) {
                    const uint32_t last = 1u << ((L - 1) & 31);
                    final = (cov & last) != 0u;
                    cov &= ~last;
                }
                g[j] = cov;
                more |= cov;
            }
            if (final) atomicMin(&s_final[level], S2 << 5 | (uint32_t)w);
            if (more == 0u) continue;
            const uint32_t at = ((uint32_t)k + beg * (uint32_t)k + it) * kStride;  // behind those of one node
            uint32_t old = 1u;
            if (PP_IN_BOUNDS(chk, S2, full + 1u)) old = atomicExch(&head[S2], at + 1u);
            if (PP_IN_BOUNDS(chk, at + W, n_rows)) {
#pragma unroll
                for (int j = 0; j < W; ++j) rows[at + j] = g[j];
                rows[at + W] = (uint32_t)w | old << 8;
            }
            if (old == 0u) {
                const uint32_t pos = to + atomicAdd(&s_added[level], 1u);
                if (PP_IN_BOUNDS(chk, pos, full + 1u)) list[pos] = S2;
            }
        }
    };

    // ---- one threshold: 0 no plan, 1 a plan of m nodes, 2 out of rows ----
    auto probe = [&](double t, int *m) -> int {
        [[maybe_unused]] uint32_t whole = 0u;  // nodes that do everything within t
        for (uint32_t i = k + tid; i < n_sets; i += NT) head[list[i]] = 0u;  // what the threshold before this one left
        if (tid < kThresholdK + 2) {
            s_added[tid] = tid == 1 ? (uint32_t)k : 0u;
            s_final[tid] = kAll;
        }
        if (tid < k * k) {
            const uint32_t b = in.bw[tid];
            count[tid] = (uint16_t)(b != 0u && tid / k != tid % k ? places_within(size_within(t, (double)b)) * W : 0);
        }
        if constexpr (CT) {
            int w = w_first, i = i_first, at = -1;
            unsigned long long work = 0ull;
            for (int e = e_first; e < e_last; ++e) {
                if (at < 0) work = work_within(t, in.speed[w]);
                const int stop = in.speed[w] ? (int)fit[e] : i;
                const unsigned long long most = in.Wp[i] + work;
                if (at < i) {
                    at = i;
#pragma unroll 1
                    for (int step = W * 16; step; step >>= 1)
                        if (at + step <= stop && in.Wp[at + step] <= most) at += step;
                }
                while (at < stop && in.Wp[at + 1] <= most) ++at;
                end[e] = (uint16_t)at;
                if (i == 0) {
                    first_row(w, at);
                    if (at == L) whole |= 1u << w;
                }
                if (++i > L) {
                    i = 0;
                    ++w;
                    at = -1;
                }
            }
        }
        __syncthreads();
        if constexpr (CT) {  // after the words are reset
            if (whole) {
                atomicMin(&s_final[1], (whole & (0u - whole)) << 5 | (uint32_t)(__ffs(whole) - 1));
            }
            __syncthreads();
        }
        const int top = k < L ? k : L;
        uint32_t beg = 0u, to = 0u;
        for (int level = 1;; ++level) {
            if (level > 1) {
                make_level(level, beg, to);
                __syncthreads();
            }
            beg = to;
            n_sets = to = beg + s_added[level];
            *m = level;
            if (s_final[level] != kAll) return 1;
            if (beg == to || level == top) return 0;
            if (to + 1u > set_cap) return 2;
        }
    };

    // ---- rounds ----
    unsigned long long lowest = d.key_floor, highest = top_key;  // the terms in question, as bits of doubles
    unsigned long long from = max(d.key_base, lowest), to = highest;  // of a round of thresholds spread over a range
    auto spread = [&](int b) -> unsigned long long {       // the last one is the end of the range
        return b >= nblk - 1 ? to : from + (unsigned long long)((double)(to - from) * ((double)b * per_block));
    };
    int n = 0;  // of the last round, whose thresholds are terms, `each` to a block: their number
    int m = 0;
    for (int round = 0; round < kThresholdRounds; ++round) {
        unsigned long long key = 0ull;
        int vote = 1;
        if (n == 0) {
            key = spread((int)blockIdx.x);
            vote = probe(__longlong_as_double((long long)key), &m);
        } else {
            const int each = (n + nblk - 1) / nblk, i1 = min(((int)blockIdx.x + 1) * each, n);
            for (int i = (int)blockIdx.x * each; i < i1; ++i) {
                key = ranked[i];
                vote = probe(__longlong_as_double((long long)key), &m);
                if (vote != 0) break;
                __syncthreads();
            }
        }
        uint32_t opens, overs;
        if (!threshold_vote(d, d.ctl->count + kThresholdWords + 2 * round, vote != 0, vote == 2, n != 0, &opens, &overs)) return kThresholdGaveUp;
        const int first = nblk - (int)opens;  // block of the smallest threshold that may have a plan
        if (round == 0 && opens == 0u) return kThresholdNoPlan;
        if (overs) {  // is it this one that ran out of rows?  Then the others near the optimum will, too
            if (!threshold_vote(d, d.ctl->count + kThresholdWords + 2 * round + 1, (int)blockIdx.x == first && vote == 2, 0u, false, &opens, &overs))
                return kThresholdGaveUp;
            if (opens) return kThresholdOpen;
        }
        if (n != 0) {
            if (opens == 0u && first == nblk) return kThresholdOpen;
            *winner = first;
            if ((int)blockIdx.x != first) return kThresholdSolved;
            // ---- backtrack: the smallest (mask, node) of the fewest nodes, then the lowest (cut, node) in front ----
            if (wid == 0) {
                uint32_t S = s_final[m] >> 5;
                int w = (int)(s_final[m] & 31u), c2 = L - 1;
                if (lane < PP_MAX_K) s_cut[lane] = s_node[lane] = -1;
                __syncwarp();
                for (int j = m - 1; j >= 0; --j) {
                    if (lane == 0) {
                        s_node[j] = w;
                        if (j < m - 1) s_cut[j] = c2;
                    }
                    if (j == 0) break;
                    S &= ~(1u << w);
                    // the rows of the set, one to a lane
                    uint32_t at = head[S], mine = 0u;
                    for (int i = 0; at != 0u && i < k; ++i) {
                        if (lane == i) mine = at;
                        if (!PP_IN_BOUNDS(chk, at - 1u + W, n_rows)) break;
                        at = rows[at - 1u + W] >> 8;
                    }
                    uint32_t pick = kAll;
                    if (mine != 0u) {
                        const uint32_t *row = rows + (mine - 1u);
                        const uint32_t v = row[W] & 0xFFu, *in_t = under + count[v * k + w];
                        const uint16_t *stop = end + w * (L + 1) + 1;
                        for (int i = 0; i < words && pick == kAll; ++i)
                            for (uint32_t x = row[i] & in_t[i]; x != 0u; x &= x - 1u) {
                                const int c = 32 * i + __ffs(x) - 1;
                                if (c >= c2) break;
                                if ((int)stop[c] > c2) {  // its segment reaches the next cut
                                    pick = (uint32_t)c << 5 | v;
                                    break;
                                }
                            }
                    }
                    pick = __reduce_min_sync(kAll, pick);
                    if (pick == kAll) {
                        m = -1;  // cannot happen on a consistent table
                        break;
                    }
                    w = (int)(pick & 31u);
                    c2 = (int)(pick >> 5);
                }
            }
            *m_out = m;
            *beta_out = __longlong_as_double((long long)key);
            return kThresholdSolved;
        }
        // ---- what is left: terms above the largest threshold without a plan, up to the next one ----
        if (first > 0) lowest = spread(first - 1) + 1ull;
        if (first < nblk) highest = spread(first);
        if (tid == 0) s_n = 0u;
        const double t_a = __longlong_as_double((long long)(lowest - 1ull)), t_b = __longlong_as_double((long long)highest);
        __syncthreads();
        if (const int e = tid; e < k * k) do {
            const int v = e / k, w = e - v * k;
            const uint32_t b = in.bw[e];
            if (v == w || b == 0u || (v > w && in.bw[w * k + v] == b)) break;  // both directions alike
            const unsigned long long most = size_within(t_b, (double)b);
            int i = lowest ? places_within(size_within(t_a, (double)b)) : 0, last = i;
            while (last < cuts && sorted[last] <= most) ++last;
            if (i < last) {
                uint32_t at = atomicAdd(&s_n, (uint32_t)(last - i));
                for (; i < last && at < (uint32_t)kCandidates; ++i, ++at) code[at] = (uint32_t)e << 16 | (uint32_t)i;
            }
        } while (false);
        if constexpr (CT) {
            int w = w_first, i = i_first;
            bool fresh = true;
            unsigned long long work_a = 0ull, work_b = 0ull;
            for (int e = e_first; e < e_last; ++e) {
                if (fresh) {
                    work_a = lowest ? work_within(t_a, in.speed[w]) : 0ull;
                    work_b = work_within(t_b, in.speed[w]);
                    fresh = false;
                }
                if (in.speed[w] != 0u) {
                    const int stop = fit[e];
                    const unsigned long long most = in.Wp[i] + work_b, least = in.Wp[i] + work_a;
                    int at = i;
                    if (lowest) {
#pragma unroll 1
                        for (int step = W * 16; step; step >>= 1)
                            if (at + step <= stop && in.Wp[at + step] <= least) at += step;
                        if (at < stop && in.Wp[at + 1] <= least) ++at;
                    }
                    int last = at;
                    while (last < stop && in.Wp[last + 1] <= most) ++last;
                    for (; at < last; ++at) {
                        // a run of the same work a layer further down, which fits: the same term
                        if (i > 0 && (int)fit[e - 1] >= at && in.Wp[at + 1] - in.Wp[i] == in.Wp[at] - in.Wp[i - 1]) continue;
                        const uint32_t to_at = atomicAdd(&s_n, 1u);
                        if (to_at < (uint32_t)kCandidates) code[to_at] = 1u << 31 | (uint32_t)w << 20 | (uint32_t)i << 10 | (uint32_t)(at + 1);
                    }
                }
                if (++i > L) {
                    i = 0;
                    ++w;
                    fresh = true;
                }
            }
        }
        __syncthreads();
        n = (int)s_n;
        if (n == 0) return kThresholdOpen;
        if (lowest >= highest) {  // one value, however many terms have it
            n = 1;
            if (tid == 0) ranked[0] = highest;
        } else if (n <= min(kCandidates, 2 * nblk)) {
            const int shift = max(32 - __clzll((long long)(highest - lowest)), 0);  // the terms to 32 bits
            for (int i = tid; i < n; i += NT) {
                const uint32_t c = code[i];
                double x;
                if (CT && c >> 31) {
                    x = __ddiv_rn((double)(in.Wp[c & 1023u] - in.Wp[c >> 10 & 1023u]), (double)in.speed[c >> 20 & 31u]);
                } else {
                    x = __ddiv_rn((double)sorted[c & 0xFFFFu], (double)in.bw[c >> 16]);
                }
                const unsigned long long y = (unsigned long long)__double_as_longlong(x);
                cand[i] = y;
                near[i] = (uint32_t)((y - lowest) >> shift);
                place[i] = 0u;
            }
            __syncthreads();
            const int wide = (n + 31) & ~31, parts = wide <= NT ? NT / wide : 1, each = (n + parts - 1) / parts;
            for (int i = tid; i < wide * parts; i += NT) {
                const int c = i % wide, o0 = i / wide * each, o1 = min(o0 + each, n);
                if (c >= n) continue;
                const unsigned long long x = cand[c];
                const uint32_t y = near[c];
                uint32_t below = 0u;
#pragma unroll 8
                for (int o = o0; o < o1; ++o) {
                    const uint32_t z = near[o];
                    below += z < y ? 1u : 0u;
                    if (z == y && o != c) below += cand[o] < x + (o < c ? 1ull : 0ull) ? 1u : 0u;
                }
                if (below) atomicAdd(&place[c], below);
            }
            __syncthreads();
            for (int i = tid; i < n; i += NT) ranked[place[i]] = cand[i];
        } else {
            n = 0;
            from = lowest;
            to = highest;
        }
        __syncthreads();
    }
    return kThresholdOpen;
}

}  // namespace pp
