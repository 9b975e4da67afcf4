// Many-instance exact search of short chains, an instance to a warp, by thresholds.
//
// Whether some plan has no quotient above t is a question about sets, not values: with L <= 32 layers the cut
// positions that a (node set, last node) reaches under t are one word, and the recurrence of the search
//   reach[S + w][w] = { c' : some c in [lo_w(c'), c' - 1] is in G },  G = OR over v in S of reach[S][v] & under_t[v][w]
// is a dozen logical instructions a row where the search on ranks works through a row of 16-bit values.  beta* is
// one of the quotients, so that a bisection over them ends with it exactly, and the table of the last feasible probe is
// what the backtrack's threshold rule asks for: no ranking of the quotients.  It starts from a lower bound, the optimum
// over the plans that may use a node again, which is one word a node.  Of k = 8, L = 24 with sizes and links drawn uniformly that is
// beta* in six of ten instances, and one probe confirms it; of log-normal ones in a third, of identical blocks or of two groups of
// nodes in one of twelve and fewer, and those take ten probes or so.
//
// A warp keeps an instance's table in shared memory, reach[S] a row of eight words.  Lane (w, q) takes the rows of
// target node w: the links into w and the windows of w are registers, a source set is two 16-byte loads, and all
// lanes walk the list of node sets of the other nodes, eight sets a trip.  No barriers but the warp's own.
// What bounds it: 15 300 warp instructions an instance of the uniform kind (3500 the bound, 1400 the staging, a trip 92, of which
// the windows 54) at 56 % of the issue slots while an SM has work (chains of dependent instructions), and then the longest instances, up
// to 15 probes or so of 7 us: 2000 instances take 118, 4096 150, 20000 483, and an SM has work 66 % of the time at 4096.
#include <algorithm>

#include "pp_blocks.cuh"

namespace pp {

namespace {

constexpr uint32_t kAll = 0xFFFFFFFFu;
constexpr int KW = 8;  // words of a row, one a node: k <= 8
constexpr int kWarpMaxL = 32;
constexpr int kSingly = 4;       // candidates above the bound that are tried one after another
constexpr int kWindowRegs = 15;  // distances of a window held in registers; longer ones come from shared memory

// Shared memory of a warp, in bytes.
struct WarpLayout {
    static constexpr int kReach = (1 << KW) * KW * 4;
    static constexpr int kRough = 33 * 8 + 32 * 8 + 8;                   // before reach takes their place: prefix sums, sizes, and
    static constexpr int kSetup = kRough + 32 * 4;                       // the sizes in order as floats, rounded down
    static constexpr int kSorted = kReach > kSetup ? kReach : kSetup;    // 32 sizes in ascending order
    static constexpr int kUnder = kSorted + 32 * 8;                      // [n] the positions of the n smallest sizes, 33 words
    static constexpr int kFar = kUnder + 36 * 4;                         // windows beyond kWindowRegs, [distance][node], 16 bits:
    static constexpr int kTotal = kFar + (31 - kWindowRegs) * KW * 2;    // the cut lies that far from the end
    static_assert(kTotal % 16 == 0, "rows are read 16 bytes at a time");
};

// Where a set's row lies.  A quarter of a warp reads, for one set s of the other nodes, the rows of the sets S_w that s is to its
// eight target nodes: s with a zero put in at bit w, so that S_w and S_{w+1} are one set or differ in a node moved from w to
// w + 1.  With the sum of the node numbers modulo 8 as the bank group the different ones among them, whose sums are
// consecutive numbers, meet in no bank (4096 x (k = 8, L = 24) 243 -> 211 us at the time).  Nodes 1, 2 and 4 are given by that
// sum and the other five.
__device__ __forceinline__ uint32_t slot_of(uint32_t S)
{
    uint32_t sum = 0;
#pragma unroll
    for (int i = 1; i < 8; ++i) sum += (S >> i & 1u) * (uint32_t)i;
    return ((S & 1u) | (S >> 2 & 2u) | (S >> 3 & 28u)) * 8u | (sum & 7u);
}
// Word of (S, v): rows of four words, a set's second four in a part of their own.
__device__ __forceinline__ int word_of(uint32_t slot, int v)
{
    return (v >> 2) * (4 << KW) + (int)slot * 4 + (v & 3);
}

constexpr int kWarps = 12, kWarpBlocks = 2;
constexpr size_t kWarpShared = (size_t)WarpLayout::kTotal * kWarps;

// t_sets: node sets of k - 1 nodes by (popcount, value), t_first[p]: the first of p nodes
__global__ void __launch_bounds__(kWarps * 32, kWarpBlocks)
k_batch_warps(const int64_t B, const int L, const int k, const uint32_t *__restrict__ t_sets, const uint32_t *__restrict__ t_first,
              const uint64_t *__restrict__ g_bits, const uint64_t *__restrict__ g_mem, const uint64_t *__restrict__ g_cap,
              const uint32_t *__restrict__ g_bw, double *__restrict__ o_beta, int32_t *__restrict__ o_m, int32_t *__restrict__ o_cuts,
              int32_t *__restrict__ o_place, int8_t *__restrict__ o_status)
{
    constexpr int QW = 32 / KW, kQuads = KW / 4, kPairs = KW * KW / 32;
    extern __shared__ __align__(16) unsigned char smem_warps[];
    // Steps of a target w: byte offset of the row of a set of the other nodes, number of the word of that set with w.
    // The sets of one size are filled up to whole trips with their last one.
    constexpr int kTrip = 2 * QW, kSteps = 152;
    __shared__ uint32_t s_step[kSteps * KW];
    __shared__ uint8_t s_first[KW + 2], s_trip[KW + 2];
    __shared__ uint32_t s_next;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, w = lane & (KW - 1), q = lane / KW;
    unsigned char *mine = smem_warps + (size_t)wid * WarpLayout::kTotal;
    uint32_t *reach = reinterpret_cast<uint32_t *>(mine);
    double *sorted = reinterpret_cast<double *>(mine + WarpLayout::kSorted);
    float *rough = reinterpret_cast<float *>(mine + WarpLayout::kRough);
    uint32_t *under = reinterpret_cast<uint32_t *>(mine + WarpLayout::kUnder);
    uint16_t *far = reinterpret_cast<uint16_t *>(mine + WarpLayout::kFar);
    unsigned long long *s_M = reinterpret_cast<unsigned long long *>(mine), *s_bits = s_M + 33;
    const double kInf = __longlong_as_double(0x7FF0000000000000ll);
    const int jmax = k < L ? k : L, cuts = L - 1;  // the last layer sends nothing
    const uint32_t last_bit = 1u << (L - 1);
    PP_BLOCK_BOUNDS(chk);
    [[maybe_unused]] constexpr int n_reach = WarpLayout::kReach / 4;
    if (threadIdx.x == 0) {
        int at = 0;
        for (int p = 0; p <= k; ++p) {
            s_first[p] = (uint8_t)t_first[p];
            s_trip[p] = (uint8_t)at;
            if (p > 0 && p < k) at += ((int)(t_first[p + 1] - t_first[p]) + kTrip - 1) / kTrip * kTrip;
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < s_trip[k] * KW; e += kWarps * 32) {
        const int i = e / KW, u = e % KW;
        int p = 1;
        while (i >= s_trip[p + 1]) ++p;
        const uint32_t s = t_sets[min(s_first[p] + i - s_trip[p], s_first[p + 1] - 1)], S = (s & ((1u << u) - 1u)) | ((s >> u) << (u + 1));
        s_step[e] = u < k ? slot_of(S) * 16u | (uint32_t)word_of(slot_of(S | (1u << u)), u) << 16 : 0u;
    }

    // ---- an instance's own: lane c has layer c, lanes (w, q) the links v -> w of their nodes v ----
    unsigned long long bits, M1, capw;  // M1: memory of layers 0..lane
    double link[kPairs], recip[kPairs];
    uint32_t win[kWindowRegs], base;    // bit c of win[d - 1]: behind a cut at c, layers c + 1 .. c + d fit node w
    int reach_d;                        // longest window
    bool bad;
    int whole;                          // the lowest node that holds the whole chain, or -1
    auto setup = [&](int64_t inst) {
        bits = lane < L ? g_bits[inst * L + lane] : 0ull;
        M1 = lane < L ? g_mem[inst * L + lane] : 0ull;
        capw = w < k ? g_cap[inst * k + w] : 0ull;
        bad = bits >= PP_MAX_BITS;
#pragma unroll
        for (int i = 0; i < kPairs; ++i) {
            const int v = q * kPairs + i;
            const uint32_t x = v < k && w < k ? g_bw[(inst * k + v) * k + w] : 0u;
            bad |= x >= PP_MAX_KBPS;
            link[i] = v != w ? (double)x : 0.0;
            recip[i] = link[i] > 0.0 ? __drcp_rn(link[i]) : 0.0;
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(kAll, M1, o);
            if (lane >= o) {
                if (y > ~0ull - M1) bad = true;  // the 64-bit sum would wrap: PP_ERR_LIMIT, as in pp_problem_create
                M1 += y;
            }
        }
        bad = __any_sync(kAll, bad);
        const unsigned long long total = __shfl_sync(kAll, M1, L - 1);
        whole = __ffs(__ballot_sync(kAll, lane < k && capw >= total)) - 1;
        if (bad || whole >= 0) return;
        // sizes in ascending order, and the positions of the n smallest ones
        if (lane == 0) s_M[0] = 0ull;
        s_M[lane + 1] = M1;
        s_bits[lane] = bits << 5 | (unsigned)lane;
        __syncwarp();
        int place = 0;
        for (int c = 0; c < cuts; ++c) place += s_bits[c] < (bits << 5 | (unsigned)lane) ? 1 : 0;
        const int at = lane < cuts ? place : lane;
        sorted[at] = lane < cuts ? (double)bits : kInf;
        rough[at] = lane < cuts ? __ull2float_rd(bits) : __uint_as_float(0x7F800000u);
        under[lane + 1] = 0u;
        __syncwarp();
        if (lane < cuts) under[place + 1] = 1u << lane;
        __syncwarp();
        uint32_t below = under[lane + 1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kAll, below, o);
            if (lane >= o) below |= y;
        }
        __syncwarp();
        under[lane + 1] = below;
        if (lane == 0) under[0] = 0u;
        // windows
        unsigned long long cap_of[KW];
#pragma unroll
        for (int u = 0; u < KW; ++u) cap_of[u] = __shfl_sync(kAll, capw, u);
        auto fits = [&](int d) -> uint32_t {
            const bool on = lane + d < L;
            const unsigned long long need = on ? s_M[lane + 1 + d] - M1 : ~0ull;
            uint32_t x = 0;
#pragma unroll
            for (int u = 0; u < KW; ++u) {
                const uint32_t hit = __ballot_sync(kAll, on && need <= cap_of[u]);
                if (u == w) x = hit;
            }
            return x;
        };
        reach_d = 0;
#pragma unroll
        for (int d = 1; d <= kWindowRegs; ++d) {
            win[d - 1] = 0u;
            if (reach_d == d - 1) {
                win[d - 1] = fits(d);
                if (__any_sync(kAll, win[d - 1] != 0u)) reach_d = d;
            }
        }
        if (reach_d == kWindowRegs)
#pragma unroll 1
            for (int d = kWindowRegs + 1; d < L; ++d) {
                const uint32_t x = fits(d);
                if (!__any_sync(kAll, x != 0u)) break;
                reach_d = d;
                if (q == 0) far[(d - kWindowRegs - 1) * KW + w] = (uint16_t)x;
            }
        base = 0u;
#pragma unroll
        for (int u = 0; u < KW; ++u) {
            const uint32_t hit = __ballot_sync(kAll, lane < L && M1 <= cap_of[u]);
            if (u == w) base = hit;
        }
        __syncwarp();
    };
    // the table before its first threshold: where the prefix sums and the sizes were
    auto clear = [&]() {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < n_reach; i += 128)
            if (i + lane * 4 < n_reach) *reinterpret_cast<uint4 *>(reach + i + lane * 4) = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        if (q == 0 && w < k && PP_IN_BOUNDS(chk, word_of(slot_of(1u << w), w), n_reach)) reach[word_of(slot_of(1u << w), w)] = base;
        __syncwarp();
    };
    // where the segment of this lane's node behind a cut in g may end; of two rows at a time
    auto span2 = [&](uint32_t g, uint32_t h, uint32_t &G, uint32_t &H) {
        uint32_t lg = 0u, lh = 0u, ng = 0u, nh = 0u;
        auto step = [&](uint32_t x) {
            lg = (lg + lg) | (g & x);
            lh = (lh + lh) | (h & x);
        };
        if (reach_d > 6) {  // two chains of shifts
            if (reach_d > 12) {
#pragma unroll 1
                for (int d = reach_d; d > kWindowRegs; --d) step(far[(d - kWindowRegs - 1) * KW + w]);
#pragma unroll
                for (int d = kWindowRegs; d > 12; --d) step(win[d - 1]);
            }
#pragma unroll
            for (int d = 12; d > 6; --d) step(win[d - 1]);
        }
#pragma unroll
        for (int d = 6; d > 0; --d) {
            ng = (ng + ng) | (g & win[d - 1]);
            nh = (nh + nh) | (h & win[d - 1]);
        }
        G = (lg << 7) | (ng << 1);
        H = (lh << 7) | (nh << 1);
    };
    auto span = [&](uint32_t g) -> uint32_t {
        uint32_t longer = 0u, near = 0u;
        auto step = [&](uint32_t x) { longer = (longer + longer) | (g & x); };
        if (reach_d > 6) {
            if (reach_d > 12) {
#pragma unroll 1
                for (int d = reach_d; d > kWindowRegs; --d) step(far[(d - kWindowRegs - 1) * KW + w]);
#pragma unroll
                for (int d = kWindowRegs; d > 12; --d) step(win[d - 1]);
            }
#pragma unroll
            for (int d = 12; d > 6; --d) step(win[d - 1]);
        }
#pragma unroll
        for (int d = 6; d > 0; --d) near = (near + near) | (g & win[d - 1]);
        return (longer << 7) | (near << 1);
    };
    // the positions that plans reach which may use a node again, by the links ok[] of this lane's node: the group of its w
    auto walks = [&](const uint32_t (&ok)[KW]) -> uint32_t {
        uint32_t A = base;
        for (int j = 2; j <= jmax; ++j) {
            uint32_t g = 0u;
#pragma unroll
            for (int v = 0; v < KW; ++v) g |= __shfl_sync(kAll, A, v, KW) & ok[v];
            const uint32_t more = span(g) & ~A;
            A |= more;
            if (!__any_sync(kAll, more != 0u)) break;
        }
        return A;
    };
    // A lower bound by the plans that may use a node again: one word a node instead of one a (set, node), so that the groups
    // of lanes take a threshold each.  Four rounds, each a fifth of the range (uniform, 4096 x (8, 24): three rounds take 4 % more, five 1 %).
    // Returns the largest threshold found to be too small, or -1.
    auto lower_bound = [&]() -> float {
        float beaten = -1.0f, slow = __uint_as_float(0x7F800000u), fast = 0.0f;
#pragma unroll
        for (int i = 0; i < kPairs; ++i)
            if (link[i] > 0.0) {
                slow = fminf(slow, (float)link[i]);
                fast = fmaxf(fast, (float)link[i]);
            }
        slow = __uint_as_float(__reduce_min_sync(kAll, __float_as_uint(slow)));
        fast = __uint_as_float(__reduce_max_sync(kAll, __float_as_uint(fast)));
        const uint32_t size = lane < cuts ? __float_as_uint(__ull2float_rd(bits)) : 0u;
        const float most = __uint_as_float(__reduce_max_sync(kAll, size));
        const float least = __uint_as_float(__reduce_min_sync(kAll, size ? size : __float_as_uint(most)));
        if (!(most > 0.0f && fast > 0.0f)) return beaten;
        float from = __log2f(least / fast), to = __log2f(most / slow);
        float mine_f[KW];
#pragma unroll
        for (int v = 0; v < KW; ++v) mine_f[v] = __shfl_sync(kAll, (float)link[v % kPairs], (v / kPairs) * KW + w);
#pragma unroll 1
        for (int r = 0; r < 4; ++r) {
            const float t = exp2f(from + (to - from) * ((float)(q + 1) / (float)(QW + 1)));
            uint32_t ok[KW];
#pragma unroll
            for (int v = 0; v < KW; ++v) {
                // what lies within a few roundings above the threshold counts as within: the bound stays one
                const float edge = __fmul_ru(__fmul_ru(t, mine_f[v]), 1.0f + 1.0f / (1 << 20));
                int c = 0;
#pragma unroll
                for (int step = 16; step; step >>= 1)
                    if (rough[c + step - 1] <= edge) c += step;
                ok[v] = mine_f[v] > 0.0f ? under[c] : 0u;
            }
            const uint32_t hit = __ballot_sync(kAll, (walks(ok) & last_bit) != 0u);
            int won = 0;  // thresholds that are too small
#pragma unroll
            for (int i = QW - 1; i >= 0; --i)
                if (won == 0 && !(hit >> (i * KW) & ((1u << KW) - 1u))) won = i + 1;
            const float step = (to - from) / (float)(QW + 1);
            if (won > 0) beaten = fmaxf(beaten, __shfl_sync(kAll, t, (won - 1) * KW));
            from += step * (float)won;
            to = won < QW ? from + step : to;
        }
        return beaten;
    };
    // the candidates of a link are sizes lo .. hi - 1 in ascending order
    int lo[kPairs], hi[kPairs], upto[kPairs];
    uint32_t okp[kPairs], ok[KW];
    // how many sizes each link moves within t, and which layers those are
    auto within = [&](double t) {
#pragma unroll
        for (int i = 0; i < kPairs; ++i) {
            const SizeBracket fits = sizes_within(t, link[i]);
            int c = 0;
#pragma unroll
            for (int step = 16; step; step >>= 1)
                if (sorted[c + step - 1] <= fits.most) c += step;
            if (!(link[i] > 0.0)) c = 0;
            while (c > 0 && sorted[c - 1] > fits.sure && quotient(sorted[c - 1], link[i], recip[i]) > t) --c;
            upto[i] = c;
            okp[i] = under[c];
        }
#pragma unroll
        for (int v = 0; v < KW; ++v) ok[v] = __shfl_sync(kAll, okp[v % kPairs], (v / kPairs) * KW + w);
    };
    unsigned long long least, most;  // bits of the smallest and the largest candidate; ~0 and 0: none
    auto extremes = [&]() {
        least = ~0ull;
        most = 0ull;
#pragma unroll
        for (int i = 0; i < kPairs; ++i)
            if (hi[i] > lo[i]) {
                least = min(least, (unsigned long long)__double_as_longlong(quotient(sorted[lo[i]], link[i], recip[i])));
                most = max(most, (unsigned long long)__double_as_longlong(quotient(sorted[hi[i] - 1], link[i], recip[i])));
            }
        const uint32_t high = __reduce_min_sync(kAll, (uint32_t)(least >> 32));
        least = (unsigned long long)high << 32 | __reduce_min_sync(kAll, (uint32_t)(least >> 32) == high ? (uint32_t)least : kAll);
        const uint32_t top = __reduce_max_sync(kAll, (uint32_t)(most >> 32));
        most = (unsigned long long)top << 32 | __reduce_max_sync(kAll, (uint32_t)(most >> 32) == top ? (uint32_t)most : 0u);
    };
    // whether there is a plan under the threshold of ok[]: its number of nodes, or 0
    auto probe = [&]() -> int {
        for (int j = 2; j <= jmax; ++j) {
            const uint32_t *step = s_step + (s_trip[j - 1] + q) * KW + w, *const end = s_step + s_trip[j] * KW;
            uint32_t got = 0u;
            for (; step < end; step += kTrip * KW) {
                const uint32_t a = step[0], b = step[QW * KW];
                const unsigned char *ra = mine + (a & 0xFFFFu), *rb = mine + (b & 0xFFFFu);
                uint32_t g = 0u, h = 0u, G = 0u, H = 0u;
#pragma unroll
                for (int i = 0; i < kQuads; ++i) {
                    if (!PP_IN_BOUNDS(chk, (a & 0xFFFFu) / 4 + i * (4 << KW) + 3, n_reach) ||
                        !PP_IN_BOUNDS(chk, (b & 0xFFFFu) / 4 + i * (4 << KW) + 3, n_reach)) break;
                    const uint4 x = *reinterpret_cast<const uint4 *>(ra + i * (16 << KW));
                    const uint4 y = *reinterpret_cast<const uint4 *>(rb + i * (16 << KW));
                    g |= x.x & ok[4 * i];
                    h |= y.x & ok[4 * i];
                    g |= x.y & ok[4 * i + 1];
                    h |= y.y & ok[4 * i + 1];
                    g |= x.z & ok[4 * i + 2];
                    h |= y.z & ok[4 * i + 2];
                    g |= x.w & ok[4 * i + 3];
                    h |= y.w & ok[4 * i + 3];
                }
                if (__any_sync(kAll, (g | h) != 0u)) span2(g, h, G, H);
                got |= G | H;
                if (w < k && PP_IN_BOUNDS(chk, a >> 16, n_reach) && PP_IN_BOUNDS(chk, b >> 16, n_reach)) {
                    reach[a >> 16] = G;
                    reach[b >> 16] = H;
                }
            }
            __syncwarp();
            if (__any_sync(kAll, (got & last_bit) != 0u)) return j;
            if (!__any_sync(kAll, got != 0u)) break;
        }
        return 0;
    };
    // the results of an instance; m nodes and more: the plan of the table, whose threshold's links are okp[]
    auto report = [&](int64_t inst, int m, double beta, int status, bool from_table) {
        int my_cut = -1, my_node = -1;  // lane j: cut and node of segment j
        if (status == (int)PP_OK && !from_table && lane == 0) my_node = whole;
        if (from_table) {
            // the smallest (mask, node) of m nodes that reaches the last layer
            uint32_t best = kAll;
            const uint32_t low = (1u << w) - 1u;
            for (int i = s_first[m - 1] + q; i < s_first[m]; i += QW) {
                const uint32_t s = t_sets[i], S2 = (s & low) | ((s & ~low) << 1) | (1u << w);
                const int at = word_of(slot_of(S2), w);
                if (w < k && PP_IN_BOUNDS(chk, at, n_reach) && (reach[at] & last_bit)) best = min(best, S2 << 3 | (uint32_t)w);
            }
            best = __reduce_min_sync(kAll, best);
            uint32_t S = best >> 3;
            int u = (int)(best & 7u), c2 = L - 1;
            // the lowest (cut, node) in front, lanes over the positions
            for (int j = m - 1; j >= 0; --j) {
                if (lane == j) {
                    my_node = u;
                    if (j < m - 1) my_cut = c2;
                }
                if (j == 0) break;
                const uint32_t from = S & ~(1u << u), slot = slot_of(from);
                const unsigned long long end = __shfl_sync(kAll, M1, c2), cap_u = __shfl_sync(kAll, capw, u);
                const uint32_t window = __ballot_sync(kAll, lane < c2 && end - M1 <= cap_u);
                uint32_t pick = kAll;
#pragma unroll
                for (int v = 0; v < KW; ++v) {
                    const uint32_t links = __shfl_sync(kAll, okp[v % kPairs], (v / kPairs) * KW + u);
                    const int at = word_of(slot, v);
                    const uint32_t x = PP_IN_BOUNDS(chk, at, n_reach) ? reach[at] & links & window : 0u;
                    if (x) pick = min(pick, (uint32_t)(__ffs(x) - 1) << 3 | (uint32_t)v);
                }
                if (pick == kAll) {  // inconsistent table: flag the instance
                    status = (int)PP_ERR_CUDA;
                    break;
                }
                S = from;
                u = (int)(pick & 7u);
                c2 = (int)(pick >> 3);
            }
        }
        if (PP_BROKEN(chk) && status != (int)PP_ERR_LIMIT) status = (int)PP_ERR_CUDA;
        if (lane < k) o_place[inst * k + lane] = my_node;
        if (o_cuts && lane < k - 1) o_cuts[inst * (k - 1) + lane] = my_cut;
        if (lane == 0) {
            o_beta[inst] = beta;
            o_m[inst] = m;
            o_status[inst] = (int8_t)status;
        }
        __syncwarp();
    };

    if (threadIdx.x == 0) s_next = 0u;
    __syncthreads();
    for (;;) {
        uint32_t n = 0u;
        if (lane == 0) n = atomicAdd(&s_next, 1u);
        const int64_t inst = blockIdx.x + (int64_t)gridDim.x * __shfl_sync(kAll, n, 0);
        if (inst >= B) break;
        setup(inst);
        if (bad || whole >= 0) {
            report(inst, bad ? 0 : 1, bad ? kInf : 0.0, bad ? (int)PP_ERR_LIMIT : (int)PP_OK, false);
            continue;
        }
        const float beaten = lower_bound();
        clear();
        within(fmax((double)beaten, 0.0));
#pragma unroll
        for (int i = 0; i < kPairs; ++i) {
            lo[i] = beaten < 0.0f ? 0 : upto[i];
            hi[i] = link[i] > 0.0 ? cuts : 0;
        }
        double first_t = 0.0;
        int m = 0, tries = 0;  // m: nodes of the plan of the smallest threshold that has one; tries: probes, from 0 down walks
        bool fresh = false;    // the table is still that one's
        for (;;) {
            extremes();
            if (least == ~0ull || (m > 0 && least == most)) break;
            // The smallest candidate; most optima that are not there lie little above it: steps that grow, up to ten times as far,
            // then whether there is a plan at all.  What counts is the longest instance, not the mean: in steps of 1.1, 1.35, 2 and then the
            // largest candidate 4096 x (k = 8, L = 24) took 7 % longer.  Between a threshold without and one with a plan the middle of their bits.
            unsigned long long key = least;
            if (m > 0) key = least + ((most - least) >> 1);
            else if (tries > 5) key = most;
            else if (tries > 0) {
                const double far_off = tries == 1 ? 1.2 : tries == 2 ? 1.7 : tries == 3 ? 2.8 : tries == 4 ? 5.0 : 10.0;
                key = (unsigned long long)__double_as_longlong(__dmul_rn(first_t, far_off));
            } else if (tries <= -kSingly) {
                key = least + min((most - least) >> 1, 1ull << min(36 - 4 * (tries + kSingly), 60));
            }
            const double t = __longlong_as_double((long long)min(max(key, least), most));
            within(t);
            bool probing = tries > 0, yes = false;
            if (!probing) {
                // The smallest candidates may still lie below the bound, which is worked out to a 625th of the range of all on its
                // logarithm.  Where quotients are close together that is hundreds of them: a few are tried one after another, then by
                // steps that grow sixteenfold and by the middle of what is left below the first that a walk gets through, as many walks
                // as bits tell them apart (1700 x (8, 24) of near-equal layers and links with one link far slower 345 -> 154 us a
                // call, spread ones 115.4 -> 116.2).
                yes = __any_sync(kAll, (walks(ok) & last_bit) != 0u);
                probing = yes && (tries > -kSingly || least == most);
                if (probing) {
                    tries = 0;
                    first_t = t;
#pragma unroll
                    for (int i = 0; i < kPairs; ++i) hi[i] = link[i] > 0.0 ? cuts : 0;
                } else --tries;
            }
            if (probing) {
                const int got = probe();
                ++tries;
                yes = fresh = got > 0;
                if (yes) m = got;
            }
#pragma unroll
            for (int i = 0; i < kPairs; ++i) {
                if (yes) hi[i] = max(lo[i], min(hi[i], upto[i]));
                else lo[i] = min(hi[i], max(lo[i], upto[i]));
            }
        }
        if (m == 0 || least == ~0ull) {
            report(inst, 0, kInf, m ? (int)PP_ERR_CUDA : (int)PP_INFEASIBLE, false);
            continue;
        }
        const double beta = __longlong_as_double((long long)least);  // a quotient, and no plan has all of its below it
        if (!fresh) {
            within(beta);
            m = probe();
        }
        report(inst, m, beta, (int)PP_OK, true);
    }
}

}  // namespace

// Whether the batches that do not go an instance to a block (batch_lanes_takes) go an instance to a warp rather than to a lane.
// A lane's time is that of its shape and, beyond kBatchLanesChunk instances, of rounds of their tables; a warp's is that of its
// instance's probes, 24 instances to an SM, and depends on the values.  The lines were therefore drawn over five families: sizes and links
// uniform, log-normal ones under rising memory, identical blocks under links of 1 to 50 Mbit/s, two groups of nodes with slow links
// between them, and chains that hardly fit.  A warp is taken where it is faster in their geometric mean and loses a tenth at most in
// any one; chains of few layers have no such line (identical blocks at a layer a node are slower in warps at all sizes up to 8000), there
// the mean decides.  us a call in lanes / in warps, uniform, log-normal, blocks, groups, tight (mean of four seeds):
//   k = 8   900 x L = 4  33 30 33 33 35 / 18 18 50 19 42        889 x 9   67 65 68 66 69 / 41 67 79 45 80
//          1300 x 14     84 83 85 84 83 / 69 86 81 79 100       1500      92 91 92 92 92 / 73 91 85 81 100
//          1500 x 16     94 92 93 93 92 / 89 90 86 90 104       1800     103 101 102 102 101 / 82 92 89 99 110
//          1700 x 24     127 125 126 126 121 / 116 122 105 144 111   2000   141 138 140 139 133 / 121 129 104 142 104
//          1300 x 32     133 131 132 132 127 / 121 158 102 140 116   1500   152 150 152 151 146 / 123 160 102 142 115
//   k = 7   900 x 6      35 35 37 35 37 / 25 39 53 28 45        900 x 9   47 47 49 47 49 / 37 51 57 40 60
//          1500 x 12     60 59 61 60 61 / 51 61 65 57 68        1700      64 63 65 64 65 / 50 63 66 58 70
//          1800 x 20     83 81 83 83 79 / 77 75 73 91 76        2100      89 87 89 88 85 / 81 77 76 93 75
//          2200 x 24     94 93 94 94 90 / 88 91 81 99 79        2500     102 100 102 102 98 / 86 94 84 104 78
//          1700 x 32     98 95 97 97 94 / 88 111 84 99 86       2000     108 106 107 106 104 / 89 111 83 100 82
//   k = 6  1777 x 6      38 38 39 37 40 / 28 36 49 28 44        1777 x 7  38 38 40 38 40 / 30 41 51 36 49
//          4000 x 11     73 73 74 73 73 / 55 74 91 69 77        4097      97 97 101 98 98 / 62 77 91 67 83
//          4096 x 24     91 90 91 91 88 / 91 104 108 120 75     4097     119 117 119 118 111 / 91 110 111 120 75
// What lies closer together than any of these families is slow in the lanes, whose ranking it makes long (1700 x (8, 24) of near-equal
// layers and links 350 / 153).
bool batch_warps_takes(int64_t B, int L, int k)
{
    if (L <= 8 && k > kLanesShortK) return true;
    if (k == 8) return B >= (L <= 9 ? 0 : L <= 14 ? 1500 : L <= 16 ? 1800 : L <= 24 ? 2000 : 1500);
    if (k == 7) return B >= (L <= 6 ? 0 : L <= 12 ? 1700 : L <= 20 ? 2100 : L <= 24 ? 2500 : 2000);
    return k == 6 && B > (L <= 6 ? 0 : kBatchLanesChunk);
}

cudaError_t launch_batch_warps(int64_t B, int L, int k, const LaneTables &others, int sms, const uint64_t *bits, const uint64_t *mem,
                               const uint64_t *cap, const uint32_t *bw, double *beta, int32_t *m, int32_t *cuts,
                               int32_t *placement, int8_t *status, cudaStream_t s)
{
    if (B <= 0) return cudaSuccess;
    if (k < 2 || k > KW || L > kWarpMaxL) return cudaErrorInvalidValue;
    const cudaError_t e = allow_shared(k_batch_warps, 6144);
    if (e != cudaSuccess) return e;
    const int64_t grid = std::min<int64_t>(B, (int64_t)sms * kWarpBlocks);
    k_batch_warps<<<(unsigned)grid, kWarps * 32, kWarpShared, s>>>(B, L, k, others.mlist, others.moff, bits, mem, cap, bw, beta, m, cuts, placement,
                                                                 status);
    return cudaGetLastError();
}

}  // namespace pp
