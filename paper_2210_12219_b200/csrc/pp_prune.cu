// The exact search as a sparse frontier with a bound, one launch for the whole solve.
//
// The dense sweep (pp_sweep*.cu) computes every state of the recurrence
//   dp[S'][w][c'] = min over c in [lo_w(c'), c'-1] of g[c],
//   g[c] = min over v in S = S'\{w} of max(dp[S][v][c], gamma[c][v][w]).
// Values never fall along a plan, so a state that is no better than a complete plan already known
// cannot be part of a better one.  The levels are walked in the order of the number of nodes used,
// and a plan with fewer nodes wins a tie; a state is therefore kept only while its value is
//   < the best final value found on a lower level, and
//   <= the best one found on the level that is being written (another node set may still win the tie).
// Likewise a state whose remaining layers need more memory than the unused nodes have together
// cannot be completed.  What is left is exact: every state on a plan of value beta* survives, so the
// final choice and the backtrack see what they would see in the dense table.  On the named
// configurations and on the paper's evaluation graphs 0.1 to 5 % of the node sets keep a state; what
// bounds the solve is then the latency of a handful of levels, not the table.
//
// Values are 32-bit keys of the fp64 quotients (one correctly rounded division per layer and link):
// 0 for +0.0, all ones for +inf, else 1 + (bits - base) >> shift, base and shift such that the
// smallest and the largest possible quotient fit.  A key stands for a class of neighbouring doubles
// (relative width about 2^-28), and since the map is monotone the minima and maxima of keys are the
// keys of the minima and maxima.  The plan found is therefore optimal and canonical unless the class
// of beta* holds a quotient smaller than the plan's own bottleneck.  That is checked at the end; if it
// does, the search runs again (block 0 alone) with keys that resolve exactly this class.  A rank
// compression as the dense search has it would be exact at once, but ranking 30 000 quotients takes
// longer (0.03 ms) than the search.
//
// One cooperative launch: blocks meet at a barrier in global memory once per level.
//   level 2   one group of lanes per ordered pair (v, w): the keys of the link (kept in `gam` for the
//             later levels), the base state of v, the row of ({v, w}, w)
//   level j   the node sets of the frontier are a list; a group of lanes takes (S, w), reads the rows
//             of S that can still matter, and writes the row of (S + w, w) if any of its states does
//   end       once a level has little work block 0 goes on alone (its barrier costs nothing); it walks
//             back by the threshold rule, checks the class of beta*, and writes the result record
// A group of G lanes holds a row, P consecutive cut positions per lane.
#include <algorithm>
#include <cstring>

#include "pp_blocks.cuh"

namespace pp {

namespace {

constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr uint32_t kInfKey = 0xFFFFFFFFu;
constexpr int kSpinLimit = 1 << 22;  // polls of a barrier before the kernel gives up
constexpr int kAloneRounds = 2;      // a level of at most this many rounds of one block is done by block 0 alone
__host__ __device__ constexpr int prune_threads(int P) { return P <= 16 ? 512 : 256; }

// Which class of doubles a key stands for.
struct KeyMap {
    unsigned long long base;
    int shift;
    uint32_t zoom;  // 0, or the class that is resolved exactly: smaller values become 0, larger ones +inf
    __device__ __forceinline__ uint32_t operator()(double x) const
    {
        const unsigned long long b = (unsigned long long)__double_as_longlong(x);
        if (b == 0ull) return 0u;
        const uint32_t key = 1u + (uint32_t)((b - base) >> shift);
        if (!zoom) return key;
        return key < zoom ? 0u : key > zoom ? kInfKey : 1u + (uint32_t)((b - base) & ((1ull << shift) - 1ull));
    }
};

// first value that is not worth keeping on `level`, given the best final state known
__device__ __forceinline__ uint32_t limit_of(unsigned long long best, int level)
{
    if (best == kNoBest) return kInfKey;
    const uint32_t val = (uint32_t)(best >> 30);
    return ((int)(best >> 25) & 31) < level ? val : val + 1u;
}

// smallest of a group's keys
template <int G>
__device__ __forceinline__ uint32_t group_min(uint32_t u)
{
    if constexpr (G == 32) {
        u = __reduce_min_sync(kFull, u);
    } else {
#pragma unroll
        for (int o = G >> 1; o; o >>= 1) u = min(u, __shfl_xor_sync(kFull, u, o, G));
    }
    return u;
}

// Shared memory: the part common to the block, then one strip per group of lanes.
struct PruneLayout {
    size_t bits, M, cap, bw, gmin, lo, code, Wp, speed, strips, total;
};
__host__ __device__ inline PruneLayout prune_layout(int L, int k, int Lp, int groups, size_t strip, bool codes, bool compute)
{
    PruneLayout p;
    size_t o = 0;
    auto take = [&o](size_t bytes) { size_t at = o; o = (o + bytes + 15) & ~(size_t)15; return at; };
    p.bits = take((size_t)Lp * 8);
    p.M = take((size_t)(L + 1) * 8);
    p.cap = take((size_t)k * 8);
    p.bw = take((size_t)k * k * 4);
    p.gmin = take((size_t)k * k * 4);
    p.lo = take((size_t)k * Lp * 2);
    p.code = take(codes ? (size_t)k * Lp * sizeof(WindowCode) : 0);
    p.Wp = take(compute ? (size_t)(L + 1) * 8 : 0);
    p.speed = take(compute ? (size_t)k * 4 : 0);
    p.strips = o;
    p.total = o + (size_t)groups * strip;
    return p;
}
// Window codes where a warp works off several rows of every node: short chains, few blocks.
template <int G, bool CT>
constexpr bool kCodes = G <= 16 && !CT;

// strip of a group: its window minima, then the ids of the source rows
template <int G, int P>
constexpr size_t kStripBytes = ((size_t)(Strip<G, P>::kSize + PP_MAX_K) * 4 + 15) & ~(size_t)15;

template <int P>
__device__ __forceinline__ void load_row(const uint32_t *p, uint32_t (&x)[P])
{
#pragma unroll
    for (int i = 0; i < P; i += 4) {
        const uint4 t = __ldcg(reinterpret_cast<const uint4 *>(p + i));
        x[i] = t.x; x[i + 1] = t.y; x[i + 2] = t.z; x[i + 3] = t.w;
    }
}
template <int P>
__device__ __forceinline__ void load_row_ca(const uint32_t *p, uint32_t (&x)[P])  // through L1: written before the last barrier
{
#pragma unroll
    for (int i = 0; i < P; i += 4) {
        const uint4 t = *reinterpret_cast<const uint4 *>(p + i);
        x[i] = t.x; x[i + 1] = t.y; x[i + 2] = t.z; x[i + 3] = t.w;
    }
}
template <int P>
__device__ __forceinline__ void store_row(uint32_t *p, const uint32_t (&x)[P])
{
#pragma unroll
    for (int i = 0; i < P; i += 4) *reinterpret_cast<uint4 *>(p + i) = make_uint4(x[i], x[i + 1], x[i + 2], x[i + 3]);
}

// All blocks of the grid; false when the wait ran out (the caller returns).
__device__ __forceinline__ bool grid_barrier(PruneCtl *ctl, uint32_t target)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t seen;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&ctl->arrived) : "memory");
        int spins = 0;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&ctl->arrived) : "memory");
        } while (seen < target && ++spins < kSpinLimit);
        s_ok = seen >= target;
        if (!s_ok) ctl->failed = 1;
    }
    __syncthreads();
    return s_ok != 0;
}

// The inputs travel as a kernel parameter (4 KB for chains of up to 128 layers, 18 KB for the longest): no
// copy to queue in front of the search and to wait for.
template <int N, bool CT>
struct PruneIn {
    unsigned long long bits[N], M[N + 1], cap[PP_MAX_K];
    uint32_t bw[PP_MAX_K * PP_MAX_K];
};
template <int N>
struct PruneIn<N, true> {
    unsigned long long bits[N], M[N + 1], cap[PP_MAX_K];
    uint32_t bw[PP_MAX_K * PP_MAX_K], speed[PP_MAX_K];
    unsigned long long Wp[N + 1];
};

// n-th (from 0) set bit of x
__device__ __forceinline__ int nth_bit(uint32_t x, int n)
{
    for (; n > 0; --n) x &= x - 1;
    return __ffs(x) - 1;
}

template <int G, int P, bool CT>
__global__ void __launch_bounds__(prune_threads(P), 1) k_prune(const PruneDev d, const __grid_constant__ PruneIn<G * P, CT> params)
{
    constexpr int kThreads = prune_threads(P), kWarps = kThreads / 32, kGroups = kThreads / G, kPerWarp = 32 / G;
    extern __shared__ __align__(16) unsigned char smem_prune[];
    const int k = d.k, L = d.L, Lp = d.Lp, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int sl = lane & (G - 1), gb = lane & ~(G - 1);  // position in the group, first lane of the group
    const int at = sl * P;                                // this lane's first cut position
    const bool in_row = at < Lp;
    const int at0 = in_row ? at : 0;
    const PruneLayout lay = prune_layout(L, k, Lp, kGroups, kStripBytes<G, P>, kCodes<G, CT>, CT);
    double *s_bits = reinterpret_cast<double *>(smem_prune + lay.bits);
    unsigned long long *s_M = reinterpret_cast<unsigned long long *>(smem_prune + lay.M);
    unsigned long long *s_cap = reinterpret_cast<unsigned long long *>(smem_prune + lay.cap);
    uint32_t *s_bw = reinterpret_cast<uint32_t *>(smem_prune + lay.bw);
    uint32_t *s_gmin = reinterpret_cast<uint32_t *>(smem_prune + lay.gmin);
    int16_t *s_lo = reinterpret_cast<int16_t *>(smem_prune + lay.lo);
    [[maybe_unused]] unsigned long long *s_Wp = reinterpret_cast<unsigned long long *>(smem_prune + lay.Wp);
    [[maybe_unused]] uint32_t *s_speed = reinterpret_cast<uint32_t *>(smem_prune + lay.speed);
    [[maybe_unused]] WindowCode *s_code = reinterpret_cast<WindowCode *>(smem_prune + lay.code);
    uint32_t *s_strip = reinterpret_cast<uint32_t *>(smem_prune + lay.strips + (size_t)(tid / G) * kStripBytes<G, P>);
    uint32_t *s_ids = s_strip + Strip<G, P>::kSize;
    __shared__ unsigned long long s_best;  // best final state the block knows of
    __shared__ unsigned int s_pick[kWarps];
    __shared__ int s_cut[PP_MAX_K], s_node[PP_MAX_K];
    __shared__ unsigned long long s_worst;  // bits of the plan's bottleneck
    __shared__ int s_zoom, s_nlinks;
    __shared__ uint16_t s_links[PP_MAX_K * PP_MAX_K];  // links with a quotient no larger than the optimum
    PruneCtl *ctl = d.ctl;
    const double kInf = __longlong_as_double(0x7FF0000000000000ll);
    const int top = k < L ? k : L;
    const uint32_t full = (1u << k) - 1u;
    const int npairs = k * (k - 1) / 2;

    unsigned long long t_start = 0;
    if (blockIdx.x == 0 && tid == 0) asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t_start));
    // ---- inputs ----
    // read through an address of their own: neighbouring threads read neighbouring words, which the constant
    // bank would serve one after another
    const PruneIn<G * P, CT> *in = &params;
    asm volatile("" : "+l"(in));
    for (int c = tid; c < Lp; c += kThreads) s_bits[c] = c < L ? (double)in->bits[c] : 0.0;
    for (int c = tid; c <= L; c += kThreads) s_M[c] = in->M[c];
    for (int e = tid; e < k * k; e += kThreads) {
        s_bw[e] = in->bw[e];
        s_gmin[e] = kInfKey;
    }
    if (tid < k) s_cap[tid] = in->cap[tid];
    if (tid == 0) s_best = kNoBest;
    if constexpr (CT) {
        for (int c = tid; c <= L; c += kThreads) s_Wp[c] = in->Wp[c];
        if (tid < k) s_speed[tid] = in->speed[tid];
    }
    if (sl == 0) s_strip[Strip<G, P>::kNone] = kInfKey;
    __syncthreads();
    auto set_window = [&](int w, int c, int l) {
        s_lo[w * Lp + c] = (int16_t)l;
        if constexpr (kCodes<G, CT>) s_code[w * Lp + c] = window_code<G, P, uint32_t>(c, l);
    };
    // window starts: lo[w][c'] = earliest previous cut c >= 0 such that layers c+1..c' fit on w, c' itself when
    // not even layer c' alone does; a lane takes a run of neighbouring positions, found by bisection for the
    // first and by stepping on for the others
    if (d.lo)  // a problem that is solved again and again has them on the device
        for (int w = wid; w < k; w += kWarps)
            for (int c = lane; c < Lp; c += 32) set_window(w, c, c < L ? (int)d.lo[w * L + c] : c);
    else
    for (int w = wid; w < k; w += kWarps) {
        const int run = (Lp + 31) / 32, c0 = lane * run, c1 = min(c0 + run, Lp);
        const unsigned long long capw = s_cap[w];
        int l = 0;
        for (int c = c0; c < c1; ++c) {
            if (c < L) {
                const unsigned long long need = s_M[c + 1], thr = need > capw ? need - capw : 0ull;
                if (c == c0) {
                    int hi = c;  // M[c + 1] >= thr
                    while (l < hi) {
                        const int mid = (l + hi) >> 1;
                        if (s_M[mid + 1] < thr) l = mid + 1; else hi = mid;
                    }
                } else {
                    while (s_M[l + 1] < thr) ++l;
                }
            } else {
                l = c;
            }
            set_window(w, c, l);
        }
    }
    __syncthreads();
    const unsigned long long total = s_M[L];
    const uint32_t tight_levels = d.tight_levels, whole = d.whole;

    KeyMap key_of{d.key_base, d.key_shift, 0u};
    bool dense = false;
    uint32_t barriers = 0;
    int nblk = gridDim.x;  // blocks that work on the search: 1 once block 0 goes on alone
    int m = 0, w_end = 0, status = (int)PP_INFEASIBLE;
    double beta = kInf;

    // base state of one node: layers 0..c on v
    auto base_key = [&](int v, int c) -> uint32_t {
        if (s_M[c + 1] > s_cap[v]) return kInfKey;
        if constexpr (CT) return s_speed[v] ? key_of(__ddiv_rn((double)s_Wp[c + 1], (double)s_speed[v])) : kInfKey;
        return 0u;
    };
    // row of (S2, w) from g: window minimum, then drop what cannot matter, note a final state; returns
    // whether the group keeps the row, and its smallest value
    auto make_row = [&](const uint32_t (&g)[P], uint32_t (&out)[P], uint32_t S2, int w, int level, uint32_t lim, bool on,
                        uint32_t &rmin) -> bool {
        if constexpr (!CT) {
            if constexpr (kCodes<G, CT>) window_min<G, P>(g, s_code + (size_t)w * Lp + at0, s_strip, sl, kInfKey, out);
            else window_min_direct<G, P>(g, s_lo + (size_t)w * Lp + at0, s_strip, sl, kInfKey, out);
        } else {
            // the compute time of the last partition depends on both its ends: every output scans its
            // window, nearest start first, until the compute time alone is too much
#pragma unroll
            for (int i = 0; i < P; ++i) s_strip[at + i] = g[i];
            __syncwarp();
            uint32_t cur[P];
            cur[0] = at > 0 ? s_strip[at - 1] : kInfKey;
#pragma unroll
            for (int i = 1; i < P; ++i) cur[i] = g[i - 1];
#pragma unroll
            for (int i = 0; i < P; ++i) out[i] = kInfKey;
            const uint32_t *seg = d.seg + (size_t)w * L * Lp + at0;
            for (int dd = 0; dd < L; ++dd) {
                uint32_t x[P];
                bool more = false;
                load_row_ca<P>(seg + (size_t)dd * Lp, x);
#pragma unroll
                for (int i = 0; i < P; ++i) {
                    out[i] = min(out[i], max(cur[i], x[i]));
                    more |= x[i] < lim;
                }
                if (!more || at + P - 2 - dd < 0) break;
#pragma unroll
                for (int i = P - 1; i > 0; --i) cur[i] = cur[i - 1];
                cur[0] = at - 2 - dd >= 0 ? s_strip[at - 2 - dd] : kInfKey;
            }
        }
        const bool tight = (tight_levels >> level) & 1u;
        double room = kInf;
        if (tight) {
            room = 0.0;
            for (uint32_t rest = full & ~S2; rest; rest &= rest - 1) room += (double)s_cap[__ffs(rest) - 1];
            room *= 1.0 + 1e-9;  // rounding of the sums must not drop a state
        }
        uint32_t least = kInfKey, x = kInfKey;
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const int c = at + i;
            if (!on || out[i] >= lim || c >= L || (tight && (double)(total - s_M[c + 1]) > room)) out[i] = kInfKey;
            least = min(least, out[i]);
            if (c == L - 1) x = out[i];
        }
        if (x != kInfKey) {
            const unsigned long long cand = pack_best(x, level, S2, w);
            if (cand < *reinterpret_cast<volatile unsigned long long *>(&s_best)) atomicMin(&s_best, cand);
        }
        rmin = group_min<G>(least);
        return rmin != kInfKey;
    };
    // end of a level: the block's best final state goes to the others; false = a barrier gave up
    auto level_end = [&](unsigned long long best_before) -> bool {
        if (nblk == 1) {
            __syncthreads();
            return true;
        }
        __syncthreads();
        if (tid == 0 && s_best < best_before)
            asm volatile("red.relaxed.gpu.global.min.u64 [%0], %1;" ::"l"(&ctl->best), "l"(s_best) : "memory");
        barriers += gridDim.x;
        if (!grid_barrier(ctl, barriers)) return false;
        const unsigned long long seen = __ldcg(&ctl->best);
        if (tid == 0 && seen < s_best) s_best = seen;
        __syncthreads();
        return true;
    };

    bool found = !CT && whole != 0;
    if (found) {
        m = 1;
        beta = 0.0;
        w_end = __ffs(whole) - 1;
        status = (int)PP_OK;
        if (tid < PP_MAX_K) {
            s_cut[tid] = -1;
            s_node[tid] = tid == 0 ? w_end : -1;
        }
    }
    while (!found) {
        const int slots = nblk * kWarps, my_slot = wid * nblk + (nblk == 1 ? 0 : (int)blockIdx.x);
        // node sets of three nodes and more start without rows (those of two nodes are all written below)
        for (uint32_t S = (nblk == 1 ? 0 : blockIdx.x) * kThreads + tid; S < (1u << k); S += nblk * kThreads)
            if (__popc(S) > 2) d.live[S] = 0u;
        uint32_t *const count = ctl->count + (key_of.zoom ? 32 : 0);
        if constexpr (CT) {
            // compute times of every run of layers: seg[(w * L + d) * Lp + c'] = layers c'-d .. c' on w
            const int n = k * L * Lp;
            for (int e = (nblk == 1 ? 0 : (int)blockIdx.x) * kThreads + tid; e < n; e += nblk * kThreads) {
                const int r = e / Lp, c2 = e - r * Lp, w = r / L, first = c2 - (r - w * L);
                uint32_t key = kInfKey;
                const uint32_t sp = s_speed[w];
                if (c2 < L && first >= 0 && sp != 0 && s_M[c2 + 1] - s_M[first] <= s_cap[w])
                    key = key_of(__ddiv_rn((double)(s_Wp[c2 + 1] - s_Wp[first]), (double)sp));
                d.seg[e] = key;
            }
            if (tid == 0)
                for (int v = 0; v < k; ++v) {
                    const uint32_t x = base_key(v, L - 1);
                    if (x != kInfKey) s_best = min(s_best, pack_best(x, 1, 1u << v, v));
                }
            if (!level_end(kNoBest)) return;
        }
        // ---- two nodes: the keys of every link, the rows of every pair ----
        if (top >= 2) {
            const unsigned long long before = s_best;
            const int items = k * (k - 1);
            for (int base = my_slot * kPerWarp; base < items; base += slots * kPerWarp) {
                const int it = base + lane / G;
                const bool on = it < items;
                const int v = on ? it / (k - 1) : 0, x = on ? it - v * (k - 1) : 0, w = x + (x >= v ? 1 : 0);
                const uint32_t link = on ? s_bw[v * k + w] : 0u;
                const double div = (double)link;
                uint32_t g[P], out[P], gm = kInfKey, rmin;
#pragma unroll
                for (int i = 0; i < P; ++i) {
                    const int c = at + i;
                    g[i] = (link != 0 && c < L) ? key_of(__ddiv_rn(s_bits[c], div)) : kInfKey;
                    if (c < L - 1) gm = min(gm, g[i]);
                }
                if (on && in_row) store_row<P>(d.gam + (size_t)(w * k + v) * Lp + at, g);
                gm = group_min<G>(gm);
                if (on && sl == 0) d.gmin[w * k + v] = gm;
#pragma unroll
                for (int i = 0; i < P; ++i) {
                    const int c = at + i;
                    g[i] = c < L ? max(g[i], base_key(v, c)) : kInfKey;
                }
                const uint32_t S2 = (1u << v) | (1u << w);
                const uint32_t lim = limit_of(*reinterpret_cast<volatile unsigned long long *>(&s_best), 2);
                const bool keep = make_row(g, out, S2, w, 2, lim, on, rmin);
                const int a = v < w ? v : w, b = v < w ? w : v;
                const int pr = a * (2 * k - a - 1) / 2 + (b - a - 1);
                const uint32_t id = 2u * (uint32_t)pr + (w == b ? 1u : 0u);
                if (keep && in_row) store_row<P>(d.rows + (size_t)id * Lp + at, out);
                if (on && sl == 0) {
                    d.rowmap[(size_t)S2 * k + w] = ((unsigned long long)rmin << 32) | id;
                    if (w == b) {
                        d.list[pr] = S2;
                        d.live[S2] = S2;
                    }
                }
                __syncwarp();
            }
            if (!level_end(before)) return;
            for (int e = tid; e < k * k; e += kThreads) s_gmin[e] = (e / k != e % k) ? __ldcg(d.gmin + e) : kInfKey;
            __syncthreads();
        }

        // ---- three nodes and more ----
        uint32_t beg = 0, cnt = (uint32_t)npairs;
        unsigned long long used = 2ull * npairs;  // rows: one per item, kept or not, so that ids need no counter
        bool alone = nblk == 1;
        for (int level = 3; level <= top && cnt; ++level) {
            const int nw = k - (level - 1);
            const unsigned long long items = (unsigned long long)cnt * nw;
            if (used + items > d.row_cap) {
                dense = true;
                break;
            }
            if (!alone && items <= (unsigned long long)(kGroups * kAloneRounds)) {
                if (blockIdx.x != 0) break;
                alone = true;
                nblk = 1;
            }
            const unsigned long long before = s_best;
            const int my = alone ? wid : my_slot, all = alone ? kWarps : slots;
            for (unsigned long long base = (unsigned long long)my * kPerWarp; base < items; base += (unsigned long long)all * kPerWarp) {
                const unsigned long long it = base + lane / G;
                const bool on = it < items;
                const uint32_t li = on ? (uint32_t)it / (uint32_t)nw : 0u;
                const uint32_t S = __ldcg(d.list + beg + li);
                const int w = nth_bit(full & ~S, on ? (int)((uint32_t)it - li * (uint32_t)nw) : 0);
                const uint32_t rows_of_S = __ldcg(d.live + S);
                const uint32_t lim = limit_of(*reinterpret_cast<volatile unsigned long long *>(&s_best), level);
                // source rows that can still matter: their smallest value and the link's smallest key
                uint32_t src = 0;
#pragma unroll
                for (int v0 = 0; v0 < PP_MAX_K; v0 += G) {
                    if (v0 >= k) break;
                    const int v = v0 + sl;
                    bool ok = false;
                    if (v < k && ((S >> v) & 1u)) {
                        const unsigned long long e = __ldcg(d.rowmap + (size_t)S * k + v);
                        s_ids[v] = (uint32_t)e;
                        ok = on && ((rows_of_S >> v) & 1u) && max((uint32_t)(e >> 32), s_gmin[w * k + v]) < lim;
                    }
                    const uint32_t hit = __ballot_sync(kFull, ok);
                    src |= (G == 32 ? hit : ((hit >> gb) & ((1u << (G & 31)) - 1u))) << v0;
                }
                if (!__any_sync(kFull, src != 0)) continue;
                __syncwarp();
                uint32_t g[P];
#pragma unroll
                for (int i = 0; i < P; ++i) g[i] = kInfKey;
                while (src != 0) {  // two sources at a time: their loads are in flight together
                    const int v = __ffs(src) - 1;
                    src &= src - 1;
                    const int v2 = src ? __ffs(src) - 1 : v;
                    src &= src - 1;
                    if (in_row) {
                        uint32_t a[P], b[P], a2[P], b2[P];
                        load_row<P>(d.rows + (size_t)s_ids[v] * Lp + at, a);
                        load_row<P>(d.gam + (size_t)(w * k + v) * Lp + at, b);
                        load_row<P>(d.rows + (size_t)s_ids[v2] * Lp + at, a2);
                        load_row<P>(d.gam + (size_t)(w * k + v2) * Lp + at, b2);
#pragma unroll
                        for (int i = 0; i < P; ++i) g[i] = min(g[i], min(max(a[i], b[i]), max(a2[i], b2[i])));
                    }
                }
                uint32_t gm = g[0], out[P], rmin;
#pragma unroll
                for (int i = 1; i < P; ++i) gm = min(gm, g[i]);
                if (!__any_sync(kFull, gm < lim)) continue;
                const uint32_t S2 = S | (1u << w);
                if (make_row(g, out, S2, w, level, lim, on, rmin)) {
                    const uint32_t id = (uint32_t)(used + it);
                    if (in_row) store_row<P>(d.rows + (size_t)id * Lp + at, out);
                    if (sl == 0) {
                        d.rowmap[(size_t)S2 * k + w] = ((unsigned long long)rmin << 32) | id;
                        if (atomicOr(d.live + S2, 1u << w) == 0u)
                            d.list[beg + cnt + atomicAdd(&count[level], 1u)] = S2;
                    }
                }
                __syncwarp();
            }
            used += items;
            if (!level_end(before)) return;
            beg += cnt;
            cnt = __ldcg(&count[level]);
        }
        if (blockIdx.x != 0 || dense) break;  // block 0 finishes
        __syncthreads();
        const unsigned long long best = s_best;
        if (best == kNoBest) break;  // no plan

        // ---- final choice, backtrack: the lowest (c, v) whose value is within the optimum's class ----
        status = (int)PP_OK;
        m = (int)(best >> 25) & 31;
        const uint32_t vstar = (uint32_t)(best >> 30);
        uint32_t S = (uint32_t)(best >> 5) & 0xFFFFFu;
        int w = (int)best & 31, c2 = L - 1;
        if (tid < PP_MAX_K) s_cut[tid] = s_node[tid] = -1;
        if (tid == 0) s_worst = 0ull;
        __syncthreads();
        for (int j = m - 1; j >= 0; --j) {
            if (tid == 0) {
                s_node[j] = w;
                if (j < m - 1) s_cut[j] = c2;
            }
            if (j == 0) break;
            const uint32_t from = S & ~(1u << w);
            const int lo = s_lo[(size_t)w * Lp + c2], np = __popc(from);
            const uint32_t rows_of = np > 1 ? __ldcg(d.live + from) : from;
            unsigned int bestk = 0xFFFFFFFFu;
            for (int vi = wid; vi < np; vi += kWarps) {
                const int v = nth_bit(from, vi);
                const unsigned long long e = np > 1 ? __ldcg(d.rowmap + (size_t)from * k + v) : 0ull;
                if (!((rows_of >> v) & 1u) || (uint32_t)(e >> 32) > vstar) continue;
                const uint32_t *row = d.rows + (size_t)(uint32_t)e * Lp, *gm = d.gam + (size_t)(w * k + v) * Lp;
                for (int c0 = lo; c0 < c2; c0 += 32) {
                    const int c = c0 + lane;
                    bool hit = false;
                    if (c < c2) {
                        uint32_t x = max(np > 1 ? __ldcg(row + c) : base_key(v, c), __ldcg(gm + c));
                        if constexpr (CT) x = max(x, __ldcg(d.seg + (size_t)(w * L + c2 - c - 1) * Lp + c2));
                        hit = x <= vstar;
                    }
                    const unsigned int hits = __ballot_sync(kFull, hit);
                    if (hits) {
                        const unsigned int kk = ((unsigned)(c0 + __ffs(hits) - 1) << 5) | (unsigned)v;
                        bestk = kk < bestk ? kk : bestk;
                        break;
                    }
                }
            }
            if (lane == 0) s_pick[wid] = bestk;
            __syncthreads();
            unsigned int pick = s_pick[lane < kWarps ? lane : 0];
            pick = __reduce_min_sync(kFull, pick);
            __syncthreads();
            if (pick == 0xFFFFFFFFu) {  // cannot happen on a consistent frontier; report, do not trap
                status = (int)PP_ERR_CUDA;
                break;
            }
            S = from;
            w = (int)(pick & 31u);
            c2 = (int)(pick >> 5);
        }
        __syncthreads();
        if (status != (int)PP_OK) break;
        // the plan's own bottleneck
        if (tid < m) {
            double x = 0.0;
            if (tid < m - 1) x = __ddiv_rn(s_bits[s_cut[tid]], (double)s_bw[s_node[tid] * k + s_node[tid + 1]]);
            if constexpr (CT) {
                const int first = tid ? s_cut[tid - 1] + 1 : 0, last = tid < m - 1 ? s_cut[tid] : L - 1;
                const double y = __ddiv_rn((double)(s_Wp[last + 1] - s_Wp[first]), (double)s_speed[s_node[tid]]);
                x = y > x ? y : x;
            }
            atomicMax(&s_worst, (unsigned long long)__double_as_longlong(x));
        }
        if (tid == 0) s_zoom = 0;
        __syncthreads();
        const unsigned long long worst = s_worst;
        beta = __longlong_as_double((long long)worst);
        if (key_of.zoom || key_of.shift == 0 || worst == 0ull) break;  // every key is one double
        // a smaller quotient in the same class?  Few links have one at all below the optimum.
        if (tid < 32) {
            int n = 0;
            for (int p0 = 0; p0 < k * k; p0 += 32) {
                const int p = p0 + lane;
                const bool has = p < k * k && s_gmin[p] <= vstar;
                const uint32_t hit = __ballot_sync(kFull, has);
                if (has) s_links[n + __popc(hit & ((1u << lane) - 1u))] = (uint16_t)p;
                n += __popc(hit);
            }
            if (lane == 0) s_nlinks = n;
        }
        __syncthreads();
#pragma unroll 4
        for (int e = tid; e < s_nlinks * L; e += kThreads) {
            const int p = s_links[e / L], c = e % L;
            if (c < L - 1 && d.gam[(size_t)p * Lp + c] == vstar) {
                const int w2 = p / k, v2 = p - w2 * k;
                if ((unsigned long long)__double_as_longlong(__ddiv_rn(s_bits[c], (double)s_bw[v2 * k + w2])) < worst) s_zoom = 1;
            }
        }
        if constexpr (CT) {
            for (int e = tid; e < k * L * Lp; e += kThreads)
                if (__ldcg(d.seg + e) == vstar) {
                    const int r = e / Lp, last = e - r * Lp, w2 = r / L, first = last - (r - w2 * L);
                    if ((unsigned long long)__double_as_longlong(__ddiv_rn((double)(s_Wp[last + 1] - s_Wp[first]), (double)s_speed[w2])) < worst)
                        s_zoom = 1;
                }
        }
        __syncthreads();
        if (!s_zoom) break;
        key_of.zoom = vstar;  // once more, this class resolved
        nblk = 1;
        if (tid == 0) s_best = kNoBest;
        __syncthreads();
    }

    // ---- result ----
    __syncthreads();
    if (blockIdx.x == 0) {
        if (!dense && tid < PP_MAX_K) {
            d.out->cuts[tid] = m ? s_cut[tid] : -1;
            d.out->placement[tid] = m ? s_node[tid] : -1;
        }
        if (tid == 0) {
            if (!dense) {
                d.out->beta_ms = beta;
                d.out->status = status;
                d.out->m = m;
            }
            unsigned long long t_end;
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t_end));
            d.note->ns = (long long)(t_end - t_start);
            d.note->dense = dense ? 1 : 0;
            ctl->dense = dense ? 1 : 0;
        }
    }
    // the last block to leave clears the counters for the next launch
    __shared__ uint32_t s_left;
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_left = atomicAdd(&ctl->left, 1u);
    }
    __syncthreads();
    if (s_left == gridDim.x - 1) {
        if (tid < 64) ctl->count[tid] = 0u;
        if (tid == 0) {
            ctl->best = kNoBest;
            ctl->arrived = 0u;
            ctl->left = 0u;
        }
    }
}

struct PruneShape {
    int G, P;
};
PruneShape prune_shape(int L)
{
    PruneShape s{4, 4};
    while (s.G * s.P < L && s.G < 32) s.G *= 2;
    while (s.G * s.P < L) s.P *= 2;
    return s;
}

template <int G, int P, bool CT>
cudaError_t launch_shape(const PruneDev &d, const PruneHost &h, int sms, cudaStream_t s)
{
    PruneIn<G * P, CT> in;
    std::memcpy(in.bits, h.bits, (size_t)d.L * 8);
    std::memcpy(in.M, h.M, (size_t)(d.L + 1) * 8);
    std::memcpy(in.cap, h.cap, (size_t)d.k * 8);
    std::memcpy(in.bw, h.bw, (size_t)d.k * d.k * 4);
    if constexpr (CT) {
        std::memcpy(in.Wp, h.Wp, (size_t)(d.L + 1) * 8);
        std::memcpy(in.speed, h.speed, (size_t)d.k * 4);
    }
    constexpr int threads = prune_threads(P), groups = threads / G;
    // blocks: one round over the targets of the widest level if it is kept whole; a single block where
    // two rounds of it do, its barrier costs next to nothing
    unsigned long long widest = 1, binom = 1;
    for (int j = 1; j <= d.k; ++j) {
        binom = binom * (unsigned)(d.k - j + 1) / (unsigned)j;  // C(k, j)
        widest = std::max(widest, binom * (unsigned)(d.k - j));
    }
    int blocks = (int)std::min<unsigned long long>((widest + groups - 1) / groups, (unsigned long long)sms);
    if (blocks <= 2) blocks = 1;
    const size_t sm = prune_layout(d.L, d.k, d.Lp, groups, kStripBytes<G, P>, kCodes<G, CT>, CT).total;
    cudaError_t e = cudaFuncSetAttribute(k_prune<G, P, CT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = blocks > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_prune<G, P, CT>, d, in);
}

}  // namespace

int prune_row_pad(int L)
{
    const int P = prune_shape(L).P;
    return (L + P - 1) / P * P;
}

void prune_ctl_init(PruneCtl *c)
{
    *c = PruneCtl{};
    c->best = kNoBest;
}

// base and shift of the keys of all values between lo and hi (the smallest and the largest positive one)
void prune_key_range(double lo, double hi, PruneDev *d)
{
    unsigned long long a, b;
    static_assert(sizeof a == sizeof lo, "doubles are 64 bits");
    std::memcpy(&a, &lo, 8);
    std::memcpy(&b, &hi, 8);
    d->key_base = a;
    d->key_shift = 0;
    while (((b - a) >> d->key_shift) >= 0x80000000ull) ++d->key_shift;
}

// The nodes that hold the whole chain, and the levels on which some choice of nodes leaves too little
// memory for some rest of it: even the k - j smallest nodes together hold everything on the others.
void prune_node_bounds(const uint64_t *cap, uint64_t total, PruneDev *d)
{
    uint64_t sorted[PP_MAX_K];
    d->whole = 0;
    for (int v = 0; v < d->k; ++v) {
        sorted[v] = cap[v];
        d->whole |= (cap[v] >= total ? 1u : 0u) << v;
    }
    std::sort(sorted, sorted + d->k);
    d->tight_levels = 0;
    double sum = 0.0;
    for (int n = 0; n <= d->k; ++n) {
        if (sum < (double)total) d->tight_levels |= 1u << (d->k - n);
        if (n < d->k) sum += (double)sorted[n];
    }
}

cudaError_t launch_prune(const PruneDev &d, const PruneHost &h, int sms, cudaStream_t s)
{
    const PruneShape sh = prune_shape(d.L);
    switch (sh.G * 100 + sh.P) {
#define PP_CASE(g, p) \
    case g * 100 + p: return d.seg ? launch_shape<g, p, true>(d, h, sms, s) : launch_shape<g, p, false>(d, h, sms, s);
        PP_CASE(4, 4) PP_CASE(8, 4) PP_CASE(16, 4) PP_CASE(32, 4) PP_CASE(32, 8)
#undef PP_CASE
        case 3216: return launch_shape<32, 16, false>(d, h, sms, s);  // Eq. 1 stops at 256 layers
        case 3232: return launch_shape<32, 32, false>(d, h, sms, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace pp
