// Partition stage of the paper's heuristic (Section 3.2.1, Eq. 6-7, Algorithm 1), many chains per
// launch: split a chain of L cut points into contiguous partitions that each fit the capacity
// kappa of a node, minimising the sum of the weights of the points a partition ends with (the
// tensor that crosses the cut; the last partition sends nothing).
//
// The paper walks an explicit graph of all feasible partitions with a memo per last point.  Here
// the same optimum is a chain recurrence over suffixes with the sliding memory window of the
// exact search:   F[i] = min over e in [i, hi(i)] of G[e],   G[e] = weight[e] + F[e + 1],  G[L-1] = 0,
// where hi(i) is the last point such that points i..hi(i) fit.  Values carry the number of
// partitions in their low bits, (cost << 11 | partitions), so that one unsigned minimum applies the
// tie rule "smaller cost, then fewer partitions"; walking forward from point 0 and always taking
// the earliest e that attains F[i] gives the lexicographically smallest cut list among those.
//
// Three kernels.  One warp per chain, chains of up to 128 points: see k_partition_warp.
// One warp per chain of any length: everything about a point that does not
// depend on the recurrence (prefix sums, weights, the last point hi of its window) is worked out by the
// lanes in parallel and kept in the warp's slice of shared memory; the recurrence itself is L dependent
// steps of one lane, a sliding minimum over a queue of candidates with ascending values (a step pushes
// one and drops the beaten and the expired ones: about 360 cycles, whatever the window's length).
// One lane per chain (chains of up to 64 points, 8192 chains or more): see k_partition_lanes.
#include "pp_internal.cuh"

#include <cstring>
#include <type_traits>

namespace pp {

namespace {

constexpr int kPartWarps = 4;
constexpr unsigned long long kInfCost = ~0ull;
constexpr int kPartsBits = 11;  // partitions <= PP_MAX_L = 1024 < 2^11

__host__ __device__ inline size_t part_words(int L) { return 3 * (size_t)L + 1 + ((size_t)L + 1) / 2; }

__global__ void __launch_bounds__(kPartWarps * 32)
k_partition_minsum(int64_t B, int L, int cap_seg, const uint64_t *__restrict__ weight,
                   const uint64_t *__restrict__ mem, const uint64_t *__restrict__ kappa,
                   uint64_t *__restrict__ o_cost, int32_t *__restrict__ o_m, int32_t *__restrict__ o_cuts,
                   uint64_t *__restrict__ o_sizes, int8_t *__restrict__ o_status)
{
    extern __shared__ unsigned long long smem_u64[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long *M = smem_u64 + (size_t)wid * part_words(L);  // [L + 1] prefix sums of the memory
    unsigned long long *G = M + (L + 1);                             // [L]
    unsigned long long *Wt = G + L;                                  // [L] weights
    uint16_t *H = reinterpret_cast<uint16_t *>(Wt + L);              // [L] points after i's window start: hi(i) + 1
    uint16_t *D = H + L;                                             // [L] queue of candidates
    for (int64_t b = (int64_t)blockIdx.x * kPartWarps + wid; b < B; b += (int64_t)gridDim.x * kPartWarps) {
        const uint64_t *w = weight + b * L, *mm = mem + b * L;
        const unsigned long long cap = kappa[b];
        __syncwarp();
        // prefix sums, 32 points at a time; a wrapping sum or a weight beyond the limit voids the chain
        bool bad = false;
        unsigned long long carry = 0;
        if (lane == 0) M[0] = 0;
        for (int base = 0; base < L; base += 32) {
            const int i = base + lane;
            unsigned long long x = i < L ? mm[i] : 0ull;
            const unsigned long long wi = i < L ? w[i] : 0ull;
            if (wi >= PP_MAX_BITS) bad = true;
            if (i < L) Wt[i] = wi;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, x, o);
                if (lane >= o) {
                    if (y > ~0ull - x) bad = true;
                    x += y;
                }
            }
            if (x > ~0ull - carry) bad = true;
            x += carry;
            if (i < L) M[i + 1] = x;
            carry = __shfl_sync(0xFFFFFFFFu, x, 31);
        }
        bad = __any_sync(0xFFFFFFFFu, bad);
        int32_t *cuts = o_cuts ? o_cuts + b * cap_seg : nullptr;
        uint64_t *sizes = o_sizes ? o_sizes + b * cap_seg : nullptr;
        for (int j = lane; j < cap_seg; j += 32) {
            if (cuts) cuts[j] = -1;
            if (sizes) sizes[j] = 0;
        }
        if (bad) {
            if (lane == 0) {
                o_cost[b] = 0;
                o_m[b] = 0;
                o_status[b] = (int8_t)PP_ERR_LIMIT;
            }
            continue;
        }
        __syncwarp();
        for (int i = lane; i < L; i += 32) {  // points i .. e fit: the prefix sums ascend
            const unsigned long long base = M[i];
            int lo = i, hi = L;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (M[mid + 1] - base <= cap) lo = mid + 1; else hi = mid;
            }
            H[i] = (uint16_t)lo;
        }
        __syncwarp();
        // backward recurrence
        unsigned long long F = kInfCost;
        if (lane == 0) {
            unsigned long long g = 1ull;  // G of the point about to be pushed: cost 0, one partition
            unsigned long long back = 0ull, front = 0ull;
            int head = 0, tail = -1, oldest = 0;  // D[head .. tail]: points in descending order, values ascending
            for (int i = L - 1; i >= 0; --i) {
                const int end = H[i];
                const unsigned long long wprev = i > 0 ? Wt[i - 1] : 0ull;
                G[i] = g;
                while (tail >= head && back >= g) {
                    --tail;
                    if (tail >= head) back = G[D[tail]];
                }
                D[++tail] = (uint16_t)i;
                back = g;
                if (tail == head) { front = g; oldest = i; }
                while (head <= tail && oldest >= end) {
                    ++head;
                    if (head <= tail) { oldest = D[head]; front = G[oldest]; }
                }
                F = head <= tail ? front : kInfCost;
                g = F == kInfCost ? kInfCost : F + (wprev << kPartsBits) + 1ull;
            }
        }
        __syncwarp();
        F = __shfl_sync(0xFFFFFFFFu, F, 0);
        if (F == kInfCost) {
            if (lane == 0) {
                o_cost[b] = 0;
                o_m[b] = 0;
                o_status[b] = (int8_t)PP_INFEASIBLE;
            }
            continue;
        }
        const int parts = (int)(F & ((1ull << kPartsBits) - 1ull));
        if (lane == 0) {
            o_cost[b] = F >> kPartsBits;
            o_m[b] = parts;
            o_status[b] = parts > cap_seg + 1 ? (int8_t)PP_ERR_LIMIT : (int8_t)PP_OK;  // cuts do not fit the caller's rows
        }
        if (parts > cap_seg + 1) continue;
        // forward walk: the earliest point that attains the optimum of the suffix
        unsigned long long target = F;
        int i = 0, nc = 0;
        for (;;) {
            const int hi = (int)H[i] - 1;
            int found = -1;
            for (int base = i; base <= hi && found < 0; base += 32) {
                const int e = base + lane;
                const unsigned int hits = __ballot_sync(0xFFFFFFFFu, e <= hi && G[e] == target);
                if (hits) found = base + __ffs(hits) - 1;
            }
            if (found < 0 || found == L - 1) break;  // found < 0 cannot happen on a consistent table
            const unsigned long long wf = Wt[found];
            if (lane == 0) {
                if (cuts) cuts[nc] = found;
                if (sizes) sizes[nc] = wf;
            }
            ++nc;
            target = target - (wf << kPartsBits) - 1ull;
            i = found + 1;
        }
    }
}

// One warp per chain of at most 32 NQ points: lane l holds the points l, l + 32, ... in registers.  A step
// of the recurrence hands the value of one point to the lanes of the points in front of it, which keep the smallest of those
// within their windows; the next point's value is then one shuffle away.  (Taking the
// minimum over a point's window by two warp reductions: 600 chains of 128 points on the device 25.1 us, 8000 of 50 37.1, 8000 of
// 100 98.5; so 21.0, 27.8, 72.1.)  The cut list is put together in registers too and leaves in one piece: the outputs may lie
// across the bus.
//
// Bound by the chain of L steps.  A call with one chain of 50 points: 31.9 us with the queue and inputs read across the bus, 10
// less with the inputs as parameters; 120 points 35.5 by reductions, 32.6 so.  Up to four points a lane.
//
// PARAMS: the inputs of all chains (weights, memory, capacities one after another) are the kernel's
// parameters; nothing is read across the bus or copied in front of the kernel.
constexpr int kParamWords = 496;  // of the 4 KB that every launch may carry
struct PartIn {
    uint64_t v[kParamWords];
};
struct PartNone {};
constexpr int kWarpMaxL = 128;
// No suffix of these chains comes near it (weights are below 2^40), and it can take more weights without wrapping.
constexpr unsigned long long kFar = 1ull << 62;

template <int NQ, bool PARAMS>
__global__ void __launch_bounds__(kPartWarps * 32)
k_partition_warp(const __grid_constant__ std::conditional_t<PARAMS, PartIn, PartNone> params, int64_t B, int L, int cap_seg,
                 const uint64_t *__restrict__ weight, const uint64_t *__restrict__ mem, const uint64_t *__restrict__ kappa,
                 uint64_t *__restrict__ o_cost, int32_t *__restrict__ o_m, int32_t *__restrict__ o_cuts,
                 uint64_t *__restrict__ o_sizes, int8_t *__restrict__ o_status)
{
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    __shared__ unsigned long long s_M[kPartWarps][32 * NQ + 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long *M = s_M[wid];
    if constexpr (PARAMS) {
        const uint64_t *in = params.v;
        // an address of its own: neighbouring lanes read neighbouring words, which the constant bank would serve
        // one after another
        asm volatile("" : "+l"(in));
        weight = in;
        mem = in + B * L;
        kappa = in + 2 * B * L;
    }
    for (int64_t b = (int64_t)blockIdx.x * kPartWarps + wid; b < B; b += (int64_t)gridDim.x * kPartWarps) {
        unsigned long long wt[NQ], x[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int i = q * 32 + lane;
            wt[q] = i < L ? weight[b * L + i] : 0ull;
            x[q] = i < L ? mem[b * L + i] : 0ull;
        }
        const unsigned long long cap = kappa[b];
        // prefix sums; a wrapping sum or a weight beyond the limit voids the chain
        bool bad = false;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1)
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const unsigned long long y = __shfl_up_sync(kAll, x[q], o);
                if (lane >= o) {
                    bad |= y > ~0ull - x[q];
                    x[q] += y;
                }
            }
        __syncwarp();
        if (lane == 0) M[0] = 0;
        unsigned long long carry = 0;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            bad |= wt[q] >= PP_MAX_BITS || x[q] > ~0ull - carry;
            x[q] += carry;
            M[q * 32 + lane + 1] = x[q];
            carry = __shfl_sync(kAll, x[q], 31);
        }
        bad = __any_sync(kAll, bad);
        __syncwarp();
        // first point beyond the window of i: points i .. end - 1 fit (the prefix sums ascend)
        int end[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) end[q] = q * 32 + lane;
#pragma unroll
        for (int step = 32 * NQ; step; step >>= 1)
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int to = end[q] + step;
                if (to <= L && M[to] - M[min(q * 32 + lane, L)] <= cap) end[q] = to;
            }
        // Backward recurrence: G of a point goes to all points in front of it whose window holds it, so that the optimum of
        // the next suffix is complete when its turn comes.
        unsigned long long G[NQ], best[NQ], g = 1ull;  // g: of the point at hand; cost 0, one partition
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            G[q] = kInfCost;
            best[q] = kFar;
        }
#pragma unroll
        for (int q = NQ - 1; q >= 0; --q) {
            const unsigned long long before = q > 0 ? __shfl_sync(kAll, wt[q > 0 ? q - 1 : 0], 31) : 0ull;
            unsigned long long wprev = __shfl_up_sync(kAll, wt[q], 1);  // lane i: weight of the point before i
            if (lane == 0) wprev = before;
            wprev = (wprev << kPartsBits) + 1ull;
#pragma unroll 4
            for (int i = min(L - 1 - q * 32, 31); i >= 0; --i) {
                if (lane == i) G[q] = g;
#pragma unroll
                for (int p = 0; p <= q; ++p) {
                    const int ahead = (q - p) * 32 + i - lane;
                    if ((unsigned)ahead < (unsigned)(end[p] - p * 32 - lane) && g < best[p]) best[p] = g;
                }
                g = __shfl_sync(kAll, best[q] + wprev, i);
            }
        }
        const unsigned long long F0 = __shfl_sync(kAll, best[0], 0), F = F0 >= kFar ? kInfCost : F0;
        const int parts = bad || F == kInfCost ? 0 : (int)(F & ((1ull << kPartsBits) - 1ull));
        const bool fits = parts <= cap_seg + 1;  // the cuts fit the caller's rows
        // forward walk: the earliest point that attains the optimum of the suffix
        int cut[NQ];
        unsigned long long size[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            cut[q] = -1;
            size[q] = 0ull;
        }
        unsigned long long target = F;
        int i = 0;
        for (int nc = 0; fits && nc < parts - 1; ++nc) {
            int e = 0, found = 0;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int x = __shfl_sync(kAll, end[q], i & 31);
                e = q == i >> 5 ? x : e;
            }
            bool none = true;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int at = q * 32 + lane;
                const uint32_t hits = __ballot_sync(kAll, at >= i && at < e && G[q] == target);
                if (none && hits) {
                    none = false;
                    found = q * 32 + __ffs(hits) - 1;
                }
            }
            unsigned long long wf = 0ull;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const unsigned long long x = __shfl_sync(kAll, wt[q], found & 31);
                wf = q == found >> 5 ? x : wf;
            }
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (nc == q * 32 + lane) {
                    cut[q] = found;
                    size[q] = wf;
                }
            target = target - (wf << kPartsBits) - 1ull;
            i = found + 1;
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int j = q * 32 + lane;
            if (o_cuts && j < cap_seg) o_cuts[b * cap_seg + j] = cut[q];
            if (o_sizes && j < cap_seg) o_sizes[b * cap_seg + j] = size[q];
        }
        for (int j = 32 * NQ + lane; j < cap_seg; j += 32) {
            if (o_cuts) o_cuts[b * cap_seg + j] = -1;
            if (o_sizes) o_sizes[b * cap_seg + j] = 0;
        }
        if (lane == 0) {
            o_cost[b] = parts ? F >> kPartsBits : 0ull;
            o_m[b] = parts;
            o_status[b] = bad || !fits ? (int8_t)PP_ERR_LIMIT : parts ? (int8_t)PP_OK : (int8_t)PP_INFEASIBLE;
        }
    }
}

// The same recurrence with one chain per lane, for short chains in bulk: every lane of a warp walks
// its own chain through the same loop, so the control of a step is paid once per 32 chains, and the
// window minimum needs no reduction across lanes.  A lane's prefix sums and G values sit in its own
// column of shared memory, element (i, lane) at word pair (i * 32 + lane): whatever index a lane
// uses, it stays in its own banks.  Same tie rules, same outputs.
constexpr int kLaneWarps = 2;
constexpr int kLaneMaxL = 64;   // (2 L + 1) * 256 bytes of shared memory per warp
constexpr int kLaneMinB = 8192;  // below this the warp-per-chain kernel has more warps to hide the steps' latency behind

__global__ void __launch_bounds__(kLaneWarps * 32)
k_partition_lanes(int64_t B, int L, int cap_seg, const uint64_t *__restrict__ weight,
                  const uint64_t *__restrict__ mem, const uint64_t *__restrict__ kappa,
                  uint64_t *__restrict__ o_cost, int32_t *__restrict__ o_m, int32_t *__restrict__ o_cuts,
                  uint64_t *__restrict__ o_sizes, int8_t *__restrict__ o_status)
{
    extern __shared__ unsigned long long smem_u64[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long *M = smem_u64 + (size_t)wid * (2 * L + 1) * 32 + lane;  // M[i * 32]: memory of points 0..i-1
    unsigned long long *G = M + (size_t)(L + 1) * 32;                          // G[e * 32]
    const int64_t groups = (B + 31) >> 5;
    for (int64_t g = (int64_t)blockIdx.x * kLaneWarps + wid; g < groups; g += (int64_t)gridDim.x * kLaneWarps) {
        const int64_t b0 = g * 32, b = b0 + lane;
        const bool act = b < B;
        const int64_t rows = (B - b0 < 32 ? B - b0 : 32) * (int64_t)cap_seg;
        // the 32 chains' output rows are one contiguous stretch: cleared by the warp together
        for (int64_t j = lane; j < rows; j += 32) {
            if (o_cuts) o_cuts[b0 * cap_seg + j] = -1;
            if (o_sizes) o_sizes[b0 * cap_seg + j] = 0;
        }
        __syncwarp();
        const uint64_t *w = weight + (act ? b : b0) * L, *mm = mem + (act ? b : b0) * L;
        const unsigned long long cap = kappa[act ? b : b0];
        bool bad = false;
        unsigned long long acc = 0;
        M[0] = 0;
        for (int i = 0; i < L; ++i) {
            const unsigned long long x = mm[i];
            if (w[i] >= PP_MAX_BITS) bad = true;
            if (x > ~0ull - acc) bad = true;  // the 64-bit sum would wrap
            acc += x;
            M[(size_t)(i + 1) * 32] = acc;
        }
        // backward recurrence
        unsigned long long F = kInfCost;
        int hi = L - 1;
        G[(size_t)(L - 1) * 32] = 1ull;  // cost 0, one partition
        unsigned long long wprev = L > 1 ? w[L - 2] : 0ull;
        for (int i = L - 1; i >= 0; --i) {
            const unsigned long long wcur = wprev;          // weight of point i - 1
            if (i >= 2) wprev = w[i - 2];                   // asked for one step ahead
            const unsigned long long Mi = M[(size_t)i * 32];
            while (hi >= i && M[(size_t)(hi + 1) * 32] - Mi > cap) --hi;
            unsigned long long best = kInfCost;
            for (int e = i; e <= hi; ++e) {
                const unsigned long long x = G[(size_t)e * 32];
                best = x < best ? x : best;
            }
            F = best;
            if (i > 0) G[(size_t)(i - 1) * 32] = F == kInfCost ? kInfCost : F + (wcur << kPartsBits) + 1ull;
        }
        if (!act) continue;
        if (bad || F == kInfCost) {
            o_cost[b] = 0;
            o_m[b] = 0;
            o_status[b] = bad ? (int8_t)PP_ERR_LIMIT : (int8_t)PP_INFEASIBLE;
            continue;
        }
        const int parts = (int)(F & ((1ull << kPartsBits) - 1ull));
        o_cost[b] = F >> kPartsBits;
        o_m[b] = parts;
        o_status[b] = parts > cap_seg + 1 ? (int8_t)PP_ERR_LIMIT : (int8_t)PP_OK;  // cuts do not fit the caller's rows
        if (parts > cap_seg + 1) continue;
        // forward walk: the earliest point that attains the optimum of the suffix
        unsigned long long target = F;
        int i = 0, nc = 0;
        for (;;) {
            int found = -1;
            const unsigned long long Mi = M[(size_t)i * 32];
            for (int e = i; e < L && M[(size_t)(e + 1) * 32] - Mi <= cap; ++e)
                if (G[(size_t)e * 32] == target) {
                    found = e;
                    break;
                }
            if (found < 0 || found == L - 1) break;  // found < 0 cannot happen on a consistent table
            const unsigned long long wf = w[found];
            if (o_cuts) o_cuts[b * cap_seg + nc] = found;
            if (o_sizes) o_sizes[b * cap_seg + nc] = wf;
            ++nc;
            target = target - (wf << kPartsBits) - 1ull;
            i = found + 1;
        }
    }
}

template <bool PARAMS, typename In, typename... Args>
void launch_warp(int L, unsigned blocks, cudaStream_t s, const In &in, Args... args)
{
    if (L <= 32) k_partition_warp<1, PARAMS><<<blocks, kPartWarps * 32, 0, s>>>(in, args...);
    else if (L <= 64) k_partition_warp<2, PARAMS><<<blocks, kPartWarps * 32, 0, s>>>(in, args...);
    else k_partition_warp<4, PARAMS><<<blocks, kPartWarps * 32, 0, s>>>(in, args...);
}

}  // namespace

bool partition_as_params(int64_t B, int L) { return L <= kWarpMaxL && B * (2 * L + 1) <= kParamWords; }

cudaError_t launch_partition_params(int64_t B, int L, int cap_seg, const uint64_t *weight, const uint64_t *mem,
                                    const uint64_t *kappa, uint64_t *cost, int32_t *m, int32_t *cuts, uint64_t *sizes,
                                    int8_t *status, cudaStream_t s)
{
    const uint64_t *none = nullptr;
    PartIn in;
    std::memcpy(in.v, weight, (size_t)(B * L) * 8);
    std::memcpy(in.v + B * L, mem, (size_t)(B * L) * 8);
    std::memcpy(in.v + 2 * B * L, kappa, (size_t)B * 8);
    launch_warp<true>(L, (unsigned)((B + kPartWarps - 1) / kPartWarps), s, in, B, L, cap_seg, none, none, none, cost, m, cuts,
                      sizes, status);
    return cudaGetLastError();
}

size_t partition_smem_bytes(int L) { return (size_t)kPartWarps * part_words(L) * sizeof(unsigned long long); }

cudaError_t launch_partition_minsum(int64_t B, int L, int cap_seg, const uint64_t *weight, const uint64_t *mem,
                                    const uint64_t *kappa, uint64_t *cost, int32_t *m, int32_t *cuts,
                                    uint64_t *sizes, int8_t *status, cudaStream_t s)
{
    if (B <= 0) return cudaSuccess;
    if (B >= kLaneMinB && L <= kLaneMaxL) {
        const size_t lsm = (size_t)kLaneWarps * (2 * (size_t)L + 1) * 32 * sizeof(unsigned long long);
        cudaError_t el = allow_shared(k_partition_lanes);
        if (el != cudaSuccess) return el;
        const int64_t groups = (B + 31) / 32;
        int64_t lblocks = (groups + kLaneWarps - 1) / kLaneWarps;
        if (lblocks > 148 * 32) lblocks = 148 * 32;
        k_partition_lanes<<<(unsigned)lblocks, kLaneWarps * 32, lsm, s>>>(B, L, cap_seg, weight, mem, kappa, cost, m, cuts,
                                                                           sizes, status);
        return cudaGetLastError();
    }
    int64_t blocks = (B + kPartWarps - 1) / kPartWarps;
    const int64_t cap = 148 * 32;
    if (blocks > cap) blocks = cap;
    if (L <= kWarpMaxL) {
        launch_warp<false>(L, (unsigned)blocks, s, PartNone{}, B, L, cap_seg, weight, mem, kappa, cost, m, cuts, sizes, status);
        return cudaGetLastError();
    }
    const size_t sm = partition_smem_bytes(L);
    cudaError_t e = allow_shared(k_partition_minsum);
    if (e != cudaSuccess) return e;
    k_partition_minsum<<<(unsigned)blocks, kPartWarps * 32, sm, s>>>(B, L, cap_seg, weight, mem, kappa, cost, m, cuts,
                                                                     sizes, status);
    return cudaGetLastError();
}

}  // namespace pp
