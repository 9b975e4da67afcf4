// Building blocks shared by the kernels that work on one instance in shared memory: the window minimum
// over a row held by a group of lanes, the ranking of an instance's quotients by one block, bit selection.
#pragma once
#include "pp_internal.cuh"

namespace pp {

__host__ __device__ constexpr int log2i(int x) { return x <= 1 ? 0 : 1 + log2i(x / 2); }

// The correctly rounded quotient x / b of integers 0 <= x < 2^40 and 0 < b < 2^24 held as doubles; r is b's correctly rounded
// reciprocal.  x r lies within two units in the last place of x / b, so its remainder is below 2^26 such units and exact, and
// what the last step rounds is off by less than 2^-50 of a unit.  No quotient comes that near to the middle m between two
// doubles: x / b - m is a multiple of half a unit over b, hence at least 2^-25 of a unit, and zero never, since m has 54
// bits, the last one set, and would have to divide x.  (pp_debug_quotients holds it against __ddiv_rn.)
__device__ __forceinline__ double quotient(double x, double b, double r)
{
    const double q = __dmul_rn(x, r);
    return __fma_rn(__fma_rn(-q, b, x), r, q);
}

// What a link of bandwidth b moves within t: every size up to `sure`, none beyond `most`; one between them is settled by its
// quotient.  The largest size whose quotient rounds to no more than t lies below t b (1 + 2^-53), which is beyond the product rounded
// down by less than 2^-10, sizes being below 2^40.
struct SizeBracket {
    double sure, most;
};
__device__ __forceinline__ SizeBracket sizes_within(double t, double b)
{
    const double sure = __dmul_rd(t, b);
    return {sure, __dadd_rn(sure, 1.0 / 1024.0)};
}

// The window minimum of a row that a group of G lanes holds, P consecutive positions a lane: out at
// position c2 = min of g over [lo, c2 - 1].  The window is the tail of the block (= lane) that holds its
// start (suffix minima, through shared memory), whole blocks in between (a sparse table over the G block
// minima), and the lane's own prefix; or, where it starts inside the lane's own block, a few of its
// registers.  Which cells those are depends on the node and the position only: a WindowCode names them, made
// once per instance, so that a position costs three loads and three minima (35 instructions where the
// cells were worked out anew for every row).
template <int G, int P>
struct Strip {  // of a group, in elements: suffix minima (odd stride: no bank conflicts), table, one "none"
    static constexpr int kLevels = log2i(G) + 1;
    static constexpr int kTable = G * (P + 1);
    static constexpr int kNone = kTable + kLevels * G;
    static constexpr int kSize = kNone + 1;
};

struct alignas(8) WindowCode {
    uint16_t tail, left, right;  // byte offsets of the cells in the strip
    uint16_t inside;             // 0, or 1 + the start's position in the lane's own block when it is there
};

// code of position c2 with window start lo (c2 itself: an empty window); T: element of the strip
template <int G, int P, typename T>
__device__ __forceinline__ WindowCode window_code(int c2, int lo)
{
    using St = Strip<G, P>;
    const int sl = c2 / P, bl = lo / P, n = sl - 1 - bl;  // n whole blocks between lo's and this one
    int tail = St::kNone, left = St::kNone, right = St::kNone, inside = 0;
    if (n >= 0) {
        tail = bl * (P + 1) + (lo & (P - 1));
        if (n > 0) {
            const int t = 31 - __clz(n);
            left = St::kTable + t * G + sl - 1;
            right = St::kTable + t * G + bl + (1 << t);
        }
    } else if (lo > sl * P) {
        inside = 1 + lo - sl * P;
    }
    return WindowCode{(uint16_t)(tail * sizeof(T)), (uint16_t)(left * sizeof(T)), (uint16_t)(right * sizeof(T)), (uint16_t)inside};
}

// What goes to the strip: suffix minima of the lane's block, minima of the last 2^t blocks.
// Returns the own prefix minima, pre[i] = min g[0 .. i - 1].
template <int G, int P, typename T>
__device__ __forceinline__ void window_strip(const uint32_t (&g)[P], T *strip, int sl, uint32_t none, uint32_t (&pre)[P])
{
    using St = Strip<G, P>;
    uint32_t s = g[P - 1];
    pre[0] = none;
#pragma unroll
    for (int i = 1; i < P; ++i) pre[i] = i > 1 ? min(pre[i - 1], g[i - 1]) : g[0];
    T *mine = strip + sl * (P + 1);
    mine[P - 1] = (T)s;
#pragma unroll
    for (int i = P - 2; i >= 0; --i) {
        s = min(s, g[i]);
        mine[i] = (T)s;
    }
    uint32_t D = s;
    strip[St::kTable + sl] = (T)D;
#pragma unroll
    for (int t = 1; t < St::kLevels; ++t) {
        D = min(D, __shfl_up_sync(0xFFFFFFFFu, D, 1 << (t - 1), G));  // a lane without a source lane gets its own back
        strip[St::kTable + t * G + sl] = (T)D;
    }
    __syncwarp();
}

// Without codes, for a kernel that asks for a handful of rows only (making the codes of a node takes as
// long as two rows of it): out[i] = min of g over [lo[i], P sl + i - 1].
template <int G, int P, typename T>
__device__ __forceinline__ void window_min_direct(const uint32_t (&g)[P], const int16_t *lo, T *strip, int sl,
                                                  uint32_t none, uint32_t (&out)[P])
{
    uint32_t pre[P];
    window_strip<G, P>(g, strip, sl, none, pre);
    const T *table = strip + Strip<G, P>::kTable;
    const int pos0 = sl * P;
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const int l = lo[i];
        const int bl = l / P, n = sl - 1 - bl;  // whole blocks between lo's and this one
        uint32_t v = pre[i];
        if (n >= 0) {
            v = min(v, (uint32_t)strip[bl * (P + 1) + (l & (P - 1))]);
            if (n > 0) {
                const int t = 31 - __clz(n);
                v = min(v, min((uint32_t)table[t * G + sl - 1], (uint32_t)table[t * G + bl + (1 << t)]));
            }
        } else if (l > pos0) {  // the window starts inside this lane's own block
            v = none;
#pragma unroll
            for (int q = 1; q < i; ++q)
                if (q >= l - pos0) v = min(v, g[q]);
        }
        out[i] = v;
    }
}

// code: this lane's P codes, 16-byte aligned
template <int G, int P, typename T>
__device__ __forceinline__ void window_min(const uint32_t (&g)[P], const WindowCode *code, T *strip,
                                           int sl, uint32_t none, uint32_t (&out)[P])
{
    uint32_t pre[P];
    window_strip<G, P>(g, strip, sl, none, pre);
    const unsigned char *cells = reinterpret_cast<const unsigned char *>(strip);
#pragma unroll
    for (int i = 0; i < P; i += 2) {
        const uint4 two = *reinterpret_cast<const uint4 *>(code + i);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t a = h ? two.z : two.x, b = h ? two.w : two.y;
            const uint32_t tail = *reinterpret_cast<const T *>(cells + (a & 0xFFFFu));
            const uint32_t left = *reinterpret_cast<const T *>(cells + (a >> 16));
            const uint32_t right = *reinterpret_cast<const T *>(cells + (b & 0xFFFFu));
            uint32_t own = pre[i + h];
            if (const uint32_t from = b >> 16) {
                own = none;
#pragma unroll
                for (int q = 1; q < i + h; ++q)
                    if ((uint32_t)q + 1u >= from) own = min(own, g[q]);
            }
            out[i + h] = min(min(own, tail), min(left, right));
        }
    }
}

// r-th (from 0) set bit of x; r below the number of set bits
__device__ __forceinline__ int select_bit(uint32_t x, int r)
{
    int at = 0;
#pragma unroll
    for (int half = 16; half; half >>= 1) {
        const int below = __popc(x & ((1u << half) - 1u));
        const bool up = r >= below;
        r -= up ? below : 0;
        at += up ? half : 0;
        x = up ? x >> half : x;
    }
    return at;
}

constexpr int kRankBuckets = 1024;

// Ranks of the U x D quotients bits[i] / bw[u] of an instance (distinct bits, distinct bandwidths), by one
// block of kThreads: rk[u * D + i] = 1 + number of quotients strictly below.  A bucket sort: a quotient's
// bucket is its place in the range of the instance's quotients on the scale of the doubles' bits
// (monotone), counters in shared memory, their prefix sums, the quotients scattered into the order of the
// buckets, and each compared with the few that share its bucket.  Some 90 instructions per quotient where
// a staircase walk over the sorted quotient matrix took U + L dependent steps, 350.
// first(u, i) is the quotient as the first pass gets it, which may read what val[] held before.
// V holds a key and an entry number of kIdBits; key[] and val[] have n entries, hist kRankBuckets counters.
// lo_d, hi_d: bounds of all positive quotients.  Ends with the block in step.
template <int kThreads, typename V, int kIdBits, typename First>
__device__ __forceinline__ void rank_quotients(const unsigned long long *bits, const uint32_t *bw, int U, int D, First first,
                                               double lo_d, double hi_d, uint32_t *key, V *val, uint32_t *hist,
                                               uint16_t *rk, uint32_t *s_sum)
{
    const int tid = threadIdx.x, n = U * D;
    const unsigned long long lowest = (unsigned long long)__double_as_longlong(lo_d);
    const unsigned long long span = (unsigned long long)__double_as_longlong(hi_d) - lowest;
    const int shift = max(31, 64 - __clzll((long long)(span | 1ull))) - 31;  // keys of 31 bits, buckets of 10
    const uint32_t recip_D = D > 1 ? 0xFFFFFFFFu / (uint32_t)D + 1u : 0u;  // floor(e / D) by a multiplication, e < 2^16
    for (int i = tid; i < kRankBuckets; i += kThreads) hist[i] = 0u;
    __syncthreads();
    auto quotient = [&](int e) {
        const int u = D > 1 ? (int)__umulhi((uint32_t)e, recip_D) : e;
        return __ddiv_rn((double)bits[e - u * D], (double)bw[u]);
    };
    for (int e = tid; e < n; e += kThreads) {
        const int u = D > 1 ? (int)__umulhi((uint32_t)e, recip_D) : e;
        const unsigned long long q = (unsigned long long)__double_as_longlong(first(u, e - u * D));
        const uint32_t y = (uint32_t)((q > lowest ? q - lowest : 0ull) >> shift);  // 0.0 counts as the lowest
        key[e] = y;
        atomicAdd(&hist[y >> 21], 1u);
    }
    __syncthreads();
    static_assert(kThreads >= kRankBuckets / 8 && kThreads % 32 == 0, "eight buckets to a thread");
    {  // counters -> first places
        uint32_t c[8], sum = 0, upto;
        const bool on = tid < kRankBuckets / 8;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            c[i] = on ? hist[8 * tid + i] : 0u;
            sum += c[i];
        }
        upto = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, upto, o);
            if ((tid & 31) >= o) upto += y;
        }
        if ((tid & 31) == 31 && on) s_sum[tid >> 5] = upto;
        __syncthreads();
        uint32_t place = upto - sum;
        if (on) {
            for (int i = 0; i < (tid >> 5); ++i) place += s_sum[i];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                hist[8 * tid + i] = place;
                place += c[i];
            }
        }
    }
    __syncthreads();
    for (int e = tid; e < n; e += kThreads) {
        const uint32_t y = key[e];
        val[atomicAdd(&hist[y >> 21], 1u)] = ((V)y << kIdBits) | (V)e;
    }
    __syncthreads();
    // a counter now holds the end of its bucket, that is the start of the next one
    constexpr V kId = ((V)1 << kIdBits) - 1;
    for (int e = tid; e < n; e += kThreads) {
        const uint32_t y = key[e], bk = y >> 21;
        const V mine = ((V)y << kIdBits) | (V)e;
        const int start = bk ? (int)hist[bk - 1] : 0, end = (int)hist[bk];
        int below = start;
        for (int q = start; q < end; ++q) {
            const V other = val[q];
            if ((other ^ mine) > kId) below += other < mine;
            else if (other != mine) below += quotient((int)(other & kId)) < quotient(e);  // one key: the doubles decide
        }
        rk[e] = (uint16_t)(1 + below);
    }
    __syncthreads();
}

}  // namespace pp
