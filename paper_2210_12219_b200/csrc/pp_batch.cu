// Many-instance exact search: one thread block per instance, the whole state table in shared
// memory as 16-bit ranks.  Same recurrence, final choice and backtrack rule as the single-instance path
// (see pp_sweep.cu); global memory sees the inputs once and the result record once.
//
// Per instance the block
//   1. stages the inputs, builds the memory prefix sums and the window table lo[w][c'] (binary searches);
//   2. rank-compresses gamma (Eq. 3): distinct bandwidths and distinct transfer sizes listed, one fp64
//      division per pair of them, ranked by rank_quotients;
//   3. sweeps the popcount levels: a group of G lanes takes a target row (P + w, w), P positions a lane,
//      forms g[c] = min_v max(dp[P][v][c], rank[v][w][c]) on packed pairs of positions and takes the
//      window minimum over [lo_w(c'), c'-1] (window_min); one block barrier a level;
//   4. walks back from the smallest final state (value, popcount, mask, node) by the threshold rule, one warp,
//      lanes over the positions, and takes beta from the plan's own quotients.
// An instance is a chain of some twenty short phases; what bounds a batch of a few hundred is the length of
// that chain.  300 x (k = 7, L = 45), us in the kernel: 66 with a walk of U + L steps per rank and windows
// scanned position by position, about 40 with the phases above.  Of 93 000 cycles 26 000 then went to the
// inputs (three dependent trips over the bus, contended 64-bit maxima in shared memory): 9 000 with all loads
// of a thread in flight and warp reductions, 74 000 in all.  A call from host arrays 88.2 -> 85.8 us, 155 x (k = 8,
// L = 47) 138.7 -> 133.4, 1616 x (k = 5, L = 53) on the device 72.0 -> 68.3.  Levels take half of it, bound by
// instruction issue: 8 positions a lane where 4 fit 92.8 us, blocks of 512 threads 91.9, of 256 87.0.
#include <algorithm>

#include "pp_blocks.cuh"

namespace pp {

namespace {

// Blocks of 384 threads, three to an SM.  Where the batch does not fit the GPU so and the instances are small (k <= 6, whose
// levels do not fill twelve warps) blocks of 192, up to six to an SM: us a call, 888 x (k = 4, L = 24) 23.7 -> 16.6, (k = 6, L = 24)
// 39.1 -> 30.9, 1616 x (k = 5, L = 53) 68.5 -> 54.2, 4000 x (k = 4, L = 45) 109 -> 74, 3000 x (k = 6, L = 60) 194 -> 170; 444 x (k = 6, L = 24) 20.9, 22.7, 1000 x (k = 7, L = 45) 112, 117.
// (256 threads, four to an SM: 22.8, 38.7, 61.3 and 20.7, 125; 384, four to an SM: 24.8, 41.1, 63.4.)
constexpr int kWideThreads = 384, kWideBlocks = 3;
constexpr int kNarrowThreads = 192, kNarrowBlocks = 6, kNarrowMaxK = 6, kNarrowMaxP = 8;
constexpr uint32_t kInf16 = 0xFFFFu;

// Lanes and positions a lane of a row of L positions.
struct BatchShape {
    int G, P;
};
__host__ __device__ inline BatchShape batch_shape(int L)
{
    BatchShape s{4, 4};
    while (s.G * s.P < L && s.G < 32) s.G *= 2;
    while (s.G * s.P < L) s.P *= 2;
    return s;
}

struct BatchLayout {
    size_t dp, key, val, rk, hist, rank, M, cap, bits, dbits, bw, ubw, rowoff, pair_u, cls, lo, code, strips, total;
    int Ls;  // row stride: whole pieces of four positions
    int Lc;  // row stride of the window codes: a lane reads those of all its P positions
};

__host__ __device__ inline BatchLayout batch_layout(int L, int k, int threads)
{
    BatchLayout b;
    const size_t rows = (size_t)k << (k - 1);
    const size_t U = (size_t)k * (k - 1) > 0 ? (size_t)k * (k - 1) : 1;
    const size_t Ls = ((size_t)L + 3) & ~(size_t)3;
    const BatchShape sh = batch_shape(L);
    b.Ls = (int)Ls;
    b.Lc = (L + sh.P - 1) / sh.P * sh.P;
    size_t o = 0;
    auto up16 = [](size_t x) { return (x + 15) & ~(size_t)15; };
    auto take = [&](size_t bytes) { size_t at = o; o = up16(o + bytes); return at; };
    b.M = take((size_t)(L + 1) * sizeof(uint64_t));
    b.cap = take((size_t)k * sizeof(uint64_t));
    b.bits = take((size_t)L * sizeof(uint64_t));
    b.dbits = take((size_t)L * sizeof(uint64_t));
    b.bw = take((size_t)k * k * sizeof(uint32_t));
    b.ubw = take(U * sizeof(uint32_t));
    b.rowoff = take(((size_t)1 << k) * sizeof(uint16_t));
    b.lo = take((size_t)k * Ls * sizeof(int16_t));
    b.rank = take((size_t)k * k * Ls * sizeof(uint16_t));
    b.pair_u = take((size_t)k * k * sizeof(int16_t));
    b.cls = take((size_t)L * sizeof(uint16_t));
    b.code = take((size_t)k * b.Lc * sizeof(WindowCode));
    // The scratch of the ranking is dead before the first state is written: it shares the bytes of the state
    // table and the strips.
    const size_t table = up16(rows * Ls * sizeof(uint16_t));
    const size_t strip = (size_t)sh.G * (sh.P + 1) + (size_t)(log2i(sh.G) + 1) * sh.G + 1;
    b.dp = o;
    b.strips = o + table;
    const size_t end = b.strips + up16((size_t)(threads / sh.G) * strip * sizeof(uint16_t));
    size_t q = b.dp;
    b.hist = q; q += up16((size_t)kRankBuckets * sizeof(uint32_t));
    b.val = q;  q += up16(U * L * sizeof(unsigned long long));
    b.key = q;  q += up16(U * L * sizeof(uint32_t));
    b.rk = q;   q += up16(U * L * sizeof(uint16_t));
    b.total = end > q ? end : q;
    return b;
}

}  // namespace

PP_CHECKS_OF(batch)

size_t batch_smem_bytes(int L, int k)
{
    if (k > 12) return (size_t)1 << 40;  // compact rows are 16-bit numbers
    if ((size_t)k * (k - 1) * L + 1 > 65534) return (size_t)1 << 40;  // ranks must fit 16 bits
    return batch_layout(L, k, kWideThreads).total;
}

int batch_block_threads(bool narrow) { return narrow ? kNarrowThreads : kWideThreads; }

// Blocks that an SM holds at a time: as many as the registers are shared out for, or as fit its 228 KB.
int batch_blocks_per_sm(int L, int k, bool narrow)
{
    const size_t fit = (size_t)(228 << 10) / (batch_layout(L, k, batch_block_threads(narrow)).total + 1024);
    return (int)std::max<size_t>(1, std::min<size_t>(narrow ? kNarrowBlocks : kWideBlocks, fit));
}

// Whether the instances of a batch go to narrow blocks: where these take fewer waves.  That is no matter of the batch's
// size alone: the tables of a longer chain leave room for five narrow blocks, four, or no more than wide ones.  Four are 24
// warps against 36, which the levels of k > 4 feel: there it has to be a third fewer.  Ratio of the times, narrow to wide,
// at 500, 600, 900, 1500, 4000 instances (888 are two waves either way from five on, 1.07 to 1.15):
//   six to an SM    (k = 6, L = 45) 0.82, 0.88, 0.91, 0.85, 0.83
//   five            (k = 6, L = 60) 0.83, 0.86, 0.93, 0.94, 0.88
//   four            (k = 6, L = 80) 0.91, 1.19, 1.01, 1.03, 1.03; (k = 5, L = 110) 0.87, 1.20, 0.98, 1.01, 1.00;
//                   (k = 4, L = 160) 0.77, 1.11, 0.92, 0.93, 0.93
//   as many as wide (k = 6, L = 100), three, 1.37, 1.26, 1.29, 1.20, 1.23; (k = 6, L = 140), two, 1.24 to 1.31;
//                   (k = 6, L = 200), one, 1.48 to 1.50
bool batch_narrow(int64_t B, int L, int k, int sms)
{
    if (k > kNarrowMaxK || batch_shape(L).P > kNarrowMaxP) return false;
    const int held = batch_blocks_per_sm(L, k, true);
    const auto waves = [&](int blocks) { return (B + (int64_t)sms * blocks - 1) / ((int64_t)sms * blocks); };
    const int64_t wide = waves(batch_blocks_per_sm(L, k, false)), narrow = waves(held);
    return held > 4 || k < 5 ? narrow < wide : 3 * narrow <= 2 * wide;
}

namespace {

// t_rowoff, t_rows, t_first: compact row of (S, lowest node of S), rows ordered by (popcount, mask, node);
// source mask and target node of every row; first row of each popcount
template <int NT, int G, int P>
__global__ void __launch_bounds__(NT, P > 8 ? 1 : NT == kWideThreads ? kWideBlocks : kNarrowBlocks)
k_batch(int64_t B, int L, int k, const uint32_t *__restrict__ t_rowoff, const uint32_t *__restrict__ t_rows,
        const uint32_t *__restrict__ t_first, const uint64_t *__restrict__ g_bits, const uint64_t *__restrict__ g_mem,
        const uint64_t *__restrict__ g_cap, const uint32_t *__restrict__ g_bw, double *__restrict__ o_beta,
        int32_t *__restrict__ o_m, int32_t *__restrict__ o_cuts, int32_t *__restrict__ o_place, int8_t *__restrict__ o_status)
{
    // The next piece of a batch that is launched in pieces shares nothing with this one and may start beside it.
    asm volatile("griddepcontrol.launch_dependents;");
    constexpr int kGroups = NT / G;
    extern __shared__ __align__(16) unsigned char smem[];
    const BatchLayout lay = batch_layout(L, k, NT);
    unsigned long long *M = reinterpret_cast<unsigned long long *>(smem + lay.M);
    unsigned long long *cap = reinterpret_cast<unsigned long long *>(smem + lay.cap);
    unsigned long long *s_bits = reinterpret_cast<unsigned long long *>(smem + lay.bits);
    unsigned long long *dbits = reinterpret_cast<unsigned long long *>(smem + lay.dbits);
    uint32_t *s_bw = reinterpret_cast<uint32_t *>(smem + lay.bw);
    uint32_t *ubw = reinterpret_cast<uint32_t *>(smem + lay.ubw);
    uint16_t *rowoff = reinterpret_cast<uint16_t *>(smem + lay.rowoff);
    uint16_t *dp = reinterpret_cast<uint16_t *>(smem + lay.dp);      // [compact row][Ls]
    uint16_t *rank = reinterpret_cast<uint16_t *>(smem + lay.rank);  // [v][w][Ls]
    uint16_t *rk = reinterpret_cast<uint16_t *>(smem + lay.rk);
    int16_t *pair_u = reinterpret_cast<int16_t *>(smem + lay.pair_u);
    uint16_t *cls = reinterpret_cast<uint16_t *>(smem + lay.cls);
    int16_t *lo = reinterpret_cast<int16_t *>(smem + lay.lo);        // [w][Ls]
    __shared__ unsigned long long s_best;
    __shared__ uint32_t s_least, s_most;  // sizes as floats, rounded down and up
    __shared__ uint32_t s_slow, s_fast, s_U, s_D;
    __shared__ uint32_t s_sum[(NT / 32)];

    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int sl = lane & (G - 1), at = sl * P;
    const int Ls = lay.Ls, Lc = lay.Lc;
    const bool in_row = at < Ls;
    const int at0 = in_row ? at : 0;
    WindowCode *code = reinterpret_cast<WindowCode *>(smem + lay.code);  // [w][Lc]
    uint16_t *strip = reinterpret_cast<uint16_t *>(smem + lay.strips) + (size_t)(tid / G) * Strip<G, P>::kSize;
    const double kInf = __longlong_as_double(0x7FF0000000000000ll);
    const uint32_t FULL = 0xFFFFFFFFu;
    const int kk = k * k, jmax = k < L ? k : L;
    PP_BLOCK_BOUNDS(chk);
    [[maybe_unused]] const size_t n_dp = ((size_t)k << (k - 1)) * Ls, n_rank = (size_t)kk * Ls;  // entries of the tables
    for (uint32_t S = tid; S < (1u << k); S += NT) rowoff[S] = (uint16_t)t_rowoff[S];

    for (int64_t inst = blockIdx.x; inst < B; inst += gridDim.x) {
        const uint64_t *bits = g_bits + inst * L, *mem = g_mem + inst * L;
        const uint32_t *bw = g_bw + inst * kk;
        // ---- 1. stage inputs, bounds of the values ----
        // The arrays may lie across the bus: every thread asks for its words of all of them before it uses one.
        unsigned long long x_bits = 0ull, x_mem = 0ull, x_cap = 0ull;
        uint32_t x_bw = 0u;
        if (tid < L) {
            x_bits = bits[tid];
            x_mem = mem[tid];
        }
        if (tid < kk) x_bw = bw[tid];
        if (tid < k) x_cap = g_cap[inst * k + tid];
        __syncthreads();  // the instance before this one is done
        if (tid == 0) {
            s_least = 0x7F800000u;
            s_most = 0u;
            s_slow = FULL;
            s_fast = s_U = s_D = 0u;
            s_best = kNoBest;
            M[0] = 0ull;
            PP_RESET(chk);
        }
        __syncthreads();
        bool bad = false;
        {
            uint32_t least = 0x7F800000u, most = 0u;
            for (int i = tid; i < L; i += NT) {
                if (i >= NT) {
                    x_bits = bits[i];
                    x_mem = mem[i];
                }
                s_bits[i] = x_bits;
                M[i + 1] = x_mem;
                bad |= x_bits >= PP_MAX_BITS;
                if (x_bits) least = min(least, __float_as_uint(__ull2float_rd(x_bits)));
                most = max(most, __float_as_uint(__ull2float_ru(x_bits)));
            }
            uint32_t usable = 0u;
            if (tid < kk) {  // k <= 12
                bad |= x_bw >= PP_MAX_KBPS;
                usable = tid / k != tid - tid / k * k ? x_bw : 0u;
                s_bw[tid] = usable;
            }
            if (tid < k) cap[tid] = x_cap;
            if (wid * 32 < L) {
                least = __reduce_min_sync(FULL, least);
                most = __reduce_max_sync(FULL, most);
                if (lane == 0) {
                    atomicMin(&s_least, least);
                    atomicMax(&s_most, most);
                }
            }
            if (wid * 32 < kk) {
                const uint32_t slow = __reduce_min_sync(FULL, usable ? usable : FULL), fast = __reduce_max_sync(FULL, usable);
                if (lane == 0) {
                    atomicMin(&s_slow, slow);
                    atomicMax(&s_fast, fast);
                }
            }
        }
        __syncthreads();
        // ---- prefix sums of the memory: the first warp, while the others look for equal values ----
        if (wid == 0) {
            unsigned long long carry = 0;
            for (int base = 0; base < L; base += 32) {
                unsigned long long x = base + lane < L ? M[base + lane + 1] : 0ull;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned long long y = __shfl_up_sync(FULL, x, o);
                    if (lane >= o) {
                        if (y > ~0ull - x) bad = true;  // the 64-bit sum would wrap: PP_ERR_LIMIT, as in pp_problem_create
                        x += y;
                    }
                }
                if (carry > ~0ull - x) bad = true;
                x += carry;
                if (base + lane < L) M[base + lane + 1] = x;
                carry = __shfl_sync(FULL, x, 31);
            }
        }
        // ---- distinct bandwidths and sizes: a value's class is that of its first appearance, and the first
        // appearances are numbered as they come ----
        for (int p = tid - 32; p >= 0 && p < kk; p += NT) {
            const uint32_t x = s_bw[p];
            int f = p;
            for (int q = p - 1; q >= 0; --q) f = s_bw[q] == x ? q : f;
            int u = -1;
            if (x != 0u && f == p) {
                u = (int)atomicAdd(&s_U, 1u);
                ubw[u] = x;
            }
            pair_u[p] = (int16_t)(x == 0u ? -1 : f == p ? u : -2 - f);  // -2 - f: as pair f
        }
        for (int c = NT - 1 - tid; wid > 0 && c < L; c += NT - 32) {
            const unsigned long long x = s_bits[c];
            int f = c;
            for (int q = c - 1; q >= 0; --q) f = s_bits[q] == x ? q : f;
            uint32_t d = 0x8000u | (uint32_t)f;  // as layer f
            if (f == c) {
                d = atomicAdd(&s_D, 1u);
                dbits[d] = x;
            }
            cls[c] = (uint16_t)d;
        }
        bad = __syncthreads_or(bad);
        // windows: lo = max(c* - 1, 0), c* = first start layer from which the segment ending at layer c2 fits
        for (int w = wid; w < k; w += NT / 32) {
            const unsigned long long capw = cap[w];
            for (int c2 = lane; c2 < Lc; c2 += 32) {
                int a = 0, b = c2;
                if (c2 < L) {
                    const unsigned long long need = M[c2 + 1];
                    b = c2 + 1;  // first index in [0, c2 + 1] with M[idx] >= need - cap
                    const unsigned long long thr = need > capw ? need - capw : 0ull;
                    while (a < b) {
                        const int mid = (a + b) >> 1;
                        if (M[mid] < thr) a = mid + 1; else b = mid;
                    }
                    a = a > 0 ? a - 1 : 0;
                } else {
                    a = c2;  // the pad: an empty window
                }
                if (c2 < Ls) lo[w * Ls + c2] = (int16_t)a;
                code[w * Lc + c2] = window_code<G, P, uint16_t>(c2, a);
            }
        }
        __syncthreads();
        const int U = (int)s_U, D = (int)s_D;
        // ---- 2. ranks of the quotients, spread out as rank[v][w][c] ----
        rank_quotients<NT, unsigned long long, 16>(
            dbits, ubw, U, D, [&](int u, int d) { return __ddiv_rn((double)dbits[d], (double)ubw[u]); }, __ddiv_rd((double)__uint_as_float(s_least), (double)s_fast),
            __ddiv_ru((double)__uint_as_float(s_most), (double)s_slow),
            reinterpret_cast<uint32_t *>(smem + lay.key), reinterpret_cast<unsigned long long *>(smem + lay.val),
            reinterpret_cast<uint32_t *>(smem + lay.hist), rk, s_sum);
        for (int pr = wid; pr < kk; pr += (NT / 32)) {
            int u = pair_u[pr];
            if (u < -1) u = pair_u[-2 - u];
            for (int c = lane; c < Ls; c += 32) {
                uint32_t r = kInf16;
                if (u >= 0 && c < L) {
                    uint32_t d = cls[c];
                    if (d & 0x8000u) d = cls[d & 0x7FFFu];
                    if (PP_IN_BOUNDS(chk, u * D + (int)d, U * D)) r = rk[u * D + (int)d];
                }
                if (PP_IN_BOUNDS(chk, pr * Ls + c, n_rank)) rank[pr * Ls + c] = (uint16_t)r;
            }
        }
        __syncthreads();  // the per-entry ranks share their bytes with the state table
        // ---- base frontier ----
        for (int v = wid; v < k; v += (NT / 32))
            for (int c = lane; c < Ls; c += 32) {
                const bool fits = c < L && M[c + 1] <= cap[v];
                if (PP_IN_BOUNDS(chk, (size_t)rowoff[1u << v] * Ls + c, n_dp)) dp[(size_t)rowoff[1u << v] * Ls + c] = (uint16_t)(fits ? 0u : kInf16);
                if (fits && c == L - 1) atomicMin(&s_best, pack_best(0u, 1, 1u << v, v));
            }
        __syncthreads();
        // ---- 3. levels ----
        if (sl == 0) strip[Strip<G, P>::kNone] = kInf16;  // the strips share bytes with the ranking's scratch
        for (int j = 2; j <= jmax; ++j) {
            const uint32_t first = t_first[j], items = t_first[j + 1] - first;
            for (uint32_t base = (uint32_t)(wid * (32 / G)); base < items; base += kGroups) {
                const uint32_t it = base + (uint32_t)(lane / G), row = first + (it < items ? it : items - 1);  // spare groups repeat the last row
                const uint32_t info = t_rows[row], S = info & 0xFFFFu;
                const int w = (int)(info >> 16);
                uint32_t g2[P / 2];
#pragma unroll
                for (int i = 0; i < P / 2; ++i) g2[i] = 0xFFFFFFFFu;
                if (in_row) {
                    const uint16_t *src = dp + (size_t)rowoff[S] * Ls + at, *rw = rank + w * Ls + at;
                    for (uint32_t rem = S; rem; rem &= rem - 1, src += Ls) {
                        const int v = __ffs(rem) - 1;
#pragma unroll
                        for (int i = 0; i < P / 2; i += 2) {
                            if (at + 2 * i >= Ls) break;
                            if (!PP_IN_BOUNDS(chk, src - dp + 2 * i + 3, n_dp) || !PP_IN_BOUNDS(chk, rw - rank + v * k * Ls + 2 * i + 3, n_rank)) break;
                            const uint2 a = *reinterpret_cast<const uint2 *>(src + 2 * i);
                            const uint2 b = *reinterpret_cast<const uint2 *>(rw + v * k * Ls + 2 * i);
                            g2[i] = __vminu2(g2[i], __vmaxu2(a.x, b.x));
                            g2[i + 1] = __vminu2(g2[i + 1], __vmaxu2(a.y, b.y));
                        }
                    }
                }
                uint32_t g[P], out[P];
#pragma unroll
                for (int i = 0; i < P; ++i) g[i] = (i & 1) ? g2[i / 2] >> 16 : g2[i / 2] & 0xFFFFu;
                __syncwarp();  // the previous row's readers are done
                window_min<G, P>(g, code + w * Lc + at0, strip, sl, kInf16, out);
                const uint32_t S2 = S | (1u << w);
                uint16_t *dst = dp + (size_t)row * Ls + at;
#pragma unroll
                for (int i = 0; i < P; i += 4)
                    if (at + i < Ls && PP_IN_BOUNDS(chk, dst - dp + i + 3, n_dp)) {
                        *reinterpret_cast<uint2 *>(dst + i) = make_uint2(out[i] | (out[i + 1] << 16), out[i + 2] | (out[i + 3] << 16));
#pragma unroll
                        for (int q = i; q < i + 4; ++q)
                            if (at + q == L - 1 && out[q] != kInf16) {
                                const unsigned long long cand = pack_best(out[q], j, S2, w);
                                if (cand < *reinterpret_cast<volatile unsigned long long *>(&s_best)) atomicMin(&s_best, cand);
                            }
                    }
            }
            __syncthreads();
        }
        // ---- 4. backtrack from the smallest (value, popcount, mask, node) at c = L - 1 ----
        const unsigned long long key = s_best;
        int32_t *cuts = o_cuts ? o_cuts + inst * (k - 1) : nullptr;
        int32_t *place = o_place + inst * k;
        if (bad || key == kNoBest) {
            if (tid < k) place[tid] = -1;
            if (cuts && tid < k - 1) cuts[tid] = -1;
            if (tid == 0) {
                o_beta[inst] = kInf;
                o_m[inst] = 0;
                o_status[inst] = bad ? (int8_t)PP_ERR_LIMIT : PP_BROKEN(chk) ? (int8_t)PP_ERR_CUDA : (int8_t)PP_INFEASIBLE;
            }
            continue;
        }
        const uint32_t rstar = (uint32_t)(key >> 30);
        const int m = (int)((key >> 25) & 31);
        uint32_t S = (uint32_t)((key >> 5) & 0xFFFFF);
        int w = (int)(key & 31), c2 = L - 1, status = (int)PP_OK;
        if (wid > 0) continue;
        // One warp: a step is a handful of candidates, and a barrier costs more than they do.  Lanes over the
        // positions, every lane walks the nodes in ascending order: the smallest (position, node) within the
        // threshold wins.
        int my_cut = -1, my_node = -1;  // lane j: cut and node of segment j
        for (int j = m - 1; j >= 0; --j) {
            if (lane == j) {
                my_node = w;
                if (j < m - 1) my_cut = c2;
            }
            if (j == 0) break;
            const uint32_t from = S & ~(1u << w);
            unsigned int pick = FULL;
            for (int c0 = lo[w * Ls + c2]; c0 < c2 && pick == FULL; c0 += 32) {
                const int c = min(c0 + lane, c2 - 1);
                const uint16_t *row = dp + (size_t)rowoff[from] * Ls + c, *rw = rank + (size_t)w * Ls + c;
                for (uint32_t rem = from; rem; rem &= rem - 1, row += Ls) {
                    const int v = __ffs(rem) - 1;
                    if (PP_IN_BOUNDS(chk, row - dp, n_dp) && PP_IN_BOUNDS(chk, rw - rank + v * k * Ls, n_rank) &&
                        max((uint32_t)*row, (uint32_t)rw[v * k * Ls]) <= rstar) pick = min(pick, ((unsigned)c << 5) | (unsigned)v);
                }
                pick = __reduce_min_sync(FULL, pick);
            }
            if (pick == FULL) {  // inconsistent table: flag the instance, keep going
                status = (int)PP_ERR_CUDA;
                break;
            }
            S = from;
            w = (int)(pick & 31u);
            c2 = (int)(pick >> 5);
        }
        if (PP_BROKEN(chk)) status = (int)PP_ERR_CUDA;
        // beta* is the bottleneck of the plan: no link of it ranks above the optimum, and no plan is better
        const int next = __shfl_down_sync(FULL, my_node, 1);
        double x = 0.0;
        if (status == (int)PP_OK && lane < m - 1) x = __ddiv_rn((double)s_bits[my_cut], (double)s_bw[my_node * k + next]);
        unsigned long long worst = (unsigned long long)__double_as_longlong(x);  // order like the values
#pragma unroll
        for (int o = 8; o; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(FULL, worst, o);
            worst = other > worst ? other : worst;
        }
        if (lane < k) place[lane] = my_node;
        if (cuts && lane < k - 1) cuts[lane] = my_cut;
        if (lane == 0) {
            o_beta[inst] = __longlong_as_double((long long)worst);
            o_m[inst] = m;
            o_status[inst] = (int8_t)status;
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");  // no launch is complete before the one in front of it
}

template <int NT, int G, int P>
cudaError_t launch_shape(int64_t B, int L, int k, const LaneTables &lt, int sms, const uint64_t *bits, const uint64_t *mem,
                         const uint64_t *cap, const uint32_t *bw, double *beta, int32_t *m, int32_t *cuts,
                         int32_t *placement, int8_t *status, bool early, cudaStream_t s)
{
    const size_t sm = batch_layout(L, k, NT).total;
    cudaError_t e = allow_shared(k_batch<NT, G, P>, 1024);
    if (e != cudaSuccess) return e;
    // a block per instance while they fit a few rounds of the GPU; beyond that blocks take several in turn
    const int64_t grid = std::min<int64_t>(B, (int64_t)sms * 16);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_batch<NT, G, P>, B, L, k, lt.rowoff, lt.rows, lt.first, bits, mem, cap, bw, beta, m, cuts,
                              placement, status);
}

}  // namespace

cudaError_t launch_batch(int64_t B, bool narrow, int L, int k, const LaneTables &lt, int sms, const uint64_t *bits, const uint64_t *mem,
                         const uint64_t *cap, const uint32_t *bw, double *beta, int32_t *m, int32_t *cuts,
                         int32_t *placement, int8_t *status, bool early, cudaStream_t s)
{
    if (B <= 0) return cudaSuccess;
    const BatchShape sh = batch_shape(L);
    switch (sh.G * 100 + sh.P) {
#define PP_LAUNCH(nt, g, p) launch_shape<nt, g, p>(B, L, k, lt, sms, bits, mem, cap, bw, beta, m, cuts, placement, status, early, s)
#define PP_CASE(g, p) \
    case g * 100 + p: return narrow ? PP_LAUNCH(kNarrowThreads, g, p) : PP_LAUNCH(kWideThreads, g, p);
        PP_CASE(4, 4) PP_CASE(8, 4) PP_CASE(16, 4) PP_CASE(32, 4) PP_CASE(32, 8)
#undef PP_CASE
        case 3216: return PP_LAUNCH(kWideThreads, 32, 16);
        case 3232: return PP_LAUNCH(kWideThreads, 32, 32);
#undef PP_LAUNCH
    }
    return cudaErrorInvalidValue;
}

}  // namespace pp
