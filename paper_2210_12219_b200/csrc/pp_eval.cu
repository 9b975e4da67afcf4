// Batched beta evaluator: one thread per candidate plan.
// gamma_j = bits[e_j] / bw[n_j][n_{j+1}] (Eq. 3), beta = max_j gamma_j (Eq. 2); validity
// rules as documented in pp.h.
//
// A plan is a loop over its cuts of integer instructions; with staging, sorting and the division it takes 113 warp
// instructions a cut (262 144 plans of k = 18: 7.9 million, 8.0 us at the busiest scheduler, which issues in 82 % of its
// cycles), so the kernel is bound by instruction issue first.  What can be saved there is lanes that wait for the longest
// plan of their warp.  A block therefore takes its 256 plans in the order of their number of segments (a
// counting sort in shared memory): with 1 to 18 segments the lanes of a warp then differ by one or two.
// The rows of the block come into shared memory as a whole first, so that the loop waits for no global
// load.  The largest quotient is kept as a fraction: bit counts are below 2^40 and bandwidths below 2^24,
// so two fractions compare exactly by cross multiplication in 64 bits, and since rounding is monotone the
// one division at the end gives the largest of the rounded quotients.  Whether a segment fits its node
// is one look into the table of forward windows.  One pass over a row collects all
// flags; an index that is out of range reads a padding entry and has raised its flag already.
// 262 144 compressed plans of k = 18, L = 200, a queued call: 21.7 us with a thread to a plan as they come, a
// division a cut and the row read along the way, 11.9 so, 11.4 with the tables fetched while the launch in
// front runs out.  256 threads, five blocks per SM: 128 or 512 threads, four, six or seven blocks 12.0 to 13.8.
#include "pp_internal.cuh"

namespace pp {

PP_CHECKS_OF(eval)

namespace {

constexpr int kEvalThreads = 256;

struct EvalLayout {
    size_t ends, nodes, total;
};
__host__ __device__ inline EvalLayout eval_layout(int L, int k)
{
    EvalLayout l;
    l.ends = plan_tables(L, k).total;
    l.nodes = l.ends + (((size_t)kEvalThreads * k * 2 + 16 + 15) & ~(size_t)15);  // rows of the block's plans
    l.total = l.nodes + (((size_t)kEvalThreads * k + 16 + 15) & ~(size_t)15);
    return l;
}

// x * y for x below 2^40, y below 2^24
__device__ __forceinline__ unsigned long long times(unsigned long long x, uint32_t y)
{
    return (unsigned long long)(uint32_t)x * y + ((unsigned long long)((uint32_t)(x >> 32) * y) << 32);
}

// PACKED: plan b owns the entries [off[b], off[b + 1]) of 16-bit `ends` and 8-bit `nodes`; a block's plans
// own one stretch of them when the offsets ascend, else a plan's row is read where it is.  Otherwise rows
// of k 32-bit entries, of which the part that a plan uses is staged in the compressed types (a value
// they cannot hold becomes the largest code, which is out of range as well).
template <bool PACKED, typename E, typename N>
__global__ void __launch_bounds__(kEvalThreads, 5)
k_eval(const int L, const int k, const unsigned char *__restrict__ tables, const int64_t B, const int64_t total, const uint8_t *__restrict__ nseg, const uint32_t *__restrict__ off,
       const E *__restrict__ ends, const N *__restrict__ nodes, double *__restrict__ beta, uint8_t *__restrict__ status)
{
    extern __shared__ __align__(16) unsigned char smem_eval[];
    const int k1 = k + 1, tid = threadIdx.x;
    const EvalLayout lay = eval_layout(L, k);
    const PlanTables tab = plan_tables(L, k);
    const unsigned long long *s_bits = reinterpret_cast<const unsigned long long *>(smem_eval + tab.bits);
    const uint32_t *s_bw = reinterpret_cast<const uint32_t *>(smem_eval + tab.bw);
    const uint16_t *s_fwd = reinterpret_cast<const uint16_t *>(smem_eval + tab.fwd);
    uint16_t *s_ends = reinterpret_cast<uint16_t *>(smem_eval + lay.ends);
    uint8_t *s_nodes = smem_eval + lay.nodes;
    PP_BLOCK_BOUNDS(chk);
    [[maybe_unused]] const size_t n_fwd = (size_t)k1 * L + 1, n_bw = (size_t)k1 * k1;  // entries of the tables
    __shared__ uint8_t s_order[kEvalThreads], s_m[kEvalThreads];
    __shared__ uint32_t s_start[kEvalThreads];  // PACKED: first entry of the row within the staged stretch, or kFar
    __shared__ uint32_t s_first[2][32];
    constexpr uint32_t kFar = 0xFFFFFFFFu;
    const int mmax = k < L ? k : L;
    const double kInf = __longlong_as_double(0x7FF0000000000000ll);
    // what a batch needs to know before its rows can be fetched; asked for one batch ahead
    struct Ahead {
        int m = 0;
        uint32_t from = 0, to = 0, o0 = 0, o1 = 0;
    } next;
    auto look_ahead = [&](int64_t base) {
        if (base >= B) return;
        const int rows = B - base < kEvalThreads ? (int)(B - base) : kEvalThreads;
        next.m = tid < rows ? nseg[base + tid] : 0;
        if constexpr (PACKED) {
            next.from = off[base];
            next.to = off[base + rows];
            if (tid < rows) {
                next.o0 = off[base + tid];
                next.o1 = off[base + tid + 1];
            }
        }
    };
    if (tid < 32) s_first[0][tid] = s_first[1][tid] = 0u;
    for (int i = tid; i < (int)(tab.total / 16); i += kEvalThreads)
        reinterpret_cast<uint4 *>(smem_eval)[i] = reinterpret_cast<const uint4 *>(tables)[i];
    // launched as a dependent of whatever writes the plans: only now is it complete (the tables are
    // older than that, see launch_eval)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    look_ahead((int64_t)blockIdx.x * kEvalThreads);
    int turn = 0;
    for (int64_t base = (int64_t)blockIdx.x * kEvalThreads; base < B; base += (int64_t)gridDim.x * kEvalThreads, turn ^= 1) {
        const int rows = B - base < kEvalThreads ? (int)(B - base) : kEvalThreads;
        // ---- number of segments of the plans; 0 = nothing of the row is read ----
        int m = next.m > mmax ? 0 : next.m;
        __syncthreads();  // the tables are there, the previous plans are done
        if (tid < 32) s_first[turn ^ 1][tid] = 0u;
        if constexpr (PACKED) {
            const uint32_t from = next.from, to = next.to, n = to - from, lead = from & 3u;
            const bool whole = from <= to && (int64_t)to <= total && n <= (uint32_t)(kEvalThreads * k);
            if (m) {
                if (next.o1 < next.o0 || (int64_t)next.o1 > total || next.o1 - next.o0 < (uint32_t)m) m = 0;  // does not hold nseg entries
                s_start[tid] = whole && next.o0 >= from && next.o1 <= to ? next.o0 - from + lead : kFar;
            }
            if (whole) {
                if ((reinterpret_cast<uintptr_t>(nodes) & 3u) == 0 && (reinterpret_cast<uintptr_t>(ends) & 7u) == 0) {
                    // words of four entries; the first and the last one may be cut
                    const uint32_t first = from - lead, words = (lead + n + 3) >> 2;
                    for (uint32_t i = tid; i < words; i += kEvalThreads) {
                        const uint32_t e0 = first + 4 * i;
                        if (e0 >= from && e0 + 4 <= to) {
                            reinterpret_cast<uint32_t *>(s_nodes)[i] = *reinterpret_cast<const uint32_t *>(nodes + e0);
                            reinterpret_cast<uint2 *>(s_ends)[i] = *reinterpret_cast<const uint2 *>(ends + e0);
                        } else {
                            for (uint32_t q = 0; q < 4; ++q)
                                if (e0 + q >= from && e0 + q < to) {
                                    s_nodes[4 * i + q] = nodes[e0 + q];
                                    s_ends[4 * i + q] = ends[e0 + q];
                                }
                        }
                    }
                } else {
                    for (uint32_t i = tid; i < n; i += kEvalThreads) {
                        s_nodes[lead + i] = nodes[from + i];
                        s_ends[lead + i] = ends[from + i];
                    }
                }
            }
        }
        s_m[tid] = (uint8_t)m;
        const uint32_t place = atomicAdd(&s_first[turn][m], 1u);
        look_ahead(base + (int64_t)gridDim.x * kEvalThreads);
        __syncthreads();
        if constexpr (!PACKED) {
            int r = tid / k, c = tid - r * k;
            const int dr = kEvalThreads / k, dc = kEvalThreads - dr * k;
#pragma unroll 4
            for (int i = tid; i < rows * k; i += kEvalThreads) {
                const int mr = s_m[r];
                if (c < mr) {
                    const uint32_t n = (uint32_t)nodes[base * k + i], e = c < mr - 1 ? (uint32_t)ends[base * k + i] : 0u;
                    s_nodes[i] = (uint8_t)min(n, 0xFFu);  // negative values are large ones here
                    s_ends[i] = (uint16_t)min(e, 0xFFFFu);
                }
                r += dr;
                c += dc;
                if (c >= k) { c -= k; ++r; }
            }
        }
        {  // counts -> first places, by every warp for its own plans
            const uint32_t n = s_first[turn][tid & 31];
            uint32_t x = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
                if ((tid & 31) >= o) x += y;
            }
            s_order[__shfl_sync(0xFFFFFFFFu, x - n, m) + place] = (uint8_t)tid;
        }
        __syncthreads();
        // ---- score ----
        const int mine = s_order[tid];
        if (mine >= rows) continue;
        const int64_t b = base + mine;
        m = s_m[mine];
        int flags = PP_PLAN_BAD_NSEG;
        double bt = kInf;
        auto score = [&](auto node_at, auto end_at) {
            uint32_t used = 1u << k, den = 1;  // the largest quotient so far: num / den
            unsigned long long num = 0;
            bool twice = false, late = false, full = false, dead = false;
            int first = 0, n = min(node_at(0), k);
            for (int j = 0; j < m - 1; ++j) {
                const int e = min(end_at(j), L - 1), next = min(node_at(j + 1), k);
                twice = twice || ((used >> n) & 1u);  // node n again, or no such node
                used |= 1u << n;
                late = late || (uint32_t)(e - first) >= (uint32_t)(L - 1 - first);
                if (!PP_IN_BOUNDS(chk, n * L + first, n_fwd) || !PP_IN_BOUNDS(chk, n * k1 + next, n_bw) || !PP_IN_BOUNDS(chk, e, L)) break;
                full = full || (uint32_t)(e - first) >= s_fwd[n * L + first];
                const uint32_t link = s_bw[n * k1 + next];
                dead = dead || link == 0u;
                const unsigned long long bits = s_bits[e];
                if (times(bits, den) > times(num, link)) {
                    num = bits;
                    den = link;
                }
                first = e + 1;
                n = next;
            }
            twice = twice || ((used >> n) & 1u);
            if (PP_IN_BOUNDS(chk, n * L + first, n_fwd)) full = full || (uint32_t)(L - 1 - first) >= s_fwd[n * L + first];
            flags = (twice ? PP_PLAN_BAD_NODE : 0) | (late ? PP_PLAN_BAD_ENDS : 0);
            if (!flags) flags = (full ? PP_PLAN_MEMORY : 0) | (dead ? PP_PLAN_DEAD_LINK : 0);
            if (!flags) bt = __ddiv_rn((double)num, (double)den);
        };
        if (m != 0) {
            const uint32_t at = PACKED ? s_start[mine] : (uint32_t)(mine * k);
            if (!PACKED || at != kFar) {
                score([&](int j) { return (int)s_nodes[at + j]; }, [&](int j) { return (int)s_ends[at + j]; });
            } else if constexpr (PACKED) {
                const uint32_t far = off[b];
                score([&](int j) { return (int)nodes[(size_t)far + j]; }, [&](int j) { return (int)ends[(size_t)far + j]; });
            }
        }
        if (PP_BROKEN(chk)) flags = 255;
        beta[b] = bt;
        status[b] = (uint8_t)flags;
    }
}

template <bool PACKED, typename E, typename N>
cudaError_t launch(const Dev &d, const unsigned char *tables, int64_t B, int64_t total, const uint8_t *nseg, const uint32_t *off, const E *ends,
                   const N *nodes, double *beta, uint8_t *status, bool early, cudaStream_t s)
{
    if (B <= 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_eval<PACKED, E, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, 80 * 1024);
    if (e != cudaSuccess) return e;  // 68 KB at k = 20, L = 1024
    int64_t blocks = (B + kEvalThreads - 1) / kEvalThreads;
    const int64_t cap = 148 * 12;  // five of them fit an SM at a time; a block's tables are staged once for all its plans
    if (blocks > cap) blocks = cap;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kEvalThreads);
    cfg.dynamicSmemBytes = eval_layout(d.L, d.k).total;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_eval<PACKED, E, N>, d.L, d.k, tables, B, total, nseg, off, ends, nodes, beta, status);
}

}  // namespace

cudaError_t launch_eval_packed(const Dev &d, const unsigned char *tables, int64_t B, int64_t total, const uint8_t *nseg, const uint32_t *off,
                               const uint16_t *ends, const uint8_t *nodes, double *beta, uint8_t *status,
                               bool early, cudaStream_t s)
{
    return launch<true>(d, tables, B, total, nseg, off, ends, nodes, beta, status, early, s);
}

cudaError_t launch_eval(const Dev &d, const unsigned char *tables, int64_t B, const uint8_t *nseg, const int32_t *ends,
                        const int32_t *nodes, double *beta, uint8_t *status, bool early, cudaStream_t s)
{
    return launch<false>(d, tables, B, 0, nseg, static_cast<const uint32_t *>(nullptr), ends, nodes, beta, status, early, s);
}

}  // namespace pp
