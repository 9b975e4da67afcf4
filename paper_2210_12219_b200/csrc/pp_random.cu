// Random comparison baseline of Section 4 (the "random algorithm" of the paper's comparison list),
// many plans per launch for one problem: one thread per plan.  Step s of a plan takes a random
// node among the nodes not used yet (draw 2 s) and a random segment among those that start at
// the next unassigned layer and fit the node's memory (draw 2 s + 1), until the chain is used up.
// The 32-bit draws are inputs; draw d picks index floor(d * n / 2^32) among n candidates in
// ascending order.  Bandwidths play no part: the plans go to the evaluator afterwards.  No plan
// (nseg = 0, rows of -1) when the chosen node holds not even the next layer, or when all k
// nodes are used and layers are left over.
//
// A plan is a chain of dependent steps, so with the tens of thousands of plans of a call the kernel is
// bound by the latency of a step and by getting the rows in and out.  How many layers from a given one
// on fit a node is looked up (a table of k * L counts, made once per problem) instead of
// bisected over the prefix sums, and the r-th free node is found by counting bits in halves: a step is
// some forty instructions for every lane alike (a bisection and a walk over the free nodes before:
// 100 003 plans of k = 14, L = 50 in 14.4 us).
#include "pp_blocks.cuh"

namespace pp {

PP_CHECKS_OF(random)

constexpr int kRandomThreads = 128;

// Rows travel through shared memory so that global memory sees whole contiguous blocks: the draws
// of the block's plans on the way in, their two output rows on the way out, a pair of words at a time.  A
// thread's outputs overwrite its own draws: step s has read pair s before segment n <= s + 1 goes to pair
// n - 1 as (cut, node).  The row stride is an odd number of pairs, which keeps the threads of a warp, each
// on its own row, on different banks.
__global__ void __launch_bounds__(kRandomThreads)
k_random_plans(const int L, const int k, const uint16_t *__restrict__ fwd, const int64_t P, const uint32_t *__restrict__ draws,
               uint8_t *nseg, int32_t *ends, int32_t *nodes)
{
    extern __shared__ uint2 smem_pairs[];
    const int stride = k | 1, tid = threadIdx.x;
    uint2 *sd = smem_pairs;  // [threads][stride]: draws in, (cut, node) pairs out
    uint16_t *s_fwd = reinterpret_cast<uint16_t *>(smem_pairs + kRandomThreads * stride);  // [k][L]
    PP_BLOCK_BOUNDS(chk);
    for (int i = tid; i < k * L; i += kRandomThreads) s_fwd[i] = fwd[i];
    // whatever wrote the draws, or reads or writes the plans, is complete (fwd is older, see launch_eval)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const int64_t p0 = (int64_t)blockIdx.x * kRandomThreads;
    const int np = P - p0 < kRandomThreads ? (int)(P - p0) : kRandomThreads;
    const int r0 = tid / k, c0 = tid - r0 * k, dr = kRandomThreads / k, dc = kRandomThreads - dr * k;
    const uint32_t *src = draws + p0 * 2 * k;
    const bool pairs = (reinterpret_cast<uintptr_t>(draws) & 7u) == 0;
    {
        int at = r0 * stride + c0, c = c0;
        const int step = dr * stride + dc, carry = stride - k;
#pragma unroll 4
        for (int i = tid; i < np * k; i += kRandomThreads) {
            sd[at] = pairs ? reinterpret_cast<const uint2 *>(src)[i] : make_uint2(src[2 * i], src[2 * i + 1]);
            at += step;
            c += dc;
            if (c >= k) { c -= k; at += carry; }
        }
    }
    __syncthreads();
    if (tid < np) {
        uint2 *row = sd + tid * stride;
        uint32_t free_nodes = (1u << k) - 1u;
        int first = 0, n = 0;
        bool done = false;
        for (int step = 0; step < k; ++step) {
            const uint2 draw = row[step];
            const int node = select_bit(free_nodes, (int)__umulhi(draw.x, (unsigned)(k - step)));
            if (!PP_IN_BOUNDS(chk, node * L + first, k * L)) break;
            const uint32_t count = s_fwd[node * L + first];  // segments [first, e] that fit
            if (count == 0) break;
            const int last = first + (int)__umulhi(draw.y, count);
            free_nodes &= ~(1u << node);
            done = last == L - 1;
            row[n] = make_uint2(done ? 0xFFFFFFFFu : (uint32_t)last, (uint32_t)node);  // the last segment has no cut
            ++n;
            if (done) break;
            first = last + 1;
        }
        if (!done) n = 0;
        nseg[p0 + tid] = PP_BROKEN(chk) ? (uint8_t)255 : (uint8_t)n;
        for (int i = n; i < k; ++i) row[i] = make_uint2(0xFFFFFFFFu, 0xFFFFFFFFu);
    }
    __syncthreads();
    {
        int32_t *de = ends + p0 * k, *dn = nodes + p0 * k;
        int at = r0 * stride + c0, c = c0;
        const int step = dr * stride + dc, carry = stride - k;
#pragma unroll 4
        for (int i = tid; i < np * k; i += kRandomThreads) {
            const uint2 x = sd[at];
            de[i] = (int32_t)x.x;
            dn[i] = (int32_t)x.y;
            at += step;
            c += dc;
            if (c >= k) { c -= k; at += carry; }
        }
    }
}

cudaError_t launch_random_plans(const Dev &d, const unsigned char *tables, int64_t P, const uint32_t *draws, uint8_t *nseg,
                                int32_t *ends, int32_t *nodes, bool early, cudaStream_t s)
{
    const int64_t blocks = (P + kRandomThreads - 1) / kRandomThreads;
    if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
    const size_t smem = (size_t)kRandomThreads * (d.k | 1) * sizeof(uint2) + (size_t)d.k * d.L * sizeof(uint16_t);
    cudaError_t e = cudaFuncSetAttribute(k_random_plans, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
    if (e != cudaSuccess) return e;  // at most 62 KB (k = 20, L = 1024)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kRandomThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_random_plans, d.L, d.k, reinterpret_cast<const uint16_t *>(tables + plan_tables(d.L, d.k).fwd), P, draws, nseg, ends, nodes);
}

}  // namespace pp
