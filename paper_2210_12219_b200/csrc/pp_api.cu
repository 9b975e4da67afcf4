// C-ABI of libpp (see include/pp.h) and the host orchestration behind it: validation,
// memory prefix sums, window table, mask lists, launch sequence, result download.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <limits>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <vector>

#include "pp_internal.cuh"

using namespace pp;

struct pp_problem {
    int L = 0, k = 0;
    std::vector<uint64_t> bits, mem, cap, M;
    std::vector<uint32_t> bw;
    std::vector<int16_t> lo;
    std::vector<uint16_t> fwd;
    unsigned char *d_inputs = nullptr;  // one allocation: see bind_inputs
    unsigned char *d_spare = nullptr;   // the one of pp_problem_create where the inputs are elsewhere: see upload_inputs
    unsigned char *mallocs[4] = {};     // of the kept buffers those that are not of the pool
    int n_mallocs = 0;
    size_t inputs_bytes = 0;
    bool uploaded = false;              // the inputs have been copied (queued on `stream`)
    bool tables_ready = false;          // a launch may read them before the work in front of it on `stream` is done:
                                        // the copy is complete, or another launch is ordered behind it
    unsigned char *d_sparse = nullptr;  // scratch of the bounded search when there is no workspace
    unsigned char *d_work = nullptr;    // workspace (own or caller's): either search runs in it
    uint64_t work_bytes = 0;
    bool own_work = false;
    int sms = 0;                        // multiprocessors of the device the problem lives on
    cudaStream_t stream = nullptr;
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};  // of the dense search, created by its first run
    pp_solution *d_sol = nullptr;
    PruneNote *d_note = nullptr;
    unsigned char *d_tables = nullptr;  // PlanTables, in d_inputs
    PruneDev prune{};
    bool solved = false, profiled = false;
    bool sparse_ran = false;            // the last solve ran the bounded search
    bool table_whole = false;           // ... the dense one: its table holds every state
    PruneNote note{};                   // of the last synchronous bounded search
    bool note_on_device = false;
    int force_generic = -1;
    bool profiling = false;             // record events between the phases of a solve

    // what only the dense search needs, prepared by its first run
    bool dense_dims = false, dense_ready = false;
    int Lpad = 0, U = 0, elem = 2;
    std::vector<uint32_t> ubw;
    std::vector<int16_t> pair_u;
    unsigned char *d_dense = nullptr;
    Dev d{};
    int sweep_launches = 0, total_launches = 0, fast_used = 0, pair_levels = 0;
    std::vector<signed char> pair_lvl;  // per level: 1 = two-mask kernel, 0 = one-mask, -1 = not decided yet
};

namespace {

// Mask lists depend on k only: built once per k and process, then copied.  Level j (popcount j)
// lists its masks in revolving-door order: A(n, j) = A(n-1, j), then the masks of A(n-1, j-1) in
// reverse, each with node n-1 added.  Neighbours in that list differ by one node swapped for
// another, which is what the two-mask sweep kernel pairs up.
struct MaskList {
    std::vector<uint32_t> masks, level_off;
    bool swaps = true;  // every two neighbours of a level differ by exactly one swap (checked)
};
void revolving_door(int n, int j, uint32_t add, bool reversed, std::vector<uint32_t> &out)
{
    if (j == 0) { out.push_back(add); return; }
    if (j == n) { out.push_back(add | ((1u << n) - 1u)); return; }
    if (!reversed) {
        revolving_door(n - 1, j, add, false, out);
        revolving_door(n - 1, j - 1, add | (1u << (n - 1)), true, out);
    } else {
        revolving_door(n - 1, j - 1, add | (1u << (n - 1)), false, out);
        revolving_door(n - 1, j, add, true, out);
    }
}
const MaskList &mask_list(int k)
{
    static std::mutex mu;
    static std::map<int, MaskList> cache;
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(k);
    if (it != cache.end()) return it->second;
    MaskList ml;
    const uint32_t nm = 1u << k;
    ml.level_off.assign(k + 2, 0);
    ml.masks.reserve(nm - 1);
    for (int j = 1; j <= k; ++j) {
        ml.level_off[j] = (uint32_t)ml.masks.size();
        revolving_door(k, j, 0u, false, ml.masks);
        for (size_t i = ml.level_off[j] + 1; i < ml.masks.size(); ++i)
            if (__builtin_popcount(ml.masks[i] ^ ml.masks[i - 1]) != 2) ml.swaps = false;
    }
    ml.level_off[k + 1] = (uint32_t)ml.masks.size();
    ml.level_off[0] = 0;
    return cache.emplace(k, std::move(ml)).first->second;
}

// Test hook (pp_debug_fail_alloc): the n-th device allocation from now on reports out of memory
// without asking the driver, so that the out-of-memory paths can be exercised on a healthy device.
std::atomic<int> g_fail_alloc_countdown{0};
bool alloc_should_fail()
{
    int c = g_fail_alloc_countdown.load();
    while (c > 0 && !g_fail_alloc_countdown.compare_exchange_weak(c, c - 1)) {}
    return c == 1;
}

// Test hook (pp_debug_starve).
std::atomic<int> g_starved_polls{0};
// Test hook (pp_debug_late): block << 32 | polls.
std::atomic<uint64_t> g_late{0};

// Whether the stream is being recorded into a graph (the legacy stream cannot be).
bool recording(cudaStream_t s)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    return s && cudaStreamIsCapturing(s, &st) == cudaSuccess && st != cudaStreamCaptureStatusNone;
}

// What a handle or the process keeps must not become part of a graph that happens to be recorded when it is first
// needed: such memory comes from cudaMalloc and is filled through copy_stream(), which this thread may use meanwhile.
struct OutsideCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    OutsideCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~OutsideCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// A stream of the library's own for copies to memory that no stream owns, one per device, kept.
cudaError_t copy_stream(cudaStream_t *out)
{
    static std::mutex mu;
    static cudaStream_t streams[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    *out = nullptr;
    if (e != cudaSuccess || dev < 0 || dev >= 64) return e;
    std::lock_guard<std::mutex> lock(mu);
    if (!streams[dev]) e = cudaStreamCreateWithFlags(&streams[dev], cudaStreamNonBlocking);
    *out = streams[dev];
    return e;
}

// A copy from pageable memory that is complete when the call returns.  cudaMemcpy may return while the last
// bytes are still under way, which a stream that does not wait for the legacy stream would not notice.
// via: the legacy stream for memory of the pool, copy_stream() for memory of cudaMalloc.
cudaError_t copy_in(void *dst, const void *src, size_t n, cudaStream_t via)
{
    const cudaError_t e = cudaMemcpyAsync(dst, src, n, cudaMemcpyHostToDevice, via);
    const cudaError_t e2 = cudaStreamSynchronize(via);
    return e != cudaSuccess ? e : e2;
}

// Device copy of a mask list, uploaded once per (device, k) and kept for the life of the process:
// masks [2^k - 1] followed (256-byte aligned) by level_off [k + 2].
struct DeviceMasks {
    uint32_t *masks = nullptr, *level_off = nullptr;
};
cudaError_t device_masks(int k, const MaskList &ml, DeviceMasks *out)
{
    static std::mutex mu;
    static std::map<std::pair<int, int>, DeviceMasks> cache;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find({dev, k});
    if (it == cache.end()) {
        const size_t mb = (ml.masks.size() * 4 + 255) / 256 * 256, lb = ml.level_off.size() * 4;
        unsigned char *buf = nullptr;
        OutsideCapture outside;
        cudaStream_t via = nullptr;
        e = copy_stream(&via);
        if (e != cudaSuccess) return e;
        e = alloc_should_fail() ? cudaErrorMemoryAllocation : cudaMalloc(reinterpret_cast<void **>(&buf), mb + lb);
        if (e != cudaSuccess) return e;
        e = copy_in(buf, ml.masks.data(), ml.masks.size() * 4, via);
        if (e == cudaSuccess) e = copy_in(buf + mb, ml.level_off.data(), lb, via);
        if (e != cudaSuccess) {
            cudaFree(buf);
            return e;
        }
        DeviceMasks dm;
        dm.masks = reinterpret_cast<uint32_t *>(buf);
        dm.level_off = reinterpret_cast<uint32_t *>(buf + mb);
        it = cache.emplace(std::make_pair(dev, k), dm).first;
    }
    *out = it->second;
    return cudaSuccess;
}

// The tables of LaneTables are made by the first batch of that k on a device and kept.
cudaError_t lane_tables(int k, LaneTables *out)
{
    static std::mutex mu;
    static std::map<std::pair<int, int>, LaneTables> cache;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find({dev, k});
    if (it == cache.end()) {
        const uint32_t nm = 1u << k;
        const size_t n_rows = (size_t)k << (k - 1);
        std::vector<uint32_t> host(2 * (size_t)nm + 2 * ((size_t)k + 2) + n_rows);
        uint32_t *rowoff = host.data(), *mlist = rowoff + nm, *moff = mlist + nm, *first = moff + k + 2, *row = first + k + 2;
        uint32_t rows = 0, masks = 0;
        for (int pc = 0; pc <= k; ++pc) {
            moff[pc] = masks;
            first[pc] = rows;
            for (uint32_t S = 0; S < nm; ++S)
                if (__builtin_popcount(S) == pc) {
                    rowoff[S] = rows;
                    mlist[masks++] = S;
                    for (uint32_t rem = S; rem; rem &= rem - 1) {
                        const uint32_t w = (uint32_t)__builtin_ctz(rem);
                        row[rows++] = (S & ~(1u << w)) | (w << 16);
                    }
                }
        }
        moff[k + 1] = masks;
        first[k + 1] = rows;
        uint32_t *buf = nullptr;
        OutsideCapture outside;
        cudaStream_t via = nullptr;
        e = copy_stream(&via);
        if (e != cudaSuccess) return e;
        e = alloc_should_fail() ? cudaErrorMemoryAllocation
                                : cudaMalloc(reinterpret_cast<void **>(&buf), host.size() * 4);
        if (e != cudaSuccess) return e;
        e = copy_in(buf, host.data(), host.size() * 4, via);
        if (e != cudaSuccess) {
            cudaFree(buf);
            return e;
        }
        LaneTables lt;
        lt.rowoff = buf;
        lt.mlist = buf + nm;
        lt.moff = buf + 2 * (size_t)nm;
        lt.first = lt.moff + k + 2;
        lt.rows = lt.first + k + 2;
        it = cache.emplace(std::make_pair(dev, k), lt).first;
    }
    *out = it->second;
    return cudaSuccess;
}

// Staging buffers and small scratch come from a pool of the library's own that keeps up to
// kPoolKeepBytes between calls (the default pool would hand everything back at every
// synchronisation); what is free beyond that goes back to the device at the next one.
constexpr unsigned long long kPoolKeepBytes = 1ull << 30;
cudaError_t staging_alloc(void **ptr, size_t bytes, cudaStream_t s)
{
    static std::mutex mu;
    static cudaMemPool_t pools[64] = {};
    if (alloc_should_fail()) return cudaErrorMemoryAllocation;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaMalloc(ptr, bytes);
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!pools[dev]) {
            cudaMemPoolProps props = {};
            props.allocType = cudaMemAllocationTypePinned;
            props.handleTypes = cudaMemHandleTypeNone;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            e = cudaMemPoolCreate(&pools[dev], &props);
            if (e != cudaSuccess) return e;
            unsigned long long keep = kPoolKeepBytes;
            e = cudaMemPoolSetAttribute(pools[dev], cudaMemPoolAttrReleaseThreshold, &keep);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaMallocFromPoolAsync(ptr, bytes, pools[dev], s);
}

pp_status from_cuda(cudaError_t e)
{
    if (e == cudaSuccess) return PP_OK;
    cudaGetLastError();  // clear the sticky-less error state
    return e == cudaErrorMemoryAllocation ? PP_ERR_NOMEM : PP_ERR_CUDA;
}

#define PP_CUDA(call)                                   \
    do {                                                \
        cudaError_t e__ = (call);                       \
        if (e__ != cudaSuccess) return from_cuda(e__);  \
    } while (0)

// Multiprocessors of a device, asked for once.
cudaError_t multiprocessors(int dev, int *sms)
{
    static std::atomic<int> known[64];
    if (dev >= 0 && dev < 64 && (*sms = known[dev].load(std::memory_order_relaxed)) > 0) return cudaSuccess;
    const cudaError_t e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && dev >= 0 && dev < 64) known[dev].store(*sms, std::memory_order_relaxed);
    return e;
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

struct WorkLayout {
    size_t pos, order, gu, cnt, rk, inv, rank, table, total;
};

WorkLayout work_layout(int L, int k, int Lpad, int U, int elem)
{
    WorkLayout w;
    size_t o = 0;
    w.pos = o;   o = align_up(o + (size_t)L * 2, 256);
    w.order = o; o = align_up(o + (size_t)L * 2, 256);
    w.gu = o;    o = align_up(o + (size_t)std::max(U, 1) * L * 8, 256);
    w.cnt = o;   o = align_up(o + (size_t)std::max(U, 1) * L * 4, 256);
    w.rk = o;    o = align_up(o + (size_t)std::max(U, 1) * L * 4, 256);
    w.inv = o;   o = align_up(o + ((size_t)std::max(U, 1) * L + 2) * 4, 256);
    w.rank = o;  o = align_up(o + (size_t)k * k * Lpad * elem, 256);
    w.table = o; o = align_up(o + ((size_t)k << k) * Lpad * elem, 256);
    w.total = o;
    return w;
}

pp_status validate(int32_t L, const uint64_t *bits, const uint64_t *mem, int32_t k,
                   const uint64_t *cap, const uint32_t *bw)
{
    if (!bits || !mem || !cap || !bw) return PP_ERR_ARG;
    if (L < 1 || k < 1) return PP_ERR_ARG;
    if (L > PP_MAX_L || k > PP_MAX_K) return PP_ERR_LIMIT;
    for (int i = 0; i < L; ++i)
        if (bits[i] >= PP_MAX_BITS) return PP_ERR_LIMIT;
    for (int i = 0; i < k * k; ++i)
        if (bw[i] >= PP_MAX_KBPS) return PP_ERR_LIMIT;
    uint64_t acc = 0;
    for (int i = 0; i < L; ++i) {
        if (mem[i] > std::numeric_limits<uint64_t>::max() - acc) return PP_ERR_LIMIT;
        acc += mem[i];
    }
    return PP_OK;
}

// ---- the bounded search (pp_prune.cu) ----------------------------------------------------------

// Rows of the dense programme: (node set, last node) over all sets of two nodes and more.
unsigned long long rows_all(int k) { return ((unsigned long long)k << (k - 1)); }

// A synchronous solve gives the bounded search up after this many rows and lets the dense sweep do the
// rest, which moves more rows per microsecond once the frontier is not sparse.  Up to k = 14 it is never
// reached.  An asynchronous solve cannot look at the outcome: it has room for every row.
constexpr unsigned long long kSparseRows = 160000;
// Without a workspace of the caller the rows live in pooled scratch of at most this size.
constexpr unsigned long long kSparseScratchBytes = 128ull << 20;

size_t sparse_bytes(int k, int Lp, unsigned long long limit)
{
    const unsigned long long rows = std::min(rows_all(k), limit / ((unsigned long long)Lp * 4));
    return sparse_layout(k, Lp).rows + (size_t)rows * Lp * 4;
}

void bind_sparse(PruneDev &q, unsigned char *b, uint64_t bytes)
{
    const SparseLayout w = sparse_layout(q.k, q.Lp);
    q.live = reinterpret_cast<uint32_t *>(b + w.live);
    q.rowmap = reinterpret_cast<unsigned long long *>(b + w.rowmap);
    q.list = reinterpret_cast<uint32_t *>(b + w.list);
    q.gam = reinterpret_cast<uint32_t *>(b + w.gam);
    q.gmin = reinterpret_cast<uint32_t *>(b + w.gmin);
    q.rows = reinterpret_cast<uint32_t *>(b + w.rows);
    q.row_cap = (bytes - w.rows) / ((size_t)q.Lp * 4);
}

// lo[w][c'] = earliest previous cut c >= 0 such that layers c+1..c' fit on w; c' itself when not even
// layer c' alone fits.  fwd[w][c] = layers from c on that fit w.
void window_table(int L, int k, const uint64_t *M, const uint64_t *cap, int16_t *lo, uint16_t *fwd)
{
    for (int w = 0; w < k; ++w, lo += L, fwd += L) {
        int a = 0;  // first layer such that layers a .. c2 fit
        for (int c2 = 0; c2 < L; ++c2) {
            for (; a <= c2 && M[c2 + 1] - M[a] > cap[w]; ++a) fwd[a] = (uint16_t)(c2 - a);
            lo[c2] = (int16_t)std::max(a - 1, 0);
        }
        for (; a < L; ++a) fwd[a] = (uint16_t)(L - a);
    }
}

// Range of the keys: the smallest and the largest positive quotient of Eq. 3 the inputs allow.
void quotient_range(int L, const uint64_t *num, int n, const uint32_t *den, double *lo, double *hi)
{
    uint64_t a = ~0ull, b = 0;
    uint32_t c = ~0u, e = 0;
    for (int i = 0; i < L; ++i) {
        if (num[i]) a = std::min(a, num[i]);
        b = std::max(b, num[i]);
    }
    for (int i = 0; i < n; ++i) {
        if (den[i]) c = std::min(c, den[i]);
        e = std::max(e, den[i]);
    }
    if (!b || !e) return;  // no positive quotient
    *lo = std::min(*lo, (double)a / (double)e);
    *hi = std::max(*hi, (double)b / (double)c);
}

// Device memory that the handle keeps: of the pool, ordered on its stream, else of cudaMalloc.
cudaError_t kept_alloc(pp_problem *p, unsigned char **out, size_t bytes, bool rec)
{
    if (!rec) return staging_alloc(reinterpret_cast<void **>(out), bytes, p->stream);
    if (alloc_should_fail()) return cudaErrorMemoryAllocation;
    OutsideCapture outside;
    const cudaError_t e = cudaMalloc(reinterpret_cast<void **>(out), bytes);
    if (e == cudaSuccess) p->mallocs[p->n_mallocs++] = *out;
    return e;
}

// The parts of the buffer of the inputs: the inputs, the counters of the searches, a result record, the tables of the
// scoring calls.
size_t bind_inputs(pp_problem *p, unsigned char *b)
{
    const int L = p->L, k = p->k;
    const size_t bytes[10] = {(size_t)L * 8, (size_t)(L + 1) * 8, (size_t)k * 8, (size_t)k * k * 4, (size_t)k * L * 2,
                              sizeof(PruneCtl), 8 /* best */, 4 /* err */, sizeof(pp_solution) + sizeof(PruneNote),
                              plan_tables(L, k).total};
    size_t off[10], total = 0;
    for (int i = 0; i < 10; ++i) { off[i] = total; total = align_up(total + bytes[i], i < 4 ? 16 : 128); }
    if (!b) return total;
    p->d_inputs = b;
    Dev &d = p->d;
    d.bits = reinterpret_cast<uint64_t *>(b + off[0]);
    d.M = reinterpret_cast<uint64_t *>(b + off[1]);
    d.cap = reinterpret_cast<uint64_t *>(b + off[2]);
    d.bw = reinterpret_cast<uint32_t *>(b + off[3]);
    d.lo = reinterpret_cast<int16_t *>(b + off[4]);
    p->prune.ctl = reinterpret_cast<PruneCtl *>(b + off[5]);
    d.best = reinterpret_cast<unsigned long long *>(b + off[6]);
    d.err = reinterpret_cast<int32_t *>(b + off[7]);
    p->d_sol = reinterpret_cast<pp_solution *>(b + off[8]);
    p->d_note = reinterpret_cast<PruneNote *>(b + off[8] + sizeof(pp_solution));
    p->d_tables = b + off[9];
    return total;
}

void ensure_windows(pp_problem *p)
{
    if (!p->lo.empty()) return;
    std::vector<int16_t> lo((size_t)p->k * p->L);
    std::vector<uint16_t> fwd((size_t)p->k * p->L);
    window_table(p->L, p->k, p->M.data(), p->cap.data(), lo.data(), fwd.data());
    p->lo.swap(lo);
    p->fwd.swap(fwd);
}

// PlanTables of the problem at `out` (zeros so far).  They come out of the pass that makes the window starts and go
// up with the inputs.  Made by a kernel of the first scoring call they cost that call an allocation, a launch and
// the overlap with the launch in front (k = 14, L = 50, 100 003 plans: first call 32.3 us so, 21.4 now; with
// create and set stream 59.5 and 54.7).
void fill_plan_tables(const pp_problem *p, unsigned char *out)
{
    const int L = p->L, k = p->k;
    const PlanTables t = plan_tables(L, k);
    std::memcpy(out + t.bits, p->bits.data(), (size_t)L * 8);
    uint32_t *bw = reinterpret_cast<uint32_t *>(out + t.bw);
    for (int v = 0; v < k; ++v) std::memcpy(bw + (size_t)v * (k + 1), p->bw.data() + (size_t)v * k, (size_t)k * 4);
    std::memcpy(out + t.fwd, p->fwd.data(), p->fwd.size() * 2);
}

// Copies the inputs to the device, ordered on the problem's stream.  The staging memory may go as soon
// as the call returns: copies from pageable memory leave it first.
pp_status upload_inputs(pp_problem *p, bool wait)
{
    if (p->uploaded) return PP_OK;
    const bool rec = recording(p->stream);
    if (rec && !p->d_spare) {  // the buffer of pp_problem_create is ordered on the legacy stream, which is out of reach now
        unsigned char *b = nullptr;
        PP_CUDA(kept_alloc(p, &b, p->inputs_bytes, true));
        p->d_spare = p->d_inputs;
        bind_inputs(p, b);
    }
    const int L = p->L, k = p->k;
    std::vector<unsigned char> st;
    try {
        ensure_windows(p);
        st.assign(p->inputs_bytes, 0);
    } catch (const std::bad_alloc &) {
        return PP_ERR_NOMEM;
    }
    auto put = [&](const void *dst, const void *src, size_t n) {
        std::memcpy(st.data() + (static_cast<const unsigned char *>(dst) - p->d_inputs), src, n);
    };
    put(p->d.bits, p->bits.data(), (size_t)L * 8);
    put(p->d.M, p->M.data(), (size_t)(L + 1) * 8);
    put(p->d.cap, p->cap.data(), (size_t)k * 8);
    put(p->d.bw, p->bw.data(), (size_t)k * k * 4);
    put(p->d.lo, p->lo.data(), (size_t)k * L * 2);
    PruneCtl ctl;
    prune_ctl_init(&ctl);
    put(p->prune.ctl, &ctl, sizeof ctl);
    fill_plan_tables(p, st.data() + (p->d_tables - p->d_inputs));
    if (rec) {
        OutsideCapture outside;
        cudaStream_t via = nullptr;
        PP_CUDA(copy_stream(&via));
        PP_CUDA(copy_in(p->d_inputs, st.data(), st.size(), via));
    } else if (wait) {
        PP_CUDA(copy_in(p->d_inputs, st.data(), st.size(), nullptr));
    } else PP_CUDA(cudaMemcpyAsync(p->d_inputs, st.data(), st.size(), cudaMemcpyHostToDevice, p->stream));
    p->uploaded = true;
    p->tables_ready = wait || rec;
    return PP_OK;
}

// Whether a launch over plans may start before the one in front of it has ended.
bool early(pp_problem *p)
{
    const bool was = p->tables_ready;
    p->tables_ready = true;  // for the launch behind this one
    return was;
}

// Page-locked memory of the synchronous calls, one slot per call in flight: the kernel writes its result
// straight into host memory.  Chunks of kSlots; all but one chunk are given back when unused.
struct HostSlot {
    pp_solution sol;
    PruneNote note;
    MatchOut match;
    PruneCtl *ctl;             // counters of a search, on the chunk's device
    unsigned long long *records;  // of the placement stage, on the chunk's device: MatchDev::records
    int half;
    alignas(256) unsigned char small[15 * 1024];  // inputs and results of a small call as a whole
};
constexpr int kSlots = 8;
class HostSlots {
public:
    HostSlot *take()
    {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
        std::lock_guard<std::mutex> lock(mu_);
        for (auto &c : chunks_)
            if (c.free && c.dev == dev) return from(c);
        int sms = 0;
        if (multiprocessors(dev, &sms) != cudaSuccess) return nullptr;
        Chunk c{nullptr, nullptr, nullptr, (1u << kSlots) - 1u, dev};
        const size_t records = match_record_bytes(sms);
        try {
            chunks_.reserve(chunks_.size() + 1);
        } catch (const std::bad_alloc &) {
            return nullptr;
        }
        PruneCtl init[kSlots];
        for (auto &x : init) prune_ctl_init(&x);
        cudaError_t e = cudaHostAlloc(reinterpret_cast<void **>(&c.base), kSlots * sizeof(HostSlot),
                                      cudaHostAllocPortable | cudaHostAllocMapped);
        if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void **>(&c.ctl), sizeof init);
        if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void **>(&c.records), kSlots * records);
        cudaStream_t via = nullptr;
        if (e == cudaSuccess) e = copy_stream(&via);
        if (e == cudaSuccess) e = cudaMemsetAsync(c.records, 0, kSlots * records, via);
        if (e == cudaSuccess) e = copy_in(c.ctl, init, sizeof init, via);  // the same stream: both are complete
        if (e != cudaSuccess) {
            cudaFreeHost(c.base);
            cudaFree(c.ctl);
            cudaFree(c.records);
            cudaGetLastError();
            return nullptr;
        }
        for (int i = 0; i < kSlots; ++i) {
            c.base[i].ctl = c.ctl + i;
            c.base[i].records = reinterpret_cast<unsigned long long *>(c.records + i * records);
            c.base[i].half = 0;
        }
        chunks_.push_back(c);
        return from(chunks_.back());
    }
    void give(HostSlot *s)
    {
        std::lock_guard<std::mutex> lock(mu_);
        for (size_t i = 0; i < chunks_.size(); ++i) {
            Chunk &c = chunks_[i];
            const ptrdiff_t at = s - c.base;
            if (at < 0 || at >= kSlots) continue;
            c.free |= 1u << at;
            bool another = false;  // the first chunk of a device stays
            for (size_t j = 0; j < i; ++j) another |= chunks_[j].dev == c.dev;
            if (another && c.free == (1u << kSlots) - 1u) {
                cudaFreeHost(c.base);
                cudaFree(c.ctl);
                cudaFree(c.records);
                chunks_.erase(chunks_.begin() + (long)i);
            }
            return;
        }
    }

private:
    struct Chunk {
        HostSlot *base;
        PruneCtl *ctl;
        unsigned char *records;
        uint32_t free;
        int dev;
    };
    static HostSlot *from(Chunk &c)
    {
        const int at = __builtin_ctz(c.free);
        c.free &= ~(1u << at);
        return c.base + at;
    }
    std::mutex mu_;
    std::vector<Chunk> chunks_;
};
HostSlots g_slots;
// Page-locked staging memory of the host-pointer calls of middling size: at most kPinnedKeep buffers stay
// for later calls, of any thread; what is handed back beyond that is freed.
constexpr size_t kPinnedBytes = 1 << 20;
constexpr size_t kPinnedKeep = 4;
class PinnedBuffers {
public:
    unsigned char *take()
    {
        {
            std::lock_guard<std::mutex> lock(mu_);
            if (n_ > 0) return free_[--n_];
        }
        void *ptr = nullptr;
        if (cudaHostAlloc(&ptr, kPinnedBytes, cudaHostAllocPortable | cudaHostAllocMapped) == cudaSuccess)
            return static_cast<unsigned char *>(ptr);
        cudaGetLastError();
        return nullptr;
    }
    void give(unsigned char *p)
    {
        {
            std::lock_guard<std::mutex> lock(mu_);
            if (n_ < kPinnedKeep) {
                free_[n_++] = p;
                return;
            }
        }
        cudaFreeHost(p);
    }

private:
    std::mutex mu_;
    unsigned char *free_[kPinnedKeep] = {};
    size_t n_ = 0;
};
PinnedBuffers g_pinned;

struct SlotLease {  // a slot for the duration of a call
    HostSlot *slot = g_slots.take();
    ~SlotLease() { if (slot) g_slots.give(slot); }
};

// ---- the dense search (pp_rank.cu, pp_sweep*.cu) ------------------------------------------------

// Sizes of its tables: distinct usable bandwidths, element width, row stride.
void dense_dims(pp_problem *p)
{
    if (p->dense_dims) return;
    const int k = p->k, L = p->L;
    std::map<uint32_t, int> seen;
    p->ubw.clear();
    p->pair_u.assign((size_t)k * k, -1);
    for (int v = 0; v < k; ++v)
        for (int w = 0; w < k; ++w) {
            uint32_t b = p->bw[(size_t)v * k + w];
            if (v == w || b == 0) continue;
            auto it = seen.find(b);
            if (it == seen.end()) {
                it = seen.emplace(b, (int)p->ubw.size()).first;
                p->ubw.push_back(b);
            }
            p->pair_u[(size_t)v * k + w] = (int16_t)it->second;
        }
    p->U = (int)p->ubw.size();
    if (p->ubw.empty()) p->ubw.push_back(0);  // keep the upload non-empty; U stays 0
    // 16-bit ranks when 0, 1..L*U and the +inf code all fit
    p->elem = ((uint64_t)L * (uint64_t)std::max(p->U, 1) + 1 <= 65534) ? 2 : 4;
    const int per32 = 32 / p->elem;
    p->Lpad = (L + per32 - 1) / per32 * per32;
    Dev &d = p->d;
    d.Lpad = p->Lpad; d.U = p->U; d.elem = p->elem;
    p->dense_dims = true;
}

// Bytes of a workspace that either search can run in.
uint64_t workspace_bytes(pp_problem *p)
{
    dense_dims(p);
    return std::max<uint64_t>(work_layout(p->L, p->k, p->Lpad, p->U, p->elem).total,
                              sparse_bytes(p->k, p->prune.Lp, ~0ull));
}

void bind_work(pp_problem *p)
{
    WorkLayout w = work_layout(p->L, p->k, p->Lpad, p->U, p->elem);
    unsigned char *b = p->d_work;
    p->d.pos = reinterpret_cast<int16_t *>(b + w.pos);
    p->d.order = reinterpret_cast<int16_t *>(b + w.order);
    p->d.gu = reinterpret_cast<double *>(b + w.gu);
    p->d.cnt = reinterpret_cast<uint32_t *>(b + w.cnt);
    p->d.rk = reinterpret_cast<uint32_t *>(b + w.rk);
    p->d.inv = reinterpret_cast<uint32_t *>(b + w.inv);
    p->d.rank = b + w.rank;
    p->d.table = b + w.table;
    p->d.rank_elems = (uint64_t)p->k * p->k * p->Lpad;
    p->d.table_elems = ((uint64_t)p->k << p->k) * p->Lpad;
}

pp_status ensure_work(pp_problem *p)
{
    if (p->d_work) return PP_OK;
    void *ptr = nullptr;
    if (alloc_should_fail()) return PP_ERR_NOMEM;
    const uint64_t bytes = workspace_bytes(p);
    OutsideCapture outside;
    PP_CUDA(cudaMalloc(&ptr, bytes));
    p->d_work = static_cast<unsigned char *>(ptr);
    p->work_bytes = bytes;
    p->own_work = true;
    bind_work(p);
    bind_sparse(p->prune, p->d_work, bytes);
    return PP_OK;
}

// Window constants of the register-tiled kernels, the list of node sets and the bandwidth classes on
// the device, and which kernel takes which level.
pp_status dense_prepare(pp_problem *p)
{
    if (p->dense_ready) return PP_OK;
    const int L = p->L, k = p->k;
    Dev &d = p->d;
    try {
        dense_dims(p);
        ensure_windows(p);
        const MaskList &ml = mask_list(k);
        // constants of the register-tiled sweep, when the instance is inside its envelope
        std::vector<unsigned char> fmeta(fast_meta_bytes()), pmeta;
        std::vector<uint32_t> gmeta;
        const bool tiled = p->elem == 2 && p->Lpad <= 240 && k >= 2;
        const bool has_fast = tiled && fast_meta_build(L, k, p->lo.data(), fmeta.data());
        if (has_fast && ml.swaps) {
            pmeta.resize(pair_meta_bytes());
            if (!pair_meta_build(L, k, p->lo.data(), pmeta.data())) pmeta.clear();
        }
        if (!has_fast && tiled) {
            gmeta.resize((size_t)k * p->Lpad);
            d.gen_levels = gen_meta_build(L, k, p->Lpad, p->lo.data(), gmeta.data());
        }
        struct Part { const void *src; size_t bytes; size_t off; };
        Part parts[5] = {{p->pair_u.data(), p->pair_u.size() * 2, 0}, {p->ubw.data(), p->ubw.size() * 4, 0},
                         {fmeta.data(), fmeta.size(), 0}, {gmeta.data(), gmeta.size() * 4, 0}, {pmeta.data(), pmeta.size(), 0}};
        size_t total = 0;
        for (auto &q : parts) { q.off = total; total = align_up(total + q.bytes, 256); }
        // one staging buffer, one copy: the parts are small and a copy per part costs more than the bytes
        std::vector<unsigned char> staging(total, 0);
        for (auto &q : parts)
            if (q.bytes) std::memcpy(staging.data() + q.off, q.src, q.bytes);
        DeviceMasks dmasks;
        PP_CUDA(device_masks(k, ml, &dmasks));
        {
            const bool rec = recording(p->stream);
            OutsideCapture outside;
            cudaStream_t via = nullptr;
            if (rec) PP_CUDA(copy_stream(&via));
            if (!p->d_dense) {
                if (rec) PP_CUDA(kept_alloc(p, &p->d_dense, total, true));
                else PP_CUDA(staging_alloc(reinterpret_cast<void **>(&p->d_dense), total, nullptr));
            }
            PP_CUDA(copy_in(p->d_dense, staging.data(), total, via));
        }
        for (auto &e : p->ev)
            if (!e) PP_CUDA(cudaEventCreate(&e));
        unsigned char *b = p->d_dense;
        d.pair_u = reinterpret_cast<int16_t *>(b + parts[0].off);
        d.ubw = reinterpret_cast<uint32_t *>(b + parts[1].off);
        d.fast_meta = has_fast ? b + parts[2].off : nullptr;
        d.gen_meta = gmeta.empty() ? nullptr : reinterpret_cast<uint32_t *>(b + parts[3].off);
        d.pair_meta = pmeta.empty() ? nullptr : b + parts[4].off;
        d.masks = dmasks.masks;  // shared by every problem of this k on this device
        d.level_off = dmasks.level_off;
        p->pair_lvl.assign(k + 2, -1);
    } catch (const std::bad_alloc &) {
        return PP_ERR_NOMEM;
    }
    p->dense_ready = true;
    return PP_OK;
}

// The kernels the dense search of this problem consists of (also what pp_last_solve_profile reports).
void dense_plan(pp_problem *p, bool *fast)
{
    const Dev &d = p->d;
    *fast = p->force_generic != 1 && fast_sweep_supported(d);
    p->pair_levels = 0;
    const int top = std::min(p->k, p->L);
    for (int level = 2; level <= top; ++level) {
        if (!*fast || p->force_generic == 2) continue;
        if (p->pair_lvl[level] < 0) p->pair_lvl[level] = pair_sweep_takes(d, level, p->force_generic == 3) ? 1 : 0;
        p->pair_levels += p->pair_lvl[level];
    }
    p->fast_used = *fast ? (d.fast_meta ? 1 : 2) : 0;
}

pp_status queue_dense(pp_problem *p, pp_solution *sol_dev)
{
    pp_status st = ensure_work(p);
    if (st == PP_OK) st = upload_inputs(p, false);
    if (st == PP_OK) st = dense_prepare(p);
    if (st != PP_OK) return st;
    cudaStream_t s = p->stream;
    bool fast = false;
    dense_plan(p, &fast);
    const Dev &d = p->d;
    int launches = 0;
    PP_CUDA(cudaEventRecord(p->ev[0], s));
    PP_CUDA(launch_rank_base(d, s, &launches));
    // an event between two kernels ends the programmatic overlap of their launches: only on request
    if (p->profiling) PP_CUDA(cudaEventRecord(p->ev[1], s));
    int sweep = 0;
    const int top = std::min(p->k, p->L);
    for (int level = 2; level <= top; ++level) {
        const bool first = level == 2;
        if (!fast) PP_CUDA(launch_sweep_generic(d, level, s));
        else if (p->force_generic != 2 && p->pair_lvl[level]) PP_CUDA(launch_sweep_pair(d, level, s, first));
        else PP_CUDA(launch_sweep_fast(d, level, s, first));
        ++sweep;
    }
    if (p->profiling) PP_CUDA(cudaEventRecord(p->ev[2], s));
    PP_CUDA(launch_finalize(d, sol_dev, s, true));
    PP_CUDA(cudaEventRecord(p->ev[3], s));
    p->sweep_launches = sweep;
    p->total_launches += launches + sweep + 1;
    p->solved = true;
    p->profiled = p->profiling;
    p->table_whole = true;
    return PP_OK;
}

// The bounded search is the way an ordinary solve takes; a caller that pins a sweep kernel or asks for
// the times of the dense search's phases gets the dense search.
bool takes_sparse(const pp_problem *p) { return p->force_generic == -1 && !p->profiling; }

// Scratch of the bounded search: the workspace, else a pooled buffer of its own.
pp_status ensure_sparse(pp_problem *p)
{
    if (p->d_work || p->d_sparse) return PP_OK;
    const size_t bytes = sparse_bytes(p->k, p->prune.Lp, kSparseScratchBytes);
    PP_CUDA(kept_alloc(p, &p->d_sparse, bytes, recording(p->stream)));
    bind_sparse(p->prune, p->d_sparse, bytes);
    return PP_OK;
}

// row_limit: rows after which the search gives up (note->dense).
pp_status queue_sparse(pp_problem *p, PruneCtl *ctl, pp_solution *sol, PruneNote *note, unsigned long long row_limit)
{
    PruneDev q = p->prune;
    q.ctl = ctl;
    q.lo = p->uploaded ? p->d.lo : nullptr;
    q.out = sol;
    q.note = note;
    q.row_cap = std::min(q.row_cap, row_limit);
    q.fallback = row_limit != ~0ull;
    const PruneHost h{p->bits.data(), p->M.data(), p->cap.data(), p->bw.data(), nullptr, nullptr};
    PP_CUDA(launch_prune(q, h, p->sms, p->stream));
    p->total_launches = 1;
    p->sweep_launches = 1;
    p->solved = true;
    p->profiled = false;
    p->sparse_ran = true;
    p->table_whole = false;
    return PP_OK;
}

}  // namespace

int pp::starved_polls() { return g_starved_polls.load(std::memory_order_relaxed) ? g_starved_polls.exchange(0) : 0; }
// What the search by thresholds did in the calling thread's last synchronous solve (pp_debug_thresholds).
static thread_local int32_t t_thresholds = 0;
int pp::late_polls(int *block)
{
    const uint64_t late = g_late.load(std::memory_order_relaxed) ? g_late.exchange(0) : 0;
    *block = (int)(late >> 32);
    return (int)(uint32_t)late;
}

extern "C" {

const char *pp_status_str(pp_status s)
{
    switch (s) {
        case PP_OK: return "ok";
        case PP_INFEASIBLE: return "infeasible: no plan exists";
        case PP_ERR_ARG: return "bad argument";
        case PP_ERR_LIMIT: return "size or value above the library limits";
        case PP_ERR_NOMEM: return "out of memory";
        case PP_ERR_CUDA: return "CUDA runtime error";
        case PP_ERR_TIMEOUT: return "timeout";
    }
    return "unknown status";
}

pp_status pp_problem_create(int32_t L, const uint64_t *layer_out_bits,
                            const uint64_t *layer_mem_bytes, int32_t k,
                            const uint64_t *node_mem_bytes, const uint32_t *bw_kbps,
                            pp_problem **out)
{
    if (!out) return PP_ERR_ARG;
    pp_status st = validate(L, layer_out_bits, layer_mem_bytes, k, node_mem_bytes, bw_kbps);
    if (st != PP_OK) return st;
    pp_problem *p = new (std::nothrow) pp_problem();
    if (!p) return PP_ERR_NOMEM;
    try {
        p->L = L;
        p->k = k;
        p->bits.assign(layer_out_bits, layer_out_bits + L);
        p->mem.assign(layer_mem_bytes, layer_mem_bytes + L);
        p->cap.assign(node_mem_bytes, node_mem_bytes + k);
        p->bw.assign(bw_kbps, bw_kbps + (size_t)k * k);
        // memory prefix sums: segment first..last needs M[last+1] - M[first] bytes
        p->M.assign(L + 1, 0);
        for (int i = 0; i < L; ++i) p->M[i + 1] = p->M[i] + p->mem[i];
    } catch (const std::bad_alloc &) {
        delete p;
        return PP_ERR_NOMEM;
    }
    // one device buffer; the copy is queued by pp_problem_set_stream or by the first call that needs it
    p->inputs_bytes = bind_inputs(p, nullptr);
    int dev = 0;
    unsigned char *b = nullptr;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = multiprocessors(dev, &p->sms);
    if (e == cudaSuccess) e = staging_alloc(reinterpret_cast<void **>(&b), p->inputs_bytes, nullptr);
    if (e != cudaSuccess) {
        pp_status rc = from_cuda(e);
        pp_problem_destroy(p);
        return rc;
    }
    p->d.L = L; p->d.k = k;
    bind_inputs(p, b);
    PruneDev &q = p->prune;
    q.L = L; q.k = k; q.Lp = prune_row_pad(L, k);
    double lo = std::numeric_limits<double>::max(), hi = 0.0;
    quotient_range(L, p->bits.data(), k * k, p->bw.data(), &lo, &hi);
    prune_key_range(hi > 0.0 ? lo : 1.0, hi > 0.0 ? hi : 1.0, &q);
    prune_node_bounds(p->cap.data(), p->M[L], &q);
    *out = p;
    return PP_OK;
}

void pp_problem_destroy(pp_problem *p)
{
    if (!p) return;
    if (p->own_work && p->d_work) cudaFree(p->d_work);
    for (unsigned char *q : {p->d_inputs, p->d_spare, p->d_sparse, p->d_dense})
        if (q && std::find(p->mallocs, p->mallocs + p->n_mallocs, q) == p->mallocs + p->n_mallocs)
            cudaFreeAsync(q, p->stream);  // ordered after the problem's queued work
    for (int i = 0; i < p->n_mallocs; ++i) cudaFree(p->mallocs[i]);
    for (auto &e : p->ev)
        if (e) cudaEventDestroy(e);
    delete p;
}

pp_status pp_problem_set_stream(pp_problem *p, void *cuda_stream)
{
    if (!p) return PP_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    if (s != p->stream && (p->uploaded || p->d_sparse) && !recording(p->stream)) {  // copies and scratch are ordered there
        if (p->stream || !recording(s)) {  // waiting for the legacy stream would end the recording
            OutsideCapture outside;
            PP_CUDA(cudaStreamSynchronize(p->stream));
            p->tables_ready = p->uploaded;
        }
    }
    p->stream = s;
    return upload_inputs(p, s != nullptr);  // the legacy stream, on which the buffer was allocated, has it in order
}

pp_status pp_problem_workspace_bytes(const pp_problem *p, uint64_t *bytes)
{
    if (!p || !bytes) return PP_ERR_ARG;
    try {
        *bytes = workspace_bytes(const_cast<pp_problem *>(p));
    } catch (const std::bad_alloc &) {
        return PP_ERR_NOMEM;
    }
    return PP_OK;
}

pp_status pp_problem_set_workspace(pp_problem *p, void *device_buffer, uint64_t bytes)
{
    if (!p || !device_buffer) return PP_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(device_buffer) % 256) return PP_ERR_ARG;
    uint64_t need = 0;
    pp_status st = pp_problem_workspace_bytes(p, &need);
    if (st != PP_OK) return st;
    if (bytes < need) return PP_ERR_NOMEM;
    if (p->own_work && p->d_work) {
        cudaStreamSynchronize(p->stream);
        cudaFree(p->d_work);
    }
    p->d_work = static_cast<unsigned char *>(device_buffer);
    p->work_bytes = bytes;
    p->own_work = false;
    p->solved = false;
    bind_work(p);
    bind_sparse(p->prune, p->d_work, bytes);
    return PP_OK;
}

pp_status pp_problem_force_generic(pp_problem *p, int32_t mode)
{
    if (!p || mode < -1 || mode > 3) return PP_ERR_ARG;
    p->force_generic = mode;
    if (p->dense_ready) p->pair_lvl.assign(p->k + 2, -1);
    return PP_OK;
}

pp_status pp_problem_set_profiling(pp_problem *p, int32_t on)
{
    if (!p) return PP_ERR_ARG;
    p->profiling = on != 0;
    return PP_OK;
}

pp_status pp_solve_exact_dev(pp_problem *p, pp_solution *solution_dev)
{
    if (!p || !solution_dev) return PP_ERR_ARG;
    try {
        p->total_launches = 0;
        p->sparse_ran = false;
        if (!takes_sparse(p)) return queue_dense(p, solution_dev);
        // room for every row: pooled scratch where that is small, else a workspace
        pp_status st = PP_OK;
        if (!prune_in_shared(p->L, p->k, false))
            st = sparse_bytes(p->k, p->prune.Lp, ~0ull) <= kSparseScratchBytes ? ensure_sparse(p) : ensure_work(p);
        if (st == PP_OK) st = upload_inputs(p, false);  // the counters
        if (st == PP_OK) st = queue_sparse(p, p->prune.ctl, solution_dev, p->d_note, ~0ull);
        p->note_on_device = true;
        return st;
    } catch (const std::bad_alloc &) {
        return PP_ERR_NOMEM;
    }
}

// The bounded search with its result in page-locked memory.  PP_ERR_LIMIT: the frontier outgrew its
// rows, the dense search has to run.
static pp_status solve_sparse(pp_problem *p, pp_solution *sol)
{
    pp_status st = prune_in_shared(p->L, p->k, false) ? PP_OK : ensure_sparse(p);
    if (st != PP_OK) return st;
    HostSlot *slot = g_slots.take();
    if (!slot) return PP_ERR_NOMEM;
    st = queue_sparse(p, slot->ctl, &slot->sol, &slot->note, kSparseRows);
    const cudaError_t e = cudaStreamSynchronize(p->stream);
    if (st == PP_OK) st = from_cuda(e);
    if (st == PP_OK) {
        p->note = slot->note;
        p->note_on_device = false;
        t_thresholds = slot->note.thresholds;
        *sol = slot->sol;
        if (p->note.dense) st = PP_ERR_LIMIT;
        else if (sol->status != PP_OK && sol->status != PP_INFEASIBLE) st = PP_ERR_CUDA;
    }
    g_slots.give(slot);
    return st;
}

pp_status pp_solve_exact(pp_problem *p, double *beta_ms, int32_t *m, int32_t *cuts,
                         int32_t *placement)
{
    if (!p || !beta_ms || !m || !placement || (!cuts && p->k > 1)) return PP_ERR_ARG;
    pp_solution sol{};
    try {
        p->total_launches = 0;
        p->sparse_ran = false;
        t_thresholds = 0;
        pp_status st = takes_sparse(p) ? solve_sparse(p, &sol) : PP_ERR_LIMIT;
        if (st == PP_ERR_LIMIT) {
            int32_t err = 0;
            st = upload_inputs(p, false);
            if (st != PP_OK) return st;
            PP_CUDA(cudaMemsetAsync(p->d.err, 0, sizeof(int32_t), p->stream));
            st = queue_dense(p, p->d_sol);
            if (st != PP_OK) return st;
            PP_CUDA(cudaMemcpyAsync(&sol, p->d_sol, sizeof sol, cudaMemcpyDeviceToHost, p->stream));
            PP_CUDA(cudaMemcpyAsync(&err, p->d.err, sizeof err, cudaMemcpyDeviceToHost, p->stream));
            PP_CUDA(cudaStreamSynchronize(p->stream));
            if (err) return PP_ERR_CUDA;
        } else if (st != PP_OK) {
            return st;
        }
    } catch (const std::bad_alloc &) {
        return PP_ERR_NOMEM;
    }
    *beta_ms = sol.beta_ms;
    *m = sol.m;
    for (int j = 0; j < p->k - 1; ++j) cuts[j] = sol.cuts[j];
    for (int j = 0; j < p->k; ++j) placement[j] = sol.placement[j];
    return static_cast<pp_status>(sol.status);
}

pp_status pp_last_solve_profile(pp_problem *p, pp_profile *out)
{
    if (!p || !out || !p->solved) return PP_ERR_ARG;
    PP_CUDA(cudaStreamSynchronize(p->stream));
    pp_status st = dense_prepare(p);
    if (st != PP_OK) return st;
    bool fast = false;
    dense_plan(p, &fast);
    out->ms_rank = out->ms_sweep = out->ms_finalize = out->ms_total = 0.0f;
    if (p->sparse_ran) {
        if (p->note_on_device) PP_CUDA(cudaMemcpy(&p->note, p->d_note, sizeof p->note, cudaMemcpyDeviceToHost));
        out->ms_total = (float)((double)p->note.ns * 1e-6);
    }
    if (p->table_whole) {
        float ms = 0.0f;
        PP_CUDA(cudaEventElapsedTime(&ms, p->ev[0], p->ev[3]));
        out->ms_total += ms;
    }
    if (p->profiled) {
        PP_CUDA(cudaEventElapsedTime(&out->ms_rank, p->ev[0], p->ev[1]));
        PP_CUDA(cudaEventElapsedTime(&out->ms_sweep, p->ev[1], p->ev[2]));
        PP_CUDA(cudaEventElapsedTime(&out->ms_finalize, p->ev[2], p->ev[3]));
    }
    out->sweep_launches = p->sweep_launches;
    out->total_launches = p->total_launches;
    out->state_bytes = p->elem;
    out->fast_path = p->fast_used;
    out->pair_levels = p->pair_levels;
    return PP_OK;
}

pp_status pp_eval_plans_dev(pp_problem *p, int64_t B, const uint8_t *nseg, const int32_t *ends,
                            const int32_t *nodes, double *beta_ms, uint8_t *plan_status)
{
    if (!p || B < 0) return PP_ERR_ARG;
    if (B == 0) return PP_OK;
    if (!nseg || !ends || !nodes || !beta_ms || !plan_status) return PP_ERR_ARG;
    pp_status st = upload_inputs(p, false);
    if (st != PP_OK) return st;
    PP_CUDA(launch_eval(p->d, p->d_tables, B, nseg, ends, nodes, beta_ms, plan_status, early(p), p->stream));
    return PP_OK;
}

pp_status pp_eval_plans(pp_problem *p, int64_t B, const uint8_t *nseg, const int32_t *ends,
                        const int32_t *nodes, double *beta_ms, uint8_t *plan_status)
{
    if (!p || B < 0) return PP_ERR_ARG;
    if (B == 0) return PP_OK;
    if (!nseg || !ends || !nodes || !beta_ms || !plan_status) return PP_ERR_ARG;
    const size_t k = p->k;
    const size_t b_nseg = (size_t)B, b_rows = (size_t)B * k * 4, b_beta = (size_t)B * 8;
    size_t o_ends = align_up(b_nseg, 256), o_nodes = align_up(o_ends + b_rows, 256);
    size_t o_beta = align_up(o_nodes + b_rows, 256), o_st = align_up(o_beta + b_beta, 256);
    size_t total = o_st + (size_t)B;
    pp_status st = upload_inputs(p, false);
    if (st != PP_OK) return st;
    unsigned char *buf = nullptr;
    cudaStream_t s = p->stream;
    PP_CUDA(staging_alloc(reinterpret_cast<void **>(&buf), total, s));
    cudaError_t e = cudaMemcpyAsync(buf, nseg, b_nseg, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(buf + o_ends, ends, b_rows, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(buf + o_nodes, nodes, b_rows, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = launch_eval(p->d, p->d_tables, B, buf, reinterpret_cast<int32_t *>(buf + o_ends),
                        reinterpret_cast<int32_t *>(buf + o_nodes),
                        reinterpret_cast<double *>(buf + o_beta), buf + o_st, early(p), s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(beta_ms, buf + o_beta, b_beta, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(plan_status, buf + o_st, (size_t)B, cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(buf, s);
    cudaError_t e2 = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return from_cuda(e);
    return from_cuda(e2);
}

pp_status pp_eval_plans_packed_dev(pp_problem *p, int64_t B, int64_t total, const uint8_t *nseg,
                                   const uint32_t *plan_off, const uint16_t *ends, const uint8_t *nodes,
                                   double *beta_ms, uint8_t *plan_status)
{
    if (!p || B < 0 || total < 0) return PP_ERR_ARG;
    if (B == 0) return PP_OK;
    if (!nseg || !plan_off || !beta_ms || !plan_status || ((!ends || !nodes) && total > 0)) return PP_ERR_ARG;
    pp_status st = upload_inputs(p, false);
    if (st != PP_OK) return st;
    PP_CUDA(launch_eval_packed(p->d, p->d_tables, B, total, nseg, plan_off, ends, nodes, beta_ms, plan_status, early(p), p->stream));
    return PP_OK;
}

pp_status pp_eval_plans_packed(pp_problem *p, int64_t B, int64_t total, const uint8_t *nseg,
                               const uint32_t *plan_off, const uint16_t *ends, const uint8_t *nodes,
                               double *beta_ms, uint8_t *plan_status)
{
    if (!p || B < 0 || total < 0) return PP_ERR_ARG;
    if (B == 0) return PP_OK;
    if (!nseg || !plan_off || !beta_ms || !plan_status || ((!ends || !nodes) && total > 0)) return PP_ERR_ARG;
    const size_t nB = (size_t)B, nT = (size_t)total;
    const size_t o_off = align_up(nB, 256), o_ends = align_up(o_off + (nB + 1) * 4, 256);
    const size_t o_nodes = align_up(o_ends + nT * 2, 256), o_beta = align_up(o_nodes + nT, 256);
    const size_t o_st = align_up(o_beta + nB * 8, 256), bytes = o_st + nB;
    pp_status st = upload_inputs(p, false);
    if (st != PP_OK) return st;
    unsigned char *buf = nullptr;
    cudaStream_t s = p->stream;
    PP_CUDA(staging_alloc(reinterpret_cast<void **>(&buf), bytes, s));
    cudaError_t e = cudaMemcpyAsync(buf, nseg, nB, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(buf + o_off, plan_off, (nB + 1) * 4, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && nT) e = cudaMemcpyAsync(buf + o_ends, ends, nT * 2, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && nT) e = cudaMemcpyAsync(buf + o_nodes, nodes, nT, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = launch_eval_packed(p->d, p->d_tables, B, total, buf, reinterpret_cast<uint32_t *>(buf + o_off),
                               reinterpret_cast<uint16_t *>(buf + o_ends), buf + o_nodes,
                               reinterpret_cast<double *>(buf + o_beta), buf + o_st, early(p), s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(beta_ms, buf + o_beta, nB * 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(plan_status, buf + o_st, nB, cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(buf, s);
    cudaError_t e2 = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return from_cuda(e);
    return from_cuda(e2);
}

pp_status pp_random_plans_dev(pp_problem *p, int64_t P, const uint32_t *draws, uint8_t *nseg, int32_t *ends,
                              int32_t *nodes)
{
    if (!p || P < 0) return PP_ERR_ARG;
    if (P == 0) return PP_OK;
    if (!draws || !nseg || !ends || !nodes) return PP_ERR_ARG;
    pp_status st = upload_inputs(p, false);
    if (st != PP_OK) return st;
    PP_CUDA(launch_random_plans(p->d, p->d_tables, P, draws, nseg, ends, nodes, early(p), p->stream));
    return PP_OK;
}

pp_status pp_random_plans(pp_problem *p, int64_t P, const uint32_t *draws, uint8_t *nseg, int32_t *ends,
                          int32_t *nodes)
{
    if (!p || P < 0) return PP_ERR_ARG;
    if (P == 0) return PP_OK;
    if (!draws || !nseg || !ends || !nodes) return PP_ERR_ARG;
    const size_t k = p->k;
    const size_t b_draws = (size_t)P * 2 * k * 4, b_rows = (size_t)P * k * 4;
    const size_t o_ends = align_up(b_draws, 256), o_nodes = align_up(o_ends + b_rows, 256);
    const size_t o_nseg = align_up(o_nodes + b_rows, 256), total = o_nseg + (size_t)P;
    pp_status st = upload_inputs(p, false);
    if (st != PP_OK) return st;
    unsigned char *buf = nullptr;
    cudaStream_t s = p->stream;
    PP_CUDA(staging_alloc(reinterpret_cast<void **>(&buf), total, s));
    cudaError_t e = cudaMemcpyAsync(buf, draws, b_draws, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = launch_random_plans(p->d, p->d_tables, P, reinterpret_cast<uint32_t *>(buf), buf + o_nseg,
                                reinterpret_cast<int32_t *>(buf + o_ends),
                                reinterpret_cast<int32_t *>(buf + o_nodes), early(p), s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(nseg, buf + o_nseg, (size_t)P, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(ends, buf + o_ends, b_rows, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(nodes, buf + o_nodes, b_rows, cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(buf, s);
    cudaError_t e2 = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return from_cuda(e);
    return from_cuda(e2);
}

// What solves a batch: an instance to a lane, to a warp, or to a block, and there to a narrow one or a wide one.
struct BatchRoute {
    bool lanes, warps, narrow;
};

// pieces: of a batch that lies in page-locked host memory, 0 for one on the device.
// The pieces of short chains run side by side, so that all the batch's instances count for the width of the blocks.
// Pieces of chains of more than 32 layers hold fewer instances: up to 36 layers two of them meet on the GPU, and beyond
// that wide blocks are done with one when the host has copied the next.  A call from host arrays, narrow and wide, us
// (three seeds; the runs of one side lie within 2 %):
//   (k = 6, L = 33)  500 73.9, 75.7; 600 80.7, 79.0; 740 94.3, 90.7; 888 103.0, 99.3; 1000 110.1, 114.3; 1100 116.4, 119.5
//   (6, 36)          500 75.2, 77.0; 600 83.3, 81.0; 740 97.7, 93.1; 888 106.7, 101.3; 1000 113.4, 115.2; 1100 120.9, 121.6
//   (6, 40), (6, 50) 500 79.9, 75.8 and 87.8, 82.5; 740 100.8, 95.0 and 110.1, 105.3; 1000 x (6, 40) 118.0, 117.3
//   (5, 33), (5, 50) 600 67.6, 64.1 and 84.1, 81.3; 1000 92.7, 93.0 and 113.7, 112.8; (4, 33) to (4, 60) within 2 %
// (two pieces of 222 fill a wave of wide blocks, 500 and 1000 instances come in pieces of 250).
static BatchRoute batch_route(int64_t B, int L, int k, int sms, int64_t pieces)
{
    const int64_t each = pieces ? (B + pieces - 1) / pieces : B;
    const int64_t together = !pieces || L <= 32 ? B : L <= 36 ? std::min(B, 2 * each) : each;
    const bool shared = !pieces && batch_lanes_takes(B, L, k, sms), warps = shared && batch_warps_takes(B, L, k);
    return {shared && !warps, warps, batch_narrow(together, L, k, sms)};
}

// These are the batch whose route it is, or a piece of it.  early: behind another piece of the same batch.
static pp_status queue_exact_batch(int64_t B, int32_t L, int32_t k, const uint64_t *out_bits, const uint64_t *mem,
                                   const uint64_t *node_mem, const uint32_t *bw, double *beta_ms, int32_t *m, int32_t *cuts,
                                   int32_t *placement, int8_t *status, int sms, BatchRoute route, bool early, cudaStream_t s)
{
    if (batch_smem_bytes(L, k) + 1024 > kBlockShared) return PP_ERR_LIMIT;
    LaneTables lt;
    if (route.warps) {
        PP_CUDA(lane_tables(k - 1, &lt));
        PP_CUDA(launch_batch_warps(B, L, k, lt, sms, out_bits, mem, node_mem, bw, beta_ms, m, cuts, placement, status, s));
        return PP_OK;
    }
    PP_CUDA(lane_tables(k, &lt));
    if (!route.lanes) {
        PP_CUDA(launch_batch(B, route.narrow, L, k, lt, sms, out_bits, mem, node_mem, bw, beta_ms, m, cuts, placement, status, early,
                             s));
        return PP_OK;
    }
    // Instance-per-lane path: the tables of a chunk of instances live in scratch memory from the
    // library's pool, ordered on the caller's stream; chunks follow one another on that stream.
    const int64_t chunk = std::min<int64_t>(B, kBatchLanesChunk);
    const size_t G = (size_t)((chunk + 31) / 32);
    BatchLanes t;
    t.LH = batch_lanes_words(L);
    t.rows = (uint32_t)k << (k - 1);
    t.rowoff = lt.rowoff;
    t.mlist = lt.mlist;
    t.moff = lt.moff;
    const size_t line = (size_t)t.LH * 32 * sizeof(uint32_t);
    const size_t b_table = G * t.rows * line, b_rank = G * (size_t)(k * k) * line, b_len = G * (size_t)k * line;
    const size_t b_win = 2 * b_len;
    const size_t b_key = G * 32 * sizeof(unsigned long long), b_flag = align_up(G * 32, 256), b_err = 256;
    unsigned char *buf = nullptr;
    PP_CUDA(staging_alloc(reinterpret_cast<void **>(&buf), b_table + b_rank + b_len + b_win + b_key + b_flag + b_err, s));
    t.table = reinterpret_cast<uint32_t *>(buf);
    t.rank = reinterpret_cast<uint32_t *>(buf + b_table);
    t.len = reinterpret_cast<uint32_t *>(buf + b_table + b_rank);
    t.win = reinterpret_cast<uint32_t *>(buf + b_table + b_rank + b_len);
    t.key = reinterpret_cast<unsigned long long *>(buf + b_table + b_rank + b_len + b_win);
    t.flag = reinterpret_cast<int8_t *>(buf + b_table + b_rank + b_len + b_win + b_key);
    t.err = reinterpret_cast<int32_t *>(buf + b_table + b_rank + b_len + b_win + b_key + b_flag);
    t.table_words = b_table / 4;
    t.rank_words = b_rank / 4;
    t.len_words = b_len / 4;
    t.win_words = b_win / 4;
#ifdef PP_DEBUG_BOUNDS
    {  // the bounds-checking build records violations here; k_lanes_back turns them into PP_ERR_CUDA
        cudaError_t ez = cudaMemsetAsync(t.err, 0, sizeof(int32_t), s);
        if (ez != cudaSuccess) {
            cudaFreeAsync(buf, s);
            return from_cuda(ez);
        }
    }
#endif
    cudaError_t e = cudaSuccess;
    for (int64_t b0 = 0; b0 < B && e == cudaSuccess; b0 += chunk) {
        const int64_t n = std::min<int64_t>(chunk, B - b0);
        e = launch_batch_prep(n, L, k, out_bits + b0 * L, mem + b0 * L, node_mem + b0 * k, bw + b0 * k * k, t, s);
        if (e == cudaSuccess)
            e = launch_batch_lanes(n, L, k, out_bits + b0 * L, bw + b0 * k * k, t, beta_ms + b0, m + b0,
                                   cuts ? cuts + b0 * (k - 1) : nullptr, placement + b0 * k, status + b0, s);
    }
    cudaFreeAsync(buf, s);
    PP_CUDA(e);
    return PP_OK;
}

// Multiprocessors of the current device.
static cudaError_t current_sms(int *sms)
{
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    return e == cudaSuccess ? multiprocessors(dev, sms) : e;
}

pp_status pp_solve_exact_batch_dev(int64_t B, int32_t L, int32_t k, const uint64_t *out_bits,
                                   const uint64_t *mem, const uint64_t *node_mem,
                                   const uint32_t *bw, double *beta_ms, int32_t *m, int32_t *cuts,
                                   int32_t *placement, int8_t *status, void *cuda_stream)
{
    if (B < 0 || L < 1 || k < 1) return PP_ERR_ARG;
    if (L > PP_MAX_L || k > PP_MAX_K) return PP_ERR_LIMIT;
    if (B == 0) return PP_OK;
    if (!out_bits || !mem || !node_mem || !bw || !beta_ms || !m || !placement || !status ||
        (!cuts && k > 1))
        return PP_ERR_ARG;
    int sms = 0;
    PP_CUDA(current_sms(&sms));
    return queue_exact_batch(B, L, k, out_bits, mem, node_mem, bw, beta_ms, m, cuts, placement, status, sms,
                             batch_route(B, L, k, sms, 0), false, static_cast<cudaStream_t>(cuda_stream));
}

// Host-pointer form of a batched entry point: stage the inputs, run the device-pointer form on
// the legacy default stream, bring the results back.
typedef pp_status (*batch_dev_fn)(int64_t, int32_t, int32_t, const uint64_t *, const uint64_t *,
                                  const uint64_t *, const uint32_t *, double *, int32_t *, int32_t *,
                                  int32_t *, int8_t *, void *);

// in_place: the kernels read an input word once, so that a batch of up to kPinnedBytes is worked on where
// it lies in page-locked memory: one pass of the host over the inputs, no device buffer, no copies queued
// (300 x (k = 7, L = 45): 190 us with nine copies from and to pageable memory).
// Where a block takes an instance the batch goes in pieces of 128 KB and more, at most four (87.9 -> 86.1 us, 648 x
// (k = 4, L = 40) 68.0 -> 63.4; pieces of 64 KB 90.9 and 65.3: a launch costs the host what copying 80 KB does).
constexpr int64_t kHostPieces = 4;
constexpr size_t kHostPieceBytes = 128 << 10;

// A host batch's four inputs and five results: bytes of each, and where they lie in one buffer.
struct BatchArrays {
    size_t sz[9], off[10];
};
static BatchArrays batch_arrays(int64_t B, int32_t L, int32_t k)
{
    const size_t nB = (size_t)B;
    BatchArrays a = {{nB * L * 8, nB * L * 8, nB * k * 8, nB * k * k * 4, nB * 8, nB * 4, nB * (size_t)std::max(k - 1, 1) * 4,
                      nB * k * 4, nB}, {}};
    for (int i = 0; i < 9; ++i) a.off[i + 1] = align_up(a.off[i] + a.sz[i], 256);
    return a;
}
static int64_t host_pieces(const BatchArrays &a)
{
    return std::max<int64_t>(1, std::min<int64_t>(kHostPieces, (int64_t)(a.off[4] / kHostPieceBytes)));
}

static pp_status batch_from_host(batch_dev_fn run_dev, bool in_place, int64_t B, int32_t L, int32_t k,
                                 const uint64_t *out_bits, const uint64_t *mem, const uint64_t *node_mem,
                                 const uint32_t *bw, double *beta_ms, int32_t *m, int32_t *cuts,
                                 int32_t *placement, int8_t *status)
{
    if (B < 0 || L < 1 || k < 1) return PP_ERR_ARG;
    if (L > PP_MAX_L || k > PP_MAX_K) return PP_ERR_LIMIT;
    if (B == 0) return PP_OK;
    if (!out_bits || !mem || !node_mem || !bw || !beta_ms || !m || !placement || !status ||
        (!cuts && k > 1))
        return PP_ERR_ARG;
    const size_t nB = (size_t)B;
    const BatchArrays arrays = batch_arrays(B, L, k);
    const size_t *const sz = arrays.sz, *const off = arrays.off;
    if (in_place && off[9] <= kPinnedBytes) {
        struct Lease {
            unsigned char *b = g_pinned.take();
            ~Lease() { if (b) g_pinned.give(b); }
        } lease;
        unsigned char *h = lease.b;
        if (!h) return PP_ERR_NOMEM;
        int sms = 0;
        PP_CUDA(current_sms(&sms));
        const int64_t pieces = host_pieces(arrays);
        const BatchRoute route = batch_route(B, L, k, sms, pieces);
        const void *in[4] = {out_bits, mem, node_mem, bw};
        // An instance to a block: the batch goes in pieces, so that the host copies one while the GPU works on the
        // one before.  With that a batch of this size is faster so than an instance to a lane (to a warp has not been tried from
        // page-locked memory), also in several waves, us a call in lanes and in blocks: 300 x (k = 5, L = 24) 68.8, 47.5, 3600 x (4, 9) 194, 130, 1400 x (7, 24) 199, 153; two
        // blocks to an SM 600 x (8, 32) 158, 146, 1100 246, 214; 450 and 1200 x (8, 28) 128, 112, 252, 208; 1900 x (8, 9) 228, 195,
        // 2200 x (8, 4) 147, 140.  Only k = 8, L = 5 to 7 is not beyond four waves, where a piece is a wave and a bit (1800
        // and 2100 x (8, 5) 140, 144 and 158, 161, x (8, 6) 158, 162 and 178, 182; 1776 x (8, 5) 139, 130).
        pp_status st = PP_OK;
        for (int64_t p = 0; p < pieces && st == PP_OK; ++p) {
            const size_t b0 = (size_t)(B * p / pieces), n = (size_t)(B * (p + 1) / pieces) - b0;
            for (int i = 0; i < 4; ++i) {
                const size_t each = sz[i] / nB;
                std::memcpy(h + off[i] + b0 * each, static_cast<const unsigned char *>(in[i]) + b0 * each, n * each);
            }
            st = queue_exact_batch((int64_t)n, L, k, reinterpret_cast<uint64_t *>(h + off[0]) + b0 * L,
                         reinterpret_cast<uint64_t *>(h + off[1]) + b0 * L, reinterpret_cast<uint64_t *>(h + off[2]) + b0 * k,
                         reinterpret_cast<uint32_t *>(h + off[3]) + b0 * k * k, reinterpret_cast<double *>(h + off[4]) + b0,
                         reinterpret_cast<int32_t *>(h + off[5]) + b0, reinterpret_cast<int32_t *>(h + off[6]) + b0 * (k - 1),
                         reinterpret_cast<int32_t *>(h + off[7]) + b0 * k, reinterpret_cast<int8_t *>(h + off[8]) + b0,
                                   sms, route, p > 0, nullptr);
        }
        const cudaError_t e = cudaStreamSynchronize(nullptr);
        if (st != PP_OK) return st;
        if (e != cudaSuccess) return from_cuda(e);
        void *out[5] = {beta_ms, m, cuts, placement, status};
        const size_t n[5] = {sz[4], sz[5], nB * (size_t)(k - 1) * 4, sz[7], sz[8]};
        for (int i = 0; i < 5; ++i)
            if (out[i] && n[i]) std::memcpy(out[i], h + off[4 + i], n[i]);
        return PP_OK;
    }
    unsigned char *buf = nullptr;
    cudaStream_t s = nullptr;
    PP_CUDA(staging_alloc(reinterpret_cast<void **>(&buf), off[9], s));
    const void *src[4] = {out_bits, mem, node_mem, bw};
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 4 && e == cudaSuccess; ++i)
        e = cudaMemcpyAsync(buf + off[i], src[i], sz[i], cudaMemcpyHostToDevice, s);
    pp_status st = PP_OK;
    if (e == cudaSuccess)
        st = run_dev(B, L, k, reinterpret_cast<uint64_t *>(buf + off[0]),
                     reinterpret_cast<uint64_t *>(buf + off[1]), reinterpret_cast<uint64_t *>(buf + off[2]),
                     reinterpret_cast<uint32_t *>(buf + off[3]), reinterpret_cast<double *>(buf + off[4]),
                     reinterpret_cast<int32_t *>(buf + off[5]), reinterpret_cast<int32_t *>(buf + off[6]),
                     reinterpret_cast<int32_t *>(buf + off[7]), reinterpret_cast<int8_t *>(buf + off[8]), s);
    if (e == cudaSuccess && st == PP_OK) {
        void *dst[5] = {beta_ms, m, cuts, placement, status};
        for (int i = 0; i < 5 && e == cudaSuccess; ++i) {
            if (!dst[i]) continue;
            size_t n = (i == 2) ? nB * (size_t)(k - 1) * 4 : sz[4 + i];
            if (n) e = cudaMemcpyAsync(dst[i], buf + off[4 + i], n, cudaMemcpyDeviceToHost, s);
        }
    }
    cudaFreeAsync(buf, s);
    cudaError_t e2 = cudaStreamSynchronize(s);
    if (st != PP_OK) return st;
    if (e != cudaSuccess) return from_cuda(e);
    return from_cuda(e2);
}

pp_status pp_solve_exact_batch(int64_t B, int32_t L, int32_t k, const uint64_t *out_bits,
                               const uint64_t *mem, const uint64_t *node_mem, const uint32_t *bw,
                               double *beta_ms, int32_t *m, int32_t *cuts, int32_t *placement,
                               int8_t *status)
{
    return batch_from_host(pp_solve_exact_batch_dev, true, B, L, k, out_bits, mem, node_mem, bw, beta_ms, m, cuts,
                           placement, status);
}

pp_status pp_greedy_batch_dev(int64_t B, int32_t L, int32_t k, const uint64_t *out_bits,
                              const uint64_t *mem, const uint64_t *node_mem, const uint32_t *bw,
                              double *beta_ms, int32_t *m, int32_t *cuts, int32_t *placement,
                              int8_t *status, void *cuda_stream)
{
    if (B < 0 || L < 1 || k < 1) return PP_ERR_ARG;
    if (L > PP_MAX_L || k > PP_MAX_K) return PP_ERR_LIMIT;
    if (B == 0) return PP_OK;
    if (!out_bits || !mem || !node_mem || !bw || !beta_ms || !m || !placement || !status ||
        (!cuts && k > 1))
        return PP_ERR_ARG;
    PP_CUDA(launch_greedy(B, L, k, out_bits, mem, node_mem, bw, beta_ms, m, cuts, placement, status,
                          static_cast<cudaStream_t>(cuda_stream)));
    return PP_OK;
}

pp_status pp_greedy_batch(int64_t B, int32_t L, int32_t k, const uint64_t *out_bits,
                          const uint64_t *mem, const uint64_t *node_mem, const uint32_t *bw,
                          double *beta_ms, int32_t *m, int32_t *cuts, int32_t *placement, int8_t *status)
{
    return batch_from_host(pp_greedy_batch_dev, false, B, L, k, out_bits, mem, node_mem, bw, beta_ms, m, cuts,
                           placement, status);
}

pp_status pp_partition_minsum_batch_dev(int64_t B, int32_t L, const uint64_t *cut_weight, const uint64_t *mem,
                                        const uint64_t *kappa, int32_t cap_seg, uint64_t *cost, int32_t *m,
                                        int32_t *cuts, uint64_t *sizes, int8_t *status, void *cuda_stream)
{
    if (B < 0 || L < 1 || cap_seg < 0) return PP_ERR_ARG;
    if (L > PP_MAX_L) return PP_ERR_LIMIT;
    if (B == 0) return PP_OK;
    if (!cut_weight || !mem || !kappa || !cost || !m || !status || (!cuts && cap_seg > 0)) return PP_ERR_ARG;
    PP_CUDA(launch_partition_minsum(B, L, cap_seg, cut_weight, mem, kappa, cost, m, cuts, sizes, status,
                                    static_cast<cudaStream_t>(cuda_stream)));
    return PP_OK;
}

pp_status pp_partition_minsum_batch(int64_t B, int32_t L, const uint64_t *cut_weight, const uint64_t *mem,
                                    const uint64_t *kappa, int32_t cap_seg, uint64_t *cost, int32_t *m,
                                    int32_t *cuts, uint64_t *sizes, int8_t *status)
{
    if (B < 0 || L < 1 || cap_seg < 0) return PP_ERR_ARG;
    if (L > PP_MAX_L) return PP_ERR_LIMIT;
    if (B == 0) return PP_OK;
    if (!cut_weight || !mem || !kappa || !cost || !m || !status || (!cuts && cap_seg > 0)) return PP_ERR_ARG;
    const size_t nB = (size_t)B, rows = nB * (size_t)std::max(cap_seg, 1);
    const size_t sz[8] = {nB * L * 8, nB * L * 8, nB * 8, nB * 8, nB * 4, rows * 4, rows * 8, nB};
    size_t off[9];
    off[0] = 0;
    for (int i = 0; i < 8; ++i) off[i + 1] = align_up(off[i] + sz[i], 16);
    if (off[8] <= sizeof(HostSlot::small)) {
        // a few chains: the kernel reads and writes page-locked memory, nothing is copied or allocated on
        // the device (every word crosses the bus once)
        SlotLease lease;
        if (!lease.slot) return PP_ERR_NOMEM;
        unsigned char *h = lease.slot->small;
        uint64_t *o_cost = reinterpret_cast<uint64_t *>(h + off[3]), *o_sizes = reinterpret_cast<uint64_t *>(h + off[6]);
        int32_t *o_m = reinterpret_cast<int32_t *>(h + off[4]), *o_cuts = reinterpret_cast<int32_t *>(h + off[5]);
        int8_t *o_status = reinterpret_cast<int8_t *>(h + off[7]);
        if (partition_as_params(B, L)) {
            PP_CUDA(launch_partition_params(B, L, cap_seg, cut_weight, mem, kappa, o_cost, o_m, o_cuts, o_sizes, o_status, nullptr));
        } else {
            const void *in[3] = {cut_weight, mem, kappa};
            for (int i = 0; i < 3; ++i) std::memcpy(h + off[i], in[i], sz[i]);
            PP_CUDA(launch_partition_minsum(B, L, cap_seg, reinterpret_cast<uint64_t *>(h + off[0]),
                                            reinterpret_cast<uint64_t *>(h + off[1]), reinterpret_cast<uint64_t *>(h + off[2]),
                                            o_cost, o_m, o_cuts, o_sizes, o_status, nullptr));
        }
        PP_CUDA(cudaStreamSynchronize(nullptr));
        void *out[5] = {cost, m, cuts, sizes, status};
        const size_t n[5] = {sz[3], sz[4], nB * (size_t)cap_seg * 4, nB * (size_t)cap_seg * 8, sz[7]};
        for (int i = 0; i < 5; ++i)
            if (out[i] && n[i]) std::memcpy(out[i], h + off[3 + i], n[i]);
        return PP_OK;
    }
    for (int i = 0; i < 8; ++i) off[i + 1] = align_up(off[i] + sz[i], 256);
    unsigned char *buf = nullptr;
    cudaStream_t s = nullptr;
    PP_CUDA(staging_alloc(reinterpret_cast<void **>(&buf), off[8], s));
    const void *src[3] = {cut_weight, mem, kappa};
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 3 && e == cudaSuccess; ++i)
        e = cudaMemcpyAsync(buf + off[i], src[i], sz[i], cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = launch_partition_minsum(B, L, cap_seg, reinterpret_cast<uint64_t *>(buf + off[0]),
                                    reinterpret_cast<uint64_t *>(buf + off[1]), reinterpret_cast<uint64_t *>(buf + off[2]),
                                    reinterpret_cast<uint64_t *>(buf + off[3]), reinterpret_cast<int32_t *>(buf + off[4]),
                                    reinterpret_cast<int32_t *>(buf + off[5]), reinterpret_cast<uint64_t *>(buf + off[6]),
                                    reinterpret_cast<int8_t *>(buf + off[7]), s);
    if (e == cudaSuccess) {
        void *dst[5] = {cost, m, cuts, sizes, status};
        const size_t n[5] = {sz[3], sz[4], nB * (size_t)cap_seg * 4, nB * (size_t)cap_seg * 8, sz[7]};
        for (int i = 0; i < 5 && e == cudaSuccess; ++i)
            if (dst[i] && n[i]) e = cudaMemcpyAsync(dst[i], buf + off[3 + i], n[i], cudaMemcpyDeviceToHost, s);
    }
    cudaFreeAsync(buf, s);
    cudaError_t e2 = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return from_cuda(e);
    return from_cuda(e2);
}

pp_status pp_kpath_colour_batch_dev(int32_t n, const uint32_t *bw_kbps, int64_t Q, int32_t kk,
                                    const uint32_t *threshold, const int32_t *start, const int32_t *end,
                                    const uint64_t *alive, const uint8_t *colours, uint8_t *found, int32_t *path,
                                    void *cuda_stream)
{
    if (n < 1 || kk < 1 || Q < 0) return PP_ERR_ARG;
    if (n > PP_KPATH_MAX_N || kk > PP_KPATH_MAX_K) return PP_ERR_LIMIT;
    if (Q == 0) return PP_OK;
    if (!bw_kbps || !threshold || !start || !end || !alive || !colours || !found || !path) return PP_ERR_ARG;
    PP_CUDA(launch_kpath(n, kk, Q, bw_kbps, threshold, start, end, reinterpret_cast<const unsigned long long *>(alive),
                         colours, found, path, static_cast<cudaStream_t>(cuda_stream)));
    return PP_OK;
}

pp_status pp_kpath_colour_batch(int32_t n, const uint32_t *bw_kbps, int64_t Q, int32_t kk, const uint32_t *threshold,
                                const int32_t *start, const int32_t *end, const uint64_t *alive,
                                const uint8_t *colours, uint8_t *found, int32_t *path)
{
    if (n < 1 || kk < 1 || Q < 0) return PP_ERR_ARG;
    if (n > PP_KPATH_MAX_N || kk > PP_KPATH_MAX_K) return PP_ERR_LIMIT;
    if (Q == 0) return PP_OK;
    if (!bw_kbps || !threshold || !start || !end || !alive || !colours || !found || !path) return PP_ERR_ARG;
    const size_t nQ = (size_t)Q;
    const size_t sz[9] = {(size_t)n * n * 4, nQ * 4, nQ * 4, nQ * 4, nQ * 8, nQ * n, nQ, nQ * kk * 4, 0};
    size_t off[9];
    off[0] = 0;
    for (int i = 0; i < 8; ++i) off[i + 1] = align_up(off[i] + sz[i], 256);
    unsigned char *buf = nullptr;
    cudaStream_t s = nullptr;
    PP_CUDA(staging_alloc(reinterpret_cast<void **>(&buf), off[8], s));
    const void *src[6] = {bw_kbps, threshold, start, end, alive, colours};
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 6 && e == cudaSuccess; ++i)
        e = cudaMemcpyAsync(buf + off[i], src[i], sz[i], cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = launch_kpath(n, kk, Q, reinterpret_cast<uint32_t *>(buf + off[0]), reinterpret_cast<uint32_t *>(buf + off[1]),
                         reinterpret_cast<int32_t *>(buf + off[2]), reinterpret_cast<int32_t *>(buf + off[3]),
                         reinterpret_cast<unsigned long long *>(buf + off[4]), buf + off[5], buf + off[6],
                         reinterpret_cast<int32_t *>(buf + off[7]), s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(found, buf + off[6], sz[6], cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(path, buf + off[7], sz[7], cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(buf, s);
    cudaError_t e2 = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return from_cuda(e);
    return from_cuda(e2);
}

// The whole stage as one launch (pp_match.cu): one copy up, the result in page-locked memory.
constexpr size_t kMatchSharedBytes = 224 * 1024;
static pp_status match_one_launch(int32_t n, const uint32_t *bw, int32_t n_cuts, int32_t trials, const uint32_t *draws,
                                  const std::vector<MatchRun> &order, int kk, int32_t *nodes, uint32_t *cut_threshold,
                                  cudaStream_t s)
{
    int dev = 0, sms = 0;
    PP_CUDA(cudaGetDevice(&dev));
    PP_CUDA(multiprocessors(dev, &sms));
    SlotLease lease;
    if (!lease.slot) return PP_ERR_NOMEM;
    HostSlot &slot = *lease.slot;
    MatchDev d;
    d.n = n; d.n_cuts = n_cuts; d.n_runs = (int)order.size(); d.trials = trials; d.kk = kk;
    d.bw = d.draws = nullptr;
    d.runs = nullptr;
    d.records = slot.records;
    d.half = slot.half;
    d.stride = sms;
    d.out = &slot.match;
    slot.match.status = (int)PP_ERR_CUDA;
    slot.match.bounds = 0;
    const size_t nn = (size_t)n * n, at = match_runs_at(n, trials), words = at + order.size() * (sizeof(MatchRun) / 4);
    std::unique_ptr<uint32_t[]> in(new uint32_t[words]);
    std::memcpy(in.get(), bw, nn * 4);
    std::memcpy(in.get() + nn, draws, (size_t)trials * n * 4);
    std::memcpy(in.get() + at, order.data(), order.size() * sizeof(MatchRun));
    uint32_t *buf = nullptr;
    cudaError_t e = cudaSuccess;
    if (!match_as_params(words)) {
        PP_CUDA(staging_alloc(reinterpret_cast<void **>(&buf), words * 4, s));
        d.bw = buf;
        d.draws = buf + nn;
        d.runs = reinterpret_cast<MatchRun *>(buf + at);
        e = cudaMemcpyAsync(buf, in.get(), words * 4, cudaMemcpyHostToDevice, s);
    }
    if (e == cudaSuccess) e = launch_match(d, in.get(), words, s);
    if (buf) cudaFreeAsync(buf, s);
    const cudaError_t e2 = cudaStreamSynchronize(s);
    slot.half ^= 1;
    if (e != cudaSuccess || e2 != cudaSuccess || slot.match.status == (int)PP_ERR_CUDA) {
        cudaMemset(slot.records, 0, match_record_bytes(sms));  // not cleared for the next call
        cudaStreamSynchronize(nullptr);
        return e != cudaSuccess ? from_cuda(e) : e2 != cudaSuccess ? from_cuda(e2) : PP_ERR_CUDA;
    }
    const MatchOut &got = slot.match;
    if (got.bounds) return PP_ERR_CUDA;
    std::copy(got.nodes, got.nodes + n_cuts + 1, nodes);
    if (cut_threshold) std::copy(got.threshold, got.threshold + n_cuts, cut_threshold);
    return static_cast<pp_status>(got.status);
}

// Placement stage of the paper's heuristic (Section 3.2.2, Algorithms 2 and 3): classes of the cut sizes
// and the order of their runs on the host, the paths on the device.  Without the one-launch kernel every
// run is a bisection over the sorted link bandwidths whose probes are batches of colour-coding k-path
// queries (one query per trial colouring).
pp_status pp_kpath_matching(int32_t n, const uint32_t *bw_kbps, int32_t n_cuts, const uint64_t *sizes,
                            int32_t n_classes, int32_t trials, const uint32_t *draws, int32_t *nodes,
                            uint32_t *cut_threshold, void *cuda_stream)
{
    if (n < 1 || n_cuts < 0 || n_classes < 1 || trials < 1) return PP_ERR_ARG;
    if (!bw_kbps || !draws || !nodes || (!sizes && n_cuts > 0)) return PP_ERR_ARG;
    if (n > PP_KPATH_MAX_N) return PP_ERR_LIMIT;
    const int m = n_cuts + 1;
    for (int j = 0; j < m; ++j) nodes[j] = -1;
    if (cut_threshold)
        for (int j = 0; j < n_cuts; ++j) cut_threshold[j] = 0;
    if (n_cuts == 0) {
        nodes[0] = 0;
        return PP_OK;
    }
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    try {
        // classes of the sizes by rank among the distinct values, highest class served first
        std::vector<uint64_t> distinct(sizes, sizes + n_cuts);
        std::sort(distinct.begin(), distinct.end());
        distinct.erase(std::unique(distinct.begin(), distinct.end()), distinct.end());
        std::vector<int> cls(n_cuts);
        for (int j = 0; j < n_cuts; ++j) {
            const size_t rank = std::lower_bound(distinct.begin(), distinct.end(), sizes[j]) - distinct.begin();
            cls[j] = (int)(rank * (size_t)n_classes / distinct.size());
        }
        // serving order: classes from the highest down, within a class maximal runs of cuts, longest first,
        // equal lengths by first cut
        std::vector<MatchRun> order;
        int longest = 0;
        for (int X = n_classes - 1; X >= 0; --X) {
            const size_t from = order.size();
            for (int i = 0; i < n_cuts;) {
                if (cls[i] != X) { ++i; continue; }
                int j = i;
                while (j < n_cuts && cls[j] == X) ++j;
                order.push_back({i, j - i});
                longest = std::max(longest, j - i);
                i = j;
            }
            std::stable_sort(order.begin() + (long)from, order.end(),
                             [](const MatchRun &a, const MatchRun &b) { return a.cuts > b.cuts; });
        }
        // tables of bottlenecks that fit a block's shared memory: one launch for the whole stage.  Longer
        // runs (paths of ten vertices and more on large graphs) and plans with more cuts than the kernel's
        // records hold are bisected with a launch per probe.
        if (n_cuts < 64 && longest < PP_KPATH_MAX_K && match_smem_bytes(n, longest + 1) <= kMatchSharedBytes)
            return match_one_launch(n, bw_kbps, n_cuts, trials, draws, order, longest + 1, nodes, cut_threshold, s);
        // link bandwidths in descending order: the thresholds Algorithm 2 bisects over
        std::vector<uint32_t> edge_list;
        for (int v = 0; v < n; ++v)
            for (int w = 0; w < n; ++w)
                if (v != w && bw_kbps[v * n + w] > 0) edge_list.push_back(bw_kbps[v * n + w]);
        std::sort(edge_list.begin(), edge_list.end(), std::greater<uint32_t>());
        // device buffers for one batch of queries (the longest path decides their size)
        const size_t T = (size_t)trials;
        const size_t sz[8] = {(size_t)n * n * 4, T * 4, T * 4, T * 4, T * 8, T * n, T, T * PP_KPATH_MAX_K * 4};
        size_t off[9];
        off[0] = 0;
        for (int i = 0; i < 8; ++i) off[i + 1] = align_up(off[i] + sz[i], 256);
        unsigned char *buf = nullptr;
        PP_CUDA(staging_alloc(reinterpret_cast<void **>(&buf), off[8], s));
        struct Release {
            unsigned char *b; cudaStream_t st;
            ~Release() { cudaFreeAsync(b, st); cudaStreamSynchronize(st); }
        } release{buf, s};
        PP_CUDA(cudaMemcpyAsync(buf + off[0], bw_kbps, sz[0], cudaMemcpyHostToDevice, s));
        std::vector<uint32_t> h_thr(T);
        std::vector<int32_t> h_start(T), h_end(T), h_path(T * PP_KPATH_MAX_K);
        std::vector<uint64_t> h_alive(T);
        std::vector<uint8_t> h_col(T * n), h_found(T);
        uint64_t used = 0;
        {
            for (const MatchRun &run : order) {
                const int first = run.first, cuts = run.cuts, kk = cuts + 1;
                if (kk > PP_KPATH_MAX_K) return PP_ERR_LIMIT;
                const int sv = nodes[first], uv = nodes[first + cuts];
                uint64_t alive = ~used;
                if (sv >= 0) alive |= 1ull << sv;
                if (uv >= 0) alive |= 1ull << uv;
                for (size_t t = 0; t < T; ++t) {
                    h_start[t] = sv;
                    h_end[t] = uv;
                    h_alive[t] = alive;
                    for (int v = 0; v < n; ++v)
                        h_col[t * n + v] = (uint8_t)(((uint64_t)draws[t * n + v] * (uint64_t)kk) >> 32);
                }
                PP_CUDA(cudaMemcpyAsync(buf + off[2], h_start.data(), sz[2], cudaMemcpyHostToDevice, s));
                PP_CUDA(cudaMemcpyAsync(buf + off[3], h_end.data(), sz[3], cudaMemcpyHostToDevice, s));
                PP_CUDA(cudaMemcpyAsync(buf + off[4], h_alive.data(), sz[4], cudaMemcpyHostToDevice, s));
                PP_CUDA(cudaMemcpyAsync(buf + off[5], h_col.data(), sz[5], cudaMemcpyHostToDevice, s));
                size_t low = 0, high = edge_list.size();
                std::vector<int32_t> best_path;
                uint32_t best_t = 0;
                while (low < high) {
                    const size_t median = (low + high) / 2;
                    std::fill(h_thr.begin(), h_thr.end(), edge_list[median]);
                    PP_CUDA(cudaMemcpyAsync(buf + off[1], h_thr.data(), sz[1], cudaMemcpyHostToDevice, s));
                    PP_CUDA(launch_kpath(n, kk, (int64_t)T, reinterpret_cast<uint32_t *>(buf + off[0]),
                                         reinterpret_cast<uint32_t *>(buf + off[1]), reinterpret_cast<int32_t *>(buf + off[2]),
                                         reinterpret_cast<int32_t *>(buf + off[3]),
                                         reinterpret_cast<unsigned long long *>(buf + off[4]), buf + off[5], buf + off[6],
                                         reinterpret_cast<int32_t *>(buf + off[7]), s));
                    PP_CUDA(cudaMemcpyAsync(h_found.data(), buf + off[6], T, cudaMemcpyDeviceToHost, s));
                    PP_CUDA(cudaMemcpyAsync(h_path.data(), buf + off[7], T * kk * 4, cudaMemcpyDeviceToHost, s));
                    PP_CUDA(cudaStreamSynchronize(s));
                    size_t hit = T;
                    for (size_t t = 0; t < T && hit == T; ++t)
                        if (h_found[t]) hit = t;  // the first colouring that finds a path
                    if (hit == T) {
                        low = median + 1;
                    } else {
                        high = median;
                        best_path.assign(h_path.begin() + hit * kk, h_path.begin() + (hit + 1) * kk);
                        best_t = edge_list[median];
                    }
                }
                if (best_path.empty()) {
                    for (int j = 0; j < m; ++j) nodes[j] = -1;
                    return PP_INFEASIBLE;
                }
                for (int i = 0; i < kk; ++i) {
                    nodes[first + i] = best_path[i];
                    used |= 1ull << best_path[i];
                }
                if (cut_threshold)
                    for (int i = 0; i < cuts; ++i) cut_threshold[first + i] = best_t;
            }
        }
    } catch (const std::bad_alloc &) {
        return PP_ERR_NOMEM;
    }
    return PP_OK;
}

pp_status pp_solve_exact_compute(int32_t L, const uint64_t *layer_out_bits, const uint64_t *layer_mem_bytes,
                                 const uint64_t *layer_work, int32_t k, const uint64_t *node_mem_bytes,
                                 const uint32_t *bw_kbps, const uint32_t *node_speed, double *beta_ms, int32_t *m,
                                 int32_t *cuts, int32_t *placement)
{
    if (!beta_ms || !m || !placement || (!cuts && k > 1) || !layer_work || !node_speed) return PP_ERR_ARG;
    pp_status st = validate(L, layer_out_bits, layer_mem_bytes, k, node_mem_bytes, bw_kbps);
    if (st != PP_OK) return st;
    if (L > PP_COMPUTE_MAX_L || k > PP_COMPUTE_MAX_K) return PP_ERR_LIMIT;
    for (int i = 0; i < L; ++i)
        if (layer_work[i] >= PP_MAX_BITS) return PP_ERR_LIMIT;
    PruneDev q{};
    q.L = L; q.k = k; q.Lp = prune_row_pad(L, k);
    uint64_t M[PP_COMPUTE_MAX_L + 1], Wp[PP_COMPUTE_MAX_L + 1];
    M[0] = Wp[0] = 0;
    for (int i = 0; i < L; ++i) {
        M[i + 1] = M[i] + layer_mem_bytes[i];
        Wp[i + 1] = Wp[i] + layer_work[i];
    }
    const PruneHost h{layer_out_bits, M, node_mem_bytes, bw_kbps, Wp, node_speed};
    double lo = std::numeric_limits<double>::max(), hi = 0.0;
    quotient_range(L, layer_out_bits, k * k, bw_kbps, &lo, &hi);
    quotient_range(L, layer_work, k, node_speed, &lo, &hi);   // shortest run of layers: one
    quotient_range(1, Wp + L, k, node_speed, &lo, &hi);       // longest: all of them
    prune_key_range(hi > 0.0 ? lo : 1.0, hi > 0.0 ? hi : 1.0, &q);
    prune_node_bounds(node_mem_bytes, M[L], &q);
    // all nodes together cannot do all the work in less (the quotients' roundings are far below the margin)
    double speeds = 0.0;
    for (int v = 0; v < k; ++v) speeds += (double)node_speed[v];
    if (speeds > 0.0) {
        const double floor_ms = (double)Wp[L] / speeds * (1.0 - 1e-9);
        std::memcpy(&q.key_floor, &floor_ms, sizeof floor_ms);
    }
    int dev = 0, sms = 0;
    PP_CUDA(cudaGetDevice(&dev));
    PP_CUDA(multiprocessors(dev, &sms));
    cudaStream_t s = nullptr;
    HostSlot *slot = g_slots.take();
    if (!slot) return PP_ERR_NOMEM;
    const size_t head = align_up((size_t)k * L * q.Lp * 4, 256);
    cudaError_t e = cudaSuccess;
    // pooled scratch for a frontier that stays small, room for every state if it does not
    const unsigned long long limits[2] = {kSparseScratchBytes, ~0ull};
    for (int pass = 0; pass < 2 && e == cudaSuccess; ++pass) {
        unsigned char *buf = nullptr;
        if (!prune_in_shared(q, h)) {
            const size_t table = sparse_bytes(k, q.Lp, limits[pass]);
            e = staging_alloc(reinterpret_cast<void **>(&buf), head + table, s);
            if (e != cudaSuccess) break;
            q.seg = reinterpret_cast<uint32_t *>(buf);
            bind_sparse(q, buf + head, table);
        }
        q.ctl = slot->ctl;
        q.out = &slot->sol;
        q.note = &slot->note;
        e = launch_prune(q, h, sms, s);
        if (buf) cudaFreeAsync(buf, s);
        const cudaError_t e2 = cudaStreamSynchronize(s);
        if (e == cudaSuccess) e = e2;
        if (e == cudaSuccess && !slot->note.dense) break;
    }
    const pp_solution sol = slot->sol;
    const int32_t dense = slot->note.dense;
    t_thresholds = e == cudaSuccess ? slot->note.thresholds : 0;
    g_slots.give(slot);
    if (e != cudaSuccess) return from_cuda(e);
    if (dense != 0 || (sol.status != PP_OK && sol.status != PP_INFEASIBLE)) return PP_ERR_CUDA;
    *beta_ms = sol.beta_ms;
    *m = sol.m;
    for (int j = 0; j < k - 1; ++j) cuts[j] = sol.cuts[j];
    for (int j = 0; j < k; ++j) placement[j] = sol.placement[j];
    return static_cast<pp_status>(sol.status);
}

pp_status pp_debug_minmax_rate(int32_t op, int32_t iters, double *warp_instr_per_clk_per_sm)
{
    if (!warp_instr_per_clk_per_sm || op < 0 || op > 2 || iters < 1 || iters > (1 << 20)) return PP_ERR_ARG;
    int dev = 0, sms = 0;
    PP_CUDA(cudaGetDevice(&dev));
    PP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    unsigned char *buf = nullptr;
    PP_CUDA(cudaMalloc(reinterpret_cast<void **>(&buf), (size_t)sms * 8 + 256));
    long long *cycles = reinterpret_cast<long long *>(buf);
    uint32_t *sink = reinterpret_cast<uint32_t *>(buf + (size_t)sms * 8);
    std::vector<long long> h;
    cudaError_t e = cudaSuccess;
    try {
        h.resize(sms);
    } catch (const std::bad_alloc &) {
        cudaFree(buf);
        return PP_ERR_NOMEM;
    }
    for (int rep = 0; rep < 3 && e == cudaSuccess; ++rep) e = launch_probe(op, iters, sms, cycles, sink, nullptr);
    if (e == cudaSuccess) e = cudaMemcpy(h.data(), cycles, (size_t)sms * 8, cudaMemcpyDeviceToHost);
    cudaFree(buf);
    if (e != cudaSuccess) return from_cuda(e);
    std::sort(h.begin(), h.end());
    const long long med = h[sms / 2];
    if (med <= 0) return PP_ERR_CUDA;
    *warp_instr_per_clk_per_sm = probe_instr_per_block(iters) / (double)med;
    return PP_OK;
}

pp_status pp_debug_fail_alloc(int32_t nth)
{
    if (nth < 0) return PP_ERR_ARG;
    g_fail_alloc_countdown.store(nth);
    return PP_OK;
}

pp_status pp_debug_starve(int32_t polls)
{
    if (polls < 0) return PP_ERR_ARG;
    g_starved_polls.store(polls);
    return PP_OK;
}

pp_status pp_debug_late(int32_t block, int32_t polls)
{
    if (block < 0 || polls < 0) return PP_ERR_ARG;
#ifdef PP_DEBUG_BOUNDS
    g_late.store(polls ? (uint64_t)block << 32 | (uint32_t)polls : 0);
    return PP_OK;
#else
    return PP_ERR_LIMIT;
#endif
}

pp_status pp_debug_thresholds(int32_t *outcome)
{
    if (!outcome) return PP_ERR_ARG;
    *outcome = t_thresholds;
    return PP_OK;
}

pp_status pp_debug_bounds_checks(int32_t kernel, uint64_t *n)
{
    unsigned long long (*const of[5])() = {prune_checks, batch_checks, match_checks, eval_checks, random_checks};
    if (!n || kernel < 0 || kernel >= 5) return PP_ERR_ARG;
    *n = of[kernel]();
    return PP_OK;
}

pp_status pp_debug_quotients(int64_t n, const uint64_t *bits, const uint32_t *kbps, double *by_reciprocal, double *divided)
{
    if (n < 0 || n > (int64_t)1 << 28) return PP_ERR_ARG;
    if (n == 0) return PP_OK;
    if (!bits || !kbps || !by_reciprocal || !divided) return PP_ERR_ARG;
    for (int64_t i = 0; i < n; ++i)
        if (bits[i] >= PP_MAX_BITS || kbps[i] >= PP_MAX_KBPS || kbps[i] == 0) return PP_ERR_LIMIT;
    const size_t each = (size_t)n * 8;
    unsigned char *buf = nullptr;
    PP_CUDA(staging_alloc(reinterpret_cast<void **>(&buf), 4 * each, nullptr));
    uint64_t *d_bits = reinterpret_cast<uint64_t *>(buf);
    double *d_out = reinterpret_cast<double *>(buf + each);
    uint32_t *d_kbps = reinterpret_cast<uint32_t *>(buf + 3 * each);
    cudaError_t e = cudaMemcpyAsync(d_bits, bits, each, cudaMemcpyHostToDevice, nullptr);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_kbps, kbps, each / 2, cudaMemcpyHostToDevice, nullptr);
    if (e == cudaSuccess) e = launch_quotients(n, d_bits, d_kbps, d_out, d_out + n, nullptr);
    if (e == cudaSuccess) e = cudaMemcpyAsync(by_reciprocal, d_out, each, cudaMemcpyDeviceToHost, nullptr);
    if (e == cudaSuccess) e = cudaMemcpyAsync(divided, d_out + n, each, cudaMemcpyDeviceToHost, nullptr);
    cudaFreeAsync(buf, nullptr);
    const cudaError_t e2 = cudaStreamSynchronize(nullptr);
    return from_cuda(e != cudaSuccess ? e : e2);
}

pp_status pp_debug_batch_route(int64_t B, int32_t L, int32_t k, int32_t sms, int32_t host, int32_t *threads)
{
    if (!threads || B < 1 || L < 1 || k < 1 || sms < 1) return PP_ERR_ARG;
    if (L > PP_MAX_L || k > PP_MAX_K || batch_smem_bytes(L, k) + 1024 > kBlockShared) return PP_ERR_LIMIT;
    const BatchArrays a = batch_arrays(B, L, k);
    const BatchRoute route = batch_route(B, L, k, sms, host && a.off[9] <= kPinnedBytes ? host_pieces(a) : 0);
    *threads = route.lanes ? 0 : route.warps ? 32 : batch_block_threads(route.narrow);
    return PP_OK;
}

pp_status pp_debug_mask_order(int32_t k, uint32_t *masks_out, uint32_t *level_off_out)
{
    if (!masks_out || !level_off_out || k < 1) return PP_ERR_ARG;
    if (k > PP_MAX_K) return PP_ERR_LIMIT;
    try {
        const MaskList &ml = mask_list(k);
        std::copy(ml.masks.begin(), ml.masks.end(), masks_out);
        std::copy(ml.level_off.begin(), ml.level_off.end(), level_off_out);
    } catch (const std::bad_alloc &) {
        return PP_ERR_NOMEM;
    }
    return PP_OK;
}

pp_status pp_debug_read_state_row(pp_problem *p, uint32_t mask, int32_t v, double *row_out)
{
    if (!p || !row_out || !p->solved) return PP_ERR_ARG;
    if (v < 0 || v >= p->k || mask >= (1u << p->k) || !((mask >> v) & 1u)) return PP_ERR_ARG;
    if (!p->table_whole) {  // the bounded search keeps no whole table: let the dense one write it
        pp_status st = queue_dense(p, p->d_sol);
        if (st != PP_OK) return st;
    }
    PP_CUDA(cudaStreamSynchronize(p->stream));
    const int L = p->L, U = p->U;
    std::vector<uint32_t> rk((size_t)std::max(U, 1) * L);
    std::vector<double> gu((size_t)std::max(U, 1) * L);
    if (U > 0) {
        PP_CUDA(cudaMemcpy(rk.data(), p->d.rk, (size_t)U * L * 4, cudaMemcpyDeviceToHost));
        PP_CUDA(cudaMemcpy(gu.data(), p->d.gu, (size_t)U * L * 8, cudaMemcpyDeviceToHost));
    }
    std::map<uint32_t, double> val;
    for (size_t i = 0; i < (size_t)U * L; ++i) val[rk[i]] = gu[i];
    const size_t row = ((size_t)mask * p->k + v) * p->Lpad;
    std::vector<uint32_t> raw(L);
    if (p->elem == 2) {
        std::vector<uint16_t> r16(L);
        PP_CUDA(cudaMemcpy(r16.data(), static_cast<uint16_t *>(p->d.table) + row, (size_t)L * 2,
                           cudaMemcpyDeviceToHost));
        for (int c = 0; c < L; ++c) raw[c] = r16[c] == 0xFFFFu ? 0xFFFFFFFFu : r16[c];
    } else {
        PP_CUDA(cudaMemcpy(raw.data(), static_cast<uint32_t *>(p->d.table) + row, (size_t)L * 4,
                           cudaMemcpyDeviceToHost));
    }
    for (int c = 0; c < L; ++c) {
        if (raw[c] == 0) row_out[c] = 0.0;
        else if (raw[c] == 0xFFFFFFFFu) row_out[c] = std::numeric_limits<double>::infinity();
        else {
            auto it = val.find(raw[c]);
            if (it == val.end()) return PP_ERR_CUDA;
            row_out[c] = it->second;
        }
    }
    return PP_OK;
}

}  // extern "C"
