// batch_api.cu -- host side of the batched form (sl_batch_*).
//
// Planning: each buffer goes to the first tuning-table entry that matches
// its dtype and size; buffers of one entry (a size class) and one dtype form
// a group that one persistent class kernel streams.  Buffers are cut into
// work items (item_bytes); each item owns the partial slots its kernel writes
// for it, and a buffer's items (hence its slots) are contiguous.  The CUDA
// graph -- the class kernels as parallel branches, then the per-buffer combine,
// which writes the results to page-locked host memory -- is captured once and
// replayed by sl_batch_run.
#include <algorithm>
#include <cstring>
#include <map>
#include <new>
#include <vector>

#include "k_batch.cuh"

namespace sl {
const void* batch_ldg_kernel(int dtype, int k, int cta);
const void* batch_ldg_any_kernel(int k, int cta);
const void* batch_cpasync_kernel(int dtype, int d);
const void* batch_tma_kernel(int dtype, int batch, bool biased);
cudaError_t launch_batch_combine(const BufSeg* segs, uint32_t nbuf, const WarpPartial* parts, uint32_t* err,
                                 uint32_t* next, uint32_t nclasses, sl_result* out, uint32_t* host_err,
                                 cudaStream_t s);
}  // namespace sl

namespace {

using sl::BatchItem;
using sl::BufSeg;
using sl::WarpPartial;

constexpr uint64_t TIMEOUT_NS = 2000000000ull;

int bfail(int code, const char* msg) { return sl::set_error(code, msg); }

#define B_TRY(expr, what)                                   \
    do {                                                    \
        cudaError_t e_ = (expr);                            \
        if (e_ != cudaSuccess) {                            \
            (void)cudaGetLastError();                       \
            return bfail(e_ == cudaErrorMemoryAllocation ? SL_ERR_OOM : SL_ERR_CUDA, what); \
        }                                                   \
    } while (0)

struct Group {
    int entry = -1;
    int dtype = 0;
    sl_config cfg{};
    const void* fn = nullptr;
    int block = 0;
    size_t smem = 0;
    int ctas = 0;             // persistent CTAs (resident per SM x SMs, or the entry's grid)
    uint32_t slots = 0;       // partial slots per item
    uint64_t unit = 0;        // bytes an item is a multiple of (but for a buffer's last one)
    uint64_t bytes = 0;       // of all its buffers
    std::vector<BatchItem> items;
    uint64_t part_off = 0;    // offset of this group's partials
};

// One launch of the graph: a group's class kernel, or several groups of one
// LDG entry in one kernel for mixed types.
struct Unit {
    const void* fn = nullptr;
    std::vector<int> groups;
    int ctas = 0;
    uint64_t nitems = 0;
    uint64_t item_off = 0, part_off = 0;
};

}  // namespace

struct sl_batch {
    int dev = -1;
    int n = 0;
    std::vector<int32_t> class_of;
    std::vector<Group> groups;
    BatchItem* d_items = nullptr;
    BufSeg* d_segs = nullptr;
    WarpPartial* d_parts = nullptr;
    uint32_t* d_ctrl = nullptr;  // [0]: error word; [16 + g]: item counter of group g
    sl_result* h_results = nullptr;  // page-locked, written by the combine kernel
    uint32_t* h_err = nullptr;   // page-locked copy of the error word after each run
    cudaStream_t stream = nullptr;
    std::vector<cudaStream_t> branch;
    std::vector<cudaEvent_t> branch_ev;
    cudaEvent_t fork_ev = nullptr, e0 = nullptr, e1 = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

namespace {

void release(sl_batch* b) {
    if (!b) return;
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    for (auto e : b->branch_ev) cudaEventDestroy(e);
    for (auto s : b->branch) cudaStreamDestroy(s);
    if (b->fork_ev) cudaEventDestroy(b->fork_ev);
    if (b->e0) cudaEventDestroy(b->e0);
    if (b->e1) cudaEventDestroy(b->e1);
    if (b->stream) cudaStreamDestroy(b->stream);
    cudaFree(b->d_items);
    cudaFree(b->d_segs);
    cudaFree(b->d_parts);
    cudaFree(b->d_ctrl);
    cudaFreeHost(b->h_results);
    cudaFreeHost(b->h_err);
    (void)cudaGetLastError();
    delete b;
}

// Persistent CTAs of kernel fn at group g's block shape; on failure the status,
// and what failed in *why.
int plan_ctas(const void* fn, const Group& g, int sms, int* ctas, const char** why) {
    int status = SL_OK;
    const auto cuda_ok = [&](cudaError_t e, const char* what) {
        if (e == cudaSuccess) return true;
        (void)cudaGetLastError();
        status = e == cudaErrorMemoryAllocation ? SL_ERR_OOM : SL_ERR_CUDA;
        *why = what;
        return false;
    };
    const auto infeasible = [&](const char* what) {
        *why = what;
        return SL_ERR_INFEASIBLE;
    };
    cudaFuncAttributes fa;
    if (!cuda_ok(cudaFuncGetAttributes(&fa, fn), "cudaFuncGetAttributes failed")) return status;
    if (fa.localSizeBytes > 0) return infeasible("tuning entry: kernel spills registers");
    if (g.block > fa.maxThreadsPerBlock) return infeasible("tuning entry: too many threads for this kernel");
    // (raised, never lowered: classes with other rings, and other batches, launch this kernel too)
    if (static_cast<int>(g.smem) > fa.maxDynamicSharedSizeBytes &&
        !cuda_ok(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(g.smem)),
                 "cudaFuncSetAttribute failed"))
        return status;
    int res = 0;
    if (!cuda_ok(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&res, fn, g.block, g.smem), "occupancy query failed"))
        return status;
    if (res < 1) return infeasible("tuning entry: zero occupancy");
    *ctas = g.cfg.grid > 0 ? g.cfg.grid : res * sms;
    return SL_OK;
}

// Whether a TMA class of bfloat16 buffers takes the biased sum: its serial chain
// is longer than TwoSum's, so it pays where the rings leave room for 24 consumer
// warps per SM (1,024 buffers of 16 GiB, TwoSum then biased: 16 KiB x 4 at 256
// threads, 24 warps, 2,561 -> 2,415 us on the device; 16 KiB x 2 at 128 threads, 28 warps,
// 2,465 -> 2,295; 16 KiB x 4 at 128 threads, 12 warps, 2,538 -> 2,546; 16 KiB x 5 at 256, 16 warps,
// 2,717 -> 2,724; 64 KiB x 2 at 256, 8 warps, 2,744 -> 3,122), and where a stage is
// whole groups of four vectors per thread, since every single vector drops
// the bias (16 KiB x 4 at 192 threads: 2,874 -> 3,659).
bool tma_biased(const sl_config& c, int smem_optin) {
    const int64_t ring = static_cast<int64_t>(c.stages) * c.stage_bytes;
    return smem_optin / ring * (c.cta / 32) >= 24 && c.stage_bytes / 16 % (4 * c.cta) == 0;
}

// Kernel, block shape, shared memory and persistent grid of one group.
int plan_group(Group& g, int sms, int smem_optin) {
    const sl_config& c = g.cfg;
    if (c.cta < 32 || c.cta > 1024 || (c.cta & 31)) return bfail(SL_ERR_ARG, "tuning entry: bad cta");
    if (c.target_loads) return bfail(SL_ERR_ARG, "tuning entry: the batched form runs exact fixed work (target_loads 0)");
    if (c.copies != 0 && c.copies != 1)
        return bfail(SL_ERR_ARG, "tuning entry: the batched cp.async class kernel puts one copy in each commit "
                     "group (copies must be 0 or 1)");
    switch (c.mech) {
    case SL_LDG:
        g.fn = sl::batch_ldg_kernel(g.dtype, c.k, c.cta);
        if (!g.fn) return bfail(SL_ERR_ARG, "tuning entry: no batched LDG kernel (K in {1,2,3,4,6,8,12,16}, cta 128/256/512)");
        g.block = c.cta;
        g.smem = 0;
        g.slots = 1;
        g.unit = static_cast<uint64_t>(c.k) * c.cta * 16;
        break;
    case SL_CPASYNC:
        g.fn = sl::batch_cpasync_kernel(g.dtype, c.k);
        if (!g.fn) return bfail(SL_ERR_ARG, "tuning entry: cp.async depth not in 1..8");
        g.block = c.cta;
        g.smem = static_cast<size_t>(c.k) * c.cta * 16;
        g.slots = 1;
        g.unit = static_cast<uint64_t>(c.k) * c.cta * 16;
        break;
    case SL_TMA:
        if (c.stage_bytes != 4096 && c.stage_bytes != 16384 && c.stage_bytes != 65536)
            return bfail(SL_ERR_INFEASIBLE, "tuning entry: TMA stage size not 4096/16384/65536");
        if (c.stages < SL_MIN_STAGES || c.stages > SL_MAX_STAGES) return bfail(SL_ERR_ARG, "tuning entry: TMA stages");
        if (c.cta > 992) return bfail(SL_ERR_ARG, "tuning entry: TMA consumer threads > 992");
        if (c.tma_ring != SL_RING_CTA)
            return bfail(SL_ERR_ARG, "tuning entry: the batched TMA class kernel has one ring per CTA "
                         "(tma_ring must be SL_RING_CTA)");
        // consumer threads read their last 4 vectors of a stage (1 where they
        // read fewer) into registers before releasing it
        g.fn = sl::batch_tma_kernel(g.dtype, c.stage_bytes / 16 >= 4 * c.cta ? 4 : 1, tma_biased(c, smem_optin));
        g.block = c.cta + 32;
        g.smem = static_cast<size_t>(c.stages) * c.stage_bytes;
        g.slots = c.cta / 32;
        g.unit = static_cast<uint64_t>(c.stage_bytes);
        break;
    default:
        return bfail(SL_ERR_ARG, "tuning entry: bad mech");
    }
    if (g.smem > static_cast<size_t>(smem_optin)) return bfail(SL_ERR_INFEASIBLE, "tuning entry: shared memory over the limit");
    const char* why = "";
    const int rc = plan_ctas(g.fn, g, sms, &g.ctas, &why);
    return rc ? bfail(rc, why) : SL_OK;
}

// Bytes of a group's work items, a multiple of its unit (a tile, a ring of
// cp.async chunks, or a TMA stage).
//
// A CTA should get a few items, or a class ends on a few CTAs streaming alone:
// in 1 MiB items 64 buffers of 16 MiB in all took 66 us on the device, since one
// CTA needs 44-74 us for a MiB, against 19 in items of a quarter of a CTA's share
// (three to six items per CTA measure alike, twelve 15% slower).  The TMA class
// streams on from item to item without draining its ring, but its warps write a
// partial each at the end of every item: an item is a CTA's share there, at
// least 128 KiB (64 buffers, 1 GiB, four types: 243 us in items of a sixth of the
// share, 190 so) and at most 1 MiB (16 GiB of bfloat16: 2,558 us, 2,610 in
// 256 KiB items).  256 KiB is enough for the others, whose loads or copies drain at
// the end of an item, where the other CTAs of the SM cover that: with one, two, ... CTAs
// on an SM an item may have 16, 8, ... units, up to 1 MiB (16 GiB by LDG K = 12 at 512
// threads, one CTA per SM, in 256 KiB / so: uint32 2,579 / 2,243 us, bfloat16
// 2,896 / 2,383; K = 8 at 512 FP32 2,471 / 2,342, FP8 2,684 / 2,489; twice as many units are
// 2-6% slower over 1 GiB).
constexpr uint64_t ITEM_MAX = 256ull << 10, ITEM_FEW = 1ull << 20, ITEM_TMA_MIN = 128ull << 10;
constexpr uint64_t ITEM_UNITS = 16;

uint64_t item_bytes(const Group& g, int sms) {
    const bool tma = g.cfg.mech == SL_TMA;
    const uint64_t share = g.bytes / ((tma ? 1 : 4) * static_cast<uint64_t>(g.ctas));
    const uint64_t few = ITEM_UNITS / std::max<uint64_t>(1, static_cast<uint64_t>(g.ctas / sms)) * g.unit;
    const uint64_t want = tma ? std::min(std::max(share, ITEM_TMA_MIN), ITEM_FEW)
                              : std::min(share, std::min(std::max(ITEM_MAX, few), ITEM_FEW));
    return g.unit * std::max<uint64_t>(1, want / g.unit);
}

// The graph's launches.  The LDG classes that one entry has for several types
// share a kernel where they have at most two items per CTA: a parallel branch
// costs the graph about 1.5 us, more than such a class takes, while larger
// classes want the registers (CTAs per SM) of their own type's kernel.  (64
// buffers, 16 MiB, four types in two size classes: 19.6 -> 14.0 us on the device,
// 36 -> 29 per call.)
std::vector<Unit> plan_units(const std::vector<Group>& groups, int sms) {
    std::vector<Unit> units;
    std::vector<bool> taken(groups.size(), false);
    for (size_t i = 0; i < groups.size(); ++i) {
        if (taken[i] || groups[i].items.empty()) continue;
        Unit u;
        if (groups[i].cfg.mech == SL_LDG) {
            const void* any = sl::batch_ldg_any_kernel(groups[i].cfg.k, groups[i].cfg.cta);
            const char* why = "";  // (not reported: the group has its own kernel)
            if (any && plan_ctas(any, groups[i], sms, &u.ctas, &why) == SL_OK) {
                for (size_t j = i; j < groups.size(); ++j)
                    if (groups[j].entry == groups[i].entry && !groups[j].items.empty()) {
                        u.groups.push_back(static_cast<int>(j));
                        u.nitems += groups[j].items.size();
                    }
                if (u.groups.size() > 1 && u.nitems <= 2 * static_cast<uint64_t>(u.ctas)) u.fn = any;
            }
        }
        if (!u.fn) {
            u.fn = groups[i].fn;
            u.groups.assign(1, static_cast<int>(i));
            u.ctas = groups[i].ctas;
            u.nitems = groups[i].items.size();
        }
        for (int j : u.groups) taken[j] = true;
        units.push_back(u);
    }
    return units;
}

// Everything after the argument checks; the caller releases b on failure.
int build_batch(sl_batch* b, const sl_batch_desc* descs, int32_t n, const sl_tune_entry* table, int32_t ntable,
                int sms, int optin) {
    // ---- group the buffers
    std::map<std::pair<int, int>, int> gidx;  // (entry, dtype) -> group
    for (int32_t i = 0; i < n; ++i) {
        const sl_batch_desc& d = descs[i];
        if (d.dtype < SL_U32 || d.dtype > SL_FP8_E4M3) return bfail(SL_ERR_ARG, "bad dtype in a descriptor");
        if ((d.bytes & 15u) || (reinterpret_cast<uintptr_t>(d.ptr) & 15u))
            return bfail(SL_ERR_ALIGN, "a descriptor is not 16-byte aligned or its size is not a multiple of 16");
        if (d.bytes > 0 && !d.ptr) return bfail(SL_ERR_ARG, "a descriptor has a NULL pointer");
        int e = -1;
        for (int32_t j = 0; j < ntable && e < 0; ++j)
            if ((table[j].dtype < 0 || table[j].dtype == d.dtype) && d.bytes >= table[j].min_bytes &&
                d.bytes <= table[j].max_bytes)
                e = j;
        if (e < 0) return bfail(SL_ERR_ARG, "no tuning-table entry matches a buffer");
        auto key = std::make_pair(e, static_cast<int>(d.dtype));
        if (!gidx.count(key)) {
            Group g;
            g.entry = e;
            g.dtype = d.dtype;
            g.cfg = table[e].cfg;
            int rc = plan_group(g, sms, optin);
            if (rc) return rc;
            gidx[key] = static_cast<int>(b->groups.size());
            b->groups.push_back(std::move(g));
        }
        b->class_of[i] = gidx[key];
        b->groups[gidx[key]].bytes += d.bytes;
    }

    // ---- items (buffers in order), then every launch's and group's place in the
    // item and partial arrays, then each buffer's partial slots
    std::vector<uint64_t> first(n);  // index of the buffer's first item in its group
    for (int32_t i = 0; i < n; ++i) {
        Group& g = b->groups[b->class_of[i]];
        first[i] = g.items.size();
        const uint64_t bytes = descs[i].bytes, step = item_bytes(g, sms);
        const uint8_t* p = static_cast<const uint8_t*>(descs[i].ptr);
        for (uint64_t off = 0; off < bytes; off += step) {
            BatchItem it;
            it.ptr = reinterpret_cast<const uint4*>(p + off);
            it.nvec = static_cast<uint32_t>(std::min(step, bytes - off) / 16);
            it.dtype = static_cast<uint32_t>(descs[i].dtype);
            g.items.push_back(it);
        }
    }
    std::vector<BatchItem> all;
    uint64_t slots = 0;
    std::vector<Unit> units = plan_units(b->groups, sms);
    for (Unit& u : units) {
        u.item_off = all.size();
        u.part_off = slots;
        for (int j : u.groups) {
            Group& g = b->groups[j];
            g.part_off = slots;
            all.insert(all.end(), g.items.begin(), g.items.end());
            slots += g.items.size() * g.slots;
        }
    }
    // (the kernels count items, claims past the last one included, and slots in 32 bits)
    if (slots >= (1ull << 31)) return bfail(SL_ERR_ARG, "batch too large");
    std::vector<BufSeg> segs(n);
    for (int32_t i = 0; i < n; ++i) {
        const Group& g = b->groups[b->class_of[i]];
        const uint64_t step = item_bytes(g, sms);
        segs[i].pstart = static_cast<uint32_t>(g.part_off + first[i] * g.slots);
        segs[i].pcount = static_cast<uint32_t>((descs[i].bytes + step - 1) / step * g.slots);
    }

    // ---- device tables (allocated before capture)
    const size_t nu = units.size();
    const size_t ctrl_bytes = (16 + nu) * sizeof(uint32_t);
    B_TRY(cudaMalloc(&b->d_items, std::max<size_t>(all.size(), 1) * sizeof(BatchItem)), "cudaMalloc failed");
    B_TRY(cudaMalloc(&b->d_segs, std::max<size_t>(n, 1) * sizeof(BufSeg)), "cudaMalloc failed");
    B_TRY(cudaMalloc(&b->d_parts, std::max<uint64_t>(slots, 1) * sizeof(WarpPartial)), "cudaMalloc failed");
    B_TRY(cudaMalloc(&b->d_ctrl, ctrl_bytes), "cudaMalloc failed");
    B_TRY(cudaMallocHost(&b->h_results, std::max<size_t>(n, 1) * sizeof(sl_result)), "cudaMallocHost failed");
    B_TRY(cudaMallocHost(&b->h_err, sizeof(uint32_t)), "cudaMallocHost failed");
    if (!all.empty())
        B_TRY(cudaMemcpy(b->d_items, all.data(), all.size() * sizeof(BatchItem), cudaMemcpyHostToDevice), "copy failed");
    if (n > 0) B_TRY(cudaMemcpy(b->d_segs, segs.data(), n * sizeof(BufSeg), cudaMemcpyHostToDevice), "copy failed");
    *b->h_err = 0;

    // ---- streams and events, then capture the graph
    B_TRY(cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking), "stream create failed");
    B_TRY(cudaMemsetAsync(b->d_ctrl, 0, ctrl_bytes, b->stream), "memset failed");  // every run leaves it so
    B_TRY(cudaEventCreate(&b->e0), "event create failed");
    B_TRY(cudaEventCreate(&b->e1), "event create failed");
    B_TRY(cudaEventCreateWithFlags(&b->fork_ev, cudaEventDisableTiming), "event create failed");
    for (size_t g = 0; g < nu; ++g) {
        cudaStream_t s;
        cudaEvent_t e;
        B_TRY(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking), "stream create failed");
        b->branch.push_back(s);
        B_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming), "event create failed");
        b->branch_ev.push_back(e);
    }
    B_TRY(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal), "begin capture failed");
    cudaError_t ce = cudaEventRecord(b->fork_ev, b->stream);
    for (size_t g = 0; g < nu && ce == cudaSuccess; ++g) {
        const Unit& u = units[g];
        const Group& gr = b->groups[u.groups[0]];
        ce = cudaStreamWaitEvent(b->branch[g], b->fork_ev, 0);
        if (ce != cudaSuccess) break;
        sl::BArgs a{};
        a.items = b->d_items + u.item_off;
        a.nitems = static_cast<uint32_t>(u.nitems);
        a.stage_bytes = static_cast<uint32_t>(gr.cfg.stage_bytes);
        a.next = b->d_ctrl + 16 + g;
        a.parts = b->d_parts + u.part_off;
        a.err = b->d_ctrl;
        a.timeout_ns = TIMEOUT_NS;
        a.nst = gr.cfg.mech == SL_TMA ? gr.cfg.stages : 0;
        void* args[] = {&a};
        const unsigned grid = static_cast<unsigned>(std::min<uint64_t>(u.ctas, u.nitems));
        ce = cudaLaunchKernel(u.fn, dim3(grid), dim3(gr.block), args, gr.smem, b->branch[g]);
        if (ce == cudaSuccess) ce = cudaEventRecord(b->branch_ev[g], b->branch[g]);
        if (ce == cudaSuccess) ce = cudaStreamWaitEvent(b->stream, b->branch_ev[g], 0);
    }
    if (ce == cudaSuccess)
        ce = sl::launch_batch_combine(b->d_segs, static_cast<uint32_t>(n), b->d_parts, b->d_ctrl, b->d_ctrl + 16,
                                      static_cast<uint32_t>(nu), b->h_results, b->h_err, b->stream);
    cudaGraph_t graph = nullptr;
    const cudaError_t ee = cudaStreamEndCapture(b->stream, &graph);
    b->graph = graph;
    if (ce != cudaSuccess || ee != cudaSuccess) {
        (void)cudaGetLastError();
        return bfail(SL_ERR_CUDA, "capturing the batch graph failed");
    }
    B_TRY(cudaGraphInstantiate(&b->exec, b->graph, 0), "graph instantiation failed");
    return SL_OK;
}

}  // namespace

extern "C" {

int sl_batch_create(const sl_batch_desc* descs, int32_t n, const sl_tune_entry* table, int32_t ntable,
                    sl_batch** out) {
    if (!out) return bfail(SL_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (n < 0 || (n > 0 && !descs) || ntable < 1 || !table) return bfail(SL_ERR_ARG, "bad batch arguments");
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return bfail(SL_ERR_NODEV, "no CUDA device");
    }
    int sms = 0, optin = 0;
    B_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "device query failed");
    B_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev), "device query failed");
    sl_batch* b = new (std::nothrow) sl_batch();
    if (!b) return bfail(SL_ERR_OOM, "out of host memory");
    b->dev = dev;
    b->n = n;
    b->class_of.assign(n, -1);
    const int rc = build_batch(b, descs, n, table, ntable, sms, optin);
    if (rc) {
        release(b);
        return rc;
    }
    *out = b;
    return SL_OK;
}

int sl_batch_run(sl_batch* b, sl_result* per_buffer, uint64_t* total_ns) {
    if (!b) return bfail(SL_ERR_ARG, "batch is NULL");
    B_TRY(cudaEventRecord(b->e0, b->stream), "event record failed");
    B_TRY(cudaGraphLaunch(b->exec, b->stream), "graph launch failed");
    B_TRY(cudaEventRecord(b->e1, b->stream), "event record failed");
    B_TRY(cudaStreamSynchronize(b->stream), "batch run failed");
    float ms = 0.0f;
    B_TRY(cudaEventElapsedTime(&ms, b->e0, b->e1), "event timing failed");
    if (total_ns) *total_ns = static_cast<uint64_t>(static_cast<double>(ms) * 1e6 + 0.5);
    const int st = *b->h_err ? SL_ERR_TIMEOUT : SL_OK;
    if (per_buffer && b->n > 0) {
        std::memcpy(per_buffer, b->h_results, b->n * sizeof(sl_result));
        if (st != SL_OK)
            for (int i = 0; i < b->n; ++i) per_buffer[i].status = st;
    }
    if (st != SL_OK) return bfail(st, "a bounded device wait timed out");
    return SL_OK;
}

int sl_batch_info(const sl_batch* b, int32_t* nclasses, int32_t* class_of_buffer) {
    if (!b) return bfail(SL_ERR_ARG, "batch is NULL");
    if (nclasses) *nclasses = static_cast<int32_t>(b->groups.size());
    if (class_of_buffer)
        for (int i = 0; i < b->n; ++i) class_of_buffer[i] = b->class_of[i];
    return SL_OK;
}

void sl_batch_destroy(sl_batch* b) { release(b); }

}  // extern "C"
