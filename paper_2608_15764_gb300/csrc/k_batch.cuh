// k_batch.cuh -- persistent kernels of the batched form.
//
// A batch is cut into work items (contiguous pieces of one buffer, sized by
// the host: see item_bytes in batch_api.cu).  Every class kernel runs a
// persistent grid; CTA b starts on the class's items b and grid + b and claims
// the others one at a time from an atomic counter (dynamic balancing across
// uneven buffers), folds each item with the class's mechanism and writes its
// partials at the item's own slots, so the result does not depend on which CTA
// took which item.  kb_combine then adds the partials of each buffer in slot
// order, writes its result straight into page-locked host memory and leaves
// the counters at zero for the next run: a run is the class kernels and this
// one, with no memset before them and no copies after them.
#pragma once

#include "sl_device.cuh"

namespace sl {

struct __align__(16) BatchItem {
    const uint4* ptr;  // first vector of the item
    uint32_t nvec;     // 16-byte vectors in the item (> 0)
    uint32_t dtype;    // sl_dtype of the buffer
};
static_assert(sizeof(BatchItem) == 16, "BatchItem layout");

struct BufSeg {
    uint32_t pstart;  // first partial slot of the buffer
    uint32_t pcount;  // partial slots of the buffer (items x slots per item)
};

struct BArgs {
    const BatchItem* items;  // this class's items
    uint32_t nitems;
    uint32_t stage_bytes;    // TMA stage size
    uint32_t* next;          // item counter (zero before every launch)
    WarpPartial* parts;      // this class's partials, in item order
    uint32_t* err;           // device error word
    uint64_t timeout_ns;     // bound of any single device wait (TMA)
    int32_t nst;             // TMA stages
    int32_t reserved;
};

// Reduce a warp's accumulators into one partial (lane 0 holds it afterwards).
template <int DT, bool BIAS>
__device__ __forceinline__ WarpPartial warp_partial(const Acc<DT, BIAS>& acc) {
    uint32_t s = acc.s;
    uint64_t x = (static_cast<uint64_t>(acc.xh) << 32) | acc.xl, n = acc.n;
    float hi = 0.0f, lo = 0.0f;
    if constexpr (DT != SL_U32) acc.float_part(hi, lo);
    warp_merge<DT>(s, x, n, hi, lo);
    WarpPartial p;
    p.sum = s;
    p.pad = 0;
    p.xr = x;
    p.issued = n;
    p.hi = hi;
    p.lo = lo;
    return p;
}

// The block's and the grid's size, as tid_here: what is computed from the thread's
// place is kept out of the registers through stream() below, ten of them in an LDG
// kernel (K = 4 uint32 42 -> 33, K = 16 102 -> 81).
__device__ __forceinline__ uint32_t threads_here() {
    uint32_t t;
    asm volatile("mov.u32 %0, %%ntid.x;" : "=r"(t));
    return t;
}
__device__ __forceinline__ uint32_t grid_here() {
    uint32_t t;
    asm volatile("mov.u32 %0, %%nctaid.x;" : "=r"(t));
    return t;
}

// The item loop of a class kernel whose CTAs work on one item together.
// stream(item) folds an item and returns the warp's partial.  The next item's descriptor is copied to
// shared memory, and the one after it claimed, while the current item streams;
// one CTA barrier per item publishes both together with the warps' partials,
// which one warp (a different one for each item) then merges into the item's
// partial while the others go on.  (Claiming, fetching the descriptor and two
// barriers between items left every CTA idle for about 2 us per item.)  Little is kept in registers across stream():
// the item's index and its place in the loop are re-read from shared memory.
//
// What orders the shared words, with B(j) the barrier of iteration j: a word is
// written before B(j) and read after it, and its readers are done only at
// B(j + 1).  Between B(j) and B(j + 1) warps read indices j and j + 1 while
// thread 0 writes index j + 3, so there are four index words (with three,
// index j + 3 would be index j's); they read descriptor j + 1 and partials j
// while descriptor j + 2 and partials j + 1 are written: two of each.
template <bool FLOATS, typename Stream>
__device__ __forceinline__ void batch_items(const BArgs& a, Stream stream) {
    __shared__ BatchItem slot[2];
    __shared__ uint32_t sidx[4];
    __shared__ WarpPartial wp[2][32];
    volatile uint32_t* vidx = sidx;
    if (threadIdx.x == 0) {
        vidx[0] = blockIdx.x;  // the host launches at most nitems CTAs
        vidx[1] = blockIdx.x + gridDim.x;
    }
    BatchItem it = a.items[dyn_first()];
#pragma unroll 1
    for (uint32_t j = 0;; ++j) {
        // sidx[j & 3]: this item, [(j + 1) & 3]: the next, [(j + 2) & 3]: being claimed
        uint32_t claim = 0xFFFFFFFFu;
        if (tid_here() == 0) {
            const uint32_t ahead = vidx[(j + 1) & 3];
            if (ahead < a.nitems) {
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(&slot[(j + 1) & 1])),
                             "l"(a.items + ahead) : "memory");
                claim = 2 * grid_here() + atomicAdd(a.next, 1u);
            }
        }
        const WarpPartial mine = stream(it);
        const uint32_t tid = tid_here(), warp = tid >> 5, lane = tid & 31, nw = threads_here() >> 5;
        if (lane == 0) wp[j & 1][warp] = mine;
        if (tid == 0) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            vidx[(j + 2) & 3] = claim;
        }
        __syncthreads();
        const uint32_t cur = vidx[j & 3], next = vidx[(j + 1) & 3];
        if (warp == j % nw) {
            uint32_t s = 0;
            uint64_t x = 0, n = 0;
            float hi = 0.0f, lo = 0.0f;
            if (lane < nw) {
                const WarpPartial q = wp[j & 1][lane];
                s = q.sum;
                x = q.xr;
                n = q.issued;
                hi = q.hi;
                lo = q.lo;
            }
            warp_merge<FLOATS ? SL_F32 : SL_U32>(s, x, n, hi, lo);
            if (lane == 0) {
                WarpPartial q;
                q.sum = s;
                q.pad = 0;
                q.xr = x;
                q.issued = n;
                q.hi = hi;
                q.lo = lo;
                a.parts[cur] = q;
            }
        }
        if (next >= a.nitems) break;
        it = slot[(j + 1) & 1];
    }
}

// One item of an LDG class: tiles of CTA*K vectors, K independent 16-byte loads
// per thread per tile (same fold and tile layout as k_ldg), guarded ragged tail.
template <int K, int CTA, int DT>
__device__ __forceinline__ WarpPartial ldg_item(const BatchItem& it) {
    constexpr uint32_t TILE = static_cast<uint32_t>(CTA) * K;
    Acc<DT, BIASED<DT, K>> acc;
    const uint32_t nfull = it.nvec / TILE;
    const uint4* p = it.ptr + tid_here();
#pragma unroll 1
    for (uint32_t t = 0; t < nfull; ++t, p += TILE) {
        uint4 v[K];
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] = ldg16<SL_COP_CG>(p + k * CTA);
        acc.fold_n(v);
    }
    acc.n = nfull * K;
    const uint32_t rem = it.nvec - nfull * TILE;
    if (rem) {
        const uint32_t tid = tid_here();
        uint4 v[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (tid + k * CTA < rem) v[k] = ldg16<SL_COP_CG>(p + k * CTA);
            else v[k] = make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (tid + k * CTA < rem) {
                acc.fold(v[k]);
                acc.n += 1;
            }
        }
    }
    return warp_partial(acc);
}

// Minimum resident CTAs per SM asked of the compiler: what 5K + 12 registers
// (uint32) or 5K + 32 (floats) allow, the K loaded vectors, the sums and the
// fold's temporaries.  Left to itself it takes more where a CTA is lost by it (1,024
// buffers of 16 GiB: FP32 K = 6 at 512 threads 70 registers, one CTA per SM, 2,710
// us; 58, two, 2,330) or fewer than the loads in flight need.
template <int K, int CTA, int DT>
constexpr int kb_ldg_min_blocks() {
    int regs = DT == SL_U32 || (DT == SL_FP8_E4M3 && K == 1) ? 5 * K + 12 : K <= 2 ? 40 : 5 * K + 32;
    if (DT == SL_BF16 && K == 8) regs = CTA >= 256 ? 64 : 80;
    regs = regs < 32 ? 32 : regs > 128 ? 128 : (regs + 7) / 8 * 8;
    return 65536 / (CTA * regs) > 0 ? 65536 / (CTA * regs) : 1;
}

template <int K, int CTA, int DT>
__global__ void __launch_bounds__(CTA, kb_ldg_min_blocks<K, CTA, DT>()) kb_ldg(const BArgs a) {
    batch_items<DT != SL_U32>(a, [](const BatchItem& it) { return ldg_item<K, CTA, DT>(it); });
}

// The LDG classes of one tuning entry, whatever their types, in one launch (the
// host takes it for small classes: see plan_units in batch_api.cu).
template <int K, int CTA>
__global__ void __launch_bounds__(CTA) kb_ldg_any(const BArgs a) {
    batch_items<true>(a, [](const BatchItem& it) {
        switch (it.dtype) {
        case SL_F32: return ldg_item<K, CTA, SL_F32>(it);
        case SL_BF16: return ldg_item<K, CTA, SL_BF16>(it);
        case SL_FP8_E4M3: return ldg_item<K, CTA, SL_FP8_E4M3>(it);
        default: return ldg_item<K, CTA, SL_U32>(it);
        }
    });
}

}  // namespace sl
