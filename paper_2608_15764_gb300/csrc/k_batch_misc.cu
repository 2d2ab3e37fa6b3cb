// k_batch_misc.cu -- cp.async and TMA class kernels of the batched form, and
// the per-buffer combine.
#include "k_batch.cuh"
#include "sl_mbar.cuh"

namespace sl {

__device__ __forceinline__ void kb_cp_async16(uint32_t saddr, const void* gptr) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(saddr), "l"(gptr) : "memory");
}
__device__ __forceinline__ void kb_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void kb_cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// cp.async class kernel: per item, chunk j of the item is vectors
// [j*cta, (j+1)*cta); each thread copies its 16 bytes of chunk j into ring
// slot j mod D with D commit groups in flight, reads its own slot back and
// folds (as k_cpasync).  The pipeline drains at the end of each item.
//
// Registers: an SM's CTAs hide each other's latency, so the budget is that of the
// loop (32 let all 2,048 threads be resident), more where the fold would be
// squeezed into a serial chain: 1,024 buffers of 16 GiB at 256 threads, uint32 D = 6
// 48 -> 32 registers 2,350 -> 2,287 us; bfloat16 D = 2 32 -> 40 registers
// 3,021 -> 2,726, but D = 1 32 -> 40 2,946 -> 3,214; FP32 D = 2 2,343 -> 2,327 (2
// GiB: 324 -> 310).  (D and the block size are the caller's, so the cap is on
// registers, not on CTAs per SM.)
constexpr int kb_cpasync_regs(int d, int dt) {
    if (dt == SL_U32 || d == 1) return 32;
    if (dt == SL_FP8_E4M3) return d <= 4 ? 32 : 40;
    if (dt == SL_F32) return d == 3 || d == 4 ? 32 : d <= 5 ? 40 : 48;
    return d <= 5 ? 40 : 48;
}

template <int D, int DT>
__global__ void __maxnreg__(kb_cpasync_regs(D, DT)) kb_cpasync(const BArgs a) {
    extern __shared__ __align__(128) uint4 cp_ring[];  // [D][cta], 128-byte aligned (cp.async destinations)
    batch_items<DT != SL_U32>(a, [&](const BatchItem& it) {
        const uint32_t cta = blockDim.x, t = tid_here();
        const uint32_t my0 = smem_addr(cp_ring) + t * 16u, stride = cta * 16u;
        Acc<DT> acc;
#pragma unroll
        for (int g = 0; g < D - 1; ++g) {
            const uint32_t v = static_cast<uint32_t>(g) * cta + t;
            if (v < it.nvec) kb_cp_async16(my0 + g * stride, it.ptr + v);
            kb_cp_commit();
        }
        uint32_t slot = 0;
#pragma unroll 1
        for (uint32_t base = 0; base < it.nvec; base += cta) {
            const uint32_t v = base + t, ahead = v + (D - 1) * cta;
            if (ahead < it.nvec) kb_cp_async16(my0 + (slot == 0 ? D - 1 : slot - 1) * stride, it.ptr + ahead);
            kb_cp_commit();
            kb_cp_wait<D - 1>();
            if (v < it.nvec) {
                acc.fold(lds16(my0 + slot * stride));
                acc.n += 1;
            }
            slot = (slot + 1 == D) ? 0 : slot + 1;
        }
        kb_cp_wait<0>();
        return warp_partial(acc);
    });
}

// Per-stage note from the producer to the consumers of the TMA class kernel.
struct StageMeta {
    uint32_t item;   // the item this stage belongs to
    uint32_t nv;     // 16-byte vectors in the stage
    uint32_t flags;  // STAGE_LAST_OF_ITEM, STAGE_DONE
    uint32_t pad;
};
constexpr uint32_t STAGE_LAST_OF_ITEM = 1, STAGE_DONE = 2;

// TMA class kernel: lane 0 of warp 0 claims items and streams them through
// the mbarrier ring stage by stage (an item of n bytes takes ceil(n / S)
// stages; the ring does not drain between items), noting in each stage which
// item it belongs to.  Consumer warps fold every stage and write their item
// partial after the item's last stage.  When the items run out the producer
// arms one more stage marked DONE with a plain arrive (no bytes).  Waits are
// bounded and issued copies are drained before exit, as in k_tma.  As there,
// a consumer thread reads its last B vectors of a stage into registers and
// its warp releases the stage before folding them (B = 4, or 1 where a
// thread reads fewer than 4 vectors of a stage).
template <int DT, int B, bool BIAS>
__global__ void __launch_bounds__(1024) kb_tma(const BArgs a) {
    extern __shared__ __align__(128) uint8_t tma_ring[];
    __shared__ __align__(8) uint64_t full[SL_MAX_STAGES];
    __shared__ __align__(8) uint64_t empty[SL_MAX_STAGES];
    __shared__ StageMeta meta[SL_MAX_STAGES];
    __shared__ volatile int abort_flag;

    const uint32_t nst = static_cast<uint32_t>(a.nst);
    const uint32_t S = a.stage_bytes;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t ncw = (blockDim.x >> 5) - 1;
    const uint32_t ring0 = smem_addr(tma_ring);
    const uint32_t full0 = smem_addr(full), empty0 = smem_addr(empty);
    if (threadIdx.x == 0) {
        ring_init(full0, empty0, nst, ncw);
        abort_flag = 0;
    }
    __syncthreads();

    if (warp == 0) {
        if (lane == 0) {
            uint32_t armed = 0, last_par = 0, s = 0, r = 0;
            bool stop = false;
            // The next item is claimed, and its descriptor fetched, when no more
            // stages are left to issue than are in flight: claimed any earlier, items
            // are dealt out before it shows which CTAs are fast.
            uint32_t item = blockIdx.x;
            BatchItem it = a.items[item];  // the host launches at most nitems CTAs
            while (!stop) {
                const bool done = item >= a.nitems;
                uint32_t nstage = 1, nbytes = 0;
                if (!done) {
                    nbytes = it.nvec * 16u;
                    nstage = (nbytes + S - 1) / S;
                }
                const uint32_t ask = nstage > nst ? nstage - nst : 0;
                uint32_t next = 0xFFFFFFFFu;
                BatchItem it1{nullptr, 0u, 0u};
                for (uint32_t k = 0; k < nstage; ++k) {
                    if (r > 0 && !bounded_wait(empty0 + 8 * s, (r - 1) & 1u, a.err, a.timeout_ns, &abort_flag, true,
                                               DEV_ERR_TIMEOUT_EMPTY)) {
                        stop = true;
                        break;
                    }
                    if (done) {
                        // The copy this stage last carried has landed (its
                        // consumers released the stage), and the sentinel
                        // advances full[s] by one more phase: stop draining it.
                        armed &= ~(1u << s);
                        meta[s] = StageMeta{0u, 0u, STAGE_DONE, 0u};
                        mbar_arrive(full0 + 8 * s);
                    } else {
                        const uint32_t off = k * S;
                        const uint32_t len = nbytes - off < S ? nbytes - off : S;
                        meta[s] = StageMeta{item, len >> 4, k + 1 == nstage ? STAGE_LAST_OF_ITEM : 0u, 0u};
                        mbar_arrive_expect_tx(full0 + 8 * s, len);
                        bulk_g2s(ring0 + s * S, reinterpret_cast<const uint8_t*>(it.ptr) + off, len, full0 + 8 * s);
                        armed |= 1u << s;
                        last_par = (last_par & ~(1u << s)) | ((r & 1u) << s);
                    }
                    if (++s == nst) { s = 0; ++r; }
                    if (k == ask && !done) {
                        next = gridDim.x + atomicAdd(a.next, 1u);
                        if (next < a.nitems) it1 = a.items[next];
                    }
                }
                if (done) stop = true;
                item = next;
                it = it1;
            }
            for (uint32_t q = 0; q < nst; ++q)
                if (armed & (1u << q))
                    bounded_wait(full0 + 8 * q, (last_par >> q) & 1u, a.err, a.timeout_ns, &abort_flag, false,
                                 DEV_ERR_TIMEOUT_DRAIN);
        }
        __syncwarp();
    } else {
        const uint32_t ct = threadIdx.x - 32, nct = ncw * 32;
        using TAcc = Acc<DT, BIAS>;
        TAcc acc;
        uint32_t s = 0, r = 0;
        for (;;) {
            const bool got =
                bounded_wait(full0 + 8 * s, r & 1u, a.err, a.timeout_ns, &abort_flag, true, DEV_ERR_TIMEOUT_FULL);
            if (!__all_sync(FULL_MASK, got)) break;
            const StageMeta m = meta[s];  // read before the stage is released
            if (m.flags & STAGE_DONE) break;
            const uint32_t base = ring0 + s * S;
            if constexpr (BIAS) {
                // one place where vectors are folded together (its code is long)
                for (uint32_t v0 = ct & ~31u;; v0 += B * nct) {  // warp-uniform
                    const uint32_t v = v0 + lane;
                    const bool last = v0 + B * nct >= m.nv;
                    if (v0 + 31 + (B - 1) * nct < m.nv) {
                        uint4 x[B];
#pragma unroll
                        for (int u = 0; u < B; ++u) x[u] = lds16(base + 16u * (v + u * nct));
                        if (last) {
                            __syncwarp();
                            if (lane == 0) mbar_arrive(empty0 + 8 * s);
                        }
                        acc.fold_n(x);
                        acc.n += B;
                    } else {
#pragma unroll 1
                        for (uint32_t w = v; w < m.nv && w < v + B * nct; w += nct) {
                            acc.fold(lds16(base + 16u * w));
                            acc.n += 1;
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(empty0 + 8 * s);
                    }
                    if (last) break;
                }
            } else {
                uint32_t v = ct;
#pragma unroll 1
                for (; v + B * nct < m.nv; v += B * nct) {
                    uint4 x[B];
#pragma unroll
                    for (int u = 0; u < B; ++u) x[u] = lds16(base + 16u * (v + u * nct));
#pragma unroll
                    for (int u = 0; u < B; ++u) acc.fold(x[u]);
                    acc.n += B;
                }
                uint4 x[B];
#pragma unroll
                for (int u = 0; u < B; ++u)
                    if (v + u * nct < m.nv) x[u] = lds16(base + 16u * (v + u * nct));
                __syncwarp();
                if (lane == 0) mbar_arrive(empty0 + 8 * s);
#pragma unroll
                for (int u = 0; u < B; ++u)
                    if (v + u * nct < m.nv) {
                        acc.fold(x[u]);
                        acc.n += 1;
                    }
            }
            if (m.flags & STAGE_LAST_OF_ITEM) {
                const WarpPartial w = warp_partial(acc);
                if (lane == 0) a.parts[static_cast<size_t>(m.item) * ncw + (warp - 1)] = w;
                acc = TAcc();
            }
            if (++s == nst) { s = 0; ++r; }
        }
    }
    __syncthreads();
}

// Per-buffer combine: one CTA per buffer adds the buffer's partial slots in a
// fixed order (thread t takes slots t, t+128, ..., four in flight; integer parts
// exact, float parts in FP64; then the lanes, then the warps) and writes its
// sl_result to page-locked host memory.  CTA 0 publishes the device error word
// and leaves it and the class counters at zero for the next run.  (One warp per
// buffer with one slot in flight took 40 us over a 256 MiB buffer's 2,048.)
constexpr int KB_COMBINE_THREADS = 128;

__global__ void __launch_bounds__(KB_COMBINE_THREADS) kb_combine(const BufSeg* __restrict__ segs,
                                                                const WarpPartial* __restrict__ parts, uint32_t* err,
                                                                uint32_t* next, uint32_t nclasses,
                                                                sl_result* out, uint32_t* host_err) {
    struct Fin {
        uint32_t sum;
        uint64_t x, n;
        double f;
    };
    __shared__ Fin fw[KB_COMBINE_THREADS / 32];
    const uint32_t b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const BufSeg g = segs[b];
    if (b == 0 && threadIdx.x < nclasses) next[threadIdx.x] = 0;
    if (b == 0 && threadIdx.x == 0) {
        for (uint32_t i = KB_COMBINE_THREADS; i < nclasses; ++i) next[i] = 0;
        *host_err = *err;
        *err = 0;
    }
    Fin v{0u, 0ull, 0ull, 0.0};
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < g.pcount; i += KB_COMBINE_THREADS) {
        const uint4* p = reinterpret_cast<const uint4*>(parts + g.pstart + i);
        const uint4 lo4 = __ldcg(p), hi4 = __ldcg(p + 1);
        v.sum += lo4.x;
        v.x ^= (static_cast<uint64_t>(lo4.w) << 32) | lo4.z;
        v.n += (static_cast<uint64_t>(hi4.y) << 32) | hi4.x;
        v.f += static_cast<double>(__uint_as_float(hi4.z)) + static_cast<double>(__uint_as_float(hi4.w));
    }
    for (int pass = 0; pass < 2; ++pass) {
        v.sum = warp_add32(v.sum);
        v.x = warp_xor64(v.x);
        v.n = warp_add64(v.n);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v.f += __shfl_xor_sync(FULL_MASK, v.f, o);
        if (pass == 1) break;
        if (lane == 0) fw[warp] = v;
        __syncthreads();
        if (warp != 0) return;
        v = lane < KB_COMBINE_THREADS / 32 ? fw[lane] : Fin{0u, 0ull, 0ull, 0.0};
    }
    if (lane == 0) {
        sl_result r;
        r.xor_u64 = v.x;
        r.issued_loads = v.n;
        r.device_ns = 0;
        r.window_ns = 0;
        r.fsum = v.f;
        r.fsum_hi = static_cast<float>(v.f);
        r.fsum_lo = static_cast<float>(v.f - static_cast<double>(r.fsum_hi));
        r.sum_u32 = v.sum;
        r.status = SL_OK;  // the host replaces it where the run's error word is set
        r.grid = 0;
        r.cta = 0;
        r.resident_per_sm = 0;
        r.smem_bytes = 0;
        out[b] = r;
    }
}

template <int DT>
static const void* kb_cp_d(int d) {
    switch (d) {
    case 1: return reinterpret_cast<const void*>(&kb_cpasync<1, DT>);
    case 2: return reinterpret_cast<const void*>(&kb_cpasync<2, DT>);
    case 3: return reinterpret_cast<const void*>(&kb_cpasync<3, DT>);
    case 4: return reinterpret_cast<const void*>(&kb_cpasync<4, DT>);
    case 5: return reinterpret_cast<const void*>(&kb_cpasync<5, DT>);
    case 6: return reinterpret_cast<const void*>(&kb_cpasync<6, DT>);
    case 7: return reinterpret_cast<const void*>(&kb_cpasync<7, DT>);
    case 8: return reinterpret_cast<const void*>(&kb_cpasync<8, DT>);
    default: return nullptr;
    }
}

const void* batch_cpasync_kernel(int dtype, int d) {
    switch (dtype) {
    case SL_U32: return kb_cp_d<SL_U32>(d);
    case SL_F32: return kb_cp_d<SL_F32>(d);
    case SL_BF16: return kb_cp_d<SL_BF16>(d);
    case SL_FP8_E4M3: return kb_cp_d<SL_FP8_E4M3>(d);
    default: return nullptr;
    }
}

template <int B>
static const void* kb_tma_b(int dtype) {
    switch (dtype) {
    case SL_U32: return reinterpret_cast<const void*>(&kb_tma<SL_U32, B, false>);
    case SL_F32: return reinterpret_cast<const void*>(&kb_tma<SL_F32, B, false>);
    case SL_BF16: return reinterpret_cast<const void*>(&kb_tma<SL_BF16, B, false>);
    case SL_FP8_E4M3: return reinterpret_cast<const void*>(&kb_tma<SL_FP8_E4M3, B, false>);
    default: return nullptr;
    }
}

const void* batch_tma_kernel(int dtype, int batch, bool biased) {
    if (batch == 4)
        return dtype == SL_BF16 && biased ? reinterpret_cast<const void*>(&kb_tma<SL_BF16, 4, true>)
                                          : kb_tma_b<4>(dtype);
    if (batch == 1) return kb_tma_b<1>(dtype);
    return nullptr;
}

cudaError_t launch_batch_combine(const BufSeg* segs, uint32_t nbuf, const WarpPartial* parts, uint32_t* err,
                                 uint32_t* next, uint32_t nclasses, sl_result* out, uint32_t* host_err,
                                 cudaStream_t s) {
    if (nbuf == 0) return cudaSuccess;
    kb_combine<<<nbuf, KB_COMBINE_THREADS, 0, s>>>(segs, parts, err, next, nclasses, out, host_err);
    return cudaGetLastError();
}

}  // namespace sl
