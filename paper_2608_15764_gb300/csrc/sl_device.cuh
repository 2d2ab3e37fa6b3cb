// sl_device.cuh -- device-side building blocks of the streaming-load kernels:
// 16-byte global loads, the checksum / compensated-sum fold, warp reduction
// and per-warp partial output.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "sl_internal.h"

namespace sl {

constexpr unsigned FULL_MASK = 0xFFFFFFFFu;

__device__ __forceinline__ uint64_t gtimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// threadIdx.x, read by hand where it is used: the compiler would keep what it
// computes from threadIdx (addresses, lane, warp, comparisons) in registers
// through the loops between.
__device__ __forceinline__ uint32_t tid_here() {
    uint32_t t;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
    return t;
}

// One 16-byte global load (paper §3: one ld.global per offered load; §4.2
// primary cell uses .cg, which caches in L2 only).  volatile keeps every load
// in the program and in source order.
template <int COP>
__device__ __forceinline__ uint4 ldg16(const uint4* p) {
    uint4 v;
    if constexpr (COP == SL_COP_CG) {
        asm volatile("ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    } else if constexpr (COP == SL_COP_CG_L2_256) {
        asm volatile("ld.global.cg.L2::256B.v4.u32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    } else {
        asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    }
    return v;
}

__device__ __forceinline__ uint4 lds16(uint32_t saddr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(saddr));
    return v;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---- packed float pairs -------------------------------------------------------
// Two FP32 values in one 64-bit register pair (lane 0 = low word), operated on
// by the sm_100-family packed instructions add/sub.rn.f32x2: each lane is an
// ordinary IEEE round-to-nearest FP32 operation (subnormals kept), two lanes
// per instruction.
__device__ __forceinline__ uint64_t f2_pack(uint32_t lo_bits, uint32_t hi_bits) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo_bits), "r"(hi_bits));
    return d;
}
__device__ __forceinline__ float f2_lane0(uint64_t p) { return __uint_as_float(static_cast<uint32_t>(p)); }
__device__ __forceinline__ float f2_lane1(uint64_t p) { return __uint_as_float(static_cast<uint32_t>(p >> 32)); }
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// ---- per-vector FP8 sum ----------------------------------------------------------
// FP8 E4M3: 8 values per half vector.  cvt.rn.f16x2.e4m3x2 widens two codes to
// half exactly (every E4M3 value is a half), add.f32.f16 adds a half to an
// FP32 accumulator.  Every E4M3 value is an integer multiple of 2^-9 below
// 2^9, so any partial sum of 16 of them is a multiple of 2^-9 below 2^13 and
// fits the 24-bit FP32 significand: each half's sum, and their total, are
// exact in any order.
__device__ __forceinline__ float fp8_word_sum(uint32_t w, float acc) {
    asm("{\n\t.reg .b16 q0, q1, a0, a1, b0, b1;\n\t.reg .b32 h0, h1;\n\t"
        "mov.b32 {q0, q1}, %1;\n\t"
        "cvt.rn.f16x2.e4m3x2 h0, q0;\n\t"
        "cvt.rn.f16x2.e4m3x2 h1, q1;\n\t"
        "mov.b32 {a0, a1}, h0;\n\t"
        "mov.b32 {b0, b1}, h1;\n\t"
        "add.rn.f32.f16 %0, a0, %0;\n\t"
        "add.rn.f32.f16 %0, a1, %0;\n\t"
        "add.rn.f32.f16 %0, b0, %0;\n\t"
        "add.rn.f32.f16 %0, b1, %0;\n\t}"
        : "+f"(acc) : "r"(w));
    return acc;
}

// ---- register budget of the plain-load kernels --------------------------------
// Minimum resident CTAs per SM asked of the compiler for an LDG kernel
// (__launch_bounds__).  A bfloat16 fold (eight TwoSum steps per vector) with
// up to K = 8 loads in flight is held to 64 registers per thread, so that four
// 256-thread (two 512-thread) CTAs stay resident: with fewer warps its
// dependent TwoSum chains cannot hide the load latency (at K = 8 the
// unconstrained allocation of 78 registers leaves three CTAs and ~7% less
// bandwidth); above K = 8 to the 102 or 128 of five or four 128-thread CTAs
// (two of 256 threads).  A K = 1 kernel of another type is held to the 32 registers that
// let an SM's 2,048 threads be resident (its loop needs fewer; the reduction at
// its end would otherwise take two or four more and cost a quarter of the
// CTAs).  Every other kernel takes the registers it wants (K loaded vectors
// must stay in registers).
template <int K, int CTA, int DT>
constexpr int ldg_min_blocks() {
    if (DT == SL_BF16) {
        if (K <= 8) return CTA >= 256 ? 1024 / CTA : 1;
        return CTA <= 512 ? (K <= 11 ? 640 : 512) / CTA : 1;
    }
    return K == 1 ? 2048 / CTA : 1;
}

// ---- coverage audit ------------------------------------------------------------
// In the coverage instantiations (COV = true) every load of 16-byte vector i
// also adds 1 to a.cov[i]; elsewhere this compiles to nothing.
template <bool COV>
__device__ __forceinline__ void cov_count(const KArgs& a, uint64_t i) {
    if constexpr (COV) atomicAdd(a.cov + i, 1u);
}

// Whether a kernel that folds n vectors at a time takes the biased sum.
template <int DT, int N>
constexpr bool BIASED = DT == SL_BF16 && N >= 4 && N <= 16;

// ---- the fold ----------------------------------------------------------------
// Per-thread accumulator.  Integer part (every dtype): wraparound uint32 sum
// of the four words and XOR of the two little-endian uint64 halves.
//
// Float part: compensated FP32 summation in which every addition's rounding
// error is recovered exactly with TwoSum (Knuth) and added to a separate
// error sum, so the represented value is s + e with an error of order u^2
// times sum|x| (u = 2^-24) instead of the 2u sum|x| of Kahan's recurrence.
// It runs as two independent lanes of packed f32x2 arithmetic (lane 0 takes
// the even-numbered values of a vector, lane 1 the odd-numbered ones), so one
// TwoSum instruction sequence serves two elements:
//   FP32: each of the 4 values goes through TwoSum (2 packed steps);
//   BF16: each of the 8 values is widened exactly to FP32
//         and goes through TwoSum (4 packed steps), so no addition inside a
//         vector is left uncompensated, whatever the values' range;
//   FP8:  the two half-vector sums, each exact (fp8_word_sum), go through one
//         packed TwoSum step.
//
// BIAS (BF16 where a thread folds four or more vectors at a time, fold_n): the
// running sum is held as fs = C + sum with a power-of-two bias C = 1.5 * 2^k
// well above the data, so that |fs| >= |x| in every addition and its rounding
// error needs the three operations of Dekker's Fast2Sum where TwoSum needs six:
// 16 packed operations per vector (and three per fold_n) instead of 28.
// The biased sum is exact: fs + fe - C is the sum of the values added, without
// any rounding.  fs stays in [2^k, 2^(k+1)), so every error is at most
// h = 2^(k-24); fe collects the 4N errors of a fold_n, then what is large enough
// of it goes back to fs, which leaves |fe| <= h.  So |fe| < 2^L h with 2^L >= 4N + 2
// and adding to it is exact while all values are multiples of its smallest step,
// 2^(k-48+L).  fold_n therefore looks at its values' largest and smallest
// exponent first:
//   - the largest may move fs by at most a quarter of 2^k (HEAD = L + 2 below k),
//     and fs starts within a quarter of C, or C is raised;
//   - the smallest but zero is LOW = 41 - L or less below k (eight bits of
//     significand above the step).
// Otherwise C is taken anew, 2 above HEAD and 3 above the sum (enter_bias, which
// also checks that what the sum holds by then is a multiple of the step).  A
// thread whose values allow none, infinities and NaN among them, goes on with
// TwoSum from the sum it has (c = SLOW); a single vector is added by TwoSum.
// So a thread's error is 0 while its values fit and TwoSum's from there on.
// Emulated on the CPU (96 threads, 16,384 values each), no error and at most 3%
// of the groups by TwoSum on N(0,1), Laplace, Student-t with 3 degrees of freedom
// and uniform values, their absolute values, and one value in 1,000 20 times
// larger; the error of TwoSum alone (1e-12 of a thread's sum|x| at most, within the
// luck of single roundings) where values shrink by 2^-13 or more after the first
// ones or spread over more than 30 binades, most of them summed by TwoSum.
// Measured, TwoSum then biased: 16 passes over 32 MiB in L2 at K = 8 76.0 -> 60.5
// us, 1 GiB at K = 8 163 -> 155, at K = 4 178 -> 162; 1,024 buffers of 16 GiB by
// 16 KiB x 2 TMA rings 2,588 -> 2,399 on the device.  Kernels with fewer vectors
// at a time (K < 4, one copy per group) stay with TwoSum.
template <int DT, bool BIAS = false>
struct Acc {
    static constexpr uint32_t SLOW = 0xFFFFFFFFu;
    // The bias a thread starts with, 1.5 * 2^12: it fits values below 2^6 (N = 4)
    // to 2^4 (N = 16) and down to 2^-24 to 2^-22, as weights and activations mostly
    // are, so that such a thread does not run renew_bias (whose code it would have
    // to fetch: 0.7 us of a 14 us launch).
    static constexpr uint32_t START = BIAS ? (139u << 23) | 0x400000u : 0u;
    uint32_t s = 0, xl = 0, xh = 0;
    uint32_t n = 0;  // 16-byte loads folded by this thread (the host keeps it below 2^32)
    // packed (lane 0, lane 1) running sums and error sums; 0 bits = +0.0f
    uint64_t fs = (static_cast<uint64_t>(START) << 32) | START, fe = 0;
    uint32_t c = START;  // BIAS: bits of C in both lanes of fs; 0: none now; SLOW: none from here on

    // TwoSum of the packed pair x into (fs, fe), lane by lane.
    __device__ __forceinline__ void add2(uint64_t x) {
        const uint64_t t = f2_add(fs, x);
        const uint64_t bp = f2_sub(t, fs);
        const uint64_t d1 = f2_sub(fs, f2_sub(t, bp));
        const uint64_t d2 = f2_sub(x, bp);
        fe = f2_add(fe, f2_add(d1, d2));
        fs = t;
    }

    // A word's two BF16 values where |fs| >= |x| in both lanes (Fast2Sum: the
    // rounding error of t = fs + x is x - (t - fs)).  The additions that take the
    // values take them as they are (add/sub.f32.bf16, one lane each, the value
    // widened exactly): the shift and the mask that would unpack them are ALU
    // work, which bounds this fold together with fold_n's look at the codes
    // (16 passes over 32 MiB in L2 at K = 8: 70.2 us with them, 60.5 without).
    __device__ __forceinline__ void add_word_biased(uint32_t w) {
        float t0, t1, e0, e1;
        asm("{\n\t.reg .b16 l, h;\n\t"
            "mov.b32 {l, h}, %2;\n\t"
            "add.rn.f32.bf16 %0, l, %3;\n\t"
            "add.rn.f32.bf16 %1, h, %4;\n\t}"
            : "=f"(t0), "=f"(t1) : "r"(w), "f"(f2_lane0(fs)), "f"(f2_lane1(fs)));
        const uint64_t t = f2_pack(__float_as_uint(t0), __float_as_uint(t1));
        const uint64_t d = f2_sub(t, fs);
        asm("{\n\t.reg .b16 l, h;\n\t"
            "mov.b32 {l, h}, %2;\n\t"
            "sub.rn.f32.bf16 %0, l, %3;\n\t"
            "sub.rn.f32.bf16 %1, h, %4;\n\t}"
            : "=f"(e0), "=f"(e1) : "r"(w), "f"(f2_lane0(d)), "f"(f2_lane1(d)));
        fe = f2_add(fe, f2_pack(__float_as_uint(e0), __float_as_uint(e1)));
        fs = t;
    }

    // (fs, fe) without a bias: fs the rounded sum of both, fe the rest.
    __device__ __forceinline__ void normalise() {
        const uint64_t t = f2_add(fs, fe);
        const uint64_t b = f2_sub(t, fs);
        fe = f2_add(f2_sub(fs, f2_sub(t, b)), f2_sub(fe, b));
        fs = t;
    }

    __device__ __forceinline__ void leave_bias() {
        if (c != 0 && c != SLOW) {
            fs = f2_sub(fs, f2_pack(c, c));  // exact: fs is within a factor of two of C
            normalise();
            c = 0;
        }
    }

    // Take a bias for a group of largest exponent e and smallest nonzero code
    // low, or set c to SLOW.  On return with a bias, C's exponent is at least
    // HEAD + 2 above e and LOW or less above low's.
    template <int HEAD, int LOW>
    __device__ __forceinline__ void enter_bias(int e, int low) {
        normalise();
        const int f0 = (static_cast<uint32_t>(fs) >> 23) & 255u, f1 = (static_cast<uint32_t>(fs >> 32) >> 23) & 255u;
        const int k = max(e + HEAD + 2, max(f0, f1) + 3);
        c = SLOW;
        if (k > 240 || low < ((k - LOW) << 7)) return;
        const uint32_t bits = (static_cast<uint32_t>(k) << 23) | 0x400000u;
        const uint64_t t = f2_add(f2_pack(bits, bits), fs);
        const uint64_t d = f2_sub(fs, f2_sub(t, f2_pack(bits, bits)));
        // multiples of the step: unchanged by a round trip through 1.5 * 2^23 steps
        const uint32_t step = (static_cast<uint32_t>(max(k - 25 + (HEAD - 2), 1)) << 23) | 0x400000u;
        const uint64_t m = f2_pack(step, step);
        const uint64_t off = f2_sub(f2_sub(f2_add(fe, m), m), fe) | f2_sub(f2_sub(f2_add(d, m), m), d);
        if ((off & 0x7FFFFFFF7FFFFFFFull) != 0) return;
        fs = t;
        fe = f2_add(fe, d);
        c = bits;
    }

    // What fold_n does before it adds where there is no bias, the sum has outgrown
    // it, or a value is outside its range: zeros (which fit any) keep it.
    template <int N, int HEAD, int LOW>
    __device__ __forceinline__ void renew_bias(const uint4 (&v)[N], bool near) {
        // largest code and smallest nonzero code less one, signs left out.  (The
        // mask comes by way of a register that is always zero: with the constant
        // the compiler would keep fold_n's codes for this, at the price of a
        // register each.)
        uint32_t m = 0, l = 0xFFFFFFFFu, mask;
        asm volatile("mov.u32 %0, %%ctaid.z;" : "=r"(mask));
        mask ^= 0x7FFF7FFFu;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const uint32_t w[4] = {v[i].x & mask, v[i].y & mask, v[i].z & mask, v[i].w & mask};
            m = __vimax3_u16x2(__vimax3_u16x2(m, w[0], w[1]), w[2], w[3]);
#pragma unroll
            for (int j = 0; j < 4; ++j) l = __viaddmin_u16x2(w[j], 0xFFFFFFFFu, l);
        }
        const int e = max(m >> 16, m & 0xFFFFu) >> 7;
        const int low = min(l >> 16, l & 0xFFFFu) + 1;
        const int k = c >> 23;
        if (c != 0 && near && e + HEAD <= k && low >= ((k - LOW) << 7)) return;
        leave_bias();
        enter_bias<HEAD, LOW>(e, low);
    }

    // N vectors at once (N <= 16), by all lanes of the warp together.
    template <int N>
    __device__ __forceinline__ void fold_n(const uint4 (&v)[N]) {
        if constexpr (!BIAS) {
#pragma unroll
            for (int i = 0; i < N; ++i) fold(v[i]);
        } else {
            constexpr int L = N > 8 ? 7 : N > 4 ? 6 : 5;  // 4N + 2 <= 2^L
            constexpr int HEAD = L + 2, LOW = 41 - L;
#pragma unroll
            for (int i = 0; i < N; ++i) fold_int(v[i]);
            if (c != SLOW) {
                // codes without sign less that of the smallest exponent allowed, mod 2^16
                const uint32_t base = (LOW << 7) - ((c >> 23) << 7);
                const uint32_t off = __byte_perm(base, base, 0x1010);
                uint32_t r = 0;
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    r = __viaddmax_u16x2(v[i].x & 0x7FFF7FFFu, off, r);
                    r = __viaddmax_u16x2(v[i].y & 0x7FFF7FFFu, off, r);
                    r = __viaddmax_u16x2(v[i].z & 0x7FFF7FFFu, off, r);
                    r = __viaddmax_u16x2(v[i].w & 0x7FFF7FFFu, off, r);
                }
                // bits 22 and 21 differ while fs is between 1.25 and 1.75 * 2^k
                const uint32_t w0 = static_cast<uint32_t>(fs), w1 = static_cast<uint32_t>(fs >> 32);
                const bool near = ((w0 ^ (w0 << 1)) & (w1 ^ (w1 << 1)) & 0x400000u) != 0;
                constexpr uint32_t RANGE = ((LOW - HEAD + 1) << 7) - 1;
                if (c == 0 || !near || max(r >> 16, r & 0xFFFFu) > RANGE) renew_bias<N, HEAD, LOW>(v, near);
            }
            // One lane on the long way takes its warp along: both ways would be run.
            if (!__any_sync(FULL_MASK, c == SLOW)) {
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    add_word_biased(v[i].x);
                    add_word_biased(v[i].y);
                    add_word_biased(v[i].z);
                    add_word_biased(v[i].w);
                }
                const uint64_t t = f2_add(fs, fe);
                fe = f2_sub(fe, f2_sub(t, fs));
                fs = t;
            } else {
                leave_bias();
                c = SLOW;
#pragma unroll
                for (int i = 0; i < N; ++i) fold_float(v[i]);
            }
        }
    }

    __device__ __forceinline__ void fold_int(const uint4& v) {
        s += (v.x + v.y) + (v.z + v.w);
        xl ^= v.x ^ v.z;
        xh ^= v.y ^ v.w;
    }

    __device__ __forceinline__ void fold(const uint4& v) {
        if constexpr (BIAS) leave_bias();
        fold_int(v);
        fold_float(v);
    }

    __device__ __forceinline__ void fold_float(const uint4& v) {
        if constexpr (DT == SL_F32) {
            add2(f2_pack(v.x, v.y));
            add2(f2_pack(v.z, v.w));
        } else if constexpr (DT == SL_BF16) {
            // element 2i is the low half of word i, element 2i+1 the high half;
            // a bfloat16 is the top 16 bits of the FP32 with the same value
            add2(f2_pack(v.x << 16, v.x & 0xFFFF0000u));
            add2(f2_pack(v.y << 16, v.y & 0xFFFF0000u));
            add2(f2_pack(v.z << 16, v.z & 0xFFFF0000u));
            add2(f2_pack(v.w << 16, v.w & 0xFFFF0000u));
        } else if constexpr (DT == SL_FP8_E4M3) {
            const float a = fp8_word_sum(v.y, fp8_word_sum(v.x, 0.0f));
            const float b = fp8_word_sum(v.w, fp8_word_sum(v.z, 0.0f));
            add2(f2_pack(__float_as_uint(a), __float_as_uint(b)));
        }
    }

    // The float part as one double-float pair (hi, lo): the two lanes merged
    // with TwoSum and renormalised.
    __device__ __forceinline__ void float_part(float& hi, float& lo) const;
};

// Error-free sum of two floats (Knuth's TwoSum): s + e == a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// Double-float add of two partials' float parts (TwoSum, then renormalise).
__device__ __forceinline__ void df_add(float& hi, float& lo, float ohi, float olo) {
    float sh, se;
    two_sum(hi, ohi, sh, se);
    se += lo + olo;
    hi = sh + se;
    lo = se - (hi - sh);
}

template <int DT, bool BIAS>
__device__ __forceinline__ void Acc<DT, BIAS>::float_part(float& hi, float& lo) const {
    Acc a = *this;
    if constexpr (BIAS) a.leave_bias();
    hi = f2_lane0(a.fs);
    lo = f2_lane0(a.fe);
    df_add(hi, lo, f2_lane1(a.fs), f2_lane1(a.fe));
}

// ---- warp reductions ------------------------------------------------------------
// Integer parts go through the warp-reduce instructions (redux.sync: one
// instruction per 32-bit word, where a shuffle butterfly is five dependent
// shuffles and adds); double-float pairs go through shuffles.
__device__ __forceinline__ uint32_t warp_add32(uint32_t v) { return __reduce_add_sync(FULL_MASK, v); }
__device__ __forceinline__ uint64_t warp_xor64(uint64_t v) {
    const uint32_t lo = __reduce_xor_sync(FULL_MASK, static_cast<uint32_t>(v));
    const uint32_t hi = __reduce_xor_sync(FULL_MASK, static_cast<uint32_t>(v >> 32));
    return (static_cast<uint64_t>(hi) << 32) | lo;
}
// Exact 64-bit sum (mod 2^64) of one value per lane: three pieces of 22, 22
// and 20 bits, each of whose 32-lane sums fits 32 bits.
__device__ __forceinline__ uint64_t warp_add64(uint64_t v) {
    const uint32_t p0 = __reduce_add_sync(FULL_MASK, static_cast<uint32_t>(v) & 0x3FFFFFu);
    const uint32_t p1 = __reduce_add_sync(FULL_MASK, static_cast<uint32_t>(v >> 22) & 0x3FFFFFu);
    const uint32_t p2 = __reduce_add_sync(FULL_MASK, static_cast<uint32_t>(v >> 44));
    return static_cast<uint64_t>(p0) + (static_cast<uint64_t>(p1) << 22) + (static_cast<uint64_t>(p2) << 44);
}

// Reduction of one partial per lane: every lane ends with the warp total
// (integer parts exact; float pairs combined as double-float with TwoSum, in
// the butterfly's fixed order).
template <int DT>
__device__ __forceinline__ void warp_merge(uint32_t& s, uint64_t& x, uint64_t& n, float& hi, float& lo) {
    s = warp_add32(s);
    x = warp_xor64(x);
    n = warp_add64(n);
    if constexpr (DT != SL_U32) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ohi = __shfl_xor_sync(FULL_MASK, hi, o);
            const float olo = __shfl_xor_sync(FULL_MASK, lo, o);
            df_add(hi, lo, ohi, olo);
        }
    }
}

// Final combine of the partials of all CTAs that took part into one sl_result,
// run by the whole CTA that finished last: thread t folds partials t,
// t+blockDim, ... in index order (FP64 for the float part: (double)hi +
// (double)lo), then the warps and the per-warp results are merged in a fixed
// order, so the float sum has a fixed order for a given launch shape.  Integer
// parts are exact.  The device error word becomes the status and is cleared;
// the CTA counter, the chunk counter (if any) and the timing window are reset
// for the next launch.
//
// This is a chain of L2 round trips at the end of every launch, so what can
// overlap does: the window and the error word are copied to shared memory
// while the partials are read (0.4-0.5 us of every launch), and the integer
// fields are reduced by redux.sync (0.1-0.6 us, most where many warps finish
// at once).  Loops are not unrolled and each field is reduced on its own, so
// that this code needs fewer registers than the streaming loop it follows: one
// more than 32 in the leanest kernels would cost a quarter of their CTAs.
__device__ __forceinline__ void final_combine(const KArgs& a) {
    struct Fin {
        uint32_t sum;
        uint64_t x, n;
        double f;
    };
    __shared__ Fin fw[32];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    const uint32_t n = a.active;
    // the window and the error word (with its 16 bytes) are copied to shared
    // memory while the partials are read: no register holds them
    __shared__ __align__(16) uint64_t swin[2];
    __shared__ __align__(16) uint32_t serr[4];
    if (threadIdx.x == blockDim.x - 1)
        asm volatile("cp.async.cg.shared.global [%0], [%2], 16;\n\tcp.async.cg.shared.global [%1], [%3], 16;"
                     ::"r"(smem_addr(swin)), "r"(smem_addr(serr)), "l"(a.window), "l"(a.err) : "memory");
    Fin v{0u, 0ull, 0ull, 0.0};
#pragma unroll 1
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
        const uint4 lo4 = __ldcg(reinterpret_cast<const uint4*>(a.parts + i));
        const uint4 hi4 = __ldcg(reinterpret_cast<const uint4*>(a.parts + i) + 1);
        v.sum += lo4.x;
        v.x ^= (static_cast<uint64_t>(lo4.w) << 32) | lo4.z;
        v.n += (static_cast<uint64_t>(hi4.y) << 32) | hi4.x;
        v.f += static_cast<double>(__uint_as_float(hi4.z)) + static_cast<double>(__uint_as_float(hi4.w));
    }
    for (int pass = 0; pass < 2; ++pass) {  // pass 0: within warps; pass 1: across warps (warp 0)
        v.sum = warp_add32(v.sum);
        v.x = warp_xor64(v.x);
        v.n = warp_add64(v.n);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v.f += __shfl_xor_sync(FULL_MASK, v.f, o);
        if (pass == 1) break;
        if (lane == 0) fw[warp] = v;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (warp != 0) return;
        v = lane < nw ? fw[lane] : Fin{0u, 0ull, 0ull, 0.0};
    }
    if (lane == 0) {
        // field by field: a whole sl_result in registers would raise the
        // kernel's register count
        sl_result* r = a.result;
        r->xor_u64 = v.x;
        r->issued_loads = v.n;
        r->device_ns = 0;
        const uint64_t t0 = swin[0], t1 = swin[1];
        r->window_ns = t1 > t0 ? t1 - t0 : 0;
        r->fsum = v.f;
        const float hi = static_cast<float>(v.f);
        r->fsum_hi = hi;
        r->fsum_lo = static_cast<float>(v.f - static_cast<double>(hi));
        r->sum_u32 = v.sum;
        r->status = serr[0] ? SL_ERR_TIMEOUT : SL_OK;
        r->grid = 0;
        r->cta = 0;
        r->resident_per_sm = 0;
        r->smem_bytes = 0;
        *a.err = 0;
        *a.done = 0;
        if (a.next) *a.next = 0;
        a.window[0] = ~0ull;
        a.window[1] = 0;
    }
}

// This CTA's %globaltimer start, kept in shared memory by cta_start (below)
// and published by cta_finish.
__device__ __forceinline__ uint64_t& cta_start_stamp() {
    __shared__ uint64_t t0;
    return t0;
}

// End of a streaming kernel: every folding warp (all 32 lanes present)
// reduces its accumulators and lane 0 puts the warp partial in shared memory;
// after a CTA barrier warp 0 merges the warp partials (butterfly, fixed
// order) into the CTA's partial a.parts[blockIdx.x], and thread 0 raises the
// launch's end stamp to this CTA's %globaltimer.  With
// a.result set, the last of the a.active CTAs to get here then runs
// final_combine.  `fw` is
// this warp's index among the nfw (<= 32) folding warps; `cta_err`, if given,
// is a CTA-local error code (shared memory) that thread 0 publishes to *a.err.
template <int DT, bool BIAS = false>
__device__ __forceinline__ void cta_finish(const Acc<DT, BIAS>& acc, bool folds, uint32_t fw, uint32_t nfw,
                                           const KArgs& a, const uint32_t* cta_err = nullptr) {
    __shared__ WarpPartial sp[32];
    const uint32_t lane = threadIdx.x & 31;
    // A pass that started streaming before the previous launch finished
    // (a.overlap) touches the shared scratch (partials,
    // window, CTA counter) only once that launch has completed and its writes
    // are visible; without a prerequisite grid this returns at once.
    // Where launches prefetch (a.prefetch), the next one on the stream may start
    // from here on: its CTAs become resident, prefetch and wait while this
    // launch's last CTAs reduce.  Otherwise it starts as the last CTA exits: its
    // CTAs then find empty SMs and spread evenly (16 passes over 32 MiB in L2:
    // 34.6 us, 39.9 where they are placed beside this launch's, 36.9 as an
    // ordinary launch; 16 MiB 6.35 us against 6.63).
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "setp.ne.u32 p, %0, 0;\n\t"
                 "griddepcontrol.wait;\n\t"
                 "@p griddepcontrol.launch_dependents;\n\t}" ::"r"(a.prefetch) : "memory");
    if (folds) {
        uint32_t s = acc.s;
        uint64_t x = (static_cast<uint64_t>(acc.xh) << 32) | acc.xl, n = acc.n;
        float hi = 0.0f, lo = 0.0f;
        if constexpr (DT != SL_U32) acc.float_part(hi, lo);
        warp_merge<DT>(s, x, n, hi, lo);
        if (lane == 0) {
            WarpPartial p;
            p.sum = s;
            p.pad = 0;
            p.xr = x;
            p.issued = n;
            p.hi = hi;
            p.lo = lo;
            sp[fw] = p;
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        uint32_t s = 0;
        uint64_t x = 0, n = 0;
        float hi = 0.0f, lo = 0.0f;
        if (lane < nfw) {
            const WarpPartial p = sp[lane];
            s = p.sum;
            x = p.xr;
            n = p.issued;
            hi = p.hi;
            lo = p.lo;
        }
        warp_merge<DT>(s, x, n, hi, lo);
        if (lane == 0) {
            WarpPartial p;
            p.sum = s;
            p.pad = 0;
            p.xr = x;
            p.issued = n;
            p.hi = hi;
            p.lo = lo;
            a.parts[blockIdx.x] = p;
            if (cta_err && *cta_err) atomicCAS(a.err, 0u, *cta_err);  // before this CTA is counted done
            atomicMin(reinterpret_cast<unsigned long long*>(a.window), cta_start_stamp());
            atomicMax(reinterpret_cast<unsigned long long*>(a.window + 1), gtimer());
        }
    }
    if (a.result == nullptr) return;
    // Last-CTA-done: publish this CTA's partial, count it, and let the CTA
    // that completes the count combine everything.
    __shared__ int s_last;
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = (atomicAdd(a.done, 1u) == a.active - 1);
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        final_combine(a);
    }
}

// Tile cursor over the grid-stride sequence it = blockIdx.x, +gridDim.x, ...
// tm = it mod ntiles (the pass-local tile), tracked without division.  32-bit:
// the host keeps total tiles + grid below 2^32.
struct TileCursor {
    uint32_t it, tm;
    __device__ __forceinline__ void start(uint32_t ntiles) {
        it = blockIdx.x;
        tm = blockIdx.x % ntiles;
    }
    __device__ __forceinline__ void next(uint32_t ntiles) {
        it += gridDim.x;
        tm += gridDim.x;
        while (tm >= ntiles) tm -= ntiles;
    }
    __device__ __forceinline__ uint32_t tile(const KArgs& a) const {
        return a.desc ? (static_cast<uint32_t>(a.ntiles) - 1 - tm) : tm;
    }
};

// SL_DYN: first unit of the chunk that claim c stands for.
__device__ __forceinline__ uint64_t dyn_chunk(const KArgs& a, uint32_t c) {
    const uint32_t nchunks = static_cast<uint32_t>(a.ntiles);
    if (c >= nchunks) c %= nchunks;  // a later pass
    return static_cast<uint64_t>(c) * a.tile_vec;
}

// SL_DYN: a CTA's first claim is its own index, so that it starts without a
// round trip to the counter; the counter deals the rest.  (Read by hand: with
// blockIdx.x the compiler treats the first chunk apart from the others and some
// kernels take a few registers more.)
__device__ __forceinline__ uint32_t dyn_first() {
    uint32_t c;
    asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(c));
    return c;
}
__device__ __forceinline__ uint32_t dyn_claim(const KArgs& a) { return gridDim.x + atomicAdd(a.next, 1u); }

// Start of a streaming kernel.  An ordinary pass waits until the kernel before
// it on the stream has completed and its writes are visible
// (griddepcontrol.wait; returns at once unless the launch is a programmatic
// dependent one); cta_finish, or its end, lets the next launch on the stream
// begin.  In that order, so that a dependent launch never starts before everything
// ahead of this one is complete, as if this launch had been an ordinary one.
// A pass with a.overlap set (sl_enqueue_steps, whose buffers are only read)
// lets the next launch begin (1; the last pass, 2, does not: what follows it
// would only wait) and streams at once, and waits in cta_finish.
// A CTA that the launch has no tile for (index a.active or more) exits at once,
// so that a small launch does not wait for hundreds of empty partials (64 KiB,
// 8 CTAs of 608 with work: 6.2 -> 4.7 us).  Thread 0 keeps this CTA's
// %globaltimer start in shared memory (no register holds it through the
// kernel).  Nothing here touches the launch's scratch.
//
// A dependent launch with a.prefetch set first asks L2 for what the CTA will
// read first, before it waits: its CTAs are resident during the last few
// microseconds of the kernel before it, when DRAM is nearly idle.  (A prefetch
// returns no data and L2 is where that kernel's writes go, so the loads after
// the wait see them.)  The start stamp is taken before the first of these reads,
// so that the window covers all that the launch reads.  tile_bytes: bytes of one of the launch's tiles (chunks
// for SL_DYN); PF false leaves this out.
template <bool PF = true>
__device__ __forceinline__ void cta_start(const KArgs& a, uint32_t tile_bytes = 0) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .u32 b;\n\t"
                 "mov.u32 b, %%ctaid.x;\n\t"
                 "setp.ge.u32 p, b, %0;\n\t"
                 "@p exit;\n\t}" ::"r"(a.active) : "memory");
    if (PF && a.prefetch && threadIdx.x == 0) {
        cta_start_stamp() = gtimer();
        const uint32_t ntiles = static_cast<uint32_t>(a.ntiles);
        const uint32_t part = tile_bytes < a.prefetch ? tile_bytes : a.prefetch;
        uint32_t it = blockIdx.x;
        for (uint32_t n = 0; n < a.prefetch && it < ntiles; n += part, it += gridDim.x) {
            const uint64_t off = static_cast<uint64_t>(a.desc ? ntiles - 1 - it : it) * tile_bytes;
            const uint64_t left = a.nvec * 16 - off;
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;"
                         ::"l"(static_cast<const char*>(a.buf) + off), "r"(left < part ? static_cast<uint32_t>(left) : part)
                         : "memory");
        }
    }
    asm volatile("{\n\t.reg .pred p, q;\n\t"
                 "setp.eq.s32 p, %0, 0;\n\t"
                 "setp.eq.s32 q, %0, 1;\n\t"
                 "@p griddepcontrol.wait;\n\t"
                 "@q griddepcontrol.launch_dependents;\n\t}" ::"r"(a.overlap) : "memory");
    if ((threadIdx.x | (PF ? a.prefetch : 0u)) == 0) cta_start_stamp() = gtimer();
}

}  // namespace sl
