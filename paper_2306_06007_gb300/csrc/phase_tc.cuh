// Turn counts <p, r> mod 1 of tiles of point pairs on the 5th-generation tensor cores.
//
// The direct sums need the fraction of <p, r> (up to ~1e5 turns and more) to 1e-8 .. 1e-11
// turn for every pair, and forming it on the FP32 pipes was most of their cost (~20 of 28
// instructions a pair at FP32, ~40 of 73 in double-float). It is a contraction over the three
// dimensions, so here it is a matrix product: every coordinate is written in balanced
// digits of 11 bits, x = sum_i x_i 2^(a - 11 i) with whole |x_i| <= 2^10 (exact in fp16),
// and the digit products of one weight are summed by one tcgen05.mma (f16 operands, FP32
// accumulators: products of two digits and sums of up to 15 of them stay below 2^24, so
// these sums are exact). Products whose weight is a whole number of turns are left out, so
// integer turns of any size cost nothing; the products below a turn are grouped by weight
// into one accumulator per group. tcgen05 with accumulators in TMEM rather than mma.sync: the
// contraction itself is short (K = 48 or 80), but an mma.sync m16n8k16 holds up the FP32
// pipes it shares registers with for ~6 cycles and starts its accumulators with register
// moves (measured with mma.sync: 21.9 cycles for 32 pairs at FP32 and 62.6 in double-float).
//
// Digit weights (p scaled by 2^e and r by 2^-e so that |r_d| <= 1):
//  double-float (|p_d| <= 2^33): P: 2^23, 2^12, 2^1, 2^-10, 2^-21, 2^-32, 2^-43; R: 2^-10, 2^-21, ...,
//    2^-54; accumulators A (weight 2^-9 turn), B (2^-20), C1 (2^-31), each exact, and C2 (2^-42 and
//    2^-53); the dropped products are below 2^-43 turn (rms);
//  FP32 (|p_d| <= 2^28): P: 2^18, 2^7, 2^-4, R: 2^-10, 2^-21, 2^-32, and the rest of each as two fp16
//    values (one for R's rest loses 2^-12 of it, which the digit at 2^18 multiplies: 1.8e-5 radians rms
//    at 2^27.8 turns); accumulators A (weight 2^-14, exact) and B (all below, units of 2^-25, at most
//    ~0.3 turn). The dropped products are below 2^-28 turn each. Phase error, restated on the CPU over
//    uniform baselines up to 2^k turns, radians rms: 3e-8 to k = 22, 5e-8 at 24, 1.7e-7 at 26 and 6e-7 at
//    27.8, where the float pairs themselves round; 1.4e-7 to k = 22 on the FP32 pipes.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace hvox {
namespace tc {

constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23

// ------------------------------------------------------------------ digits

// Nearest whole number of x k, |x k| < 2^22, on the FMA pipe.
__device__ __forceinline__ float nearest(float x, float k) { return __fsub_rn(__fmaf_rn(x, k, kMagic), kMagic); }

// The nearest digit of x at weight w (exact inverse iw), taken off x (exactly: x and the
// digit's value share their low bits).
__device__ __forceinline__ float digit(float &x, float w, float iw) {
    const float d = nearest(x, iw);
    x = __fmaf_rn(-d, w, x);
    return d;
}

// The whole number d modulo 2^k (m = 2^k, im = 2^-k), in [-m/2, m/2].
__device__ __forceinline__ float mod_pow2(float d, float m, float im) { return __fmaf_rn(nearest(d, im), -m, d); }

__device__ __forceinline__ void two_sum_into(float &s, float &e, float b) {  // s + b = s' + e exactly
    const float a = s;
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ uint32_t half2_bits(float lo, float hi) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// One term of a digit product: digit indices of the two sides; the three dimensions follow one
// another in K. An index of -1 pads.
struct Term {
    int8_t p, r;
};

// Double-float operands. Digits P: 0 .. 6 (weights 2^23 .. 2^-43), R: 0 .. 4 (2^-10 .. 2^-54). Group
// A counts half sine-table entries of 1/1024 turn: its P digits (and the R digit of the
// largest p) only modulo 512, doubled, so that |A| < 2^22; a sixteenth product adds 1.5 2^23, so
// that A arrives as the offset that rounds the rest to whole entries.
struct DfForm {
    static constexpr int kMma = 5, kAcc = 4;
    static __host__ __device__ constexpr int acc(int m) { return m < 4 ? m : 3; }
    static __host__ __device__ constexpr Term term(int m, int c) {
        constexpr Term terms[kMma][5] = {
            {{0, 2}, {1, 1}, {2, 0}, {-1, -1}, {-1, -1}},  // A:  2^-9
            {{0, 3}, {1, 2}, {2, 1}, {3, 0}, {-1, -1}},    // B:  2^-20
            {{0, 4}, {1, 3}, {2, 2}, {3, 1}, {4, 0}},      // C1: 2^-31
            {{1, 4}, {2, 3}, {3, 2}, {4, 1}, {5, 0}},      // C2: 2^-42
            {{2, 4}, {3, 3}, {4, 2}, {5, 1}, {6, 0}},      // C2: 2^-53, the P digit scaled by 2^-11
        };
        return terms[m][c];
    }

    // R side (pixels): x = hi + lo, |x| <= 1.
    struct R {
        float d[3][5], d2m[3];
        __device__ __forceinline__ void set(int k, float hi, float lo) {
            float s = hi, e;
            d[k][0] = digit(s, 0x1p-10f, 0x1p10f);
            d[k][1] = digit(s, 0x1p-21f, 0x1p21f);
            two_sum_into(s, e, lo);
            d[k][2] = digit(s, 0x1p-32f, 0x1p32f);
            s = __fadd_rn(s, e);
            d[k][3] = digit(s, 0x1p-43f, 0x1p43f);
            d[k][4] = nearest(s, 0x1p54f);
            d2m[k] = mod_pow2(d[k][2], 0x1p9f, 0x1p-9f);
        }
        __device__ __forceinline__ float slot(int m, int s) const {
            const int c = s / 3;
            if (m == 0 && s == 15) return 2048.f;  // with the P side's 6144: 1.5 2^23
            if (!(c < 5 && term(m, c).r >= 0)) return 0.f;
            return m == 0 && c == 0 ? d2m[s - 3 * c] : d[s - 3 * c][term(m, c).r];
        }
    };

    // P side (baselines): x = hi + lo.
    struct P {
        float d[3][7];
        __device__ __forceinline__ void set(int k, float hi, float lo) {
            float s = hi, e;
            d[k][0] = digit(s, 0x1p23f, 0x1p-23f);
            d[k][1] = digit(s, 0x1p12f, 0x1p-12f);
            two_sum_into(s, e, lo);
            d[k][2] = digit(s, 0x1p1f, 0x1p-1f);
            two_sum_into(s, e, e);
            d[k][3] = digit(s, 0x1p-10f, 0x1p10f);
            s = __fadd_rn(s, e);
            d[k][4] = digit(s, 0x1p-21f, 0x1p21f);
            d[k][5] = digit(s, 0x1p-32f, 0x1p32f);
            d[k][6] = nearest(s, 0x1p43f);
        }
        __device__ __forceinline__ float slot(int m, int s) const {
            const int c = s / 3;
            if (m == 0 && s == 15) return 6144.f;
            if (!(c < 5 && term(m, c).p >= 0)) return 0.f;
            const float v = d[s - 3 * c][term(m, c).p];
            return m == 0 ? 2.f * mod_pow2(v, 0x1p9f, 0x1p-9f) : m == 4 ? v * 0x1p-11f : v;
        }
    };
};

// FP32 operands. Digits P: 0 .. 2 (2^18, 2^7, 2^-4), 3 and 4 the rest as fp16 values in units
// of 2^-15; R: 0 .. 2 (2^-10, 2^-21, 2^-32), 3 and 4 the rest in units of 2^-43. The products of weight
// 2^-3 turn count modulo 8 only.
struct F32Form {
    static constexpr int kMma = 3, kAcc = 2;
    static __host__ __device__ constexpr int acc(int m) { return m < 1 ? 0 : 1; }
    static __host__ __device__ constexpr Term term(int m, int c) {
        constexpr Term terms[kMma][5] = {
            {{0, 2}, {1, 1}, {2, 0}, {0, 1}, {1, 0}},  // A: 2^-14; the last two 2^-3 (P scaled by 2^11)
            {{0, 3}, {1, 2}, {2, 1}, {3, 0}, {4, 0}},  // B: 2^-25
            {{1, 3}, {2, 2}, {3, 1}, {3, 2}, {0, 4}},  // B: 2^-36 (R scaled by 2^-11), 2^-47 (2^-22), 2^-25
        };
        return terms[m][c];
    }

    struct R {
        float d[3][5], m8[3][2];
        __device__ __forceinline__ void set(int k, float hi, float lo) {
            float s = hi, e;
            d[k][0] = digit(s, 0x1p-10f, 0x1p10f);
            d[k][1] = digit(s, 0x1p-21f, 0x1p21f);
            two_sum_into(s, e, lo);
            d[k][2] = digit(s, 0x1p-32f, 0x1p32f);
            s = __fmul_rn(__fadd_rn(s, e), 0x1p43f);
            d[k][3] = __half2float(__float2half_rn(s));
            d[k][4] = __fsub_rn(s, d[k][3]);
            m8[k][0] = mod_pow2(d[k][0], 8.f, 0.125f);
            m8[k][1] = mod_pow2(d[k][1], 8.f, 0.125f);
        }
        __device__ __forceinline__ float slot(int m, int s) const {
            const int c = s / 3;
            if (!(c < 5 && term(m, c).r >= 0)) return 0.f;
            if (m == 0 && c >= 3) return m8[s - 3 * c][term(m, c).r];
            const float v = d[s - 3 * c][term(m, c).r];
            return m < 2 || c == 4 ? v : v * (c == 3 ? 0x1p-22f : 0x1p-11f);
        }
    };

    struct P {
        float d[3][5], m8[3][2];
        __device__ __forceinline__ void set(int k, float hi, float lo) {
            float s = hi, e;
            d[k][0] = digit(s, 0x1p18f, 0x1p-18f);
            d[k][1] = digit(s, 0x1p7f, 0x1p-7f);
            two_sum_into(s, e, lo);
            d[k][2] = digit(s, 0x1p-4f, 0x1p4f);
            s = __fmul_rn(__fadd_rn(s, e), 0x1p15f);
            d[k][3] = __half2float(__float2half_rn(s));
            d[k][4] = __fsub_rn(s, d[k][3]);
            m8[k][0] = 0x1p11f * mod_pow2(d[k][0], 8.f, 0.125f);
            m8[k][1] = 0x1p11f * mod_pow2(d[k][1], 8.f, 0.125f);
        }
        __device__ __forceinline__ float slot(int m, int s) const {
            const int c = s / 3;
            if (!(c < 5 && term(m, c).p >= 0)) return 0.f;
            return m == 0 && c >= 3 ? m8[s - 3 * c][term(m, c).p] : d[s - 3 * c][term(m, c).p];
        }
    };
};

// The digits of one point. hi, lo: its float splits; sc: the power of two of its side (2^-e for
// pixels, 2^e for baselines).
template <class Side> __device__ __forceinline__ Side point_digits(const float4 &hi, const float4 &lo, float sc) {
    Side v;
    v.set(0, hi.x * sc, lo.x * sc);
    v.set(1, hi.y * sc, lo.y * sc);
    v.set(2, hi.z * sc, lo.z * sc);
    return v;
}

// Writes a point's operands: 16 bytes (8 fp16 in K order) into each of the planes [mma][K half][row].
template <class Form, int ROWS, class Side>
__device__ __forceinline__ void write_point(uint4 (*planes)[ROWS], int row, const Side &v) {
#pragma unroll
    for (int p = 0; p < 2 * Form::kMma; ++p) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = half2_bits(v.slot(p / 2, (p & 1) * 8 + 2 * j), v.slot(p / 2, (p & 1) * 8 + 2 * j + 1));
        planes[p][row] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// ------------------------------------------------------------------ tcgen05

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Allocates / frees tensor memory columns (whole warp); the address arrives in *out (shared).
__device__ __forceinline__ void tmem_alloc(uint32_t *out, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(out)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t addr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols));
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Shared memory written by this thread becomes visible to the tensor cores' reads.
__device__ __forceinline__ void fence_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Waits up to ~20 us for the barrier's phase `parity` to complete.
__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 20000;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Tries before a wait gives up: 0.37 s measured, which no healthy launch reaches.
constexpr int kWaitLimit = 100000;

// 8 columns of this thread's row of an accumulator.
__device__ __forceinline__ void tmem_load8(float *d, uint32_t addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3]), "=f"(d[4]), "=f"(d[5]), "=f"(d[6]), "=f"(d[7])
                 : "r"(addr));
}
// Waits for this thread's loads; the operands tie the registers they fill to the wait.
__device__ __forceinline__ void tmem_load_wait(float *d) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]), "+f"(d[4]), "+f"(d[5]), "+f"(d[6]), "+f"(d[7])::"memory");
}

// Operand in shared memory without swizzle: two planes (K 0 .. 7 and 8 .. 15) of 16 bytes a row, `plane`
// bytes apart.
__device__ __forceinline__ uint64_t operand_desc(uint32_t smem, uint32_t plane) {
    return (uint64_t)((smem >> 4) & 0x3FFF) | ((uint64_t)(plane >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
}

// D (128 x N, tensor memory) = A (128 x 16) B (N x 16)^T, added to D with `add`.
template <int N> __device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, bool add) {
    constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24);  // f16 x f16 -> f32
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)add)
        : "memory");
}
// The barrier completes a phase when this thread's mmas so far have finished.
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
                 : "memory");
}

}  // namespace tc
}  // namespace hvox
