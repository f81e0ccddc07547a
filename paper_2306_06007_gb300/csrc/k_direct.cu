// Direct evaluation of sub-problems (Sect. 3.1: blocks below a size threshold are
// summed directly, O(n_pix n_vis), Sect. 2) and the point preparation kernels.
//
//   sky -> vis:  V_k += sum_n c_n exp(+isign j 2 pi <p_k, r_n>),  c_n = a_n I_n
//   vis -> sky:  I_n += Re sum_k V_k exp(-isign j 2 pi <p_k, r_n>)
//
// The phase <p, r> reaches ~1e5 turns, so it is never formed in plain FP32. Every
// coordinate is stored as a pair of floats hi + lo (hi = fl32(x), lo = fl32(x - hi)), and the
// tensor cores form the turns modulo one of a tile of pairs from their digits (phase_tc.cuh):
//  * FP32 path (eps >= 1e-6): fraction in FP32 (error ~5e-9 turn rms up to 2^22 turns, 1e-7 at 2^28),
//    hardware sin/cos approximations, FP32 accumulation;
//  * double-float path (eps < 1e-6): exp(j 2 pi f) as the hi parts of a 1024-entry table of
//    exp(j 2 pi m / 1024) plus a lo part (the table's lo parts and a short series in the
//    remainder, in plain float); sums in double-float arithmetic (Dekker 1971). A term is off by
//    1.0e-10 rms and 5.7e-10 at most (restated on the CPU; 5.3e-11 and 2.8e-10 with 2,048 entries,
//    which do not fit eightfold in shared memory) and the sums add nothing to it: rel. l2 of V within
//    1,000 wavelengths 1.3e-10 for 16, 64 and 4,000 pixels (on the FP32 pipes 1.0e-10, 1.45e-10, 2.5e-10);
//  * wide path: the double-float path on the values of an FP32 plan whose |p_d r_d| exceed 2^28
//    turns (the reach of the FP32 digits);
//  * plain path: everything in FP64 (the reference form the optimised paths replace; also, on the
//    plan's own values, for |p_d r_d| above 2^33 turns, the reach of the double-float digits).
//
// What bounds them: at FP32 the sine unit (two results a pair at 8 cycles for 32: 16 cycles of
// the 20 that 32 pairs take), in double-float the FMA pipe (60% busy), the shared-memory pipe (63%)
// and issue (64%) together. FMAs and adds go two to an instruction (f32x2) over two columns or over
// a sum's two parts: they take the FMA pipe as long as two scalar ones but half the issue slots.
// Measured on one GB300 over the 52,812 pixels x 1,435,200 baselines of the LOFAR-like step, all direct,
// both directions, pairs/s: FP32 2.00e12 and double-float 7.9e11; with the phase on the FP32 pipes 1.16e12 and
// 4.7e11, on the tensor cores but without f32x2 1.95e12 and 7.1e11.
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <mutex>
#include <string>
#include <type_traits>

#include "f32x2.cuh"
#include "hvox_internal.h"
#include "phase_tc.cuh"

namespace hvox {

namespace {

using namespace f32x2;

constexpr int kThreads = 256;
constexpr int kPerThread = 2;
constexpr int kTile = kThreads * kPerThread;  // owner points per work item of the FP64 kernels

// ------------------------------------------------------------- point preparation

__global__ void prepare_points_kernel(const double *__restrict__ xyz, const int32_t *__restrict__ perm, int64_t n,
                                      double *__restrict__ soa, float4 *__restrict__ hi, float4 *__restrict__ lo) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t src = perm[i];
    float h[3], l[3];
    for (int d = 0; d < 3; ++d) {
        double x = xyz[3 * src + d];
        soa[d * n + i] = x;
        h[d] = (float)x;
        l[d] = (float)(x - (double)h[d]);
    }
    hi[i] = make_float4(h[0], h[1], h[2], 0.f);
    lo[i] = make_float4(l[0], l[1], l[2], 0.f);
}

__global__ void gather_weight_kernel(const double *__restrict__ w, const int32_t *__restrict__ perm, int64_t n,
                                     double *__restrict__ out) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = w[perm[i]];
}

// ------------------------------------------------------------- float helpers

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ void fast_two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}

// The offset for a tile whose term magnitudes sum to at most S: 2^(floor(log2 S) + 2) > 2 S
// (S from the block's own values; tiny or zero S gives 2^-100).
__device__ __forceinline__ float tile_offset(float S) {
    const unsigned e = __float_as_uint(fmaxf(S, 0x1p-102f)) & 0x7F800000u;
    return __uint_as_float(e + (2u << 23));
}

// Kahan-compensated accumulation of per-tile partial sums: the FP32 paths sum each
// thread's terms of a tile in registers and add the tile sums here, which keeps the
// rounding error of sums over millions of terms near that of a short sum.
__device__ __forceinline__ void kahan_add(float &sum, float &comp, float x) {
    const float y = __fsub_rn(x, comp);
    const float t = __fadd_rn(sum, y);
    comp = __fsub_rn(__fsub_rn(t, sum), y);
    sum = t;
}

// Adds a tile's double-float partial sum (ih + il) into the running sum (oh + ol): the
// tile sums' lo part rounds at ~2^-24 of itself, which over millions of terms
// (1.4M baselines per pixel) grows to ~5e-9 of the result; folding every tile keeps
// that growth to one tile.
__device__ __forceinline__ void df_fold(float &oh, float &ol, float ih, float il) {
    float s, e;
    two_sum(oh, ih, s, e);
    e = __fadd_rn(e, __fadd_rn(ol, il));
    fast_two_sum(s, e, oh, ol);
}

// The next work item of this CTA, taken from the launch's counter (CTA b starts with
// item b; the counter is zero at launch): CTAs that finish early take more items, and
// with the items ordered largest first a launch ends within about one small item of its
// ideal time.
__device__ __forceinline__ int next_item(int *counter, int &s_next) {
    __syncthreads();  // every thread has read the previous s_next
    if (threadIdx.x == 0) s_next = (int)gridDim.x + atomicAdd(counter, 1);
    __syncthreads();
    return s_next;
}

// The pointers of one job of a direct launch: a plan's chunk-ordered buffers. A launch
// serves one job (BATCH false: the kernel parameter J0) or several (BATCH true: work item
// it belongs to job item_job[it] of the device table jobs, so the sums of several plans
// share one launch and its dynamic schedule).
template <bool BATCH>
__device__ __forceinline__ DirectJob job_of(const DirectJob &J0, const DirectJob *__restrict__ jobs,
                                            const int *__restrict__ item_job, int it) {
    if constexpr (BATCH)
        return jobs[item_job[it]];
    else
        return J0;
}

// ------------------------------------------------------------- tiles of pairs

// One work item: 256 owner points [o0, o1) times streamed points [s0, s1). A CTA has 16 consumer
// warps, 2 producer warps and one issuing warp, and runs as a pipeline on mbarriers:
//  * producers write the digits and values of the streamed points, 128 at a time,
//    into one of two tile buffers;
//  * the tensor cores form the digit products of a chunk of kN streamed points (columns) with
//    each block of 128 owners (rows; their digits lie in shared memory for the whole item)
//    into one of two accumulator sets in tensor memory;
//  * one thread issues those products, as soon as a tile is staged and a set has been read;
//  * two groups of four warps share a row block, a thread a row: each reads its half of a
//    chunk's columns into registers and sums them.
constexpr int kRows = 256;              // owners per work item
constexpr int kStream = 128;            // streamed points per tile
constexpr int kConsumers = 2 * kRows;   // threads
constexpr int kProducers = 64;          // threads, each staging kStream / kProducers points of a tile
constexpr int kIssuer = kConsumers + kProducers;  // first thread of the issuing warp
constexpr int kDirectThreads = kIssuer + 32;      // 608: 96 registers a thread

template <class K> struct __align__(128) DirectShared {
    uint4 own[2][K::Form::kMma * 2][128];      // [row block][mma, K half][row]
    uint4 dig[2][K::Form::kMma * 2][kStream];  // [buffer][mma, K half][point]
    typename K::Val val[2][kStream];
    float red[2][kStream / 32];                // per producer warp: sum of the values' magnitudes
    typename K::Extra extra;
    uint64_t done[2][2];                       // [row block][set]: a chunk's products have finished
    uint64_t read[2][2];                       // [row block][set]: its eight warps have read the set
    uint64_t staged[2], freed[2];              // [buffer]: tile written / tile summed by every consumer
    uint64_t drained;                          // after a wait ran out: every product issued has finished
    uint32_t tmem;
    int next, abort;
};

// Chunks and tiles so far in this CTA (the same in every thread): the n-th use of one of two
// buffers is buffer n & 1 and barrier phase n >> 1.
struct DirectPipe {
    uint32_t tmem, chunks, tiles;
};

// A bounded wait: false where it ran out, or one has run out in this CTA before (a wait under way then
// goes on to its own limit; looking at the flag between tries costs the double-float kernels 2%). Then
// nothing waits any longer, no more products are issued, the item's sums become NaN and so do those of
// every item that the CTA takes after it (an item left out would be missing from a finite result); the
// products in flight are waited for before tensor memory is given back (direct_end).
__device__ __noinline__ void give_up(int *abort, int *err) {
    *(volatile int *)abort = 1;
    if (err) atomicOr(err, kDevErrStall);
}

template <class K> __device__ __forceinline__ bool pipe_wait(DirectShared<K> &sh, uint64_t *bar, uint32_t parity, int *err) {
    if (*(volatile int *)&sh.abort) return false;
    for (int i = 0; i < tc::kWaitLimit; ++i)
        if (tc::mbar_try(bar, parity & 1u)) return true;
    give_up(&sh.abort, err);
    return false;
}

// The same for a whole warp. Its lanes poll by themselves and may leave on different tries, while the
// tensor-memory reads (.aligned) that follow need them together.
template <class K> __device__ __forceinline__ void warp_wait(DirectShared<K> &sh, uint64_t *bar, uint32_t parity, int *err) {
    pipe_wait(sh, bar, parity, err);
    __syncwarp();
}

// One producer thread: its points of the tile at s0 (the staged values' magnitudes are summed per
// warp and pass).
template <class K, int DIR>
__device__ __forceinline__ void stage_tile(const DirectJob &J, const WorkItem &w, int s0, DirectShared<K> &sh, int buf) {
    using Side = std::conditional_t<DIR == 0, typename K::Form::R, typename K::Form::P>;
    constexpr int kPasses = kStream / kProducers;
    float4 h[kPasses], l[kPasses];
    typename K::Val val[kPasses];
#pragma unroll
    for (int p = 0; p < kPasses; ++p) {  // every load in flight before the first is used
        const int n = s0 + (int)threadIdx.x - kConsumers + p * kProducers;
        h[p] = l[p] = make_float4(0.f, 0.f, 0.f, 0.f);
        val[p] = typename K::Val{};
        if (n < w.s1) {
            h[p] = J.str_hi[n];
            l[p] = J.str_lo[n];
            val[p] = K::load(J, n);
        }
    }
#pragma unroll
    for (int p = 0; p < kPasses; ++p) {
        const int i = (int)threadIdx.x - kConsumers + p * kProducers;
        tc::write_point<typename K::Form, kStream>(sh.dig[buf], i,
                                                   tc::point_digits<Side>(h[p], l[p], DIR == 0 ? J.pix_scale : J.vis_scale));
        sh.val[buf][i] = val[p];
        if constexpr (K::kMagnitudes) {
            float mag = K::magnitude(val[p]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mag += __shfl_xor_sync(0xffffffffu, mag, o);
            if ((i & 31) == 0) sh.red[buf][i >> 5] = mag;
        }
    }
    tc::fence_smem();
}

// Accumulator columns of a set (tensor memory address without lanes).
template <class K> __device__ __forceinline__ uint32_t set_columns(int block, uint32_t set) {
    return ((uint32_t)block * 2u + set) * (K::Form::kAcc * K::kN);
}

// The issuing thread: the products of every chunk of an item, in order, as tiles are staged and
// accumulator sets read.
template <class K>
__device__ __forceinline__ void issue_chunks(DirectShared<K> &sh, const DirectPipe &pipe, uint32_t chunks, int *err) {
    constexpr uint32_t kPerTile = kStream / K::kN;
    const uint64_t own0 = tc::operand_desc(tc::smem_addr(sh.own), sizeof(sh.own[0][0]));
    const uint64_t dig0 = tc::operand_desc(tc::smem_addr(sh.dig), sizeof(sh.dig[0][0]));
    for (uint32_t c = 0; c < chunks; ++c) {
        const uint32_t n = pipe.chunks + c, set = n & 1u, tile = pipe.tiles + c / kPerTile;
        bool ok = c % kPerTile != 0 || pipe_wait(sh, &sh.staged[tile & 1u], tile >> 1, err);
        const uint64_t dig = dig0 + (((tile & 1u) * sizeof(sh.dig[0]) + (c % kPerTile) * K::kN * 16) >> 4);
#pragma unroll
        for (int block = 0; block < 2; ++block) {
            ok = pipe_wait(sh, &sh.read[block][set], (n >> 1) ^ 1u, err) && ok;
            if (!ok) break;  // and no later chunk is issued: every later wait fails
            tc::fence_after();
            const uint32_t d = pipe.tmem + set_columns<K>(block, set);
#pragma unroll
            for (int m = 0; m < K::Form::kMma; ++m)
                tc::mma<K::kN>(d + K::Form::acc(m) * K::kN, own0 + ((block * sizeof(sh.own[0]) + 2 * m * sizeof(sh.own[0][0])) >> 4),
                               dig + ((2 * m * sizeof(sh.dig[0][0])) >> 4),
                               m > 0 && K::Form::acc(m) == K::Form::acc(m - 1));
            tc::mma_commit(&sh.done[block][set]);
        }
    }
}

// Sums one item; whether a wait ran out (the same in every thread).
template <class K, int DIR>
__device__ __forceinline__ bool direct_item(const DirectJob &J, const WorkItem &w, DirectShared<K> &sh, DirectPipe &pipe) {
    using Form = typename K::Form;
    using Side = std::conditional_t<DIR == 0, typename Form::P, typename Form::R>;
    constexpr uint32_t kPerTile = kStream / K::kN;
    constexpr int kHalf = K::kN / 2, kPart = 8, kParts = kHalf / kPart;  // columns of a chunk per group, per read
    static_assert(kParts % 2 == 0, "parts alternate between two register sets");
    const int tid = threadIdx.x;
    const uint32_t tiles = (uint32_t)(w.s1 - w.s0 + kStream - 1) / kStream;
    const uint32_t chunks = (uint32_t)(w.s1 - w.s0 + K::kN - 1) / K::kN;
    if (tid >= kIssuer) {
        __syncthreads();  // the owners' digits
        if (tid == kIssuer) issue_chunks(sh, pipe, chunks, J.err);
        __syncwarp();
    } else if (tid >= kConsumers) {
        __syncthreads();
        for (uint32_t t = 0; t < tiles; ++t) {
            const uint32_t n = pipe.tiles + t;
            warp_wait(sh, &sh.freed[n & 1u], (n >> 1) ^ 1u, J.err);
            stage_tile<K, DIR>(J, w, w.s0 + (int)t * kStream, sh, n & 1u);
            __syncwarp();
            if ((tid & 31) == 0) tc::mbar_arrive(&sh.staged[n & 1u]);
        }
    } else {
        const int block = tid >> 8, half = (tid >> 7) & 1, row = block * 128 + (tid & 127);
        if (half == 0) {
            float4 h = make_float4(0.f, 0.f, 0.f, 0.f), l = h;
            if (w.o0 + row < w.o1) {
                h = J.own_hi[w.o0 + row];
                l = J.own_lo[w.o0 + row];
            }
            tc::write_point<Form, 128>(sh.own[block], tid & 127,
                                       tc::point_digits<Side>(h, l, DIR == 0 ? J.vis_scale : J.pix_scale));
            tc::fence_smem();
        }
        __syncthreads();
        const uint32_t lanes = pipe.tmem + ((uint32_t)(tid & 96) << 16) + half * kHalf;  // this warp's 32 lanes
        typename K::Sum sum;
        sum.clear();
        // A part (8 columns of every accumulator) is read while the part before it is summed.
        float d[2][Form::kAcc][kPart];
        auto read_part = [&](uint32_t set, int p) {
#pragma unroll
            for (int a = 0; a < Form::kAcc; ++a)
                tc::tmem_load8(d[p & 1][a], lanes + set_columns<K>(block, set) + a * K::kN + p * kPart);
        };
        auto open_chunk = [&](uint32_t c) {  // the chunk's products are done: read its first part
            const uint32_t n = pipe.chunks + c;
            warp_wait(sh, &sh.done[block][n & 1u], n >> 1, J.err);
            tc::fence_after();
            read_part(n & 1u, 0);
        };
        open_chunk(0);
        for (uint32_t c = 0; c < chunks; ++c) {
            const uint32_t set = (pipe.chunks + c) & 1u, tile = pipe.tiles + c / kPerTile, buf = tile & 1u;
            if (c % kPerTile == 0) {
                warp_wait(sh, &sh.staged[buf], tile >> 1, J.err);
                sum.begin(sh.red[buf]);
            }
            const auto *val = &sh.val[buf][(c % kPerTile) * K::kN + half * kHalf];
#pragma unroll
            for (int p = 0; p < kParts; ++p) {
#pragma unroll
                for (int a = 0; a < Form::kAcc; ++a) tc::tmem_load_wait(d[p & 1][a]);
                if (p + 1 < kParts) {
                    read_part(set, p + 1);
                } else {
                    tc::fence_before();
                    __syncwarp();
                    if ((tid & 31) == 0) tc::mbar_arrive(&sh.read[block][set]);
                    if (c + 1 < chunks) open_chunk(c + 1);
                }
                sum.chunk(d[p & 1], val + p * kPart, p * kPart, sh.extra);
            }
            if (c % kPerTile == kPerTile - 1 || c + 1 == chunks) {
                sum.end();
                __syncwarp();
                if ((tid & 31) == 0) tc::mbar_arrive(&sh.freed[buf]);
            }
        }
        if (*(volatile int *)&sh.abort) sum.poison();
        if (w.o0 + row < w.o1) sum.store(J, w.o0 + row);
    }
    pipe.chunks += chunks;
    pipe.tiles += tiles;
    return __syncthreads_or(*(volatile int *)&sh.abort) != 0;
}

// An item that a CTA takes after one of its waits ran out.
template <class K> __device__ __forceinline__ void poison_item(const DirectJob &J, const WorkItem &w) {
    const int k = w.o0 + (int)threadIdx.x;
    if ((int)threadIdx.x < kRows && k < w.o1) {
        typename K::Sum sum;
        sum.clear();
        sum.poison();
        sum.store(J, k);
    }
    if (threadIdx.x == 0 && J.err) atomicOr(J.err, kDevErrStall);
}

// stall (DirectJob::stall): staged tiles wait for more arrivals than ever come.
template <class K> __device__ __forceinline__ DirectPipe direct_begin(DirectShared<K> &sh, int stall) {
    static_assert(4 * K::Form::kAcc * K::kN <= 512 && K::kN % 16 == 0 && kStream % K::kN == 0, "tensor memory of an SM");
    if (threadIdx.x < 32) tc::tmem_alloc(&sh.tmem, 512);
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            for (int b = 0; b < 2; ++b) {
                tc::mbar_init(&sh.done[b][i], 1);
                tc::mbar_init(&sh.read[b][i], 8);
            }
            tc::mbar_init(&sh.staged[i], kProducers / 32 + (stall ? 1 << 19 : 0));
            tc::mbar_init(&sh.freed[i], kConsumers / 32);
        }
        tc::mbar_init(&sh.drained, 1);
        sh.abort = 0;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    return {sh.tmem, 0u, 0u};
}

template <class K> __device__ __forceinline__ void direct_end(DirectShared<K> &sh, const DirectPipe &pipe, bool stopped) {
    // Without the consumers' waits, products may still be reading shared memory and writing tensor memory.
    if (stopped && threadIdx.x == kIssuer) {
        tc::mma_commit(&sh.drained);
        for (int i = 0; i < tc::kWaitLimit && !tc::mbar_try(&sh.drained, 0u); ++i) {}
    }
    __syncwarp();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (threadIdx.x < 32) tc::tmem_free(pipe.tmem, 512);
}

// ------------------------------------------------------------- FP32

// exp(j 2 pi f) for f = A 2^-14 + B 2^-25 turns (A whole, |A| < 2^24): the whole turns of A go
// exactly; the rest (|f| <~ 0.6) is rounded once, in radians, with 2 pi rounded to float (k0) or the next float (k1).
// The hardware cosine of an argument scaled by either has a mean error over a turn, which a sum of N
// positive values (a long baseline's visibility) multiplies by N while the sum itself grows as sqrt(N).
// Measured on a GB300 over 2^20 random pixels and 400 baselines against FP64: k0 alone +1.21e-8, k1 alone
// -6.28e-8, the sine below 6e-10 with either. k1 on 5 of every 32 columns leaves 4e-10 (6 of 32:
// -1.9e-9), and 1.1e-6 for 7.6e-6 on the sums of 2^20 log-normal values (tests/test_sine_mean_gpu.py).
// Two columns (j even and j + 1) at once; of a half chunk's 32, k1 takes 5, 11, 17, 23 and 29.
__device__ __forceinline__ void cis_f32(float2 A, float2 B, int j, float2 &e0, float2 &e1) {
    constexpr float k0 = 6.28318548202514648f, k1 = 6.28318595886230469f;
    const float2 k = make_float2(k0, (j + 1) % 6 == 5 ? k1 : k0);
    const float2 M = both(0x1.8p23f * 0x1p14f);  // adding it rounds to whole turns, A being in units of 2^-14
    const float2 a = sub2(A, sub2(add2(A, M), M));
    const float2 x = fma2(a, make_float2(k.x * 0x1p-14f, k.y * 0x1p-14f), mul2(B, make_float2(k.x * 0x1p-25f, k.y * 0x1p-25f)));
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(e0.x) : "f"(x.x));
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(e0.y) : "f"(x.x));
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(e1.x) : "f"(x.y));
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(e1.y) : "f"(x.y));
}

struct NoExtra {};

// sky -> vis: c cos and c sin. vis -> sky: Re(V e^{-isign j 2 pi t}) = Vr cos + isign Vi sin, a sum each.
template <int DIR> struct F32Sum {
    float re, im, cre, cim;
    float2 t;  // the tile's sums
    __device__ __forceinline__ void clear() { re = im = cre = cim = 0.f; }
    __device__ __forceinline__ void poison() { re = im = __int_as_float(0x7fc00000); }
    __device__ __forceinline__ void begin(const float *) { t = both(0.f); }
    template <int N>
    __device__ __forceinline__ void chunk(const float (&d)[2][N], const float2 *c, int j0, const NoExtra &) {
#pragma unroll
        for (int j = 0; j < N; j += 2) {
            const float4 v = *reinterpret_cast<const float4 *>(c + j);
            float2 e0, e1;
            cis_f32(make_float2(d[0][j], d[0][j + 1]), make_float2(d[1][j], d[1][j + 1]), j0 + j, e0, e1);
            t = fma2(make_float2(v.x, v.y), e0, t);
            t = fma2(make_float2(v.z, v.w), e1, t);
        }
    }
    __device__ __forceinline__ void end() {
        if constexpr (DIR == 0) {
            kahan_add(re, cre, t.x);
            kahan_add(im, cim, t.y);
        } else {
            kahan_add(re, cre, t.x + t.y);
        }
    }
    __device__ __forceinline__ void store(const DirectJob &J, int k) const {
        if constexpr (DIR == 0) {
            float2 *acc = static_cast<float2 *>(J.acc);
            atomicAdd(&acc[k].x, __fsub_rn(re, cre));
            atomicAdd(&acc[k].y, J.sgn * __fsub_rn(im, cim));
        } else {
            atomicAdd(static_cast<float *>(J.acc) + k, __fsub_rn(re, cre));
        }
    }
};

template <int DIR> struct F32Kind {
    using Form = tc::F32Form;
    using Val = float2;  // (c, c), or V with isign on its imaginary part
    using Sum = F32Sum<DIR>;
    using Extra = NoExtra;
    static constexpr int kN = 64;
    static constexpr bool kMagnitudes = false;
    static __device__ __forceinline__ Val load(const DirectJob &J, int n) {
        if constexpr (DIR == 0) {
            return both(static_cast<const float *>(J.val)[n]);
        } else {
            float2 v = static_cast<const float2 *>(J.val)[n];
            v.y *= J.sgn;
            return v;
        }
    }
};

// ------------------------------------------------------------- double-float

constexpr int kDfTab = 1024;   // entries per turn of the sine table
constexpr int kDfCopies = 8;   // one copy of each entry per lane of a quarter warp

struct DfTable {
    float4 e[kDfTab * kDfCopies];  // entry m, copy c: (cos_h, sin_h, cos_l, sin_l) of 2 pi m / 1024
};

// exp(j 2 pi f) as (reh + rel) + j (imh + iml), f = (A - 1.5 2^23) / 1024 + B 2^-20 + C1 2^-31 + C2 2^-42
// turns (A whole). The nearest 1/1024 turn to the rest joins A and picks the table entry (the
// table's hi parts, exact floats); the remainder x (in units of 2^-20 turn, |x| <= 2^9) is formed
// exactly but for its last rounding (2^-36 turn) and rotates the entry through cos x - 1 =
// -x^2/2, sin x = x - x^3/6 in plain float. tab: the shared address of this lane's copy of the table.
// Two columns at once; eh, el: (re, im) of each.
__device__ __forceinline__ void cis_df(float2 A, float2 B, float2 C1, float2 C2, uint32_t tab, float2 (&eh)[2], float2 (&el)[2]) {
    const float2 tt = fma2(fma2(C1, both(0x1p-11f), B), both(0x1p-10f), A);  // 1.5 2^23 + entry
    const float2 d = fma2(sub2(tt, A), both(-1024.f), B);
    const float2 x = fma2(C2, both(0x1p-22f), fma2(C1, both(0x1p-11f), d));
    constexpr float k = 6.28318530717958648f * 0x1p-20f;
    const float2 x2 = mul2(x, x);
    const float2 cm = mul2(x2, both(-0.5f * k * k));
    const float2 sx = mul2(x, fma2(x2, both(-k * k * k / 6.0f), both(k)));
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const uint32_t at = ((__float_as_uint(i ? tt.y : tt.x) & (kDfTab - 1)) * (16u * kDfCopies)) + tab;
        float2 l;
        asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(eh[i].x), "=f"(eh[i].y), "=f"(l.x), "=f"(l.y) : "r"(at));
        const float c = i ? cm.y : cm.x, s = i ? sx.y : sx.x;
        el[i].x = __fmaf_rn(-eh[i].y, s, __fmaf_rn(eh[i].x, c, l.x));
        el[i].y = __fmaf_rn(eh[i].x, s, __fmaf_rn(eh[i].y, c, l.y));
    }
}

// Offset double-float accumulation of one streamed tile: h += (ch + cl)(eh + el). The running
// high sum starts at a power of two M above twice the tile's sum of term magnitudes S, so
// it stays in [M - S, M + S]: h - h' is exact, and the part of both products that the two
// FMAs rounded off is recovered by FMAs on that difference and collected in l with cl eh.
// At the tile's end h - M is exact (Sterbenz). Two sums at once: the real and imaginary part of a
// visibility, or the products with the real and with the imaginary part of V of a pixel.
struct DfAcc {
    float2 h, l;  // tile sums (h offset by M)
    __device__ __forceinline__ void mac(float2 ch, float2 cl, float2 eh, float2 el) {
        const float2 s = fma2(ch, el, fma2(ch, eh, h));
        float2 u = fma2(ch, eh, sub2(h, s));
        u = fma2(cl, eh, fma2(ch, el, u));
        h = s;
        l = add2(l, u);
    }
};

template <int DIR, class T> struct DfSum {
    DfAcc a;
    float M, oh[2], ol[2];  // running sums
    __device__ __forceinline__ void clear() { oh[0] = oh[1] = ol[0] = ol[1] = 0.f; }
    __device__ __forceinline__ void poison() { oh[0] = oh[1] = __int_as_float(0x7fc00000); }
    __device__ __forceinline__ void begin(const float *red) {
        float S = 0.f;
#pragma unroll
        for (int i = 0; i < kStream / 32; ++i) S += red[i];
        M = tile_offset(1.01f * S);
        a.h = both(M);
        a.l = both(0.f);
    }
    template <int N>
    __device__ __forceinline__ void chunk(const float (&d)[4][N], const float4 *v, int, const DfTable &table) {
        const uint32_t tab = tc::smem_addr(&table.e[threadIdx.x & (kDfCopies - 1)]);
#pragma unroll
        for (int j = 0; j < N; j += 2) {
            float2 eh[2], el[2];
            cis_df(make_float2(d[0][j], d[0][j + 1]), make_float2(d[1][j], d[1][j + 1]), make_float2(d[2][j], d[2][j + 1]),
                   make_float2(d[3][j], d[3][j + 1]), tab, eh, el);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float4 c = v[j + i];
                a.mac(make_float2(c.x, c.y), make_float2(c.z, c.w), eh[i], el[i]);
            }
        }
    }
    __device__ __forceinline__ void end() {
        df_fold(oh[0], ol[0], __fsub_rn(a.h.x, M), a.l.x);
        df_fold(oh[1], ol[1], __fsub_rn(a.h.y, M), a.l.y);
    }
    __device__ __forceinline__ void store(const DirectJob &J, int k) const {
        const double re = (double)oh[0] + (double)ol[0], im = (double)oh[1] + (double)ol[1];
        T *acc = static_cast<T *>(J.acc) + (size_t)k * (DIR == 0 ? 2 : 1);
        if constexpr (DIR == 0) {
            atomicAdd(acc, (T)re);
            atomicAdd(acc + 1, (T)((double)J.sgn * im));
        } else {
            atomicAdd(acc, (T)(re + im));
        }
    }
};

// The sine table takes 128 KB: 8 copies make every read of a quarter warp conflict-free, where
// 8 lanes reading one table at random met ~2.6 times in a bank group.
// T: the plan's real type (float: the wide path).
template <int DIR, class T> struct DfKind {
    using Form = tc::DfForm;
    using Val = float4;  // (c_h, c_h, c_l, c_l), or (Vr_h, Vi_h, Vr_l, Vi_l) with isign on Vi
    using Sum = DfSum<DIR, T>;
    using Extra = DfTable;
    static constexpr int kN = 32;
    static constexpr bool kMagnitudes = true;
    static __device__ __forceinline__ Val load(const DirectJob &J, int n) {
        const T *v = static_cast<const T *>(J.val) + (size_t)n * (DIR == 0 ? 1 : 2);
        const float rh = (float)v[0], rl = (float)(v[0] - (T)rh);
        if constexpr (DIR == 0) {
            return make_float4(rh, rh, rl, rl);
        } else {
            const T vi = (T)J.sgn * v[1];
            const float ih = (float)vi;
            return make_float4(rh, ih, rl, (float)(vi - (T)ih));
        }
    }
    // each pair adds at most |c| or |Vr| + |Vi| to a sum
    static __device__ __forceinline__ float magnitude(const Val &v) {
        if constexpr (DIR == 0) return fabsf(v.x);
        else return fabsf(v.x) + fabsf(v.y);
    }
};

// gT (double-float): exp(j 2 pi m / 2048), m = 0 .. 2047, as float pairs; every other entry is kept.
template <class K, int DIR, bool BATCH>
__global__ void __launch_bounds__(kDirectThreads, 1)
    direct_kernel(const WorkItem *__restrict__ items, int n_items, int *__restrict__ counter, const DirectJob J0,
                  const DirectJob *__restrict__ jobs, const int *__restrict__ item_job, const float4 *__restrict__ gT) {
    extern __shared__ __align__(128) unsigned char direct_smem[];
    DirectShared<K> &sh = *reinterpret_cast<DirectShared<K> *>(direct_smem);
    DirectPipe pipe = direct_begin(sh, J0.stall);
    if constexpr (K::kMagnitudes)
        for (int i = threadIdx.x; i < kDfTab * kDfCopies; i += kDirectThreads) {
            const float4 e = gT[2 * (i / kDfCopies)];
            sh.extra.e[i] = make_float4(e.x, e.z, e.y, e.w);
        }
    bool stopped = false;
    for (int it = blockIdx.x; it < n_items; it = next_item(counter, sh.next)) {
        const DirectJob J = job_of<BATCH>(J0, jobs, item_job, it);
        if (stopped)
            poison_item<K>(J, items[it]);
        else
            stopped = direct_item<K, DIR>(J, items[it], sh, pipe);
    }
    direct_end(sh, pipe, stopped);
}

// ------------------------------------------------------------- FP64

template <class T> using cplx_of = std::conditional_t<sizeof(T) == 4, float2, double2>;

// Plain FP64 reference form (T: the plan's real type).
template <class T, int VPT>
__global__ void __launch_bounds__(kThreads) direct_s2v_f64(const WorkItem *__restrict__ items, int n_items, int *__restrict__ counter,
                                                           const double *__restrict__ vxyz, int64_t nv_all,
                                                           const double *__restrict__ pxyz, int64_t np_all,
                                                           const T *__restrict__ c, cplx_of<T> *__restrict__ acc,
                                                           double sgn) {
    __shared__ double sx[kThreads], sy[kThreads], sz[kThreads], sw[kThreads];
    __shared__ int s_next;
    for (int it = blockIdx.x; it < n_items; it = next_item(counter, s_next)) {
        const WorkItem w = items[it];
        double px[VPT], py[VPT], pz[VPT], are[VPT], aim[VPT];
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            int k = w.o0 + threadIdx.x + v * kThreads;
            bool ok = k < w.o1;
            px[v] = ok ? vxyz[k] : 0.0;
            py[v] = ok ? vxyz[nv_all + k] : 0.0;
            pz[v] = ok ? vxyz[2 * nv_all + k] : 0.0;
            are[v] = aim[v] = 0.0;
        }
        for (int s0 = w.s0; s0 < w.s1; s0 += kThreads) {
            __syncthreads();
            int n = s0 + threadIdx.x;
            bool ok = n < w.s1;
            sx[threadIdx.x] = ok ? pxyz[n] : 0.0;
            sy[threadIdx.x] = ok ? pxyz[np_all + n] : 0.0;
            sz[threadIdx.x] = ok ? pxyz[2 * np_all + n] : 0.0;
            sw[threadIdx.x] = ok ? (double)c[n] : 0.0;
            __syncthreads();
            const int cnt = min(kThreads, w.s1 - s0);
            for (int q = 0; q < cnt; ++q) {
#pragma unroll
                for (int v = 0; v < VPT; ++v) {
                    double t = fma(px[v], sx[q], fma(py[v], sy[q], pz[v] * sz[q]));
                    t -= rint(t);
                    double sn, cs;
                    sincospi(2.0 * t, &sn, &cs);
                    are[v] = fma(sw[q], cs, are[v]);
                    aim[v] = fma(sw[q], sn, aim[v]);
                }
            }
        }
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            int k = w.o0 + threadIdx.x + v * kThreads;
            if (k < w.o1) {
                atomicAdd(&acc[k].x, (T)are[v]);
                atomicAdd(&acc[k].y, (T)(sgn * aim[v]));
            }
        }
    }
}

template <class T, int VPT>
__global__ void __launch_bounds__(kThreads) direct_v2s_f64(const WorkItem *__restrict__ items, int n_items, int *__restrict__ counter,
                                                           const double *__restrict__ pxyz, int64_t np_all,
                                                           const double *__restrict__ vxyz, int64_t nv_all,
                                                           const cplx_of<T> *__restrict__ V, T *__restrict__ acc,
                                                           double sgn) {
    __shared__ double sx[kThreads], sy[kThreads], sz[kThreads], sr[kThreads], si[kThreads];
    __shared__ int s_next;
    for (int it = blockIdx.x; it < n_items; it = next_item(counter, s_next)) {
        const WorkItem w = items[it];
        double rx[VPT], ry[VPT], rz[VPT], a[VPT];
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            int n = w.o0 + threadIdx.x + v * kThreads;
            bool ok = n < w.o1;
            rx[v] = ok ? pxyz[n] : 0.0;
            ry[v] = ok ? pxyz[np_all + n] : 0.0;
            rz[v] = ok ? pxyz[2 * np_all + n] : 0.0;
            a[v] = 0.0;
        }
        for (int s0 = w.s0; s0 < w.s1; s0 += kThreads) {
            __syncthreads();
            int k = s0 + threadIdx.x;
            bool ok = k < w.s1;
            sx[threadIdx.x] = ok ? vxyz[k] : 0.0;
            sy[threadIdx.x] = ok ? vxyz[nv_all + k] : 0.0;
            sz[threadIdx.x] = ok ? vxyz[2 * nv_all + k] : 0.0;
            sr[threadIdx.x] = ok ? (double)V[k].x : 0.0;
            si[threadIdx.x] = ok ? sgn * (double)V[k].y : 0.0;
            __syncthreads();
            const int cnt = min(kThreads, w.s1 - s0);
            for (int q = 0; q < cnt; ++q) {
#pragma unroll
                for (int v = 0; v < VPT; ++v) {
                    double t = fma(sx[q], rx[v], fma(sy[q], ry[v], sz[q] * rz[v]));
                    t -= rint(t);
                    double sn, cs;
                    sincospi(2.0 * t, &sn, &cs);
                    a[v] = fma(sr[q], cs, fma(si[q], sn, a[v]));
                }
            }
        }
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            int n = w.o0 + threadIdx.x + v * kThreads;
            if (n < w.o1) atomicAdd(&acc[n], (T)a[v]);
        }
    }
}

}  // namespace

// ------------------------------------------------------------- launchers

void launch_prepare_points(const double *xyz, const int32_t *perm, int64_t n, double *soa, float4 *hi, float4 *lo,
                           cudaStream_t s) {
    if (n <= 0) return;
    prepare_points_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(xyz, perm, n, soa, hi, lo);
    check_cuda(cudaGetLastError(), "prepare_points");
}

void launch_gather_weight(const double *w, const int32_t *perm, int64_t n, double *out, cudaStream_t s) {
    if (n <= 0) return;
    gather_weight_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(w, perm, n, out);
    check_cuda(cudaGetLastError(), "gather_weight");
}

int direct_tile(int kind) { return kind == kDirectF64 ? kTile : kRows; }

int direct_owners_per_thread(int kind) { return kind == kDirectF64 ? kPerThread : 1; }

static int sm_count() {
    static std::atomic<int> sms[256];
    const int dev = current_device();
    int n = dev < 256 ? sms[dev].load() : 0;
    if (n == 0) {
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 152;
        if (dev < 256) sms[dev].store(n);
    }
    return n;
}

// A persistent grid: the CTAs that are resident together (per_sm on every SM), at most one per item.
static unsigned grid_for(int64_t n_items, int per_sm) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(n_items, (int64_t)sm_count() * per_sm));
}

// Dynamic shared memory of a kernel (Kernel names it).
template <class Kernel, class F> static void allow_smem(F kernel, size_t bytes) {
    static OncePerDevice once;
    once.run(current_device(), [&] {
        check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes),
                   "cudaFuncSetAttribute");
    });
}

template <class K, int DIR, bool BATCH> struct DirectOnce {};

template <class K, int DIR, bool BATCH>
static void launch_one(const WorkItem *items, int64_t n, int *counter, const DirectJob &J, const DirectJob *jobs,
                       const int *item_job, const float4 *tab, cudaStream_t s) {
    constexpr size_t smem = sizeof(DirectShared<K>);
    static_assert(smem <= 226 * 1024, "shared memory of an SM");
    allow_smem<DirectOnce<K, DIR, BATCH>>(direct_kernel<K, DIR, BATCH>, smem);
    direct_kernel<K, DIR, BATCH><<<grid_for(n, 1), kDirectThreads, smem, s>>>(items, (int)n, counter, J, jobs,
                                                                                 item_job, tab);
    check_cuda(cudaGetLastError(), "direct sums");
}

template <bool BATCH>
static void launch_kind(int kind, int dir, const WorkItem *items, int64_t n, int *counter, const DirectJob &J,
                        const DirectJob *jobs, const int *item_job, const float4 *tab, cudaStream_t s) {
#define HVOX_DIRECT(...)                                                                            \
    if (dir == 0)                                                                                   \
        launch_one<__VA_ARGS__(0), 0, BATCH>(items, n, counter, J, jobs, item_job, tab, s);         \
    else                                                                                            \
        launch_one<__VA_ARGS__(1), 1, BATCH>(items, n, counter, J, jobs, item_job, tab, s)
#define HVOX_F32(D) F32Kind<D>
#define HVOX_DF(D) DfKind<D, double>
#define HVOX_WIDE(D) DfKind<D, float>
    if (kind == kDirectF32) {
        HVOX_DIRECT(HVOX_F32);
    } else if (kind == kDirectDf) {
        HVOX_DIRECT(HVOX_DF);
    } else {
        HVOX_DIRECT(HVOX_WIDE);
    }
#undef HVOX_DIRECT
#undef HVOX_F32
#undef HVOX_DF
#undef HVOX_WIDE
}

void launch_direct(int kind, int dir, const WorkItem *items, int64_t n, int *counter, const DirectJob &J,
                   const float4 *tab, cudaStream_t s) {
    if (n > 0) launch_kind<false>(kind, dir, items, n, counter, J, nullptr, nullptr, tab, s);
}

void launch_direct_batch(int kind, int dir, const WorkItem *items, int64_t n, int *counter, const DirectJob *jobs,
                         const int *item_job, const float4 *tab, bool stall, cudaStream_t s) {
    DirectJob all{};
    all.stall = stall;
    if (n > 0) launch_kind<true>(kind, dir, items, n, counter, all, jobs, item_job, tab, s);
}

template <class T>
static void launch_f64(int dir, const WorkItem *items, int64_t n, int *counter, const double *vxyz, int64_t nv,
                       const double *pxyz, int64_t np, const void *src, void *acc, double sgn, cudaStream_t s) {
    if (dir == 0)
        direct_s2v_f64<T, kPerThread><<<grid_for(n, 4), kThreads, 0, s>>>(
            items, (int)n, counter, vxyz, nv, pxyz, np, static_cast<const T *>(src), static_cast<cplx_of<T> *>(acc), sgn);
    else
        direct_v2s_f64<T, kPerThread><<<grid_for(n, 4), kThreads, 0, s>>>(
            items, (int)n, counter, pxyz, np, vxyz, nv, static_cast<const cplx_of<T> *>(src), static_cast<T *>(acc), sgn);
    check_cuda(cudaGetLastError(), "direct sums (FP64)");
}

void launch_direct_f64(int prec, int dir, const WorkItem *items, int64_t n, int *counter, const double *vxyz, int64_t nv,
                       const double *pxyz, int64_t np, const void *src, void *acc, int isign, cudaStream_t s) {
    if (n <= 0) return;
    const auto launch = prec == 1 ? launch_f64<float> : launch_f64<double>;
    launch(dir, items, n, counter, vxyz, nv, pxyz, np, src, acc, (double)isign, s);
}

}  // namespace hvox

// ============================================================================
// Direct sky -> vis evaluation that allocates nothing.
//
// For callers that cannot call cudaMalloc: code that runs inside another framework
// which has reserved the device's memory for its own pool (a cudaMalloc there fails or
// fragments that pool), and iteration loops such as calibration solvers that predict
// visibilities from a sky model every step, where an allocation (and the device
// synchronisation cudaFree brings) is not allowed. The caller passes device pointers
// for everything; the only working memory is the static array below. CUDA reserves it on
// a device when it loads this file's device code there (lazily by default: at the first
// call of the entry point or the first direct-sum launch of any plan on that device) and
// keeps it until the process exits.
// ============================================================================

namespace hvox {

namespace {

constexpr int64_t kNoAllocMaxPoints = int64_t(1) << 19;  // n_pix + n_vis <= 524,288

// hi and lo float splits of the pixel and baseline coordinates: 2 * 524,288 float4 = 16 MiB; then
// the largest |coordinate| of the pixels and of the baselines of the call as float bits.
__device__ __align__(256) float4 g_noalloc_scratch[2 * kNoAllocMaxPoints + 1];

// One launch before the sums: coordinate splits of pixels and baselines, V cleared, and the
// largest |coordinate| of each set (non-negative floats order as integers; top[0..1] zero at launch).
__global__ void noalloc_prepare_kernel(const double *__restrict__ pix, int64_t n_pix, const double *__restrict__ uvw,
                                       int64_t n_vis, float4 *__restrict__ scratch, unsigned *__restrict__ top,
                                       float2 *__restrict__ V) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    float m = 0.f;
    const bool p = i < n_pix;
    if (i < n_pix + n_vis) {
        const int64_t k = p ? i : i - n_pix;
        const double *xyz = (p ? pix : uvw) + 3 * k;
        float4 *hi = p ? scratch : scratch + 2 * n_pix, *lo = hi + (p ? n_pix : n_vis);
        float h[3], l[3];
        for (int d = 0; d < 3; ++d) {
            h[d] = (float)xyz[d];
            l[d] = (float)(xyz[d] - (double)h[d]);
            m = fmaxf(m, fabsf(h[d]));
        }
        hi[k] = make_float4(h[0], h[1], h[2], 0.f);
        lo[k] = make_float4(l[0], l[1], l[2], 0.f);
        if (!p) V[k] = make_float2(0.f, 0.f);
    }
    const unsigned bits = __float_as_uint(m);
    const unsigned mp = __reduce_max_sync(0xffffffffu, p ? bits : 0u), mv = __reduce_max_sync(0xffffffffu, p ? 0u : bits);
    if ((threadIdx.x & 31) == 0 && mp != 0u) atomicMax(top, mp);
    if ((threadIdx.x & 31) == 0 && mv != 0u) atomicMax(top + 1, mv);
}

// The FP32 direct sums (beyond the FP32 digits' reach the wide form, beyond that FP64) over items in a fixed order
// instead of a work list; the segments' sums meet in V through atomicAdd, so their order (and
// the last bits of the result) is not deterministic.
template <class K>
__device__ __forceinline__ void noalloc_items(const DirectJob &J, int n_vis, int n_pix, int seg, unsigned char *smem) {
    DirectShared<K> &sh = *reinterpret_cast<DirectShared<K> *>(smem);
    DirectPipe pipe = direct_begin(sh, J.stall);
    if constexpr (K::kMagnitudes)
        for (int i = threadIdx.x; i < kDfTab; i += kDirectThreads) {
            double sn, cs;
            sincospi(2.0 * i / kDfTab, &sn, &cs);
            const float ch = (float)cs, sh_ = (float)sn;
            const float4 e = make_float4(ch, sh_, (float)(cs - (double)ch), (float)(sn - (double)sh_));
            for (int c = 0; c < kDfCopies; ++c) sh.extra.e[i * kDfCopies + c] = e;
        }
    const int tiles = (n_vis + kRows - 1) / kRows, items = tiles * ((n_pix + seg - 1) / seg);
    bool stopped = false;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {  // direct_item ends in a barrier
        const int o0 = it % tiles * kRows, s0 = it / tiles * seg;
        const WorkItem w{o0, min(o0 + kRows, n_vis), s0, min(s0 + seg, n_pix)};
        if (stopped)
            poison_item<K>(J, w);
        else
            stopped = direct_item<K, 0>(J, w, sh, pipe);
    }
    direct_end(sh, pipe, stopped);
}

// The same in FP64, an owner to a thread: correct where the digits end, and not tuned (no instrument has 2^33
// turns).
__device__ __noinline__ void noalloc_items_f64(const double *__restrict__ pix, const double *__restrict__ uvw,
                                               const float *__restrict__ c, float2 *__restrict__ acc, double sgn,
                                               int n_vis, int n_pix, int seg) {
    const int tiles = (n_vis + kRows - 1) / kRows, items = tiles * ((n_pix + seg - 1) / seg);
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int k = it % tiles * kRows + (int)threadIdx.x, s0 = it / tiles * seg;
        if ((int)threadIdx.x >= kRows || k >= n_vis) continue;
        double re = 0.0, im = 0.0;
        for (int n = s0; n < min(s0 + seg, n_pix); ++n) {
            double t = fma(uvw[3 * (int64_t)k], pix[3 * (int64_t)n],
                           fma(uvw[3 * (int64_t)k + 1], pix[3 * (int64_t)n + 1], uvw[3 * (int64_t)k + 2] * pix[3 * (int64_t)n + 2]));
            t -= rint(t);
            double sn, cs;
            sincospi(2.0 * t, &sn, &cs);
            re = fma((double)c[n], cs, re);
            im = fma((double)c[n], sn, im);
        }
        atomicAdd(&acc[k].x, (float)re);
        atomicAdd(&acc[k].y, (float)(sgn * im));
    }
}

__global__ void __launch_bounds__(kDirectThreads, 1)
    direct_noalloc_kernel(DirectJob J, int n_vis, int n_pix, int seg, const unsigned *__restrict__ top,
                          const double *__restrict__ pix, const double *__restrict__ uvw) {
    extern __shared__ __align__(128) unsigned char direct_smem[];
    coord_scales(__uint_as_float(top[0]), J.pix_scale, J.vis_scale);
    const float far = __uint_as_float(top[1]) * J.vis_scale;
    if (far <= kF32Reach)
        noalloc_items<F32Kind<0>>(J, n_vis, n_pix, seg, direct_smem);
    else if (far <= kDfReach)
        noalloc_items<DfKind<0, float>>(J, n_vis, n_pix, seg, direct_smem);
    else
        noalloc_items_f64(pix, uvw, static_cast<const float *>(J.val), static_cast<float2 *>(J.acc), (double)J.sgn, n_vis,
                          n_pix, seg);
}

std::mutex g_noalloc_mu;
void *g_noalloc_ptr[256] = {nullptr};

// Device address of the static scratch for the current device. The first call on a
// device looks it up (cudaGetSymbolAddress, no allocation) with that device current.
float4 *noalloc_scratch_for_current_device() {
    int dev = 0;
    check_cuda(cudaGetDevice(&dev), "cudaGetDevice");
    if (dev < 0 || dev >= 256) fail(HVOX_EUNSUPPORTED, "hvox_direct_synthesize_noalloc: device index out of range");
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *ptr = nullptr;
        check_cuda(cudaGetSymbolAddress(&ptr, g_noalloc_scratch), "cudaGetSymbolAddress");
        g_noalloc_ptr[dev] = ptr;
    }
    return static_cast<float4 *>(g_noalloc_ptr[dev]);
}

bool on_device(const void *p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

}  // namespace hvox

extern "C" hvox_status hvox_direct_synthesize_noalloc(const double *pix_xyz, int64_t n_pix, const double *uvw,
                                                      int64_t n_vis, const float *I, float *V, int isign,
                                                      void *stream) {
    using namespace hvox;
    try {
        if (!pix_xyz || !uvw || !I || !V) fail(HVOX_EINVAL, "hvox_direct_synthesize_noalloc: NULL pointer");
        if (n_pix < 1 || n_vis < 1) fail(HVOX_EINVAL, "hvox_direct_synthesize_noalloc: need n_pix, n_vis >= 1");
        if (n_pix + n_vis > kNoAllocMaxPoints)
            fail(HVOX_EINVAL, "hvox_direct_synthesize_noalloc: n_pix + n_vis = " + std::to_string(n_pix + n_vis) +
                                  " exceeds the static limit of " + std::to_string(kNoAllocMaxPoints) + " points");
        if (isign != 1 && isign != -1) fail(HVOX_EINVAL, "hvox_direct_synthesize_noalloc: isign must be +1 or -1");
        if (!on_device(pix_xyz) || !on_device(uvw) || !on_device(I) || !on_device(V))
            fail(HVOX_EINVAL, "hvox_direct_synthesize_noalloc: every pointer must be device memory");
        cudaStream_t s = (cudaStream_t)stream;
        float4 *scratch = noalloc_scratch_for_current_device();
        float4 *rh = scratch, *rl = scratch + n_pix;
        float4 *vh = scratch + 2 * n_pix, *vl = vh + n_vis;
        unsigned *top = reinterpret_cast<unsigned *>(scratch + 2 * kNoAllocMaxPoints);
        check_cuda(cudaMemsetAsync(top, 0, 2 * sizeof(unsigned), s), "clear coordinate maxima");
        noalloc_prepare_kernel<<<(unsigned)((n_pix + n_vis + 255) / 256), 256, 0, s>>>(
            pix_xyz, n_pix, uvw, n_vis, scratch, top, reinterpret_cast<float2 *>(V));
        check_cuda(cudaGetLastError(), "noalloc_prepare");
        const int64_t tiles = (n_vis + kRows - 1) / kRows;
        const int64_t seg = direct_segment(tiles, n_pix), items = tiles * ((n_pix + seg - 1) / seg);
        const DirectJob J{vh, vl, rh, rl, I, V, (float)isign, 1.f, 1.f, nullptr, fault_hit("stall")};
        constexpr size_t smem = sizeof(DirectShared<DfKind<0, float>>);
        static_assert(smem >= sizeof(DirectShared<F32Kind<0>>), "either form");
        allow_smem<DirectJob>(direct_noalloc_kernel, smem);
        direct_noalloc_kernel<<<grid_for(items, 1), kDirectThreads, smem, s>>>(J, (int)n_vis, (int)n_pix, (int)seg, top,
                                                                                     pix_xyz, uvw);
        check_cuda(cudaGetLastError(), "direct_noalloc");
        set_error("");
        return HVOX_OK;
    } catch (const Error &e) {
        set_error(e.msg);
        return e.code;
    } catch (const std::exception &e) {
        set_error(std::string("internal error: ") + e.what());
        return HVOX_EINTERNAL;
    }
}
