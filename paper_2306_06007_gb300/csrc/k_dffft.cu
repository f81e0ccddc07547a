// Double-float FFT for the FP64 grids of NUFFT sub-problems (eps < 1e-6), the uniform FFT of
// step 2 of the type-3 transform (Sect. 3).
//
// GB300 runs FP64 at 1/63 of its FP32 rate, and cuFFT's Z2Z transforms of these grids are
// bound by the FP64 units (~17x the C2C time per cell). Here every value is an unevaluated
// pair of floats (hi + lo, ~48 bits; Dekker 1971 with FMA products) and every 1-D transform
// runs in shared memory on the FP32 pipes: Stockham auto-sorting stages of radix 4, 2, 3, 5
// and 7 (the odd radices through the symmetric form X_k, X_{r-k} = A_k +- s i B_k, half the
// multiplications of a plain DFT), with twiddles exp(2 pi i q / n) computed in FP64 on the
// host and stored as float pairs. One pass per dimension; each reads and writes only what the n1
// band leaves (the grid is zero outside it before the transform, unread outside it after):
//   rows (x): one band row per CTA, multiplied by 1/Psi and padded from the FP64 n1 grid on the way in
//     (sky -> vis), or cropped into it and multiplied on the way out (vis -> sky);
//   columns (y): two adjacent columns per CTA (32-byte sectors), every column of a band plane;
//   columns (z): 64 adjacent columns per CTA, the planes of a batch interleaved.
// A pass's first stage reads the grid and its last one writes it: two barriers and two trips
// through shared memory less than staging the whole sequence, and no deconvolution pass. Measured
// over both directions of a 2160 x 2240 x 28 grid with the band 1436 x 1472 x 16: FFT and deconvolution
// 10.2 -> 8.7 ms. What bounds the passes: FP32 issue and its latency (rows and columns 60 to 66%
// of the issue slots, 47% of the warps an SM can hold), not HBM.
// Transforms are unnormalised, sign s = -1 or +1: X_k = sum_q x_q exp(s 2 pi i q k / n).
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "dfloat.cuh"
#include "hvox_internal.h"

namespace hvox {

namespace {

using namespace df;

// 256 threads per CTA, held to 64 registers so that four CTAs fit an SM where shared memory
// allows (a fourth CTA hides more of each CTA's load phase and stage barriers).
constexpr int kFftThreads = 256;

struct DC {
    DF re, im;
};

__device__ __forceinline__ DC cadd(const DC &a, const DC &b) { return {dadd(a.re, b.re), dadd(a.im, b.im)}; }
__device__ __forceinline__ DC csub(const DC &a, const DC &b) { return {dadd(a.re, dneg(b.re)), dadd(a.im, dneg(b.im))}; }

// Sums and products whose results only feed further sums (within one butterfly) skip their
// renormalisation (dadd_lazy); the outputs a butterfly stores are renormalised.
__device__ __forceinline__ DC cadd_lazy(const DC &a, const DC &b) {
    return {dadd_lazy(a.re, b.re), dadd_lazy(a.im, b.im)};
}
__device__ __forceinline__ DC csub_lazy(const DC &a, const DC &b) {
    return {dadd_lazy(a.re, dneg(b.re)), dadd_lazy(a.im, dneg(b.im))};
}

// a * (c + j s) for real double-float c, s (unnormalised, it feeds the butterfly's sums).
__device__ __forceinline__ DC cmul_lazy(const DC &a, DF c, DF s) {
    return {dmul2_lazy(a.re, c, a.im, s, -1.f), dmul2_lazy(a.re, s, a.im, c, 1.f)};
}

// a * (j SG) for SG = +-1 (sign flips only).
template <int SG> __device__ __forceinline__ DC times_j(const DC &a) {
    if constexpr (SG > 0) return {dneg(a.im), a.re};
    else return {a.im, dneg(a.re)};
}

__device__ __forceinline__ DC from4(float4 v) { return {{v.x, v.y}, {v.z, v.w}}; }
__device__ __forceinline__ float4 to4(const DC &c) { return make_float4(c.re.h, c.re.l, c.im.h, c.im.l); }

__device__ __forceinline__ float4 load_f64(const double2 *p) {
    const double2 v = *p;
    const DF re = split_bits(v.x), im = split_bits(v.y);
    return make_float4(re.h, re.l, im.h, im.l);
}
// A grid cell in either format: FP64 (double2) or, between the passes of one transform, the
// double-float form itself (float4 of the same 16 bytes; zero is all-zero bits in both).
template <bool F64> __device__ __forceinline__ float4 load_cell(double2 *p) {
    if constexpr (F64) return load_f64(p);
    else return *reinterpret_cast<const float4 *>(p);
}

// Twiddle exp(SG 2 pi i e / n) from the table of exp(2 pi i q / n) (cos h, cos l, sin h, sin l).
template <int SG> __device__ __forceinline__ void twiddle(const float4 *__restrict__ tw, int e, DF &c, DF &s) {
    const float4 t = __ldg(tw + e);
    c = {t.x, t.y};
    s = SG > 0 ? DF{t.z, t.w} : DF{-t.z, -t.w};
}

// One Stockham stage of radix R over TX interleaved sequences: butterfly j (of n / R) reads
// elements j + q n / R, twiddles them by exp(s 2 pi i q k span / n) (k = j mod Ns) and writes
// the R outputs to (j / Ns) Ns R + k + q Ns. q k span < n, so the table index needs no wrap.
// The sign SG of the exponent is a template parameter: its flips fold into the operands.
// ld(e, t) reads element e of sequence t, st(e, t, v) writes it: shared memory between
// stages, the grid itself in the first and the last stage of a pass.
template <int R, int TX, int SG, class Ld, class St>
__device__ __forceinline__ void stage(Ld ld, St st, const DfftDev &d, int Ns, unsigned magic) {
    const int n = d.n, m = n / R, span = n / (Ns * R);
    for (int wk = threadIdx.x; wk < m * TX; wk += blockDim.x) {
        const int j = wk / TX, t = wk - j * TX;
        DC v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = from4(ld(j + q * m, t));
        const int jn = Ns == 1 ? j : (int)__umulhi((unsigned)j, magic), k = j - jn * Ns;
        if (k != 0) {
#pragma unroll
            for (int q = 1; q < R; ++q) {
                DF c, s;
                twiddle<SG>(d.tw, q * k * span, c, s);
                v[q] = cmul_lazy(v[q], c, s);
            }
        }
        DC y[R];
        if constexpr (R == 2) {
            y[0] = cadd(v[0], v[1]);
            y[1] = csub(v[0], v[1]);
        } else if constexpr (R == 4) {
            const DC a0 = cadd_lazy(v[0], v[2]), a1 = csub_lazy(v[0], v[2]);
            const DC b0 = cadd_lazy(v[1], v[3]), b1 = times_j<SG>(csub_lazy(v[1], v[3]));
            y[0] = cadd(a0, b0);
            y[1] = cadd(a1, b1);
            y[2] = csub(a0, b0);
            y[3] = csub(a1, b1);
        } else {
            // odd R: s_q = v_q + v_{R-q}, d_q = v_q - v_{R-q} (q = 1 .. H); X_0 = v_0 + sum s_q;
            // A_k = v_0 + sum s_q cos(2 pi q k / R), B_k = sum d_q sin(2 pi q k / R);
            // X_k = A_k + s j B_k, X_{R-k} = A_k - s j B_k. The coefficients come from the
            // kernel parameters at compile-time offsets (constant-bank operands).
            constexpr int H = R / 2;
            constexpr int off = R == 3 ? 0 : (R == 5 ? 1 : 5);
            DC sq[H], dq[H];
#pragma unroll
            for (int q = 1; q <= H; ++q) {
                sq[q - 1] = cadd_lazy(v[q], v[R - q]);
                dq[q - 1] = csub_lazy(v[q], v[R - q]);
            }
            {
                DAcc re = acc_of(v[0].re), im = acc_of(v[0].im);
#pragma unroll
                for (int q = 0; q < H; ++q) {
                    acc_add(re, sq[q].re.h, sq[q].re.l);
                    acc_add(im, sq[q].im.h, sq[q].im.l);
                }
                y[0] = {acc_done(re), acc_done(im)};
            }
#pragma unroll
            for (int kk = 1; kk <= H; ++kk) {
                DAcc ar = acc_of(v[0].re), ai = acc_of(v[0].im), br, bi;
#pragma unroll
                for (int q = 1; q <= H; ++q) {
                    const float4 cs = d.odd[off + (q - 1) * H + (kk - 1)];
                    const DF c = {cs.x, cs.y}, sn = {cs.z, cs.w};
                    acc_fma(ar, sq[q - 1].re, c);
                    acc_fma(ai, sq[q - 1].im, c);
                    if (q == 1) {
                        br = acc_mul(dq[0].re, sn);
                        bi = acc_mul(dq[0].im, sn);
                    } else {
                        acc_fma(br, dq[q - 1].re, sn);
                        acc_fma(bi, dq[q - 1].im, sn);
                    }
                }
                const DC A = {acc_lazy(ar), acc_lazy(ai)};
                const DC jb = times_j<SG>({acc_lazy(br), acc_lazy(bi)});
                y[kk] = cadd(A, jb);
                y[R - kk] = csub(A, jb);
            }
        }
        const int base = jn * Ns * R + k;
#pragma unroll
        for (int q = 0; q < R; ++q) st(base + q * Ns, t, to4(y[q]));
    }
}

// Element accessors: shared memory (element e of sequence t at e TX + t) and a tile of TX
// grid columns (columns t >= valid of a ragged tile read as 0, never written).
template <int TX> struct SmemLd {
    const float4 *a;
    __device__ __forceinline__ float4 operator()(int e, int t) const { return a[e * TX + t]; }
};
template <int TX> struct SmemSt {
    float4 *b;
    __device__ __forceinline__ void operator()(int e, int t, float4 v) const { b[e * TX + t] = v; }
};
// Elements outside the band [0, h) and [n - h, n) (gap = n - 2 h) read as zero and are not written.
__device__ __forceinline__ bool in_band(int e, int h, int gap) { return (unsigned)(e - h) >= (unsigned)gap; }
template <bool F64> struct ColLd {
    double2 *base;
    int64_t stride;
    int valid, h, gap;
    __device__ __forceinline__ float4 operator()(int e, int t) const {
        return t < valid && in_band(e, h, gap) ? load_cell<F64>(base + e * stride + t) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
};
struct ColSt {
    double2 *base;
    int64_t stride;
    int valid, h, gap;
    __device__ __forceinline__ void operator()(int e, int t, float4 v) const {
        if (t < valid && in_band(e, h, gap)) *reinterpret_cast<float4 *>(base + e * stride + t) = v;
    }
};
// A row of the n2 grid, and the row of the n1 grid it comes from (FP64, multiplied by 1/Psi and padded) or
// goes to (float pairs, cropped and multiplied): band element e is n1 element e + h or e - h - gap.
struct RowLd {
    const double2 *row;
    __device__ __forceinline__ float4 operator()(int e, int) const { return *reinterpret_cast<const float4 *>(row + e); }
};
struct RowSt {
    double2 *row;
    __device__ __forceinline__ void operator()(int e, int, float4 v) const { *reinterpret_cast<float4 *>(row + e) = v; }
};
struct BandLd {
    const double2 *in;
    const double *px;
    double fyz;
    int h, gap;
    __device__ __forceinline__ float4 operator()(int e, int) const {
        if (!in_band(e, h, gap)) return make_float4(0.f, 0.f, 0.f, 0.f);
        const int i = e < h ? e + h : e - h - gap;
        const double2 g = in[i];
        const double f = px[i] * fyz;
        const DF re = split_bits(g.x * f), im = split_bits(g.y * f);
        return make_float4(re.h, re.l, im.h, im.l);
    }
};
struct BandSt {
    float4 *out;
    const double *px;
    double fyz;
    int h, gap;
    __device__ __forceinline__ void operator()(int e, int, float4 v) const {
        if (!in_band(e, h, gap)) return;
        const int i = e < h ? e + h : e - h - gap;
        const DF f = split_bits(px[i] * fyz);
        const DF re = dmul({v.x, v.y}, f), im = dmul({v.z, v.w}, f);
        out[i] = make_float4(re.h, re.l, im.h, im.l);
    }
};

template <int TX, int SG, class Ld, class St>
__device__ __forceinline__ void run_stage(int r, Ld ld, St st, const DfftDev &d, int Ns, unsigned mg) {
    switch (r) {
        case 4: stage<4, TX, SG>(ld, st, d, Ns, mg); break;
        case 2: stage<2, TX, SG>(ld, st, d, Ns, mg); break;
        case 3: stage<3, TX, SG>(ld, st, d, Ns, mg); break;
        case 5: stage<5, TX, SG>(ld, st, d, Ns, mg); break;
        default: stage<7, TX, SG>(ld, st, d, Ns, mg); break;
    }
}

// Transforms of TX interleaved sequences of length n held in the grid: the first stage
// reads the grid, the last writes it back, the stages between ping-pong through the
// shared buffers a and b (a only for two stages, none for one). The grid is read only in
// the first stage and written only in the last, with a barrier between them (one stage:
// each thread reads every input of the butterflies it writes), so in-place is safe.
template <int TX, int SG, class GLd, class GSt>
__device__ __forceinline__ void fft_pass(float4 *a, float4 *b, const DfftDev &d, GLd gld, GSt gst) {
    const int S = d.stages;
    if (S == 1) {
        run_stage<TX, SG>(d.radix[0], gld, gst, d, 1, d.ns_magic[0]);
        return;
    }
    run_stage<TX, SG>(d.radix[0], gld, SmemSt<TX>{a}, d, 1, d.ns_magic[0]);
    __syncthreads();
    int Ns = d.radix[0];
    for (int st = 1; st < S - 1; ++st) {
        run_stage<TX, SG>(d.radix[st], SmemLd<TX>{a}, SmemSt<TX>{b}, d, Ns, d.ns_magic[st]);
        __syncthreads();
        float4 *tmp = a;
        a = b;
        b = tmp;
        Ns *= d.radix[st];
    }
    run_stage<TX, SG>(d.radix[S - 1], SmemLd<TX>{a}, gst, d, Ns, d.ns_magic[S - 1]);
}

// Shared buffers a pass needs for a transform of s stages (see fft_pass).
inline int pass_buffers(int s) { return s >= 3 ? 2 : s - 1; }

// Linear index of a band plane (the n1 band's z planes of a batch: the lower slab's
// half K planes, then the upper slab's) -> plane number in the interleaved layout.
__device__ __forceinline__ int64_t band_plane(int64_t P, int64_t halfK, int64_t n2z, int64_t K, int64_t half) {
    return P < halfK ? P : (n2z - half) * K + (P - halfK);
}

// Rows (x): sequence s = (band plane P, band row R), R < 2 h1y. OUT false: n1 grid -> n2 rows, true: n2 rows ->
// n1 grid.
template <int SG, bool OUT>
__global__ void __launch_bounds__(kFftThreads, 4)
    dfft_rows_kernel(double2 *__restrict__ g, DfftDev d, int n2y, int n2z, int K, int h1x, int h1y, int h1z,
                     const NufftDev *__restrict__ descs, void *__restrict__ g1, const double *__restrict__ ipsi) {
    extern __shared__ float4 smem[];
    const int n = d.n, rows = 2 * h1y;
    const int64_t P = blockIdx.x / rows;
    const int R = (int)(blockIdx.x - P * rows);
    const int iz2 = (int)(P / K), grid = (int)(P - (int64_t)iz2 * K);  // lower slab, then upper slab
    const int jz = iz2 < h1z ? iz2 : n2z - 2 * h1z + iz2, jy = R < h1y ? R : n2y - rows + R;
    const int iz = iz2 < h1z ? iz2 + h1z : iz2 - h1z, iy = R < h1y ? R + h1y : R - h1y;
    const NufftDev &b = descs[grid];
    const double *px = ipsi + b.psi_off, *py = px + 2 * h1x, *pz = py + rows;
    const double fyz = py[iy] * pz[iz];
    const int64_t band = b.g1_off + ((int64_t)iz * rows + iy) * 2 * h1x;
    double2 *row = g + (((int64_t)jz * K + grid) * n2y + jy) * n;
    if constexpr (OUT)
        fft_pass<1, SG>(smem, smem + n, d, RowLd{row}, BandSt{static_cast<float4 *>(g1) + band, px, fyz, h1x, n - 2 * h1x});
    else
        fft_pass<1, SG>(smem, smem + n, d, BandLd{static_cast<const double2 *>(g1) + band, px, fyz, h1x, n - 2 * h1x}, RowSt{row});
}

// Columns: TX adjacent columns starting at column c0 of a plane (y: columns of one band plane,
// stride n2x; z: every column of the batch, stride K n2x n2y), element q at c + q * stride.
// (hi, gi): band of the input, (ho, go): of the output.
struct ColBands {
    int hi, gi, ho, go;
};
template <int TX, int SG, bool IN64>
__global__ void __launch_bounds__(kFftThreads, 4) dfft_cols_kernel(double2 *__restrict__ g, DfftDev d, int64_t stride,
                                                                 int64_t ncols, int64_t plane_cells, int64_t halfK,
                                                                 int64_t n2z, int64_t K, int64_t half, int band, ColBands b) {
    extern __shared__ float4 smem[];
    const int64_t tiles = (ncols + TX - 1) / TX;
    const int64_t P = blockIdx.x / tiles, c0 = (blockIdx.x - P * tiles) * TX;
    double2 *base = g + (band ? band_plane(P, halfK, n2z, K, half) * plane_cells : 0) + c0;
    const int valid = ncols - c0 < TX ? (int)(ncols - c0) : TX;
    fft_pass<TX, SG>(smem, smem + (size_t)d.n * TX, d, ColLd<IN64>{base, stride, valid, b.hi, b.gi},
                     ColSt{base, stride, valid, b.ho, b.go});
}

constexpr size_t kFftSmemMax = 220 * 1024;

template <typename K> void allow_smem(K kernel) {
    check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFftSmemMax),
               "cudaFuncSetAttribute");
}

template <int TX, int SG> void allow_cols() {
    allow_smem(dfft_cols_kernel<TX, SG, false>);
    allow_smem(dfft_cols_kernel<TX, SG, true>);
}

template <int SG> void allow_sign() {
    allow_smem(dfft_rows_kernel<SG, true>);
    allow_smem(dfft_rows_kernel<SG, false>);
    allow_cols<1, SG>();
    allow_cols<2, SG>();
    allow_cols<8, SG>();
    allow_cols<64, SG>();
}

void set_fft_attrs() {
    static OncePerDevice once;
    once.run(current_device(), [] {
        allow_sign<1>();
        allow_sign<-1>();
    });
}

// Columns per CTA for a column transform of length n: as many as the shared memory holds
// (two buffers of n TX cells of 16 bytes), at most `want`.
int cols_per_cta(int n, int want) {
    for (int tx : {64, 8, 2, 1})
        if (tx <= want && (size_t)2 * n * tx * 16 <= kFftSmemMax) return tx;
    return 0;
}

template <int TX, int SG>
void launch_cols(bool in64, double2 *g, const DfftDev &d, int64_t stride, int64_t ncols, int64_t plane_cells, int64_t planes,
                 int64_t halfK, int64_t n2z, int64_t K, int64_t half, int band, ColBands b, cudaStream_t s) {
    const int64_t tiles = (ncols + TX - 1) / TX;
    const size_t smem = (size_t)pass_buffers(d.stages) * d.n * TX * sizeof(float4);
    const auto kernel = in64 ? dfft_cols_kernel<TX, SG, true> : dfft_cols_kernel<TX, SG, false>;
    kernel<<<(unsigned)(planes * tiles), kFftThreads, smem, s>>>(g, d, stride, ncols, plane_cells, halfK, n2z, K, half, band, b);
    check_cuda(cudaGetLastError(), "dfft_cols");
}

template <int SG, class... A> void cols_sign(int tx, A... a) {
    switch (tx) {
        case 64: launch_cols<64, SG>(a...); break;
        case 8: launch_cols<8, SG>(a...); break;
        case 2: launch_cols<2, SG>(a...); break;
        default: launch_cols<1, SG>(a...); break;
    }
}

}  // namespace

namespace {
float4 cis_pair(int m, int r) {
    const double ang = 2.0 * M_PI * (double)m / (double)r;
    const double c = std::cos(ang), s = std::sin(ang);
    const float ch = (float)c, sh = (float)s;
    return make_float4(ch, (float)(c - (double)ch), sh, (float)(s - (double)sh));
}
}  // namespace

bool dfft_factor(int n, DfftDev &d) {
    d.n = n;
    d.stages = 0;
    int m = n;
    for (int r : {4, 2, 3, 5, 7})
        while (m % r == 0) {
            if (d.stages == kDfftMaxStages) return false;
            d.radix[d.stages++] = r;
            m /= r;
        }
    long long Ns = 1;
    for (int st = 0; st < d.stages; ++st) {
        d.ns_magic[st] = Ns >= 2 ? (unsigned)((1ull << 32) / (unsigned long long)Ns + 1) : 0u;
        Ns *= d.radix[st];
    }
    int at = 0;
    for (int r : {3, 5, 7})
        for (int q = 1; q <= r / 2; ++q)
            for (int k = 1; k <= r / 2; ++k) d.odd[at++] = cis_pair((q * k) % r, r);
    return m == 1 && n >= 2;
}

bool dfft_supported(const int64_t n2[3]) {
    DfftDev d;
    for (int k = 0; k < 3; ++k)
        if (n2[k] > (int64_t)(kFftSmemMax / 32) || !dfft_factor((int)n2[k], d)) return false;
    return cols_per_cta((int)n2[1], 2) > 0 && cols_per_cta((int)n2[2], 64) > 0;
}

void dfft_twiddles(int n, std::vector<float> &tab) {
    tab.resize(4 * (size_t)n);
    for (int q = 0; q < n; ++q) {
        const double ang = 2.0 * M_PI * (double)q / (double)n;
        const double c = std::cos(ang), s = std::sin(ang);
        const float ch = (float)c, sh = (float)s;
        tab[4 * q + 0] = ch;
        tab[4 * q + 1] = (float)(c - (double)ch);
        tab[4 * q + 2] = sh;
        tab[4 * q + 3] = (float)(s - (double)sh);
    }
}

int dfft_batch(const FftBatch &f, const NufftDev *descs, void *g1, const double *ipsi, int sign, bool s2v, cudaStream_t s) {
    set_fft_attrs();
    double2 *g = static_cast<double2 *>(f.g2);
    const int64_t n2x = f.n2[0], n2y = f.n2[1], n2z = f.n2[2], K = f.K, half = f.half;
    const int64_t halfK = half * K, band_planes = 2 * halfK, plane = n2x * n2y;
    // The grids are FP64 before the first pass (written by the spreading) and hold double-float values
    // after it: the last pass leaves them for the double-float gathers.
    auto rows = [&] {
        const size_t smem = (size_t)pass_buffers(f.dx.stages) * n2x * sizeof(float4);
        const unsigned grid = (unsigned)(band_planes * f.n1[1]);
        const auto kernel = sign > 0 ? (s2v ? dfft_rows_kernel<1, false> : dfft_rows_kernel<1, true>)
                                     : (s2v ? dfft_rows_kernel<-1, false> : dfft_rows_kernel<-1, true>);
        kernel<<<grid, kFftThreads, smem, s>>>(g, f.dx, (int)n2y, (int)n2z, (int)K, (int)(f.n1[0] / 2), (int)(f.n1[1] / 2),
                                               (int)half, descs + f.first, g1, ipsi);
        check_cuda(cudaGetLastError(), "dfft_rows");
    };
    auto bands = [&](int64_t n, int64_t h) {  // the n1 band of the pass's input (sky -> vis) or output
        const int hh = (int)h, gap = (int)(n - 2 * h);
        return s2v ? ColBands{hh, gap, 0, 0} : ColBands{0, 0, hh, gap};
    };
    auto cols = [&](int tx, auto... a) { return sign > 0 ? cols_sign<1>(tx, a..., s) : cols_sign<-1>(tx, a..., s); };
    // y columns: two adjacent columns per CTA (32-byte segments) unless that leaves fewer than
    // two CTAs per SM (long columns), then one (twice the DRAM sectors, at ~15 % of HBM).
    const int ty = (size_t)2 * n2y * 2 * sizeof(float4) <= kFftSmemMax / 2 ? 2 : 1;
    auto ycols = [&] {
        cols(cols_per_cta((int)n2y, ty), false, g, f.dy, n2x, n2x, plane, band_planes, halfK, n2z, K, half, 1,
             bands(n2y, f.n1[1] / 2));
    };
    auto zcols = [&](bool in64) {
        cols(cols_per_cta((int)n2z, 64), in64, g, f.dz, K * plane, K * plane, (int64_t)0, (int64_t)1, halfK, n2z, K, half, 0,
             bands(n2z, half));
    };
    if (s2v) {  // only the band rows of the band planes are nonzero
        rows();
        ycols();
        zcols(false);
    } else {  // only the band rows of the band planes are read afterwards
        zcols(true);
        ycols();
        rows();
    }
    return 3;
}

}  // namespace hvox
