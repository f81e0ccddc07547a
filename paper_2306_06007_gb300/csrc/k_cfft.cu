// FP32 FFT of the NUFFT grids (step 2 of the type-3 transform, Sect. 3), with the deconvolution
// passes of step 1 folded into it.
//
// Between spreading and interpolation a grid is deconvolved and padded from its n1 band to n2
// cells, and transformed; only the band is nonzero before the transform (sky -> vis) or read
// after it (vis -> sky). One pass per dimension, each reading and writing only what the band
// leaves (b = n1 / n2 per dimension, cells of the n2 grid):
//   sky -> vis  rows:    n1 grid x 1/Psi, padded in registers, x transform -> band rows    b_x b_y b_z + b_y b_z
//               columns: band rows -> y transform -> band planes                        b_y b_z + b_z
//               columns: band planes -> z transform -> the grid                         b_z + 1
//   vis -> sky  the same backwards, the last pass cropping x and multiplying by 1/Psi into the n1 grid.
// The library form moved every padded cell through a deconvolution pass (the zeros too), full 2-D
// transforms of the band planes (0.31 ms for each of the two slabs' y pass, which read two columns,
// 16 bytes, at a time) and a full z pass. Measured, one direction of a 2160 x 2240 x 18 grid with a
// band of 1436 x 1466 x 12: 1.20 -> 0.61 ms (rows 0.16, y columns 0.27, z columns 0.16); of
// 2016 x 2016 x 96, band 1612 x 1612 x 74: 4.7 -> 3.5 ms.
// What bounds it: the z columns HBM (6.8 TB/s). Rows and y columns move 2.8 to 3 TB/s: 110
// instructions a cell (48 of them FP32, three stages), issued at 60%, in CTAs that alternate
// between loads, exchanges and stores, two on an SM for their 56 registers. Packed f32x2
// butterflies spill at 56 registers: rows and y columns 2% faster, z columns 5% slower, not kept.
//
// A pass: Stockham stages of radix up to 16 in registers (three stages for most lengths of ~2,000, so
// two trips through shared memory), the first stage reading the grid and the last one writing
// it. A stage between them exchanges elements in place through one shared buffer, a
// butterfly a thread, which halves the shared memory of a CTA. Columns are taken in tiles of
// 4 or more neighbours (whole 32-byte sectors), rows two or more to a CTA. Columns of up to
// 32 elements (most z lengths) are transformed in one thread's registers.
// Elements in shared memory carry one cell of padding per first-stage radix R0 where that is
// even: the first stage's stores (R0 apart) then fall on different banks, and as every later
// stride and offset is a multiple of R0 a butterfly's addresses stay base + q step. Twiddles are
// stored as the stages read them, two to a 16-byte load.
// The inverse sign is the forward transform of the conjugate, conjugated on load and store.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "hvox_internal.h"

namespace hvox {

namespace {

constexpr int kThreads2 = 576, kThreads1 = 1024;        // threads of a CTA, two or one of them on an SM
constexpr int kSmem2 = 100 * 1024, kSmem1 = 200 * 1024;  // and their shared memory
constexpr int kRadices[] = {16, 15, 14, 12, 10, 9, 8, 7, 6, 5, 4, 3, 2};

// ------------------------------------------------------------------ butterflies

constexpr double kPi = 3.14159265358979323846;
constexpr double taylor(double x, int first) {  // cos (first = 0) or sin (first = 1), |x| <= pi
    double term = first ? x : 1.0, sum = term;
    for (int i = first + 1; i < 40; i += 2) {
        term *= -x * x / ((double)i * (i + 1));
        sum += term;
    }
    return sum;
}
constexpr double turn(int k, int n) {  // 2 pi k / n in (-pi, pi]
    k %= n;
    return 2.0 * kPi * (2 * k > n ? k - n : k) / n;
}
template <int K, int N> struct W {  // exp(-2 pi j K / N)
    static constexpr float re = (float)taylor(turn(K, N), 0), im = (float)-taylor(turn(K, N), 1);
};

__device__ __forceinline__ float2 add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 mj(float2 a) { return make_float2(a.y, -a.x); }  // -j a

template <int K, int N> __device__ __forceinline__ float2 twist(float2 a) {  // a exp(-2 pi j K / N)
    if constexpr (K % N == 0) return a;
    else if constexpr (4 * K == N) return mj(a);
    else if constexpr (2 * K == N) return make_float2(-a.x, -a.y);
    else return mul(a, make_float2(W<K, N>::re, W<K, N>::im));
}

// Forward DFT of R values in place (natural order).
template <int R> struct Dft;
template <> struct Dft<2> {
    static __device__ __forceinline__ void run(float2 *v) {
        const float2 a = v[0];
        v[0] = add(a, v[1]);
        v[1] = sub(a, v[1]);
    }
};
template <> struct Dft<4> {
    static __device__ __forceinline__ void run(float2 *v) {
        const float2 a = add(v[0], v[2]), b = sub(v[0], v[2]), c = add(v[1], v[3]), d = mj(sub(v[1], v[3]));
        v[0] = add(a, c);
        v[1] = add(b, d);
        v[2] = sub(a, c);
        v[3] = sub(b, d);
    }
};
// Odd primes by the symmetric form X_k, X_{R-k} = A_k -+ j B_k.
template <int R, int K, int Q> __device__ __forceinline__ void odd_terms(const float2 *s, const float2 *d, float2 &a, float2 &b) {
    if constexpr (Q <= R / 2) {
        constexpr float c = W<Q * K, R>::re, n = -W<Q * K, R>::im;
        a.x = fmaf(s[Q].x, c, a.x);
        a.y = fmaf(s[Q].y, c, a.y);
        b.x = fmaf(d[Q].x, n, b.x);
        b.y = fmaf(d[Q].y, n, b.y);
        odd_terms<R, K, Q + 1>(s, d, a, b);
    }
}
template <int R, int K> __device__ __forceinline__ void odd_outputs(float2 v0, const float2 *s, const float2 *d, float2 *v) {
    if constexpr (K <= R / 2) {
        float2 a = v0, b = make_float2(0.f, 0.f);
        odd_terms<R, K, 1>(s, d, a, b);
        v[K] = add(a, mj(b));
        v[R - K] = sub(a, mj(b));
        odd_outputs<R, K + 1>(v0, s, d, v);
    }
}
template <int R> struct OddDft {
    static __device__ __forceinline__ void run(float2 *v) {
        float2 s[R / 2 + 1], d[R / 2 + 1], sum = v[0];
#pragma unroll
        for (int q = 1; q <= R / 2; ++q) {
            s[q] = add(v[q], v[R - q]);
            d[q] = sub(v[q], v[R - q]);
            sum = add(sum, s[q]);
        }
        const float2 v0 = v[0];
        v[0] = sum;
        odd_outputs<R, 1>(v0, s, d, v);
    }
};
template <> struct Dft<3> : OddDft<3> {};
template <> struct Dft<5> : OddDft<5> {};
template <> struct Dft<7> : OddDft<7> {};
// N = A B: B transforms of length A, twiddles, A transforms of length B.
template <int N, int K1, int N2, int A, int B> __device__ __forceinline__ void twist_row(float2 *t) {
    if constexpr (K1 < A) {
        t[K1] = twist<K1 * N2, N>(t[K1]);
        twist_row<N, K1 + 1, N2, A, B>(t);
    }
}
template <int A, int B, int N2> __device__ __forceinline__ void first_half(const float2 *v, float2 (*t)[A]) {
    if constexpr (N2 < B) {
#pragma unroll
        for (int i = 0; i < A; ++i) t[N2][i] = v[B * i + N2];
        Dft<A>::run(t[N2]);
        twist_row<A * B, 1, N2, A, B>(t[N2]);
        first_half<A, B, N2 + 1>(v, t);
    }
}
template <int A, int B> struct PairDft {
    static __device__ __forceinline__ void run(float2 *v) {
        float2 t[B][A];
        first_half<A, B, 0>(v, t);
#pragma unroll
        for (int k = 0; k < A; ++k) {
            float2 u[B];
#pragma unroll
            for (int i = 0; i < B; ++i) u[i] = t[i][k];
            Dft<B>::run(u);
#pragma unroll
            for (int i = 0; i < B; ++i) v[k + A * i] = u[i];
        }
    }
};
template <> struct Dft<6> : PairDft<3, 2> {};
template <> struct Dft<8> : PairDft<4, 2> {};
template <> struct Dft<9> : PairDft<3, 3> {};
template <> struct Dft<10> : PairDft<5, 2> {};
template <> struct Dft<12> : PairDft<4, 3> {};
template <> struct Dft<14> : PairDft<7, 2> {};
template <> struct Dft<15> : PairDft<5, 3> {};
template <> struct Dft<16> : PairDft<4, 4> {};
template <> struct Dft<18> : PairDft<6, 3> {};
template <> struct Dft<20> : PairDft<5, 4> {};
template <> struct Dft<24> : PairDft<8, 3> {};
template <> struct Dft<28> : PairDft<7, 4> {};
template <> struct Dft<30> : PairDft<6, 5> {};
template <> struct Dft<32> : PairDft<8, 4> {};

// ------------------------------------------------------------------ stages

// Conjugates for the inverse sign (sg = +-1).
__device__ __forceinline__ float2 with_sign(float2 v, float sg) { return make_float2(v.x, sg * v.y); }

// Element e lies in the band [0, h) or [n - h, n), gap = n - 2 h.
__device__ __forceinline__ bool in_band(int e, int h, int gap) { return (unsigned)(e - h) >= (unsigned)gap; }

// Shared-memory position of element e, in elements.
__device__ __forceinline__ int padded(const CfftDev &d, int e) { return e + d.pad * (int)__umulhi((unsigned)e, d.r0_magic); }

enum Role { kMiddle = 0, kFirst = 1, kLast = 2, kOnly = 3 };

// One Stockham stage of a CTA's sequences: butterfly j reads elements j + q m (m = n / R), twiddles them by
// exp(-2 pi i k q / (Ns R)), k = j mod Ns, and writes (j - k) R + k + q Ns. The first stage (Ns = 1) reads
// the grid and the last one (m = Ns, so k = j) writes it (io); a stage between them exchanges in
// place, a butterfly a thread: every element is read before any is overwritten.
// Io::split(wk, m, t, j): butterfly wk of the CTA is butterfly j of sequence t; Io::cell(t, d): the first
// shared cell of a sequence; 1 << Io::lt() cells from one of its elements to the next.
template <int R, int ROLE, class Io>
__device__ __forceinline__ void run_stage(const CfftDev &d, const Io &io, float2 *smem, int st, int Ns) {
    const int n = d.n, m = n / R, total = m * io.seqs(), lt = io.lt();
    const int rstep = (ROLE & kFirst) ? 0 : padded(d, m) << lt;
    const int wstep = (ROLE & kLast) ? 0 : ((ROLE & kFirst) ? 1 : padded(d, Ns)) << lt;
    const float4 *tw = d.tw + d.tw_at[st];
    for (int w0 = threadIdx.x; ROLE == kMiddle ? w0 == (int)threadIdx.x : w0 < total; w0 += blockDim.x) {
        const int wk = ROLE == kMiddle ? min(w0, total - 1) : w0;
        int t, j;
        io.split(wk, m, t, j);
        float2 v[R];
        int k = 0;
        if constexpr ((ROLE & kFirst) != 0) {
            io.load(v, std::integral_constant<int, R>(), j, t, m);
        } else {
            k = ROLE == kLast ? j : j - (int)__umulhi((unsigned)j, d.ns_magic[st]) * Ns;
            const float2 *src = smem + (io.cell(t, d) + (padded(d, j) << lt));
#pragma unroll
            for (int q = 0; q < R; ++q) v[q] = src[q * rstep];
#pragma unroll
            for (int q = 1; q < R; q += 2) {
                const float4 w = __ldg(tw + (q / 2 * Ns + k));
                v[q] = mul(v[q], make_float2(w.x, w.y));
                if (q + 1 < R) v[q + 1] = mul(v[q + 1], make_float2(w.z, w.w));
            }
        }
        Dft<R>::run(v);
        if (ROLE == kMiddle) __syncthreads();
        if constexpr ((ROLE & kLast) != 0) {
            io.store(v, std::integral_constant<int, R>(), j, t, m);
        } else if (ROLE != kMiddle || w0 < total) {
            // first stage: elements j R + q, j (R + pad) + q with the padding
            const int at = (ROLE & kFirst) ? j * (R + d.pad) : padded(d, (j - k) * R + k);
            float2 *dst = smem + (io.cell(t, d) + (at << lt));
#pragma unroll
            for (int q = 0; q < R; ++q) dst[q * wstep] = v[q];
        }
    }
    if (!(ROLE & kLast)) __syncthreads();
}

template <int ROLE, class Io>
__device__ __forceinline__ void any_stage(const CfftDev &d, const Io &io, float2 *smem, int st, int Ns) {
    switch (d.radix[st]) {
        case 16: run_stage<16, ROLE>(d, io, smem, st, Ns); break;
        case 15: run_stage<15, ROLE>(d, io, smem, st, Ns); break;
        case 14: run_stage<14, ROLE>(d, io, smem, st, Ns); break;
        case 12: run_stage<12, ROLE>(d, io, smem, st, Ns); break;
        case 10: run_stage<10, ROLE>(d, io, smem, st, Ns); break;
        case 9: run_stage<9, ROLE>(d, io, smem, st, Ns); break;
        case 8: run_stage<8, ROLE>(d, io, smem, st, Ns); break;
        case 7: run_stage<7, ROLE>(d, io, smem, st, Ns); break;
        case 6: run_stage<6, ROLE>(d, io, smem, st, Ns); break;
        case 5: run_stage<5, ROLE>(d, io, smem, st, Ns); break;
        case 4: run_stage<4, ROLE>(d, io, smem, st, Ns); break;
        case 3: run_stage<3, ROLE>(d, io, smem, st, Ns); break;
        default: run_stage<2, ROLE>(d, io, smem, st, Ns); break;
    }
}

template <class Io> __device__ __forceinline__ void transform(const CfftDev &d, const Io &io, float2 *smem) {
    if (d.stages == 1) {
        any_stage<kOnly>(d, io, smem, 0, 1);
        return;
    }
    any_stage<kFirst>(d, io, smem, 0, 1);
    int Ns = d.radix[0];
    for (int st = 1; st + 1 < d.stages; ++st) {
        any_stage<kMiddle>(d, io, smem, st, Ns);
        Ns *= d.radix[st];
    }
    any_stage<kLast>(d, io, smem, d.stages - 1, Ns);
}

// ------------------------------------------------------------------ rows (x)

// `rows` rows of a batch, starting at r0 of its n1y n1z K band rows; OUT false: n1 grid -> n2 band rows
// (deconvolved, padded), true: n2 band rows -> n1 grid (cropped, deconvolved).
template <bool OUT> struct RowIo {
    const NufftDev *descs;  // the batch's K sub-problems
    float2 *g1, *g2;        // the lane's buffers
    const float *ipsi;
    int64_t r0, n_rows;
    int rows, n1x, n1y, n1z, n2x, n2y, n2z, K;
    float sg;

    struct Row {
        const float *px;
        float f;
        int64_t c1, c2;  // first cells of the row in g1 and g2
    };
    Row *row;  // shared, one per row of the CTA

    __device__ __forceinline__ void begin() const {
        if ((int)threadIdx.x < rows) {
            const int64_t r = min(r0 + (int)threadIdx.x, n_rows - 1);
            const int iy = (int)(r % n1y);
            const int64_t gz = r / n1y;
            const int g = (int)(gz % K), iz = (int)(gz / K);
            const NufftDev &b = descs[g];
            const float *px = ipsi + b.psi_off, *py = px + n1x, *pz = py + n1y;
            const int ly = iy - n1y / 2, lz = iz - n1z / 2;
            const int jy = ly < 0 ? ly + n2y : ly, jz = lz < 0 ? lz + n2z : lz;
            row[threadIdx.x] = {px, py[iy] * pz[iz], b.g1_off + ((int64_t)iz * n1y + iy) * n1x,
                                b.g2_off + (int64_t)jz * b.zs2 + (int64_t)jy * n2x};
        }
        __syncthreads();
    }
    __device__ __forceinline__ int seqs() const { return rows; }
    __device__ __forceinline__ int lt() const { return 0; }
    __device__ __forceinline__ void split(int wk, int m, int &t, int &j) const {
        t = wk / m;
        j = wk - t * m;
    }
    __device__ __forceinline__ int cell(int t, const CfftDev &d) const { return t * padded(d, d.n); }
    // The n1 band holds the padded row's elements [n2x - h, n2x) then [0, h), h = n1x / 2.
    template <int R> __device__ __forceinline__ void load(float2 *v, std::integral_constant<int, R>, int j, int t, int m) const {
        const Row &r = row[t];
        if constexpr (OUT) {
            const float2 *p = g2 + (r.c2 + j);
#pragma unroll
            for (int q = 0; q < R; ++q) v[q] = p[q * m];
#pragma unroll
            for (int q = 0; q < R; ++q) v[q] = with_sign(v[q], sg);
        } else {
            const int h = n1x / 2, gap = n2x - n1x;
            const float2 *p = g1 + r.c1;
            const float fx = r.f, fy = sg * r.f;
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const int e = j + q * m;
                v[q] = make_float2(0.f, 0.f);
                if (in_band(e, h, gap)) v[q] = p[e < h ? e + h : e - h - gap];
            }
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const int e = j + q * m;
                const float w = in_band(e, h, gap) ? r.px[e < h ? e + h : e - h - gap] : 0.f;
                v[q] = make_float2(v[q].x * (w * fx), v[q].y * (w * fy));
            }
        }
    }
    template <int R> __device__ __forceinline__ void store(const float2 *v, std::integral_constant<int, R>, int j, int t, int m) const {
        if (r0 + t >= n_rows) return;
        const Row &r = row[t];
        if constexpr (!OUT) {
            float2 *p = g2 + (r.c2 + j);
#pragma unroll
            for (int q = 0; q < R; ++q) p[q * m] = with_sign(v[q], sg);
        } else {
            const int h = n1x / 2, gap = n2x - n1x;
            float2 *p = g1 + r.c1;
            const float fx = r.f, fy = sg * r.f;
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const int e = j + q * m, i = e < h ? e + h : e - h - gap;
                if (in_band(e, h, gap)) {
                    const float w = r.px[i];
                    p[i] = make_float2(v[q].x * (w * fx), v[q].y * (w * fy));
                }
            }
        }
    }
};

constexpr int kMaxRows = 32;  // rows of a CTA

// Parameters stay in constant memory (__grid_constant__): a copy of the radix table on the stack made
// every stride of a stage a per-thread load.
template <bool OUT, int T>
__global__ void __launch_bounds__(T, T == kThreads2 ? 2 : 1)
    cfft_rows_kernel(const __grid_constant__ CfftDev d, const __grid_constant__ RowIo<OUT> in) {
    extern __shared__ float2 cfft_smem[];
    __shared__ typename RowIo<OUT>::Row row[kMaxRows];
    RowIo<OUT> io = in;
    io.row = row;
    io.r0 = (int64_t)blockIdx.x * io.rows;
    io.begin();
    transform(d, io, cfft_smem);
}

// ------------------------------------------------------------------ columns (y and z)

// A tile of 2^lt neighbouring columns: element e of column t at base + e stride + t. Elements outside
// the input band (half-width hi, gap gi) are zero, those outside the output band are not written.
struct ColIo {
    float2 *base;
    int64_t stride;
    int lt_, valid, hi, gi, ho, go;
    float sg;

    __device__ __forceinline__ int seqs() const { return 1 << lt_; }
    __device__ __forceinline__ int lt() const { return lt_; }
    __device__ __forceinline__ void split(int wk, int, int &t, int &j) const {
        t = wk & ((1 << lt_) - 1);
        j = wk >> lt_;
    }
    __device__ __forceinline__ int cell(int t, const CfftDev &) const { return t; }
    template <int R> __device__ __forceinline__ void load(float2 *v, std::integral_constant<int, R>, int j, int t, int m) const {
        const float2 *p = base + (j * stride + min(t, valid - 1));
        const int64_t step = m * stride;
#pragma unroll
        for (int q = 0; q < R; ++q) {
            v[q] = make_float2(0.f, 0.f);
            if (in_band(j + q * m, hi, gi)) v[q] = p[q * step];
        }
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = with_sign(v[q], sg);
    }
    template <int R> __device__ __forceinline__ void store(const float2 *v, std::integral_constant<int, R>, int j, int t, int m) const {
        if (t >= valid) return;
        float2 *p = base + (j * stride + t);
        const int64_t step = m * stride;
#pragma unroll
        for (int q = 0; q < R; ++q)
            if (in_band(j + q * m, ho, go)) p[q * step] = with_sign(v[q], sg);
    }
};

struct ColBand {
    int hi, gi, ho, go;
};

// planes x tiles CTAs; plane P of the batch at g + plane_of(P) plane_cells.
template <int T>
__global__ void __launch_bounds__(T, T == kThreads2 ? 2 : 1)
    cfft_cols_kernel(const __grid_constant__ CfftDev d, float2 *__restrict__ g, int64_t stride, int64_t ncols, int64_t plane_cells,
                     int64_t low_planes, int64_t skip, int lt, ColBand b, float sg) {
    extern __shared__ float2 cfft_smem[];
    const int64_t tiles = (ncols + (1 << lt) - 1) >> lt;
    const int64_t P = blockIdx.x / tiles, c0 = (blockIdx.x - P * tiles) << lt;
    const int64_t plane = P < low_planes ? P : P + skip;  // the band's planes: a lower and an upper slab
    const int64_t left = ncols - c0;
    const ColIo io{g + plane * plane_cells + c0, stride, lt, left < (1 << lt) ? (int)left : 1 << lt, b.hi, b.gi, b.ho, b.go, sg};
    transform(d, io, cfft_smem);
}

// Columns of N elements, one to a thread: no shared memory, every load of a column in flight.
// N >= 2 kernel widths, so most NUFFT grids' z length (18 at 1e-6, eight-degree fields) is one of these.
template <int N>
__global__ void __launch_bounds__(256) cfft_line_kernel(float2 *__restrict__ g, int64_t stride, ColBand b, float sg) {
    const int64_t c = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (c >= stride) return;
    float2 *p = g + c, v[N];
#pragma unroll
    for (int e = 0; e < N; ++e) v[e] = in_band(e, b.hi, b.gi) ? p[e * stride] : make_float2(0.f, 0.f);
#pragma unroll
    for (int e = 0; e < N; ++e) v[e] = with_sign(v[e], sg);
    Dft<N>::run(v);
#pragma unroll
    for (int e = 0; e < N; ++e)
        if (in_band(e, b.ho, b.go)) p[e * stride] = with_sign(v[e], sg);
}

// ------------------------------------------------------------------ host

size_t smem_bytes(const CfftDev &d, int seqs) {
    if (d.stages == 1) return 0;
    return (size_t)(d.n + d.pad * (d.n / d.radix[0])) * seqs * sizeof(float2);
}

// Threads of a CTA with `seqs` sequences: one butterfly of the stages that exchange in place, about
// 16 elements of the others.
int threads_for(const CfftDev &d, int seqs) {
    int t = (d.n * seqs + 15) / 16;
    for (int s = 1; s + 1 < d.stages; ++s) t = std::max(t, d.n / d.radix[s] * seqs);
    return (t + 31) / 32 * 32;
}

// A CTA of this many sequences can share its SM with another (2), has it alone (1) or does not fit (0).
int ctas_fit(const CfftDev &d, int seqs) {
    const size_t smem = smem_bytes(d, seqs);
    const int threads = threads_for(d, seqs);
    return threads <= kThreads2 && smem <= (size_t)kSmem2 ? 2 : threads <= kThreads1 && smem <= (size_t)kSmem1 ? 1 : 0;
}

// log2 of the columns per CTA: tiles of about 8,192 cells and 4 to 64 columns, two CTAs to an SM if
// 4 columns allow it.
int cols_log2(const CfftDev &d) {
    for (int lt = 6; lt > 2; --lt)
        if (((int64_t)d.n << lt) <= 8192 && ctas_fit(d, 1 << lt) == 2) return lt;
    return ctas_fit(d, 4) > 0 ? 2 : -1;  // fewer would move half sectors
}

int rows_per_cta(const CfftDev &d) {
    int rows = 1;
    while (rows < kMaxRows && d.n * rows < 4096 && ctas_fit(d, 2 * rows) == 2) rows *= 2;
    return rows;
}

void set_attrs() {
    static OncePerDevice once;
    once.run(current_device(), [] {
        auto allow = [](auto k, int bytes) {
            check_cuda(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes), "cudaFuncSetAttribute");
        };
        allow(cfft_rows_kernel<false, kThreads2>, kSmem2);
        allow(cfft_rows_kernel<false, kThreads1>, kSmem1);
        allow(cfft_rows_kernel<true, kThreads2>, kSmem2);
        allow(cfft_rows_kernel<true, kThreads1>, kSmem1);
        allow(cfft_cols_kernel<kThreads2>, kSmem2);
        allow(cfft_cols_kernel<kThreads1>, kSmem1);
    });
}

template <bool OUT>
void launch_rows(const FftBatch &f, const NufftDev *descs, void *g1, void *g2, const float *ipsi, float sg, cudaStream_t s) {
    RowIo<OUT> io{};
    io.descs = descs + f.first;
    io.g1 = static_cast<float2 *>(g1);
    io.g2 = static_cast<float2 *>(g2);
    io.ipsi = ipsi;
    io.n1x = (int)f.n1[0];
    io.n1y = (int)f.n1[1];
    io.n1z = (int)f.n1[2];
    io.n2x = (int)f.n2[0];
    io.n2y = (int)f.n2[1];
    io.n2z = (int)f.n2[2];
    io.K = (int)f.K;
    io.n_rows = f.n1[1] * f.n1[2] * f.K;
    io.rows = rows_per_cta(f.cx);
    io.sg = sg;
    const unsigned grid = (unsigned)((io.n_rows + io.rows - 1) / io.rows);
    const auto kernel = ctas_fit(f.cx, io.rows) == 2 ? cfft_rows_kernel<OUT, kThreads2> : cfft_rows_kernel<OUT, kThreads1>;
    kernel<<<grid, threads_for(f.cx, io.rows), smem_bytes(f.cx, io.rows), s>>>(f.cx, io);
    check_cuda(cudaGetLastError(), "cfft_rows");
}

// band: half-width of the band on input (in) or output.
ColBand col_band(int n, int64_t half, bool in) {
    const ColBand all{0, 0, 0, 0};
    ColBand b = all;
    (in ? b.hi : b.ho) = (int)half;
    (in ? b.gi : b.go) = n - 2 * (int)half;
    return b;
}

void launch_cols(const CfftDev &d, float2 *g, int64_t stride, int64_t ncols, int64_t plane_cells, int64_t planes,
                 int64_t low_planes, int64_t skip, ColBand b, float sg, cudaStream_t s) {
    const int lt = cols_log2(d);
    const int64_t tiles = (ncols + (1 << lt) - 1) >> lt;
    const auto kernel = ctas_fit(d, 1 << lt) == 2 ? cfft_cols_kernel<kThreads2> : cfft_cols_kernel<kThreads1>;
    kernel<<<(unsigned)(planes * tiles), threads_for(d, 1 << lt), smem_bytes(d, 1 << lt), s>>>(d, g, stride, ncols, plane_cells,
                                                                                             low_planes, skip, lt, b, sg);
    check_cuda(cudaGetLastError(), "cfft_cols");
}

// The columns of one plane set (plane z at g + z stride): by registers where a kernel of this length is built.
void launch_z(const CfftDev &d, float2 *g, int64_t stride, ColBand b, float sg, cudaStream_t s) {
    const unsigned grid = (unsigned)((stride + 255) / 256);
    switch (d.n) {
        case 8: cfft_line_kernel<8><<<grid, 256, 0, s>>>(g, stride, b, sg); break;
        case 10: cfft_line_kernel<10><<<grid, 256, 0, s>>>(g, stride, b, sg); break;
        case 12: cfft_line_kernel<12><<<grid, 256, 0, s>>>(g, stride, b, sg); break;
        case 14: cfft_line_kernel<14><<<grid, 256, 0, s>>>(g, stride, b, sg); break;
        case 16: cfft_line_kernel<16><<<grid, 256, 0, s>>>(g, stride, b, sg); break;
        case 18: cfft_line_kernel<18><<<grid, 256, 0, s>>>(g, stride, b, sg); break;
        case 20: cfft_line_kernel<20><<<grid, 256, 0, s>>>(g, stride, b, sg); break;
        case 24: cfft_line_kernel<24><<<grid, 256, 0, s>>>(g, stride, b, sg); break;
        case 28: cfft_line_kernel<28><<<grid, 256, 0, s>>>(g, stride, b, sg); break;
        case 30: cfft_line_kernel<30><<<grid, 256, 0, s>>>(g, stride, b, sg); break;
        case 32: cfft_line_kernel<32><<<grid, 256, 0, s>>>(g, stride, b, sg); break;
        default: return launch_cols(d, g, stride, stride, 0, 1, 1, 0, b, sg, s);
    }
    check_cuda(cudaGetLastError(), "cfft_line");
}

// Fewest stages (then the largest radices first).
bool search_radices(int n, int at, int left, int *out) {
    if (n == 1) return left == 0;
    if (left == 0) return false;
    for (int r : kRadices) {
        if (n % r != 0 || (at > 0 && r > out[at - 1])) continue;
        out[at] = r;
        if (search_radices(n / r, at + 1, left - 1, out)) return true;
    }
    return false;
}

unsigned divisor_magic(unsigned long long n) { return n >= 2 ? (unsigned)((1ull << 32) / n + 1) : 0u; }

}  // namespace

// The largest radix goes to a stage in between (fewest threads there).
bool cfft_factor(int n, CfftDev &d) {
    d.n = n;
    for (int s = 1; s <= kCfftMaxStages; ++s)
        if (search_radices(n, 0, s, d.radix)) {
            d.stages = s;
            if (s > 2) std::swap(d.radix[0], d.radix[s - 2]);
            d.pad = d.radix[0] % 2 == 0 ? 1 : 0;
            d.r0_magic = divisor_magic(d.radix[0]);
            int Ns = 1, at = 0;
            for (int k = 0; k < s; ++k) {
                d.ns_magic[k] = divisor_magic(Ns);
                d.tw_at[k] = at;
                if (k > 0) at += Ns * (d.radix[k] / 2);
                Ns *= d.radix[k];
            }
            return true;
        }
    return false;
}

// Rows and columns of these lengths fit a CTA, the y columns in tiles of whole 32-byte sectors
// (4 or more): no y length above 4,096, and below that not those whose stage in between would need
// more than 1,024 threads (1,750 = 5 5 14 5, 2,000, 2,058, 2,430, ...: its radix under n / 256). The rest
// stays with cuFFT, and takes every grid of its plan along (Plan::cf_grids). Indices inside a CTA stay
// below 2^16, where the divisions by multiplication are exact.
bool cfft_supported(const int64_t n2[3]) {
    CfftDev d[3];
    for (int k = 0; k < 3; ++k)
        if (n2[k] < 2 || n2[k] > 16384 || !cfft_factor((int)n2[k], d[k])) return false;
    return ctas_fit(d[0], 1) > 0 && cols_log2(d[1]) >= 2 && cols_log2(d[2]) >= 2;
}

// Per stage after the first, exp(-2 pi i k q / (Ns R)) for q = 1 .. R - 1 in pairs: [q / 2][k][2].
void cfft_twiddles(int n, std::vector<float> &tab) {
    CfftDev d;
    cfft_factor(n, d);
    tab.clear();
    int Ns = 1;
    for (int s = 0; s < d.stages; ++s) {
        const int R = d.radix[s];
        if (s > 0)
            for (int h = 0; h < R / 2; ++h)
                for (int k = 0; k < Ns; ++k)
                    for (int q = 2 * h + 1; q <= 2 * h + 2; ++q) {
                        const double a = 2.0 * M_PI * (double)k * (double)q / ((double)Ns * R);
                        tab.push_back((float)std::cos(a));
                        tab.push_back((float)-std::sin(a));
                    }
        Ns *= R;
    }
    if (tab.empty()) tab.resize(4);
}

// Deconvolution, padding and transform of a batch's grids (sky -> vis), or transform, crop and
// deconvolution (vis -> sky). sign: of the exponent. Returns the number of launches.
int cfft_batch(const FftBatch &f, const NufftDev *descs, void *g1, void *g2, const float *ipsi, int sign, bool s2v,
               cudaStream_t s) {
    set_attrs();
    const int64_t n2x = f.n2[0], n2y = f.n2[1], n2z = f.n2[2], K = f.K, plane = n2x * n2y;
    const int64_t half = f.n1[2] / 2 * K;  // planes of a slab of the band
    const float sg = sign < 0 ? 1.f : -1.f;
    float2 *g = static_cast<float2 *>(f.g2);
    auto ycols = [&] {
        launch_cols(f.cy, g, n2x, n2x, plane, 2 * half, half, n2z * K - 2 * half, col_band((int)n2y, f.n1[1] / 2, s2v), sg, s);
    };
    auto zcols = [&] { launch_z(f.cz, g, K * plane, col_band((int)n2z, f.n1[2] / 2, s2v), sg, s); };
    if (s2v) {
        launch_rows<false>(f, descs, g1, g2, ipsi, sg, s);
        ycols();
        zcols();
    } else {
        zcols();
        ycols();
        launch_rows<true>(f, descs, g1, g2, ipsi, sg, s);
    }
    return 3;
}

}  // namespace hvox
