// Transforms of the image step and of W stacking with the passes around them
// folded in (Sec. 2: I_D / n = F^-1[grid] / c; Sec. 4.3: the slices).
//
// The shifted transform of even N is, with a' = a - N/2 (mod N),
//   grid -> image:  I[a] = (-1)^a' sum_c G[c] exp(2 pi i c a' / N),
//   image -> grid:  G[c] = sum_a' (-1)^a' I[a] exp(-2 pi i c a' / N),
// so the shift is a reordering on the image side and a sign there: no pass
// over the grids is needed for it.  The column transforms run on the grid
// side, and the rows where the image side's reordering, sign, grid correction,
// slice phases and the sum over the slices all fold into the one load or store
// of a row.  (sepw_image towards the grid has no transform here: it runs cuFFT
// between two passes over the grid.)
//
// What that saves: the passes are bound by memory.  Per direction the slice
// grids were read and written by a sign pass, by the row transform and by the
// combine (or split) pass; now they are read (or written) once.  15 grids of
// 4096^2: sign 0.69 + rows 0.64 + combine 0.40 ms -> 0.79 ms one way and
// 0.69 + 0.64 + 0.38 -> 0.82 ms the other, now bound by the transform's and the
// phases' arithmetic (2.5 TB/s).
//
// A block transforms a row of N = 256 R points (R = 2, 4, 8, 16) in registers,
// 16 points per thread, as 16 x 16 x R (n = t + T k, T = N / 16, t = t0 + R k2;
// f = 256 m3 + 16 m2 + m): radix 16 over k, twiddles w_N^(t m); radix 16 over
// k2, twiddles w_T^(t0 m2); radix R over t0; two exchanges through shared
// memory.  Twiddles w^1, w^2, w^3, w^4, w^8, w^12 come from tables rounded
// from float64, the others are one product of two.
#include "sepw_internal.cuh"

namespace sepw {
namespace {

constexpr int kTw = 6;  // tabulated powers: 1, 2, 3, 4, 8, 12

__device__ __forceinline__ float2 operator+(float2 a, float2 b)
{
    return make_float2(a.x + b.x, a.y + b.y);
}
__device__ __forceinline__ float2 operator-(float2 a, float2 b)
{
    return make_float2(a.x - b.x, a.y - b.y);
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a times conj(b) for the inverse transform (tables hold exp(-i ...))
template <bool INV>
__device__ __forceinline__ float2 twmul(float2 a, float2 b)
{
    return INV ? make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y) : cmul(a, b);
}
// a times -i (forward) or i (inverse)
template <bool INV>
__device__ __forceinline__ float2 quarter(float2 a)
{
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

template <bool INV>
__device__ __forceinline__ void dft2(float2 &a, float2 &b)
{
    const float2 t = a - b;
    a = a + b;
    b = t;
}
template <bool INV>
__device__ __forceinline__ void dft4(float2 &a, float2 &b, float2 &c, float2 &d)
{
    const float2 s0 = a + c, s1 = a - c, s2 = b + d, s3 = quarter<INV>(b - d);
    a = s0 + s2;
    b = s1 + s3;
    c = s0 - s2;
    d = s1 - s3;
}
// v[0 .. R-1] -> its transform in order, R = 2, 4, 8, 16
template <int R, bool INV>
__device__ __forceinline__ void dft(float2 *v)
{
    if constexpr (R == 2) {
        dft2<INV>(v[0], v[1]);
    } else if constexpr (R == 4) {
        dft4<INV>(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 8) {
        constexpr float h = 0.70710678118654752f;  // cos(pi / 4)
#pragma unroll
        for (int k = 0; k < 4; ++k)
            dft2<INV>(v[k], v[k + 4]);
        v[5] = twmul<INV>(v[5], make_float2(h, -h));
        v[6] = quarter<INV>(v[6]);
        v[7] = twmul<INV>(v[7], make_float2(-h, -h));
        dft4<INV>(v[0], v[1], v[2], v[3]);
        dft4<INV>(v[4], v[5], v[6], v[7]);
        // f = 2 m' + (0, 1)
        const float2 y[8] = {v[0], v[4], v[1], v[5], v[2], v[6], v[3], v[7]};
#pragma unroll
        for (int k = 0; k < 8; ++k)
            v[k] = y[k];
    } else {
        constexpr float h = 0.70710678118654752f;
        constexpr float c = 0.92387953251128674f, s = 0.38268343236508977f;  // cos, sin(pi / 8)
#pragma unroll
        for (int k = 0; k < 4; ++k)  // over x[k], x[k+4], x[k+8], x[k+12] -> m'
            dft4<INV>(v[k], v[k + 4], v[k + 8], v[k + 12]);
        // w_16^(k m'), v[k + 4 m']
        v[5] = twmul<INV>(v[5], make_float2(c, -s));
        v[6] = twmul<INV>(v[6], make_float2(h, -h));
        v[7] = twmul<INV>(v[7], make_float2(s, -c));
        v[9] = twmul<INV>(v[9], make_float2(h, -h));
        v[10] = quarter<INV>(v[10]);
        v[11] = twmul<INV>(v[11], make_float2(-h, -h));
        v[13] = twmul<INV>(v[13], make_float2(s, -c));
        v[14] = twmul<INV>(v[14], make_float2(-h, -h));
        v[15] = twmul<INV>(v[15], make_float2(-c, s));
#pragma unroll
        for (int m = 0; m < 4; ++m)  // over k -> m'' of f = m' + 4 m''
            dft4<INV>(v[4 * m], v[4 * m + 1], v[4 * m + 2], v[4 * m + 3]);
        // v[4 m' + m''] -> v[m' + 4 m'']
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = a + 1; b < 4; ++b) {
                const float2 t = v[4 * a + b];
                v[4 * a + b] = v[4 * b + a];
                v[4 * b + a] = t;
            }
    }
}

// v[m] *= w^m, w^(1, 2, 3, 4, 8, 12) = tab[0 .. 5][i] at stride n
template <bool INV>
__device__ __forceinline__ void twiddle16(float2 (&v)[16], const float2 *__restrict__ tab, int n,
                                          int i)
{
    float2 lo[4], hi[4];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lo[k + 1] = __ldg(tab + k * n + i);
        hi[k + 1] = __ldg(tab + (k + 3) * n + i);
    }
#pragma unroll
    for (int m = 1; m < 16; ++m) {
        const float2 w = m < 4 ? lo[m] : m % 4 == 0 ? hi[m / 4] : cmul(hi[m / 4], lo[m % 4]);
        v[m] = twmul<INV>(v[m], w);
    }
}

template <int R>
struct Rows {
    static constexpr int N = 256 * R, T = N / 16;
    static constexpr int BPS = 32 / R;      // resident blocks per SM: 128 registers
    static constexpr int P1 = T + R;        // exchange strides, see row_fft
    static constexpr int P2 = 17 * R + (R == 16 ? 1 : R == 8 ? 9 : R == 4 ? 13 : 15);
    static constexpr int kShm = 16 * (P1 > P2 ? P1 : P2);  // float2
};

// Transform of the block's row.  In: thread t holds x[t + T k] in v[k]; out:
// v[m3 + R h], h < 16 / R, is frequency 256 m3 + t + T h.  shm: kShm float2,
// free on entry; on return other threads may still read it.
template <int R, bool INV>
__device__ __forceinline__ void row_fft(float2 (&v)[16], const float2 *__restrict__ tab,
                                        float2 *shm)
{
    using W = Rows<R>;
    const int t = threadIdx.x;
    dft<16, INV>(v);
    twiddle16<INV>(v, tab, W::T, t);
    // [m][t], rows padded so that the R-wide reads below hit different banks
#pragma unroll
    for (int m = 0; m < 16; ++m)
        shm[m * W::P1 + t] = v[m];
    __syncthreads();
    {
        const int m = t / R, t0 = t % R;
#pragma unroll
        for (int k = 0; k < 16; ++k)
            v[k] = shm[m * W::P1 + t0 + R * k];
        dft<16, INV>(v);
        twiddle16<INV>(v, tab + kTw * W::T, 16, t0);
        __syncthreads();
        // [m][t0][m2]: odd strides (mod 16) along m and t0
#pragma unroll
        for (int k = 0; k < 16; ++k)
            shm[m * W::P2 + t0 * 17 + k] = v[k];
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 16 / R; ++h) {
        const int q = t + W::T * h, m2 = q >> 4, m = q & 15;
#pragma unroll
        for (int k = 0; k < R; ++k)
            v[k + R * h] = shm[m * W::P2 + k * 17 + m2];
        dft<R, INV>(v + R * h);
    }
}

// ---------------------------------------------------------------------------
// Column transforms in place: a block takes four columns (32 bytes of every
// row, a whole sector) of one of `grids` grids at a time, thread (t, c) =
// (id >> 2, id & 3) the points t + T k of column c, in registers as a row
// above.  The next four columns are copied into shared memory while these are
// transformed (cp.async), so that the loads run on; the exchanges take half
// the room by moving real and imaginary parts one after the other.  Columns
// that are all zero transform to zero and are left alone: in W stacking's
// grids most columns lie beyond the uv coverage.  4096^2: cuFFT's strided
// batch took 92 us a grid, with nothing in flight while it computes; this
// 85 us, and 45 us for grids with two thirds of their columns
// empty.
// ---------------------------------------------------------------------------
template <int R>
struct Cols {
    static constexpr int N = Rows<R>::N, T = Rows<R>::T, kThreads = 4 * T;
    static constexpr int BPS = 16 / R;  // 1024 threads of 64 registers per SM
    static constexpr int kBuf = 4 * N;               // float2
    static constexpr int kX = 4 * Rows<R>::kShm;     // float
    static constexpr int kShm = sizeof(float2) * kBuf + sizeof(float) * kX;
};

// v[k] -> its value at exchange place `to(k)`, read from place `from(k)`
template <typename A, typename B>
__device__ __forceinline__ void exchange(float2 (&v)[16], float *x, int c, A to, B from)
{
    float re[16];
#pragma unroll
    for (int k = 0; k < 16; ++k)
        x[4 * to(k) + c] = v[k].x;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k)
        re[k] = x[4 * from(k) + c];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k)
        x[4 * to(k) + c] = v[k].y;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k)
        v[k] = make_float2(re[k], x[4 * from(k) + c]);
}

template <int R, bool INV>
__global__ void __launch_bounds__(Cols<R>::kThreads, Cols<R>::BPS) columns_kernel(
    int grids, float2 *g, const float2 *__restrict__ tab)
{
    using W = Rows<R>;
    constexpr int N = W::N, T = W::T, kThreads = Cols<R>::kThreads;
    extern __shared__ float4 dyn[];
    float2 *const buf = reinterpret_cast<float2 *>(dyn);
    float *const x = reinterpret_cast<float *>(buf + Cols<R>::kBuf);
    const int c = threadIdx.x & 3, t = threadIdx.x >> 2;
    const int64_t tiles = (int64_t)grids * (N / 4);
    auto first = [&](int64_t tile) {  // the tile's first cell
        return g + tile / (N / 4) * ((int64_t)N * N) + tile % (N / 4) * 4;
    };
    auto fetch = [&](int64_t tile) {  // 16-byte halves of its rows
        const unsigned dst = (unsigned)__cvta_generic_to_shared(buf) + 16u * threadIdx.x;
        const float2 *from = first(tile) + (threadIdx.x >> 1) * N + (threadIdx.x & 1) * 2;
#pragma unroll
        for (int k = 0; k < 2 * N / kThreads; ++k)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * kThreads * k),
                         "l"(from + (int64_t)(kThreads / 2) * k * N)
                         : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (blockIdx.x < tiles)
        fetch(blockIdx.x);
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // the tile has landed; the last one is done with x
        float2 v[16];
        bool any = false;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            v[k] = buf[(t + T * k) * 4 + c];
            any |= !(v[k].x == 0.f) || !(v[k].y == 0.f);  // (a NaN is not zero)
        }
        any = __syncthreads_or(any);
        if (tile + gridDim.x < tiles)
            fetch(tile + gridDim.x);
        if (!any)
            continue;
        dft<16, INV>(v);
        twiddle16<INV>(v, tab, T, t);
        const int m = t / R, t0 = t % R;
        exchange(v, x, c, [&](int k) { return k * W::P1 + t; },
                 [&](int k) { return m * W::P1 + t0 + R * k; });
        dft<16, INV>(v);
        twiddle16<INV>(v, tab + kTw * T, 16, t0);
        __syncthreads();
        // v[k + R h] is point k of the h-th transform, frequencies 256 m3 + q
        exchange(v, x, c, [&](int k) { return m * W::P2 + t0 * 17 + k; },
                 [&](int k) {
                     const int q = t + T * (k / R);
                     return (q & 15) * W::P2 + (k % R) * 17 + (q >> 4);
                 });
        float2 *const out = first(tile) + c;
#pragma unroll
        for (int h = 0; h < 16 / R; ++h) {
            dft<R, INV>(v + R * h);
#pragma unroll
            for (int k = 0; k < R; ++k)
                out[(int64_t)(256 * k + t + T * h) * N] = v[k + R * h];
        }
    }
}

// tables: [kTw][T] powers of w_N^t, then [kTw][16] powers of w_T^t0 (t0 < R)
__global__ void fft_tables_kernel(int N, int OS, const double2 *__restrict__ tw, float2 *tab)
{
    const int T = N / 16, i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kTw * (T + 16))
        return;
    const bool first = i < kTw * T;
    const int k = first ? i / T : (i - kTw * T) / 16, t = first ? i % T : (i - kTw * T) % 16;
    const int power = k < 3 ? k + 1 : 4 * (k - 2);
    const int64_t j = (int64_t)t * power * (first ? 1 : 16) % N;
    const double2 w = tw[j * OS];
    tab[i] = make_float2((float)w.x, (float)w.y);
}

// Pixel a of the image side at transform index f, and the pixel's terms.
struct Pixels {
    int N;
    float fov_over_n, l0, m0;
    const float *taper;

    __device__ __forceinline__ int shift(int f) const { return f < N / 2 ? f + N / 2 : f - N / 2; }
    // sign (-1)^(f + g) times n / (c c) (MODE 1) or 1 / (n c c) (MODE 2) at
    // pixel (a, b) = shift(f, g); nm1 = n - 1 without cancellation
    __device__ __forceinline__ float scale(int mode, int f, int g, float &nm1) const
    {
        const int a = shift(f), b = shift(g);
        const float l = (float)(a - N / 2) * fov_over_n + l0;
        const float m = (float)(b - N / 2) * fov_over_n + m0;
        const float r2 = l * l + m * m;
        const float n = sqrtf(1.f - r2);
        nm1 = -r2 / (1.f + n);
        const float cc = __ldg(taper + a) * __ldg(taper + b);
        const float s = ((f + g) & 1) ? -1.f : 1.f;
        return mode == 1 ? s * n / cc : s / (n * cc);
    }
};

// exp(sgn 2 pi i w_c (n - 1)) with the argument reduced to [-1/2, 1/2] turns
__device__ __forceinline__ float2 slice_phase(float wc, float nm1, float sgn)
{
    float x = wc * nm1;
    x -= rintf(x);
    float sn, cs;
    sincospif(2.f * x, &sn, &cs);
    return make_float2(cs, sgn * sn);
}

// thread's k-th point of a row before (DIR_IN) and after the transform
template <int R>
__device__ __forceinline__ int index_in(int k) { return threadIdx.x + Rows<R>::T * k; }
template <int R>
__device__ __forceinline__ int index_out(int k)
{
    return 256 * (k % R) + threadIdx.x + Rows<R>::T * (k / R);
}

// Inverse rows in place, rows g and g + N/2 by one block (each lands in the
// other's place): buf[b][a] = scale * transform.
template <int R>
__global__ void __launch_bounds__(Rows<R>::T, Rows<R>::BPS) rows_to_image_kernel(
    Pixels px, int mode, float2 *buf, const float2 *__restrict__ tab)
{
    __shared__ float2 shm[Rows<R>::kShm];
    const int N = Rows<R>::N;
    float2 v[2][16];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int k = 0; k < 16; ++k)
            v[h][k] = buf[(int64_t)(blockIdx.x + h * (N / 2)) * N + index_in<R>(k)];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int g = blockIdx.x + h * (N / 2);
        __syncthreads();
        row_fft<R, true>(v[h], tab, shm);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int f = index_out<R>(k);
            float nm1;
            const float s = px.scale(mode, f, g, nm1);
            buf[(int64_t)px.shift(g) * N + px.shift(f)] = make_float2(s * v[h][k].x, s * v[h][k].y);
        }
    }
}

// Inverse rows of all slices, the slice phase and the sum: one block per row.
// The next slice's row is copied into shared memory while this one's is
// transformed (cp.async), so that the loads stay in flight.
template <int R>
__global__ void __launch_bounds__(Rows<R>::T, Rows<R>::BPS) slices_to_image_kernel(
    Pixels px, int L, const float *__restrict__ wc, const float2 *__restrict__ g,
    float2 *__restrict__ image, const float2 *__restrict__ tab)
{
    extern __shared__ float4 dyn[];
    float2 *const shm = reinterpret_cast<float2 *>(dyn);
    float2 *const next = shm + ((Rows<R>::kShm + 1) & ~1);  // N float2, 16-byte aligned
    float *const nm1 = reinterpret_cast<float *>(next + Rows<R>::N);  // n - 1, N floats
    const int N = Rows<R>::N, T = Rows<R>::T;
    const int64_t n2 = (int64_t)N * N;
    const int row = blockIdx.x;
    float2 acc[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        acc[k] = make_float2(0.f, 0.f);
        px.scale(1, index_out<R>(k), row, nm1[index_out<R>(k)]);  // read by this thread alone
    }
    const float2 *src = g + (int64_t)row * N;
    auto fetch = [&](int c) {
        const unsigned dst = (unsigned)__cvta_generic_to_shared(next) + 16u * threadIdx.x;
        const char *from = reinterpret_cast<const char *>(src + c * n2) + 16 * threadIdx.x;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * T * k),
                         "l"(from + 16 * T * k)
                         : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(0);
    for (int c = 0; c < L; ++c) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // the row has landed; the last transform is done with shm
        float2 v[16];
#pragma unroll
        for (int k = 0; k < 16; ++k)
            v[k] = next[index_in<R>(k)];
        __syncthreads();
        if (c + 1 < L)
            fetch(c + 1);
        row_fft<R, true>(v, tab, shm);
        const float w = __ldg(wc + c);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const float2 e = slice_phase(w, nm1[index_out<R>(k)], 1.f);
            acc[k].x += v[k].x * e.x - v[k].y * e.y;
            acc[k].y += v[k].x * e.y + v[k].y * e.x;
        }
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int f = index_out<R>(k);
        float n;
        const float s = px.scale(1, f, row, n);
        image[(int64_t)px.shift(row) * N + px.shift(f)] = make_float2(s * acc[k].x, s * acc[k].y);
    }
}

// Forward rows of all slices from one load of the image's row.
template <int R>
__global__ void __launch_bounds__(Rows<R>::T, Rows<R>::BPS) image_to_slices_kernel(
    Pixels px, int L, const float *__restrict__ wc, const float2 *__restrict__ image,
    float2 *__restrict__ g, const float2 *__restrict__ tab)
{
    __shared__ float2 shm[Rows<R>::kShm];
    const int N = Rows<R>::N;
    const int64_t n2 = (int64_t)N * N;
    const int row = blockIdx.x;
    float2 x[16];
    float nm1[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int f = index_in<R>(k);
        const float s = px.scale(2, f, row, nm1[k]);
        const float2 y = image[(int64_t)px.shift(row) * N + px.shift(f)];
        x[k] = make_float2(s * y.x, s * y.y);
    }
    for (int c = 0; c < L; ++c) {
        const float w = __ldg(wc + c);
        float2 v[16];
#pragma unroll
        for (int k = 0; k < 16; ++k)
            v[k] = cmul(x[k], slice_phase(w, nm1[k], -1.f));
        __syncthreads();
        row_fft<R, false>(v, tab, shm);
        float2 *const out = g + c * n2 + (int64_t)row * N;
#pragma unroll
        for (int k = 0; k < 16; ++k)
            out[index_out<R>(k)] = v[k];
    }
}

Pixels pixels(const DevParams &p, const float *taper)
{
    return {p.N, (float)(p.fov / p.N), (float)p.l0, (float)p.m0, taper};
}

}  // namespace

bool rows_supported(int N) { return N == 512 || N == 1024 || N == 2048 || N == 4096; }

size_t rows_table_bytes(int N) { return sizeof(float2) * kTw * (N / 16 + 16); }

cudaError_t launch_rows_tables(const DevParams &p, const double2 *tw, float2 *tab, cudaStream_t s)
{
    const int n = kTw * (p.N / 16 + 16);
    fft_tables_kernel<<<(n + 255) / 256, 256, 0, s>>>(p.N, p.OS, tw, tab);
    return cudaGetLastError();
}

#define SEPW_FOR_EACH_ROWS(X) X(2) X(4) X(8) X(16)

cudaError_t launch_columns(const DevParams &p, bool inverse, int grids, const float2 *tab,
                           float2 *g, int num_sms, cudaStream_t s)
{
    switch (p.N / 256) {
#define X(R)                                                                                    \
    case R: {                                                                                   \
        auto *kernel = inverse ? columns_kernel<R, true> : columns_kernel<R, false>;            \
        cudaError_t e = cudaFuncSetAttribute(                                                   \
            kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Cols<R>::kShm);                \
        if (e != cudaSuccess)                                                                   \
            return e;                                                                           \
        const int64_t tiles = (int64_t)grids * (p.N / 4), fit = (int64_t)num_sms * Cols<R>::BPS; \
        kernel<<<(unsigned)(tiles < fit ? tiles : fit), Cols<R>::kThreads, Cols<R>::kShm, s>>>( \
            grids, g, tab);                                                                     \
        break;                                                                                  \
    }
        SEPW_FOR_EACH_ROWS(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_rows_to_image(const DevParams &p, int mode, const float *taper,
                                 const float2 *tab, float2 *buf, cudaStream_t s)
{
    switch (p.N / 256) {
#define X(R)                                                                                  \
    case R:                                                                                   \
        rows_to_image_kernel<R><<<p.N / 2, Rows<R>::T, 0, s>>>(pixels(p, taper), mode, buf, tab); \
        break;
        SEPW_FOR_EACH_ROWS(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_slices_to_image(const DevParams &p, int L, const float *taper, const float *wc,
                                   const float2 *tab, const float2 *g, float2 *image,
                                   cudaStream_t s)
{
    switch (p.N / 256) {
#define X(R)                                                                                   \
    case R: {                                                                                  \
        const int shm =                                                                        \
            sizeof(float2) * (((Rows<R>::kShm + 1) & ~1) + Rows<R>::N) +                       \
            sizeof(float) * Rows<R>::N;                                                        \
        cudaError_t e = cudaFuncSetAttribute(slices_to_image_kernel<R>,                        \
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, shm); \
        if (e != cudaSuccess)                                                                  \
            return e;                                                                          \
        slices_to_image_kernel<R>                                                              \
            <<<p.N, Rows<R>::T, shm, s>>>(pixels(p, taper), L, wc, g, image, tab);             \
        break;                                                                                 \
    }
        SEPW_FOR_EACH_ROWS(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_image_to_slices(const DevParams &p, int L, const float *taper, const float *wc,
                                   const float2 *tab, const float2 *image, float2 *g,
                                   cudaStream_t s)
{
    switch (p.N / 256) {
#define X(R)                                                                                     \
    case R:                                                                                      \
        image_to_slices_kernel<R>                                                                \
            <<<p.N, Rows<R>::T, 0, s>>>(pixels(p, taper), L, wc, image, g, tab);                 \
        break;
        SEPW_FOR_EACH_ROWS(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace sepw
