// Stored correction of the separable kernel (Sec. 7): the difference
// F_w - F~_w between the exact 2-D W-projection kernel and the separable one,
// kept in a full 2-D table, and a second gridding / degridding pass that
// applies it on top of the separable pass.
//
// Table: res[p][ovr][our][k][j] for the Sr x Sr central footprint cells
// (first at k0 = (S - Sr)/2) and OSr oversample offsets per axis (coarse
// entry c stands for the fine offset c * OS / OSr).  Built in float64:
//   F_w(d_u, d_v) = (1/N^2) sum_{a,b} c1(nu_a) c1(nu_b) exp(2 pi i w (n_ab - 1))
//                   exp(-2 pi i (d_u nu_a + d_v nu_b))
// minus the outer product of the 1-D taps at the same offsets.
//
// The build is bound by the FP64 pipe (about 1.3 operations per clock and SM),
// so the sum is folded by its symmetries.  With alpha = a - N/2 and
// h(alpha, beta) = c1 c1 exp(2 pi i w (n - 1)), even in alpha and in beta and
// symmetric in the two, only alpha = -N/2 (and beta = -N/2) has no partner:
//   F_w = A(|d_v|, |d_u|) + e(d_v) B(|d_u|) + e(d_u) B(|d_v|)
//         + e(d_v) e(d_u) h(N/2, N/2),                     e(d) = exp(pi i d),
//   A(x, y) = sum_{alpha, beta = 0}^{N/2 - 1} C(x, beta) h(alpha, beta) C(y, alpha),
//   B(x)    = sum_{beta = 0}^{N/2 - 1} C(x, beta) h(N/2, beta),
//   C(x, beta) = (beta ? 2 : 1) cos(2 pi x beta / N)  (real).
// The offsets are the multiples of 1/OSr from -Sr/2 + 1/OSr to Sr/2, so |d|
// takes R/2 + 1 values for R = OSr Sr; and A(x, y) = M(x, y) + M(y, x) with M
// summed over beta <= alpha alone (the diagonal by half).  That leaves a
// thirty-second of the direct sum's multiply-adds (real by complex, too) and an
// eighth of its screen values, since one thread accumulates all rows of its
// alpha (up to 33).  N = 1024, 32 planes, 8 x 8 cells, 8 x 8 offsets: the
// direct sum took 62.1 ms, all alpha and beta 2.4 ms (rows 2.21, columns 0.12,
// edge 0.06, table 0.01), this 1.3 ms in all.
//
// Pass: each warp takes work items of the plan; per visibility the lanes
// cover the Sr^2 cells.  Gridding adds W V R (conj(R) for w < 0) with float2
// atomics; degridding adds W sum conj(kernel) X to the visibility (the
// separable degridding pass writes it first).
#include "sepw_internal.cuh"

namespace sepw {

// exp(-2 pi i d nu) at d * OS = dos (an integer) and nu = (b - N/2)/N
__device__ __forceinline__ double2 dft_tw(const double2 *tw, int64_t M, int64_t dos, int b,
                                          int N)
{
    int64_t m = (dos * (int64_t)(b - N / 2)) % M;
    if (m < 0)
        m += M;
    return tw[m];
}

// integer d * OS of table row r = (coarse offset c, tap t)
__device__ __forceinline__ int64_t row_dos(const DevParams &p, int Sr, int OSr, int r)
{
    const int c = r / Sr, t = r % Sr;
    const int kk = (p.S - Sr) / 2 + t;
    return (int64_t)(kk - p.S / 2 + 1) * p.OS - (int64_t)c * (p.OS / OSr);
}

// C[beta][x] for x = 0 .. R2 - 1 (offset x / OSr), beta < N/2; row stride R2
__global__ void __launch_bounds__(256) residual_cos_kernel(DevParams p, int OSr, int R2,
                                                           const double2 *tw, double *C)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)(p.N / 2) * R2)
        return;
    const int beta = (int)(e / R2), x = (int)(e % R2);
    const int64_t M = (int64_t)p.N * p.OS;
    const int64_t m = ((int64_t)x * (p.OS / OSr) * beta) % M;
    C[e] = (beta ? 2.0 : 1.0) * tw[m].x;
}

__device__ __forceinline__ double n_minus_1(double l, double m)
{
    const double r2 = l * l + m * m;
    return -r2 / (1.0 + sqrt(1.0 - r2));
}

__device__ __forceinline__ double2 screen(double wp, double nm1)
{
    double s, c;
    sincospi(2.0 * (wp * nm1), &s, &c);
    return make_double2(c, s);
}

// The pixels' n - 1 once for all planes (its square root and division are a
// fifth of the rows' FP64 operations): nm1[beta][alpha], beta <= alpha < N/2,
// for N up to kNm1MaxN (2 N^2 bytes); beyond, the rows compute it.
constexpr int kNm1MaxN = 8192;

__global__ void __launch_bounds__(256) residual_nm1_kernel(DevParams p, double *nm1)
{
    const int H = p.N / 2, alpha = blockIdx.x * blockDim.x + threadIdx.x, beta = blockIdx.y;
    if (alpha < H && beta <= alpha)
        nm1[(int64_t)beta * H + alpha] = n_minus_1((double)alpha / (double)p.N * p.fov,
                                                   (double)beta / (double)p.N * p.fov);
}

__device__ __forceinline__ double plane_w(const DevParams &p, int plane)
{
    return p.P > 1 ? (double)plane * p.w_max / (double)(p.P - 1) : 0.0;
}

// Rows: Y[p][z][x][alpha] = sum over the z-th part of beta <= alpha of C(x, beta)
// h(alpha, beta) (beta = alpha by half), for G values of x from x0 (x >= R2: not
// written).  grid (ceil(N/2 / 64), P, parts * groups), the long sums first;
// block 64
constexpr int kResRowThreads = 64;

template <int G>
__global__ void __launch_bounds__(kResRowThreads) residual_rows_kernel(
    DevParams p, int R2, int parts, const double *__restrict__ taper64,
    const double *__restrict__ C, const double *__restrict__ nm1, double2 *__restrict__ Y)
{
    const int H = p.N / 2;
    const int alpha = (gridDim.x - 1 - blockIdx.x) * kResRowThreads + threadIdx.x;
    const int plane = blockIdx.y;
    const int z = blockIdx.z % parts, x0 = (blockIdx.z / parts) * G;
    if (alpha >= H)
        return;
    const int len = (H + parts - 1) / parts;
    const int b0 = z * len, b1 = min(alpha + 1, b0 + len);
    const double wp = plane_w(p, plane);
    const double l = (double)alpha / (double)p.N * p.fov;
    const double ca = taper64[H + alpha];
    double2 acc[G];
#pragma unroll
    for (int q = 0; q < G; ++q)
        acc[q] = make_double2(0.0, 0.0);
    for (int beta = b0; beta < b1; ++beta) {
        const double x = nm1 ? __ldg(nm1 + (int64_t)beta * H + alpha)
                             : n_minus_1(l, (double)beta / (double)p.N * p.fov);
        const double2 e = screen(wp, x);
        const double t = ca * taper64[H + beta] * (beta == alpha ? 0.5 : 1.0);
        const double hr = t * e.x, hi = t * e.y;
        const double *c = C + (int64_t)beta * R2 + x0;
#pragma unroll
        for (int q = 0; q < G; ++q) {
            const double cq = x0 + q < R2 ? __ldg(c + q) : 0.0;
            acc[q].x = fma(cq, hr, acc[q].x);
            acc[q].y = fma(cq, hi, acc[q].y);
        }
    }
    double2 *y = Y + (((int64_t)plane * parts + z) * R2 + x0) * H + alpha;
#pragma unroll
    for (int q = 0; q < G; ++q)
        if (x0 + q < R2)
            y[(int64_t)q * H] = acc[q];
}

// B[p][x] = sum_beta C(x, beta) h(N/2, beta); B[p][R2] = h(N/2, N/2).
// grid (P); block 256
__global__ void __launch_bounds__(256) residual_edge_kernel(DevParams p, int R2,
                                                            const double *__restrict__ taper64,
                                                            const double *__restrict__ C,
                                                            double2 *__restrict__ B)
{
    __shared__ double2 h[1024];
    const int H = p.N / 2, plane = blockIdx.x;
    const double wp = plane_w(p, plane);
    const double l = 0.5 * p.fov, ca = taper64[0];
    for (int xb = 0; xb < R2; xb += blockDim.x) {
        const int x = xb + threadIdx.x;
        double2 acc = make_double2(0.0, 0.0);
        for (int c0 = 0; c0 < H; c0 += 1024) {
            __syncthreads();
            for (int i = threadIdx.x; i < 1024 && c0 + i < H; i += blockDim.x) {
                const double2 e = screen(wp, n_minus_1(l, (double)(c0 + i) / (double)p.N * p.fov));
                const double t = ca * taper64[H + c0 + i];
                h[i] = make_double2(t * e.x, t * e.y);
            }
            __syncthreads();
            const int lim = min(1024, H - c0);
            if (x < R2)
                for (int i = 0; i < lim; ++i) {
                    const double cq = __ldg(C + (int64_t)(c0 + i) * R2 + x);
                    acc.x = fma(cq, h[i].x, acc.x);
                    acc.y = fma(cq, h[i].y, acc.y);
                }
        }
        if (x < R2)
            B[(int64_t)plane * (R2 + 1) + x] = acc;
    }
    if (threadIdx.x == 0) {
        const double2 e = screen(wp, n_minus_1(l, l));
        B[(int64_t)plane * (R2 + 1) + R2] = make_double2(ca * ca * e.x, ca * ca * e.y);
    }
}

// Columns: M[p][x][y] = sum_alpha Y[p][.][x][alpha] C(y, alpha).  A block
// takes one (plane, x): the parts of Y are summed into shared memory, then
// thread (g, y) sums its quarter of each chunk of alphas.
// grid (R2, P); block (64, 4)
__global__ void __launch_bounds__(256) residual_cols_kernel(DevParams p, int R2, int parts,
                                                            const double *__restrict__ C,
                                                            const double2 *__restrict__ Y,
                                                            double2 *__restrict__ M)
{
    constexpr int kCh = 512;
    __shared__ double2 ys[kCh];
    __shared__ double2 red[4][64];
    const int H = p.N / 2, x = blockIdx.x, plane = blockIdx.y;
    const int g = threadIdx.y, tid = g * 64 + threadIdx.x;
    const double2 *y0 = Y + ((int64_t)plane * parts * R2 + x) * H;
    for (int yb = 0; yb < R2; yb += 64) {
        const int y = yb + threadIdx.x;
        double2 acc = make_double2(0.0, 0.0);
        for (int c0 = 0; c0 < H; c0 += kCh) {
            __syncthreads();
            for (int i = tid; i < kCh && c0 + i < H; i += 256) {
                double2 v = y0[c0 + i];
                for (int z = 1; z < parts; ++z) {
                    const double2 w = y0[(int64_t)z * R2 * H + c0 + i];
                    v.x += w.x;
                    v.y += w.y;
                }
                ys[i] = v;
            }
            __syncthreads();
            const int lim = min(kCh, H - c0);
            if (y < R2)
                for (int i = g; i < lim; i += 4) {
                    const double cq = __ldg(C + (int64_t)(c0 + i) * R2 + y);
                    acc.x = fma(cq, ys[i].x, acc.x);
                    acc.y = fma(cq, ys[i].y, acc.y);
                }
        }
        red[g][threadIdx.x] = acc;
        __syncthreads();
        if (g == 0 && y < R2) {
            for (int q = 1; q < 4; ++q) {
                acc.x += red[q][threadIdx.x].x;
                acc.y += red[q][threadIdx.x].y;
            }
            M[((int64_t)plane * R2 + x) * R2 + y] = acc;
        }
    }
}

// F_w from M and B, minus the separable product; writes the table.
// grid (ceil(R*R / 256), P); block 256
__global__ void __launch_bounds__(256) residual_table_kernel(
    DevParams p, int Sr, int OSr, int R2, const double2 *__restrict__ tw,
    const double2 *__restrict__ M2, const double2 *__restrict__ B,
    const double2 *__restrict__ taps64, double2 *out64, float2 *out32)
{
    const int R = OSr * Sr;
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int plane = blockIdx.y;
    if (e >= (int64_t)R * R)
        return;
    const int rv = (int)(e / R), ru = (int)(e % R);
    const int64_t M = (int64_t)p.N * p.OS;
    const int step = p.OS / OSr, k0 = (p.S - Sr) / 2;
    const int64_t dv = row_dos(p, Sr, OSr, rv), du = row_dos(p, Sr, OSr, ru);
    const int xv = (int)((dv < 0 ? -dv : dv) / step), xu = (int)((du < 0 ? -du : du) / step);
    const double2 ev = dft_tw(tw, M, dv, 0, p.N), eu = dft_tw(tw, M, du, 0, p.N);
    const double2 *b = B + (int64_t)plane * (R2 + 1);
    const double2 bu = b[xu], bv = b[xv], h = b[R2];
    const double2 *m2 = M2 + (int64_t)plane * R2 * R2;
    const double2 a0 = m2[(int64_t)xv * R2 + xu], a1 = m2[(int64_t)xu * R2 + xv];
    const double2 a = make_double2(a0.x + a1.x, a0.y + a1.y);
    // e(dv) (B(du) + e(du) h) + e(du) B(dv) + A
    const double tr = bu.x + (eu.x * h.x - eu.y * h.y), ti = bu.y + (eu.x * h.y + eu.y * h.x);
    double kr = a.x + (ev.x * tr - ev.y * ti) + (eu.x * bv.x - eu.y * bv.y);
    double ki = a.y + (ev.x * ti + ev.y * tr) + (eu.x * bv.y + eu.y * bv.x);
    const double inv = 1.0 / ((double)p.N * (double)p.N);
    kr *= inv;
    ki *= inv;
    // separable product at the same offsets: taps[p][o][kk]
    const int cv = rv / Sr, k = rv % Sr, cu = ru / Sr, j = ru % Sr;
    const double2 tv = taps64[((int64_t)plane * p.OS + cv * step) * p.S + k0 + k];
    const double2 tu = taps64[((int64_t)plane * p.OS + cu * step) * p.S + k0 + j];
    kr -= tv.x * tu.x - tv.y * tu.y;
    ki -= tv.x * tu.y + tv.y * tu.x;
    const int64_t idx = (((int64_t)plane * OSr + cv) * OSr + cu) * Sr * Sr + k * Sr + j;
    if (out64)
        out64[idx] = make_double2(kr, ki);
    if (out32)
        out32[idx] = make_float2((float)kr, (float)ki);
}

// workspace: Y, M and B (double2), then C and n - 1 (double)
struct ResidualWork {
    int R2, parts;
    size_t nC, nY, nA, nB, nNm1;
    size_t bytes() const { return sizeof(double2) * (nY + nA + nB) + sizeof(double) * (nC + nNm1); }
};

static ResidualWork residual_work(const DevParams &p, int Sr, int OSr)
{
    ResidualWork w;
    const size_t H = p.N / 2;
    w.R2 = OSr * Sr / 2 + 1;
    // parts of the beta sum: enough warps for the FP64 pipes, at most 4 (the
    // partial sums then take no more memory than the R x N sums they replace)
    const size_t threads = (size_t)p.P * H;
    w.parts = threads >= 200000 ? 1 : threads >= 100000 ? 2 : 4;
    w.nC = H * w.R2;
    w.nY = (size_t)p.P * w.parts * w.R2 * H;
    w.nA = (size_t)p.P * w.R2 * w.R2;
    w.nB = (size_t)p.P * (w.R2 + 1);
    w.nNm1 = p.N <= kNm1MaxN ? H * H : 0;
    return w;
}

size_t residual_work_bytes(const DevParams &p, int Sr, int OSr)
{
    return residual_work(p, Sr, OSr).bytes();
}

cudaError_t launch_residual_table(const DevParams &p, int Sr, int OSr, const double *taper64,
                                  const double2 *tw, const double2 *taps64, void *work,
                                  double2 *out64, float2 *out32, cudaStream_t s)
{
    const ResidualWork w = residual_work(p, Sr, OSr);
    double2 *Y = (double2 *)work, *A = Y + w.nY, *B = A + w.nA;
    double *C = (double *)(B + w.nB);
    const int R = OSr * Sr, R2 = w.R2, H = p.N / 2;
    cudaError_t e;
    residual_cos_kernel<<<(unsigned)(((int64_t)H * R2 + 255) / 256), 256, 0, s>>>(p, OSr, R2, tw,
                                                                                C);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    double *nm1 = nullptr;
    if (w.nNm1) {
        nm1 = C + w.nC;
        residual_nm1_kernel<<<dim3((H + 255) / 256, H), 256, 0, s>>>(p, nm1);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return e;
    }
    const unsigned gx = (H + kResRowThreads - 1) / kResRowThreads;
    if (R2 <= 9)
        residual_rows_kernel<9><<<dim3(gx, p.P, w.parts), kResRowThreads, 0, s>>>(
            p, R2, w.parts, taper64, C, nm1, Y);
    else if (R2 <= 17)
        residual_rows_kernel<17><<<dim3(gx, p.P, w.parts), kResRowThreads, 0, s>>>(
            p, R2, w.parts, taper64, C, nm1, Y);
    else
        residual_rows_kernel<33><<<dim3(gx, p.P, w.parts * ((R2 + 32) / 33)), kResRowThreads, 0,
                                   s>>>(p, R2, w.parts, taper64, C, nm1, Y);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    residual_edge_kernel<<<p.P, 256, 0, s>>>(p, R2, taper64, C, B);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    residual_cols_kernel<<<dim3(R2, p.P), dim3(64, 4), 0, s>>>(p, R2, w.parts, C, Y, A);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    residual_table_kernel<<<dim3((unsigned)(((int64_t)R * R + 255) / 256), p.P), 256, 0, s>>>(
        p, Sr, OSr, R2, tw, A, B, taps64, out64, out32);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// correction passes over the plan's work items
//
// A table entry (the Sr x Sr cells of one plane and offset pair) is read once
// per visibility and used once, so the passes are bound by the L2 reads of
// the entries (8 Sr^2 bytes a visibility; the table exceeds L1).  Two things
// keep them near that:
//   * lane l owns the cell pairs l, l + 32, ... (Sr is even, so a pair never
//     straddles two rows): an entry arrives as whole 16-byte loads of
//     consecutive lanes, several visibilities' loads in flight at a time;
//   * the plan's slots come in runs of one (origin, conj) key: gridding sums a
//     run in registers and adds it to the grid once, degridding reads its
//     cells once per run.
// A warp takes one of `parts` consecutive parts of an item, so that plans with
// few items still fill the chip.  One visibility at a time with the cells
// re-read (added by atomics) for each, 8 x 8 cells at 4M visibilities took
// 1.90 ms (gridding) and 2.92 ms (degridding); 0.24 ms each so.
// ---------------------------------------------------------------------------

constexpr int kResWarps = 8;
constexpr int kResBlocksPerSM = 4;
// units a pass aims at per resident warp, and the fewest visibilities in one
constexpr int kResUnitsPerWarp = 8;
constexpr int kResMinUnit = 32;

// parts of an item such that n_items * parts units fill the grid several times
__device__ __forceinline__ int res_parts(int n_items, int chunk)
{
    const int want = gridDim.x * kResWarps * kResUnitsPerWarp;
    return max(1, min(chunk / kResMinUnit, want / max(n_items, 1)));
}

// two adjacent cells of a table entry; VEC: the table is 16-byte aligned
template <bool VEC>
__device__ __forceinline__ float4 load_pair(const float2 *p)
{
    if constexpr (VEC)
        return __ldg(reinterpret_cast<const float4 *>(p));
    const float2 a = __ldg(p), b = __ldg(p + 1);
    return make_float4(a.x, a.y, b.x, b.y);
}

// index of a record's table entry (fits 32 bits unsigned: P OSr^2 <= 2^31)
__device__ __forceinline__ uint32_t res_entry(uint64_t r, int OSr, int step)
{
    return ((uint32_t)rec_plane(r) * OSr + rec_ov(r) / step) * OSr + rec_ou(r) / step;
}

// PPL: cell pairs per lane, ceil(Sr^2 / 64)
template <int PPL, bool VEC>
__global__ void __launch_bounds__(kResWarps * 32) grid_residual_kernel(
    DevParams p, int Sr, int OSr, const WorkItem *__restrict__ items,
    const int32_t *__restrict__ nitems, int32_t *counter, const Slot *__restrict__ slots,
    const float2 *__restrict__ vis, const float *__restrict__ weight,
    const float2 *__restrict__ res, float2 *grid)
{
    __shared__ float4 s_meta[kResWarps * 32];  // entry, key, W V
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float4 *const meta = s_meta + warp * 32;
    const int n_items = *nitems;
    const int step = p.OS / OSr, k0 = (p.S - Sr) / 2, cells = Sr * Sr, pairs = cells / 2;
    const int parts = res_parts(n_items, p.chunk);
    int off[PPL];  // grid offset of the lane's pairs from the footprint's first kept cell
#pragma unroll
    for (int q = 0; q < PPL; ++q) {
        const int c = 2 * (lane + 32 * q);
        off[q] = (c / Sr) * p.N + c % Sr;
    }
    for (;;) {
        int unit = 0;
        if (lane == 0)
            unit = atomicAdd(counter, 1);
        unit = __shfl_sync(0xffffffffu, unit, 0);
        const int item = unit / parts, part = unit % parts;
        if (item >= n_items)
            break;
        const WorkItem it = items[item];
        const int len = max(kResMinUnit, (it.count + parts - 1) / parts);
        const int b0 = it.start + part * len, b1 = min(it.start + it.count, b0 + len);
        if (b0 >= b1)
            continue;
        const TileOrigin o = tile_origin(p, it.tile);
        float2 *const tg = grid + o.base + (o.gy0 + k0) * p.N + o.gx0 + k0;
        float4 acc[PPL];
#pragma unroll
        for (int q = 0; q < PPL; ++q)
            acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        int cur = -1;
        // conj visibilities accumulated conj(W V) R: conjugated here
        auto flush = [&]() {
            if (cur < 0)
                return;
            const float sg = (cur & 1) ? -1.f : 1.f;
            float2 *const g = tg + (int64_t)(cur >> 7) * p.N + ((cur >> 1) & 63);
#pragma unroll
            for (int q = 0; q < PPL; ++q) {
                if (lane + 32 * q < pairs) {
                    atomicAdd(g + off[q], make_float2(acc[q].x, sg * acc[q].y));
                    atomicAdd(g + off[q] + 1, make_float2(acc[q].z, sg * acc[q].w));
                }
                acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        };
        for (int base = b0; base < b1; base += 32) {
            const int s = base + lane;
            int kq = -1;
            if (s < b1) {
                const Slot slot = load_slot(slots + s);
                const uint64_t r = slot.rec;
                const int i = slot.vis;
                const float wt = weight ? __ldg(weight + i) : 1.0f;
                const float2 x = __ldg(vis + i);
                const bool cj = rec_conj(r);
                kq = ((rec_ly(r) * 64 + rec_lx(r)) << 1) | (cj ? 1 : 0);
                meta[lane] = make_float4(__uint_as_float(res_entry(r, OSr, step)),
                                         __int_as_float(kq), wt * x.x,
                                         cj ? -wt * x.y : wt * x.y);
            }
            __syncwarp();
            const int n = min(32, b1 - base);
            const int kp = __shfl_up_sync(0xffffffffu, kq, 1);
            const unsigned starts = __ballot_sync(0xffffffffu, lane < n && (lane == 0 || kq != kp));
            for (int q = 0; q < n;) {
                const unsigned later = starts & ~((2u << q) - 1u);
                const int q1 = later ? __ffs(later) - 1 : n;
                const int key = __float_as_int(meta[q].y);
                if (key != cur) {
                    flush();
                    cur = key;
                }
#pragma unroll(PPL <= 2 ? 4 : 1)
                for (; q < q1; ++q) {
                    const float4 m = meta[q];
                    const float2 *R = res + (size_t)__float_as_uint(m.x) * cells + 2 * lane;
#pragma unroll
                    for (int c = 0; c < PPL; ++c) {
                        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (lane + 32 * c < pairs)
                            t = load_pair<VEC>(R + 64 * c);
                        acc[c].x = fmaf(m.z, t.x, acc[c].x);
                        acc[c].x = fmaf(-m.w, t.y, acc[c].x);
                        acc[c].y = fmaf(m.z, t.y, acc[c].y);
                        acc[c].y = fmaf(m.w, t.x, acc[c].y);
                        acc[c].z = fmaf(m.z, t.z, acc[c].z);
                        acc[c].z = fmaf(-m.w, t.w, acc[c].z);
                        acc[c].w = fmaf(m.z, t.w, acc[c].w);
                        acc[c].w = fmaf(m.w, t.z, acc[c].w);
                    }
                }
            }
            __syncwarp();
        }
        flush();
    }
}

// Sum of v[e] over the 32 lanes for e = 0..7; v[0] then holds the sum for
// e = lane >> 2.
__device__ __forceinline__ void res_reduce8(float (&v)[8], int lane)
{
#pragma unroll
    for (int h = 4; h > 0; h >>= 1) {
        const bool up = lane & (4 * h);
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float send = up ? v[i] : v[i + h];
            const float keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * h);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
}

template <int PPL, bool VEC>
__global__ void __launch_bounds__(kResWarps * 32) degrid_residual_kernel(
    DevParams p, int Sr, int OSr, const WorkItem *__restrict__ items,
    const int32_t *__restrict__ nitems, int32_t *counter, const Slot *__restrict__ slots,
    const float2 *__restrict__ grid, const float *__restrict__ weight,
    const float2 *__restrict__ res, float2 *vis_out)
{
    constexpr int G = PPL == 1 ? 8 : PPL == 2 ? 4 : PPL <= 4 ? 2 : 1;  // entries in flight
    __shared__ uint2 s_meta[kResWarps * 32];  // entry, key
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint2 *const meta = s_meta + warp * 32;
    const int n_items = *nitems;
    const int step = p.OS / OSr, k0 = (p.S - Sr) / 2, cells = Sr * Sr, pairs = cells / 2;
    const int parts = res_parts(n_items, p.chunk);
    int off[PPL];
#pragma unroll
    for (int q = 0; q < PPL; ++q) {
        const int c = 2 * (lane + 32 * q);
        off[q] = (c / Sr) * p.N + c % Sr;
    }
    for (;;) {
        int unit = 0;
        if (lane == 0)
            unit = atomicAdd(counter, 1);
        unit = __shfl_sync(0xffffffffu, unit, 0);
        const int item = unit / parts, part = unit % parts;
        if (item >= n_items)
            break;
        const WorkItem it = items[item];
        const int len = max(kResMinUnit, (it.count + parts - 1) / parts);
        const int b0 = it.start + part * len, b1 = min(it.start + it.count, b0 + len);
        if (b0 >= b1)
            continue;
        const TileOrigin o = tile_origin(p, it.tile);
        const float2 *const tg = grid + o.base + (o.gy0 + k0) * p.N + o.gx0 + k0;
        float4 x[PPL];
#pragma unroll
        for (int q = 0; q < PPL; ++q)
            x[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        int cur = -1;
        for (int base = b0; base < b1; base += 32) {
            const int s = base + lane;
            int i = -1;
            float wt = 0.f;
            float2 old = make_float2(0.f, 0.f);
            if (s < b1) {
                const Slot slot = load_slot(slots + s);
                const uint64_t r = slot.rec;
                i = slot.vis;
                wt = weight ? __ldg(weight + i) : 1.0f;
                old = vis_out[i];
                meta[lane] = make_uint2(res_entry(r, OSr, step),
                                        ((rec_ly(r) * 64 + rec_lx(r)) << 1) |
                                            (rec_conj(r) ? 1 : 0));
            }
            __syncwarp();
            const int n = min(32, b1 - base);
            for (int qb = 0; qb < n; qb += 8) {
                float vr[8], vi[8];
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    vr[e] = vi[e] = 0.f;
#pragma unroll
                for (int eb = 0; eb < 8; eb += G) {
                    float4 t[G][PPL];
#pragma unroll
                    for (int e = 0; e < G; ++e) {
                        const int q = qb + eb + e;
                        const bool ok = q < n;
                        const float2 *R = res + (size_t)(ok ? meta[q].x : 0u) * cells + 2 * lane;
#pragma unroll
                        for (int c = 0; c < PPL; ++c) {
                            t[e][c] = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (ok && lane + 32 * c < pairs)
                                t[e][c] = load_pair<VEC>(R + 64 * c);
                        }
                    }
#pragma unroll
                    for (int e = 0; e < G; ++e) {
                        if (qb + eb + e >= n)
                            continue;
                        const int key = (int)meta[qb + eb + e].y;
                        if (key != cur) {
                            cur = key;
                            // plain-kernel runs work on conj(X)
                            const float sg = (cur & 1) ? 1.f : -1.f;
                            const float2 *g = tg + (int64_t)(cur >> 7) * p.N + ((cur >> 1) & 63);
#pragma unroll
                            for (int c = 0; c < PPL; ++c)
                                if (lane + 32 * c < pairs) {
                                    const float2 a = __ldg(g + off[c]), b = __ldg(g + off[c] + 1);
                                    x[c] = make_float4(a.x, sg * a.y, b.x, sg * b.y);
                                }
                        }
                        float sr = 0.f, si = 0.f;
#pragma unroll
                        for (int c = 0; c < PPL; ++c) {
                            sr = fmaf(t[e][c].x, x[c].x, sr);
                            sr = fmaf(-t[e][c].y, x[c].y, sr);
                            si = fmaf(t[e][c].x, x[c].y, si);
                            si = fmaf(t[e][c].y, x[c].x, si);
                            sr = fmaf(t[e][c].z, x[c].z, sr);
                            sr = fmaf(-t[e][c].w, x[c].w, sr);
                            si = fmaf(t[e][c].z, x[c].w, si);
                            si = fmaf(t[e][c].w, x[c].z, si);
                        }
                        vr[eb + e] = sr;
                        vi[eb + e] = si;
                    }
                }
                res_reduce8(vr, lane);
                res_reduce8(vi, lane);
                // visibility qb + e was staged by lane qb + e and summed on
                // lanes 4 e .. 4 e + 3
                const int src = 4 * (lane - qb);
                const float re = __shfl_sync(0xffffffffu, vr[0], src & 31);
                const float im = __shfl_sync(0xffffffffu, vi[0], src & 31);
                if (lane >= qb && lane < qb + 8 && i >= 0) {
                    const bool cj = meta[lane].y & 1;
                    vis_out[i] = make_float2(fmaf(wt, re, old.x), fmaf(wt, cj ? im : -im, old.y));
                }
            }
            __syncwarp();
        }
    }
}

// X(ceil(pairs / 32) bound): the instantiated pairs per lane, Sr <= 32
#define SEPW_FOR_EACH_PPL(X) X(1) X(2) X(3) X(4) X(8) X(16)

cudaError_t launch_grid_residual(const DevParams &p, int Sr, int OSr, const Plan &plan,
                                 const float2 *vis, const float *weight, const float2 *res,
                                 float2 *grid, int num_sms, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(plan.d_item_counter, 0, sizeof(int32_t), s);
    if (e != cudaSuccess)
        return e;
    const int ppl = (Sr * Sr / 2 + 31) / 32;
    const bool vec = ((uintptr_t)res & 15) == 0;
#define X(PPL)                                                                              \
    if (ppl <= PPL) {                                                                       \
        (vec ? grid_residual_kernel<PPL, true> : grid_residual_kernel<PPL, false>)          \
            <<<num_sms * kResBlocksPerSM, kResWarps * 32, 0, s>>>(                          \
                p, Sr, OSr, plan.d_items, plan.d_nitems, plan.d_item_counter, plan.d_slots, \
                vis, weight, res, grid);                                                    \
        return cudaGetLastError();                                                          \
    }
    SEPW_FOR_EACH_PPL(X)
#undef X
    return cudaErrorInvalidValue;
}

cudaError_t launch_degrid_residual(const DevParams &p, int Sr, int OSr, const Plan &plan,
                                   const float2 *grid, const float *weight, const float2 *res,
                                   float2 *vis_out, int num_sms, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(plan.d_item_counter + 1, 0, sizeof(int32_t), s);
    if (e != cudaSuccess)
        return e;
    const int ppl = (Sr * Sr / 2 + 31) / 32;
    const bool vec = ((uintptr_t)res & 15) == 0;
#define X(PPL)                                                                              \
    if (ppl <= PPL) {                                                                       \
        (vec ? degrid_residual_kernel<PPL, true> : degrid_residual_kernel<PPL, false>)      \
            <<<num_sms * kResBlocksPerSM, kResWarps * 32, 0, s>>>(                          \
                p, Sr, OSr, plan.d_items, plan.d_nitems, plan.d_item_counter + 1,           \
                plan.d_slots, grid, weight, res, vis_out);                                  \
        return cudaGetLastError();                                                          \
    }
    SEPW_FOR_EACH_PPL(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace sepw
