// Register-window gridder of the tiled FP32 form (the separable update of
// Sec. 5) for supports and densities without long runs of one origin.
//
// The plan orders a tile's visibilities by 4 x 4 blocks of footprint origins,
// down the columns of blocks.  The footprints of one block lie in a window of
// (S + 3)^2 cells, which a warp keeps in registers: lane (rg, cg) =
// (lane >> 3, lane & 7) owns the window's rows rg + 4 r (r < RPL) and columns
// cg + 8 c (c < CPL).  A visibility is added with its taps placed at its
// origin inside the block and zero elsewhere, so it touches every register of
// the warp whatever its origin, and no visibility causes any memory traffic
// but its taps.  When the next block lies d < RPL blocks further down, the
// lanes add their first d rows to the grid (float2 atomics) and shift the
// others up; any other move adds the whole window.
//
// Why: adding a register block per origin costs S^2 atomics for every run of
// visibilities with one origin, and in sparse data nearly every visibility
// has its own (63M visibilities over 128 grids of 2048^2 at S = 12: 144
// atomics each, 0.83e12 a second, 10.97 ms, after a 2.5 ms sort by origin that
// this kernel does not need; now 5.57 ms, 70% of the issue slots).  The window
// adds 4 (S + 3) cells per block of 16 origins and a whole window per column
// of blocks instead.  The price is the zero taps: (S + 3)^2 cells rounded up
// to the lanes' 4 RPL x 8 CPL, 256 for the 144 of S = 12.
//
// Taps come from two tables built per call (window_tables_kernel): u-rows
// padded with three zeros on either side, so that a lane's columns are plain
// loads at a per-visibility offset, and v-rows in the seven alignments
// rg - (origin row mod 4) that occur, each as the RPL taps of one lane in
// row pairs (re, re, im, im): paired FP32 FMAs take them as loaded.
// Pairs along columns (no register moves as the window steps down, a copy of
// the loop for each place of its first row) and scalar FMAs were slower: 7.4
// and 7.1 ms against 6.2 ms then, as was a fifth CTA per SM (48 registers, 7.9 ms).
//
// Zero taps must not meet non-finite values (Inf * 0 would spread to cells
// outside the footprint): visibilities whose W V is not below 1e30, and all
// of them when a tap is not below 1e4, go through add_footprint, which
// touches exactly the S x S cells.
#include "sepw_internal.cuh"

namespace sepw {

constexpr int kWinThreads = 256;
constexpr int kWinWarps = kWinThreads / 32;
constexpr int kWinTabBlocks = 152;  // blocks of the table build, one flag each

template <int S>
struct Win {
    static constexpr int RPL = (S + 6) / 4;   // ceil((S + 3) / 4) rows per lane
    static constexpr int CPL = (S + 10) / 8;  // ceil((S + 3) / 8) columns per lane
    static constexpr int RP = RPL / 2;        // row pairs
    static constexpr bool ODD = RPL % 2 != 0; // and a single last row
    static constexpr int UROW = 2 * (8 * CPL + 4);  // floats of a padded u-row
    // floats of one alignment of a v-row: pairs (re, re, im, im), then the
    // single row's (re, im); 16-byte multiples unless that loads more
    static constexpr int VG = RPL == 3 ? 6 : (2 * RPL + 3) & ~3;
    static constexpr int VROW = 7 * VG;
    // gridding adds a visibility's product to a cell's sum as one number: two
    // FMAs round the sum twice.  Up to S = 6 few visibilities meet in a cell,
    // and the grid was less exact than with each of them added to it alone,
    // whose sums are longer (S = 6, 2 visibilities a cell: 1.65e-7 from the
    // float64 sum, 1.47e-7 alone; S = 12 2.06e-7 and 2.56e-7).
    static constexpr bool ONE_SUM = S <= 6;
    // resident CTAs per SM the registers are limited to
    static constexpr int BPS = S <= 12 ? 4 : S <= 20 ? 3 : 2;
};

template <int S>
constexpr size_t win_row_floats()
{
    return Win<S>::UROW + Win<S>::VROW;
}

// utab[row][e] = tap e - 3 of the u-table (zero outside 0 .. S - 1);
// vtab[row][d + 3] = taps d + 4 r of the v-table in Win's order, d = -3 .. 3;
// flags[block]: some tap this block saw is not below 1e4 in magnitude.  Also
// clears the work counter.
template <int S>
__global__ void __launch_bounds__(256) window_tables_kernel(
    const float2 *utaps, const float2 *vtaps, int64_t rows,
    float *__restrict__ utab, float *__restrict__ vtab, int32_t *__restrict__ flags,
    int32_t *counter, const unsigned long long *ndrop, int64_t *dropped)
{
    pdl_enter();
    using W = Win<S>;
    constexpr int UE = W::UROW / 2, E = UE + 7 * W::RPL;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *counter = 0;
        if (dropped)
            *dropped = (int64_t)*ndrop;
    }
    int big = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < rows * E;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = i / E;
        const int e = (int)(i - row * E);
        const bool is_u = e < UE;
        const int d = is_u ? 0 : (e - UE) / W::RPL, r = is_u ? 0 : (e - UE) % W::RPL;
        const int k = is_u ? e - 3 : d - 3 + 4 * r;
        float2 t = make_float2(0.f, 0.f);
        if (k >= 0 && k < S)
            t = (is_u ? utaps : vtaps)[row * S + k];
        big |= !(fabsf(t.x) < 1e4f && fabsf(t.y) < 1e4f);
        if (is_u) {
            *reinterpret_cast<float2 *>(utab + row * W::UROW + 2 * e) = t;
        } else {
            float *v = vtab + row * W::VROW + d * W::VG + 4 * (r >> 1);
            const bool pair = r < 2 * W::RP;
            v[pair ? r & 1 : 0] = t.x;
            v[pair ? 2 + (r & 1) : 1] = t.y;
        }
    }
    big = __syncthreads_or(big);
    if (threadIdx.x == 0)
        flags[blockIdx.x] = big;
}

// Adds one visibility's exact S x S footprint (origin cell g) by atomics.
template <int S>
__device__ __noinline__ void add_footprint(const float2 *tu,
                                           const float2 *tv, float2 wv, float sg,
                                           float2 *g, int N, int lane)
{
    for (int c = lane; c < S * S; c += 32) {
        const int k = c / S, j = c % S;
        const float2 a = tu[j], b = tv[k];
        const float ay = sg * a.y, by = sg * b.y;
        const float pr = wv.x * a.x - wv.y * ay, pi = wv.x * ay + wv.y * a.x;
        atomicAdd(g + (int64_t)k * N + j, make_float2(pr * b.x - pi * by, pr * by + pi * b.x));
    }
}

__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }

// A lane's v-taps at an alignment: row pairs and the single last row.
template <int S>
__device__ __forceinline__ void window_vtaps(const float *tv,
                                             float2 (&vr)[Win<S>::RP], float2 (&vi)[Win<S>::RP],
                                             float2 &ve)
{
    using W = Win<S>;
#pragma unroll
    for (int k = 0; k < W::RP; ++k) {
        if constexpr (W::VG % 4 == 0) {
            const float4 t = reinterpret_cast<const float4 *>(tv)[k];
            vr[k] = make_float2(t.x, t.y);
            vi[k] = make_float2(t.z, t.w);
        } else {
            vr[k] = reinterpret_cast<const float2 *>(tv)[2 * k];
            vi[k] = reinterpret_cast<const float2 *>(tv)[2 * k + 1];
        }
    }
    if constexpr (W::ODD)
        ve = reinterpret_cast<const float2 *>(tv)[2 * W::RP];
}

template <int S>
__global__ void __launch_bounds__(kWinThreads, Win<S>::BPS) grid_window_kernel(
    DevParams p, const WorkItem *units, const int32_t *nunits,
    int32_t *counter, const Slot *slots,
    const float2 *vis, const float *weight,
    const float2 *taps, const float *utab,
    const float *vtab, const int32_t *flags, float2 *grid)
{
    pdl_enter(p);
    using W = Win<S>;
    constexpr int RPL = W::RPL, CPL = W::CPL, RP = W::RP;
    constexpr bool ODD = W::ODD;
    __shared__ int4 s_meta[kWinWarps * 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rg = lane >> 3, cg = lane & 7;
    int4 *const meta = s_meta + warp * 32;
    const float *const ulane = utab + 2 * cg;
    const float *const vlane = vtab + rg * W::VG;
    // window columns the block's footprints reach (the last one per lane)
    const bool last_col = cg + 8 * (CPL - 1) < S + 3;
    const int n_units = *nunits;
    bool big = false;
    for (int b = lane; b < kWinTabBlocks; b += 32)
        big |= flags[b] != 0;
    big = __any_sync(0xffffffffu, big);

    // the first unit by the warp's number, neighbours (which add to the same
    // cells) on different SMs; the others from the counter, taken when the
    // warp is free: claimed ahead they would wait for a busy one
    const int n_warps = gridDim.x * kWinWarps;
    auto next_unit = [&]() {
        const int k = lane == 0 ? atomicAdd(counter, 1) : 0;
        return n_warps + __shfl_sync(0xffffffffu, k, 0);
    };
    for (int unit = warp * gridDim.x + blockIdx.x; unit < n_units; unit = next_unit()) {
        const WorkItem it = units[unit];
        if (!work_item_ok(p, it))
            continue;  // checked build only
        const TileOrigin o = tile_origin(p, it.tile);
        const int b1 = it.start + it.count;
        // the lane's first cell of the tile's first block
        float2 *const g0 = grid + o.base + (o.gy0 + rg) * p.N + o.gx0 + cg;

        // rows 2q, 2q + 1 of the lane as pairs, the single last row
        float2 ar[RP][CPL], ai[RP][CPL], ae[CPL];
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
#pragma unroll
            for (int q = 0; q < RP; ++q)
                ar[q][c] = ai[q][c] = dup(0.f);
            ae[c] = dup(0.f);
        }
        int cur = -1;         // block: column << 8 | row
        float2 *g = nullptr;  // cell of the lane's first row and column

        // adds the first row to the grid and shifts the others up
        auto step = [&]() {
            const int y = (int)o.gy0 + 4 * (cur & 255) + rg;
            const int x = (int)o.gx0 + 4 * (cur >> 8) + cg;
#pragma unroll
            for (int c = 0; c < CPL; ++c)
                if ((c < CPL - 1 || last_col) && y < p.N && x + 8 * c < p.N)
                    atomicAdd(g + 8 * c, make_float2(ar[0][c].x, ai[0][c].x));
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
#pragma unroll
                for (int q = 0; q < RP; ++q) {
                    const bool more = q + 1 < RP;
                    ar[q][c] = make_float2(ar[q][c].y, more ? ar[more ? q + 1 : q][c].x : ae[c].x);
                    ai[q][c] = make_float2(ai[q][c].y, more ? ai[more ? q + 1 : q][c].x : ae[c].y);
                }
                if constexpr (ODD)
                    ae[c] = dup(0.f);
            }
            ++cur;
            g += 4 * p.N;
        };

        for (int base = it.start; base < b1; base += 32) {
            // lane q stages slot base + q
            const int s = base + lane;
            int blk = -1;
            bool cj = false, slow = false;
            uint64_t r = 0;
            float2 wv = make_float2(0.f, 0.f);
            if (s < b1) {
                const Slot slot = load_slot(slots + s);
                const int i = slot.vis;
                r = slot.rec;
                if (record_ok(p, r, i, o.gy0, o.gx0)) {
                    const float wt = weight ? load_once(weight + i) : 1.0f;
                    const float2 x = load_once(vis + i);
                    cj = rec_conj(r);
                    wv = make_float2(wt * x.x, wt * x.y);
                    slow = big || !(fabsf(wv.x) < 1e30f && fabsf(wv.y) < 1e30f);
                } else {
                    r = 0;  // checked build: a skipped slot adds zero
                }
                const int row = rec_plane(r) * p.OS;
                blk = (rec_lx(r) >> 2) << 8 | (rec_ly(r) >> 2);
                // conj visibilities: conj(W V) F1 F1, conjugated as it is added
                meta[lane] =
                    make_int4((row + rec_ou(r)) * W::UROW + 2 * (3 - (rec_lx(r) & 3)),
                              (row + rec_ov(r)) * W::VROW + (3 - (rec_ly(r) & 3)) * W::VG,
                              __float_as_int(slow ? 0.f : wv.x),
                              __float_as_int(slow ? 0.f : cj ? -wv.y : wv.y));
            }
            __syncwarp();
            const int n = min(32, b1 - base);
            const int prev = __shfl_up_sync(0xffffffffu, blk, 1);
            unsigned starts = __ballot_sync(0xffffffffu, lane < n && (lane == 0 || blk != prev));
            const unsigned cjs = __ballot_sync(0xffffffffu, cj);
            for (unsigned left = __ballot_sync(0xffffffffu, slow); left; left &= left - 1) {
                const int q = __ffs(left) - 1;
                const uint64_t rq = __shfl_sync(0xffffffffu, r, q);
                const float2 wq = make_float2(__shfl_sync(0xffffffffu, wv.x, q),
                                              __shfl_sync(0xffffffffu, wv.y, q));
                const float2 *t = taps + (int64_t)rec_plane(rq) * p.OS * S;
                add_footprint<S>(t + rec_ou(rq) * S, t + p.voff + rec_ov(rq) * S, wq,
                                 rec_conj(rq) ? -1.f : 1.f,
                                 grid + o.base + (o.gy0 + rec_ly(rq)) * p.N + o.gx0 + rec_lx(rq),
                                 p.N, lane);
            }
            for (int q = big ? n : 0; q < n;) {  // (0 times such a tap is no zero either)
                starts &= starts - 1;  // now the next run's start, if any
                const int q1 = starts ? __ffs(starts) - 1 : n;
                const int bq = __shfl_sync(0xffffffffu, blk, q), d = bq - cur;
                if (d != 0) {
                    if (cur >= 0) {  // d rows if further down the same column, else all
#pragma unroll 1
                        for (int k = d > 0 && d < RPL ? d : RPL; k > 0; --k)
                            step();
                    }
                    if (bq != cur) {
                        cur = bq;
                        g = g0 + 4 * ((cur & 255) * p.N + (cur >> 8));
                    }
                }
                for (; q < q1; ++q) {
                    const int4 m = meta[q];
                    // sign of the imaginary part: + 1.0f or - 1.0f
                    const float sg = __uint_as_float(0x3f800000u | (cjs >> q) << 31);
                    const float wx = __int_as_float(m.z), wy = __int_as_float(m.w);
                    const float *tu = ulane + m.x;
                    float2 vr[RP], vi[RP], ve;
                    window_vtaps<S>(vlane + m.y, vr, vi, ve);
#pragma unroll
                    for (int c = 0; c < CPL; ++c) {
                        const float2 t = *reinterpret_cast<const float2 *>(tu + 16 * c);
                        // W V F1(u), Sec. 5
                        const float pr = wx * t.x - wy * t.y, pi = wx * t.y + wy * t.x;
                        const float spr = sg * pr, spi = sg * pi;
#pragma unroll
                        for (int k = 0; k < RP; ++k) {
                            if constexpr (W::ONE_SUM) {
                                const float2 r = __ffma2_rn(vi[k], dup(-pi),
                                                            __fmul2_rn(vr[k], dup(pr)));
                                const float2 i = __ffma2_rn(vi[k], dup(spr),
                                                            __fmul2_rn(vr[k], dup(spi)));
                                ar[k][c] = __fadd2_rn(ar[k][c], r);
                                ai[k][c] = __fadd2_rn(ai[k][c], i);
                            } else {
                                ar[k][c] = __ffma2_rn(vr[k], dup(pr), ar[k][c]);
                                ar[k][c] = __ffma2_rn(vi[k], dup(-pi), ar[k][c]);
                                ai[k][c] = __ffma2_rn(vr[k], dup(spi), ai[k][c]);
                                ai[k][c] = __ffma2_rn(vi[k], dup(spr), ai[k][c]);
                            }
                        }
                        if constexpr (ODD && W::ONE_SUM) {
                            ae[c].x = __fadd_rn(ae[c].x, fmaf(-ve.y, pi, __fmul_rn(ve.x, pr)));
                            ae[c].y = __fadd_rn(ae[c].y, fmaf(ve.y, spr, __fmul_rn(ve.x, spi)));
                        } else if constexpr (ODD) {
                            ae[c].x = fmaf(ve.x, pr, ae[c].x);
                            ae[c].x = fmaf(-ve.y, pi, ae[c].x);
                            ae[c].y = fmaf(ve.x, spi, ae[c].y);
                            ae[c].y = fmaf(ve.y, spr, ae[c].y);
                        }
                    }
                }
            }
            __syncwarp();
        }
        if (cur >= 0)
#pragma unroll 1
            for (int k = 0; k < RPL; ++k)
                step();
    }
}

// ---------------------------------------------------------------------------
// Degridding with the same windows: the warp keeps the window's cells in
// registers (read once per block of origins, a row at a time as it steps
// down), sums a visibility's taps against them with paired FMAs over the
// lane's rows, and leaves a partial sum per lane in shared memory, which is
// added up for 16 visibilities at a time.  For supports without a block
// degridder, whose column kernel keeps the tile's window in shared memory and
// a CTA on every item, with the lanes of one column each: 333k visibilities at
// S = 10 took it 68 us, this kernel 58 us (bound by the latency of its short
// units); a step of 2M at S = 20 1090 us, now 734.  S = 2, 6 and 14 keep the
// column kernel (S = 14, whose window is three lanes' columns wide for 17
// cells: a step of 4M 1222 us with it, 1323 with this one).
//
// As in gridding, zero taps must not meet non-finite values: from the first
// cell of a unit that is not below 1e30 on, its visibilities go through
// degrid_footprint.
// ---------------------------------------------------------------------------
template <int S>
__device__ __noinline__ float2 degrid_footprint(const float2 *tu,
                                                const float2 *tv, float sg,
                                                const float2 *g, int N, int lane)
{
    float2 acc = make_float2(0.f, 0.f);
    for (int c = lane; c < S * S; c += 32) {
        const int k = c / S, j = c % S;
        const float2 a = tu[j], b = tv[k], x = g[(int64_t)k * N + j];
        const float ay = sg * a.y, by = sg * b.y;  // conjugated taps
        const float kr = a.x * b.x - ay * by, ki = a.x * by + ay * b.x;
        acc.x += kr * x.x - ki * x.y;
        acc.y += kr * x.y + ki * x.x;
    }
    return acc;
}

template <int S>
__global__ void __launch_bounds__(kWinThreads, Win<S>::BPS) degrid_window_kernel(
    DevParams p, const WorkItem *units, const int32_t *nunits,
    int32_t *counter, const Slot *slots,
    const float2 *grid, const float *weight,
    const float2 *taps, const float *utab,
    const float *vtab, const int32_t *flags, float2 *__restrict__ vis_out)
{
    pdl_enter(p);
    using W = Win<S>;
    constexpr int RPL = W::RPL, CPL = W::CPL, RP = W::RP;
    constexpr bool ODD = W::ODD;
    __shared__ int2 s_meta[kWinWarps * 32];
    __shared__ float2 s_part[kWinWarps][16 * 33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rg = lane >> 3, cg = lane & 7;
    int2 *const meta = s_meta + warp * 32;
    float2 *const part = s_part[warp];
    const float *const ulane = utab + 2 * cg;
    const float *const vlane = vtab + rg * W::VG;
    const bool last_col = cg + 8 * (CPL - 1) < S + 3;
    const int n_units = *nunits;
    bool big = false;
    for (int b = lane; b < kWinTabBlocks; b += 32)
        big |= flags[b] != 0;
    big = __any_sync(0xffffffffu, big);

    const int n_warps = gridDim.x * kWinWarps;
    auto next_unit = [&]() {
        const int k = lane == 0 ? atomicAdd(counter, 1) : 0;
        return n_warps + __shfl_sync(0xffffffffu, k, 0);
    };
    for (int unit = warp * gridDim.x + blockIdx.x; unit < n_units; unit = next_unit()) {
        const WorkItem it = units[unit];
        if (!work_item_ok(p, it))
            continue;  // checked build only
        const TileOrigin o = tile_origin(p, it.tile);
        const int b1 = it.start + it.count;
        const float2 *const g0 = grid + o.base + (o.gy0 + rg) * p.N + o.gx0 + cg;

        float2 xr[RP][CPL], xi[RP][CPL], xe[CPL];
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
#pragma unroll
            for (int q = 0; q < RP; ++q)
                xr[q][c] = xi[q][c] = dup(0.f);
            xe[c] = dup(0.f);
        }
        int cur = -1;  // block: column << 8 | row
        bool bad = big;
        // the lane's cells of window row rg + 4 r at block blk
        auto load_row = [&](int blk, int r, float2(&v)[CPL]) {
            const int y = 4 * ((blk & 255) + r), x = 4 * (blk >> 8);
            bool off = false;
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                v[c] = dup(0.f);
                if ((c < CPL - 1 || last_col) && o.gy0 + y + rg < p.N &&
                    o.gx0 + x + cg + 8 * c < p.N)
                    v[c] = g0[(int64_t)y * p.N + x + 8 * c];
                off |= !(fabsf(v[c].x) < 1e30f && fabsf(v[c].y) < 1e30f);
            }
            bad |= __any_sync(0xffffffffu, off);
        };
        auto step = [&]() {  // one block down: the first row leaves, a new last one comes
            float2 v[CPL];
            ++cur;
            load_row(cur, RPL - 1, v);
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
#pragma unroll
                for (int q = 0; q < RP; ++q) {
                    const bool more = q + 1 < RP;
                    const int n = more ? q + 1 : q;
                    xr[q][c] = make_float2(xr[q][c].y, more ? xr[n][c].x : ODD ? xe[c].x : v[c].x);
                    xi[q][c] = make_float2(xi[q][c].y, more ? xi[n][c].x : ODD ? xe[c].y : v[c].y);
                }
                if constexpr (ODD)
                    xe[c] = v[c];
            }
        };
        auto move_to = [&](int blk) {
            const int d = blk - cur;
            if (cur >= 0 && d > 0 && d < RPL) {
#pragma unroll 1
                for (int k = 0; k < d; ++k)
                    step();
            } else {
#pragma unroll
                for (int r = 0; r < RPL; ++r) {
                    float2 v[CPL];
                    load_row(blk, r, v);
#pragma unroll
                    for (int c = 0; c < CPL; ++c) {
                        if (r >= 2 * RP) {
                            xe[c] = v[c];
                        } else if (r & 1) {
                            xr[r >> 1][c].y = v[c].x;
                            xi[r >> 1][c].y = v[c].y;
                        } else {
                            xr[r >> 1][c].x = v[c].x;
                            xi[r >> 1][c].x = v[c].y;
                        }
                    }
                }
                cur = blk;
            }
        };

        for (int base = it.start; base < b1; base += 32) {
            const int s = base + lane;
            int blk = -1, i = -1;
            bool cj = false;
            float wt = 0.f;
            uint64_t r = 0;
            if (s < b1) {
                const Slot slot = load_slot(slots + s);
                r = slot.rec;
                i = slot.vis;
                if (record_ok(p, r, i, o.gy0, o.gx0)) {
                    wt = weight ? weight[i] : 1.0f;
                    cj = rec_conj(r);
                } else {
                    r = 0;  // checked build: no output
                    i = -1;
                }
                const int row = rec_plane(r) * p.OS;
                blk = (rec_lx(r) >> 2) << 8 | (rec_ly(r) >> 2);
                meta[lane] = make_int2((row + rec_ou(r)) * W::UROW + 2 * (3 - (rec_lx(r) & 3)),
                                       (row + rec_ov(r)) * W::VROW +
                                           (3 - (rec_ly(r) & 3)) * W::VG);
            }
            __syncwarp();
            const int n = min(32, b1 - base);
            const int prev = __shfl_up_sync(0xffffffffu, blk, 1);
            unsigned starts = __ballot_sync(0xffffffffu, lane < n && (lane == 0 || blk != prev));
            // a half of 16 starts a run of its own, so that runs end with it
            if (n > 16)
                starts |= 1u << 16;
            const unsigned cjs = __ballot_sync(0xffffffffu, cj);
            for (int q = 0; q < n;) {
                starts &= starts - 1;  // now the next run's start, if any
                const int q1 = starts ? __ffs(starts) - 1 : n;
                const int bq = __shfl_sync(0xffffffffu, blk, q);
                if (bq != cur)
                    move_to(bq);
                if (bad) {
                    for (; q < q1; ++q) {
                        const uint64_t rq = __shfl_sync(0xffffffffu, r, q);
                        const float2 *t = taps + (int64_t)rec_plane(rq) * p.OS * S;
                        part[(q & 15) * 33 + lane] = degrid_footprint<S>(
                            t + rec_ou(rq) * S, t + p.voff + rec_ov(rq) * S,
                            rec_conj(rq) ? 1.f : -1.f,
                            grid + o.base + (o.gy0 + rec_ly(rq)) * p.N + o.gx0 + rec_lx(rq), p.N,
                            lane);
                    }
                }
                for (; q < q1; ++q) {
                    const int2 m = meta[q];
                    // plain kernels take conjugated taps: sign + 1, conj ones - 1
                    const float sg = __uint_as_float(0x3f800000u | (cjs >> q) << 31);
                    const float *tu = ulane + m.x;
                    float2 vr[RP], vi[RP], ve;
                    window_vtaps<S>(vlane + m.y, vr, vi, ve);
#pragma unroll
                    for (int k = 0; k < RP; ++k)
                        vi[k] = __fmul2_rn(vi[k], dup(sg));
                    if constexpr (ODD)
                        ve.y *= sg;
                    float sr = 0.f, si = 0.f;
#pragma unroll
                    for (int c = 0; c < CPL; ++c) {
                        float2 a = dup(0.f), b = dup(0.f);  // sum conj(v) x over the rows
#pragma unroll
                        for (int k = 0; k < RP; ++k) {
                            a = __ffma2_rn(vr[k], xr[k][c], a);
                            a = __ffma2_rn(vi[k], xi[k][c], a);
                            b = __ffma2_rn(vr[k], xi[k][c], b);
                            b = __ffma2_rn(make_float2(-vi[k].x, -vi[k].y), xr[k][c], b);
                        }
                        float tr = a.x + a.y, ti = b.x + b.y;
                        if constexpr (ODD) {
                            tr = fmaf(ve.x, xe[c].x, tr);
                            tr = fmaf(ve.y, xe[c].y, tr);
                            ti = fmaf(ve.x, xe[c].y, ti);
                            ti = fmaf(-ve.y, xe[c].x, ti);
                        }
                        const float2 t = *reinterpret_cast<const float2 *>(tu + 16 * c);
                        const float uy = sg * t.y;
                        sr = fmaf(tr, t.x, sr);
                        sr = fmaf(ti, uy, sr);
                        si = fmaf(ti, t.x, si);
                        si = fmaf(-tr, uy, si);
                    }
                    part[(q & 15) * 33 + lane] = make_float2(sr, si);
                }
                if (q == 16 || q == n) {  // 16 partial sums of each lane's 32, two lanes a sum
                    __syncwarp();
                    const int h = (q - 1) & 16, e = h + (lane & 15);
                    float re = 0.f, im = 0.f;
#pragma unroll
                    for (int l = 0; l < 16; ++l) {
                        const float2 t = part[(lane & 15) * 33 + (lane & 16) + l];
                        re += t.x;
                        im += t.y;
                    }
                    re += __shfl_xor_sync(0xffffffffu, re, 16);
                    im += __shfl_xor_sync(0xffffffffu, im, 16);
                    const int ie = __shfl_sync(0xffffffffu, i, e);
                    const float we = __shfl_sync(0xffffffffu, wt, e);
                    if (lane < 16 && e < n && ie >= 0)
                        vis_out[ie] = make_float2(we * re, we * im);
                    __syncwarp();
                }
            }
            __syncwarp();
        }
    }
}

// the tables of this call, from the caller's
template <int S>
struct Tables {
    float *u, *v;
    int32_t *flags;
    Tables(const DevParams &p, float *at)
    {
        const int64_t rows = (int64_t)p.P * p.OS;
        u = at;
        v = u + Win<S>::UROW * rows;
        flags = reinterpret_cast<int32_t *>(v + Win<S>::VROW * rows);
    }
    cudaError_t build(const DevParams &p, const float2 *taps, int32_t *counter, const Plan &plan,
                      int64_t *dropped, cudaStream_t s) const
    {
        return launch_pdl(window_tables_kernel<S>, kWinTabBlocks, 256, 0, s, taps, taps + p.voff,
                          (int64_t)p.P * p.OS, u, v, flags, counter, plan.d_dropped, dropped);
    }
};

template <int S>
static cudaError_t launch_S(const DevParams &p, const Plan &plan, const float2 *vis,
                            const float *weight, const float2 *taps, float *tables, float2 *grid,
                            int num_sms, cudaStream_t s)
{
    const Tables<S> t(p, tables);
    const cudaError_t e = t.build(p, taps, plan.d_item_counter, plan, plan.dropped_out, s);
    if (e != cudaSuccess)
        return e;
    return launch_pdl(grid_window_kernel<S>, num_sms * Win<S>::BPS, kWinThreads, 0, s, p,
                      plan.d_units, plan.d_nunits, plan.d_item_counter, plan.d_slots,
                      vis, weight, taps, t.u, t.v, t.flags, grid);
}

template <int S>
static cudaError_t launch_degrid_S(const DevParams &p, const Plan &plan, const float2 *grid,
                                   const float *weight, const float2 *taps, float *tables,
                                   float2 *vis, int num_sms, cudaStream_t s)
{
    const Tables<S> t(p, tables);
    const cudaError_t e = t.build(p, taps, plan.d_item_counter + 1, plan, nullptr, s);
    if (e != cudaSuccess)
        return e;
    return launch_pdl(degrid_window_kernel<S>, num_sms * Win<S>::BPS, kWinThreads, 0, s, p,
                      plan.d_units, plan.d_nunits, plan.d_item_counter + 1, plan.d_slots,
                      grid, weight, taps, t.u, t.v, t.flags, vis);
}

// every support but 8, whose block gridder is the faster one (plan_window)
#define SEPW_FOR_EACH_WIN_S(X) \
    X(2) X(4) X(6) X(10) X(12) X(14) X(16) X(18) X(20) X(22) X(24) X(26) X(28) X(30) X(32)

// Bytes of the tables, 0 if the window gridder does not take these
// parameters: tiles above 32 (a tile has at most 64 blocks of 4 x 4 origins)
// and tables beyond 256 MB (several times the caller's own table; offsets
// stay in int32)
size_t window_tables_bytes(const DevParams &p)
{
    if (p.T > 32)
        return 0;
    size_t row = 0;
    switch (p.S) {
#define X(SS) \
    case SS: row = win_row_floats<SS>(); break;
        SEPW_FOR_EACH_WIN_S(X)
#undef X
    default: return 0;
    }
    const size_t b = sizeof(float) * (row * p.P * p.OS + kWinTabBlocks);
    return b <= ((size_t)256 << 20) ? b : 0;
}

cudaError_t launch_grid_window(const DevParams &p, const Plan &plan, const float2 *vis,
                               const float *weight, const float2 *taps, float *tables,
                               float2 *grid, int num_sms, cudaStream_t s)
{
    switch (p.S) {
#define X(SS) \
    case SS: return launch_S<SS>(p, plan, vis, weight, taps, tables, grid, num_sms, s);
        SEPW_FOR_EACH_WIN_S(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
}

// supports without a block degridder, but for 2, 6 and 14 (see the kernel)
#define SEPW_FOR_EACH_DEGRID_S(X) X(10) X(18) X(20) X(22) X(24) X(26) X(28) X(30) X(32)

// Left to the column degridder:
//   * small plans of medium density: its CTAs take parts of an item, the
//     window's warps whole units, one visibility after the other.  20k on
//     1000^2 (21 a tile), random order: S = 10 38 us with the window and 17
//     with the columns, S = 18 56 and 23; 100k on 2048^2 (24 a tile) S = 10 62
//     and 42, on tracks 31 and 29, S = 18 98 and 63, 46 and 49; 100k on 1000^2
//     (104 a tile) S = 10 45 and 31, 31 and 26.  But there S = 24 76 and 79, 47
//     and 66, and 100k on 4096^2 (6 a tile, and a tile's cells loaded for each)
//     S = 10 69 and 155;
//   * sorted plans at S = 10: 6M on 1000^2, tracks 585 and 473 us, random order
//     640 and 564; 1.5M 165 and 142, 184 and 194.  (S = 18: 1054 and 1108,
//     1124 and 1300.)
// Sparse plans in random order are slower with the window from there on (400k
// on 2048^2, S = 18: 168 and 148 us), tracks faster (114 and 149).
bool degrid_window_takes(const DevParams &p, const Plan &plan)
{
    const int64_t tiles = plan.ntiles;
    if (!plan.window || (p.S == 10 && plan.sorted) ||
        (plan.nvis <= (128 << 10) && plan.nvis >= 12 * tiles &&
         plan.nvis <= (p.S == 10 ? 512 : 64) * tiles))
        return false;
    switch (p.S) {
#define X(SS) case SS:
        SEPW_FOR_EACH_DEGRID_S(X)
#undef X
        return true;
    default: return false;
    }
}

cudaError_t launch_degrid_window(const DevParams &p, const Plan &plan, const float2 *grid,
                                 const float *weight, const float2 *taps, float *tables,
                                 float2 *vis, int num_sms, cudaStream_t s)
{
    switch (p.S) {
#define X(SS) \
    case SS: return launch_degrid_S<SS>(p, plan, grid, weight, taps, tables, vis, num_sms, s);
        SEPW_FOR_EACH_DEGRID_S(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace sepw
