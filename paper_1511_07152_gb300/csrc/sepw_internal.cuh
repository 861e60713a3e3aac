// Internal declarations shared by the CUDA translation units of libsepw.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/sepw.h"

namespace sepw {

// Device-side copy of the parameters plus derived constants.  Passed by
// value to every kernel.
struct DevParams {
    int32_t N, S, OS, P, T;
    int32_t ntx;      // tiles per axis for the tiled forms
    uint32_t t_inv;   // ceil(2^32 / T), see div_tile
    int32_t sub_log2; // log2 of the edge of a plan's blocks of origins
    int32_t sub_n;    // blocks along a tile's edge
    int32_t sub_conj; // 1: a block's conj visibilities are a bin of their own
    int32_t nsub;     // bins of a tile
    double fov;       // inverse cell size: x = u * fov + N/2
    double half;      // N/2 as a double
    double os_d;      // OS as a double
    int32_t os_log2;  // log2(OS) if OS is a power of two, else -1
    int32_t fast_elim;  // locate_axis: exponent bound of its integer path (least: off)
    int32_t fast_near;  // locate_axis: its fall-back margin, in units of 2^-32
    double plane_r;   // (P-1)/w_max (0 if P == 1)
    double w_max;
    double gamma;
    double beta;
    // image-plane faceting (Sec. 4.1): the v-direction taps sit voff elements
    // after the u-direction ones (0: one table for both); the image step takes
    // n at the facet's pixels (l0 + l, m0 + m); the facet tables use the
    // screens exp(2 pi i w a2 l^2) with a2 = a2u (u table), a2v (v table)
    int64_t voff = 0;
    int32_t facet = 0;
    // schedule of the tiled and tensor-core plans (sepw_set_schedule):
    // visibilities per work item (<= kChunk) and the parts a block-gridder
    // warp unit takes of an item (0: by the plan's density)
    int32_t chunk = 2048;
    int32_t grid_parts = 0;
    // 1: the persistent kernels trigger the next launch as they start.  On
    // large plans its blocks would only sit beside them for milliseconds (32M
    // visibilities: step 5.79 against 5.62 ms; 333k: 138 against 136 us; 20k: 52
    // against 60 us).
    int32_t early = 0;
    double l0 = 0.0, m0 = 0.0;
    double a2u = -0.5, a2v = -0.5;
    // bounds of the current plan, read only by the checked build's checks
    // (work_item_ok, record_ok): the status word they report into, the
    // plan's visibility slots and its tile count over all grids
    int32_t *chk_status = nullptr;
    int64_t chk_nvis = 0;
    int64_t chk_tiles = 0;
};

// Programmatic dependent launch: a kernel of a planned step is launched while
// the one before it still runs, and waits (pdl_wait, first thing in the
// kernel) until that one is complete and its writes are visible.  This hides
// the launch between two kernels, a microsecond or two of each of the dozen
// kernels of a small step (20k visibilities: 73 -> 51 us).  Every thread
// waits, so a kernel completes after all kernels before it; a launch without
// the attribute makes both calls no-ops.  pdl_trigger lets the next kernel's
// blocks take free places from here on.
//
// Such a kernel can be resident while the ones before it still write, and the
// non-coherent load path (ld.global.nc: __ldg, const __restrict__ arguments)
// is only defined for data that nobody writes during the reading kernel's
// life.  So the kernels launched by launch_pdl read memory with ordinary loads
// alone, also what only the caller writes (the kernel before the first of a
// chain may be the caller's and may trigger early, too).
__device__ __forceinline__ void pdl_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void pdl_trigger()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_enter()
{
    pdl_trigger();
    pdl_wait();
}
template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), int64_t blocks, int threads, size_t shm,
                              cudaStream_t s, A... args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = shm;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Result of locating one visibility.
struct Loc {
    int32_t cu, cv, ou, ov, plane;
    bool conj;
    bool keep;
};

// floor(fl(x + 0.5)), the IEEE sum rounded to nearest then floored, computed
// exactly from the bits of x without an FP64 add.  For |x| < 2^52 the sum
// x + 0.5 either is representable or rounds only within [2^k, 2^k + 1) for an
// integer power of two 2^k, which leaves its floor unchanged; the one
// exception is x = 0.5 - 2^-54, whose sum 1 - 2^-54 is a tie that rounds to
// 1.0.  So the result is floor(x + 1/2) of the exact real sum, except there.
// Returns false for NaN, +-inf and |x| >= 2^52 (outside the accepted range).
__device__ __forceinline__ bool floor_add_half_bits(double x, long long &out)
{
    const long long b = __double_as_longlong(x);
    const int eb = (int)((b >> 52) & 0x7FF);
    if (eb >= 1023 + 52)
        return false;
    if (eb < 1022) {  // |x| < 1/2: the sum lies in (0, 1)
        out = (b == 0x3FDFFFFFFFFFFFFFll) ? 1 : 0;
        return true;
    }
    const int shift = 52 - (eb - 1023);  // 1..53
    const long long mant = (b & 0x000FFFFFFFFFFFFFll) | 0x0010000000000000ll;
    const long long num = (b < 0 ? -mant : mant) + (1ll << (shift - 1));
    out = num >> shift;  // arithmetic shift: floor division by 2^shift
    return true;
}

// x * 2^k, exact: exponent add when x is normal and stays normal, IEEE
// multiply otherwise (zero, subnormal, overflow; all rounded identically).
__device__ __forceinline__ double scale_pow2(double x, int k, double os_d)
{
    const long long b = __double_as_longlong(x);
    const int eb = (int)((b >> 52) & 0x7FF);
    if (eb >= 1 && eb + k <= 2046)
        return __longlong_as_double(b + ((long long)k << 52));
    return __dmul_rn(x, os_d);
}

// |x| of the double with bits b, times 2^k, in 32.32 fixed point, the fraction
// below 2^-32 cut off; for |x| 2^k < 2^21 (ex <= 20, ex the exponent of x 2^k).
__device__ __forceinline__ void fixed_32_32(long long b, int ex, unsigned &whole, unsigned &frac)
{
    unsigned hi = ((unsigned)(b >> 32) & 0x000FFFFFu) | 0x00100000u, lo = (unsigned)b;
    int s = 20 - ex;  // >= 0: the 53-bit significand is x 2^(52 - ex + k)
    if (s >= 32) {
        lo = hi;
        hi = 0u;
        s -= 32;
    }
    frac = __funnelshift_rc(lo, hi, s);  // s >= 32: hi = 0
    whole = s < 32 ? hi >> s : 0u;
}

// Locate one axis: x = coord*fov + N/2, t = floor(x*OS + 0.5) in IEEE double
// with every operation rounded separately (no FMA contraction), then
// c = floor(t/OS), o = t - c*OS; the footprint c - S/2 + 1 .. c + S/2 must lie
// inside [0, N).  Returns false (drop) otherwise or for non-finite input.
// Only u*fov uses the FP64 pipe on the common path (+ N/2 only within the
// fall-back margin below); the power-of-two scaling, the rounded + 0.5 with
// its floor, and the range checks are exact integer operations on the bits.
//
// Integer path (OS a power of two): with y = fl(coord*fov) the IEEE product,
// t = floor(fl(y + N/2) OS + 1/2).  The exact value floor((y + N/2) OS + 1/2)
// = (N/2) OS + floor(y OS + 1/2) follows from the bits of y (y OS is exact),
// and differs from t only if fl(y + N/2) moves (y + N/2) OS + 1/2 across an
// integer: fl rounds by at most half an ulp of a sum below N, so that needs
// y OS within N OS 2^-53 of a half-integer.  |y| OS is taken in 32.32 fixed
// point; away from half-integers floor(y OS + 1/2) is |y| OS rounded to the
// nearest integer, with the sign of y.  Within fast_near (which covers the
// margin and the cut fraction), and at or beyond 2^fast_elim (which bounds the
// sum; infinities and NaN, too), the FP64 path below decides.
//
// All of it is 32-bit: with 64-bit shifts and 40 bits of fraction the locate
// pass issued 342 instructions per warp, its ALU pipe 80% busy (32M
// visibilities 384 us; 321 us so).
__device__ __forceinline__ bool locate_axis(double coord, const DevParams &p,
                                            int32_t &c, int32_t &o)
{
    const double y = __dmul_rn(coord, p.fov);
    const long long b = __double_as_longlong(y);
    const int ey = (int)((unsigned)(b >> 32) >> 20 & 0x7FFu) - 1023 + p.os_log2;
    if (ey < p.fast_elim) {  // (never for OS that is no power of two)
        unsigned whole, frac;
        fixed_32_32(b, ey, whole, frac);
        if (frac - 0x80000000u + (unsigned)p.fast_near > 2u * (unsigned)p.fast_near) {
            const int n = (int)(whole + (frac >> 31));
            const int t = ((p.N >> 1) << p.os_log2) + (b < 0 ? -n : n);
            c = t >> p.os_log2;
            o = t - (c << p.os_log2);
            return (unsigned)(c - p.S / 2 + 1) <= (unsigned)(p.N - p.S);
        }
    }
    const double x = __dadd_rn(y, p.half);
    long long ti, cc, oo;
    if (p.os_log2 >= 0) {
        if (!floor_add_half_bits(scale_pow2(x, p.os_log2, p.os_d), ti))
            return false;
        if (ti >= 1099511627776ll || ti <= -1099511627776ll)  // |t| < 2^40
            return false;
        cc = ti >> p.os_log2;  // floor division by OS = 2^k
        oo = ti - (cc << p.os_log2);
    } else {
        if (!floor_add_half_bits(__dmul_rn(x, p.os_d), ti))
            return false;
        if (ti >= 1099511627776ll || ti <= -1099511627776ll)
            return false;
        const long long OS = p.OS;
        cc = ti >= 0 ? ti / OS : -((-ti + OS - 1) / OS);
        oo = ti - cc * OS;
    }
    const long long f = cc - p.S / 2 + 1;
    if (f < 0 || f + p.S - 1 > p.N - 1)
        return false;
    c = (int32_t)cc;
    o = (int32_t)oo;
    return true;
}

// Plane: floor(fl(x + 0.5)) for x = fl(|w| r), r = (P-1)/w_max, dropped beyond
// P-1 or if not finite (for P = 1, r = 0: infinity times 0 is NaN); conj =
// (w < 0).  As floor_add_half_bits, in 32 bits: x below 2^21 in fixed point, of
// which only 0.5 - 2^-54 rounds up to 1 from below a half.
__device__ __forceinline__ Loc locate(double u, double v, double w, const DevParams &p)
{
    Loc L;
    L.cu = L.cv = L.ou = L.ov = L.plane = 0;
    L.conj = false;
    int32_t cu = 0, cv = 0, ou = 0, ov = 0;
    bool ok = locate_axis(u, p, cu, ou);
    ok = locate_axis(v, p, cv, ov) && ok;
    const long long wb = __double_as_longlong(w);
    const double x = __dmul_rn(__longlong_as_double(wb & 0x7FFFFFFFFFFFFFFFll), p.plane_r);
    const long long xb = __double_as_longlong(x);
    const int ex = (int)((unsigned)(xb >> 32) >> 20 & 0x7FFu) - 1023;
    unsigned whole, frac;
    fixed_32_32(xb, min(ex, 20), whole, frac);
    const unsigned q = whole + (frac >> 31) + (xb == 0x3FDFFFFFFFFFFFFFll ? 1u : 0u);
    ok = ok && ex <= 20 && q <= (unsigned)(p.P - 1);
    L.keep = ok;
    if (ok) {
        L.cu = cu;
        L.cv = cv;
        L.ou = ou;
        L.ov = ov;
        L.plane = (int32_t)q;
        L.conj = wb < 0 && (wb & 0x7FFFFFFFFFFFFFFFll) != 0;
    }
    return L;
}

// Tile id -> origin of the tile in its grid.  A batched plan numbers the
// tiles of grid g after those of grids 0 .. g-1 (ntx^2 tiles per grid), so the
// grid's base offset follows from the tile id as well.
struct TileOrigin {
    int64_t base;  // element offset of the tile's grid
    int64_t gy0;   // first row of the tile
    int64_t gx0;   // first column of the tile
};
__device__ __forceinline__ TileOrigin tile_origin(const DevParams &p, int tile)
{
    const int per = p.ntx * p.ntx;
    const int g = tile / per;
    const int tl = tile - g * per;
    const int ty = tl / p.ntx, tx = tl - ty * p.ntx;
    TileOrigin o;
    o.base = (int64_t)g * p.N * p.N;
    o.gy0 = (int64_t)ty * p.T;
    o.gx0 = (int64_t)tx * p.T;
    return o;
}

// Packed per-visibility record of a plan (tiled forms), in slot order:
//   bits  0..5   lx  footprint origin column inside the tile (0..T-1)
//   bits  6..11  ly  footprint origin row inside the tile
//   bits 12..19  ou
//   bits 20..27  ov
//   bits 28..42  plane
//   bit  43      conj
__host__ __device__ __forceinline__ uint64_t pack_rec(int lx, int ly, int ou, int ov,
                                                      int plane, bool conj)
{
    return (uint64_t)lx | ((uint64_t)ly << 6) | ((uint64_t)ou << 12) |
           ((uint64_t)ov << 20) | ((uint64_t)plane << 28) | ((uint64_t)conj << 43);
}
__host__ __device__ __forceinline__ int rec_lx(uint64_t r) { return (int)(r & 63); }
__host__ __device__ __forceinline__ int rec_ly(uint64_t r) { return (int)((r >> 6) & 63); }
__host__ __device__ __forceinline__ int rec_ou(uint64_t r) { return (int)((r >> 12) & 255); }
__host__ __device__ __forceinline__ int rec_ov(uint64_t r) { return (int)((r >> 20) & 255); }
__host__ __device__ __forceinline__ int rec_plane(uint64_t r) { return (int)((r >> 28) & 32767); }
__host__ __device__ __forceinline__ bool rec_conj(uint64_t r) { return (r >> 43) & 1; }

// One slot of a plan: the record and the caller's index of its visibility.
struct alignas(16) Slot {
    uint64_t rec;
    int32_t vis;
    int32_t pad;
};
// Loads of what a kernel reads once, kept out of L1 so that the tap rows, which
// are read again and again, stay there: window gridder at S = 12, 63M
// visibilities, 6076 -> 5959 us; TF32 gridder, 32M, 3335 -> 3252 us; BF16 and
// BF16 hi + lo gridders 0.1% and 0.2%, their degridders 0.5% by the slots alone.  The
// hi + lo gridder's values (loaded where they are used: 2504 -> 2578 us) and the
// degridders' weights (neighbours share a sector: BF16 1597 -> 2026 us) go through
// L1.
__device__ __forceinline__ float2 load_once(const float2 *p)
{
    float2 x;
    asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(x.x), "=f"(x.y)
                 : "l"(p));
    return x;
}
__device__ __forceinline__ float load_once(const float *p)
{
    float x;
    asm volatile("ld.global.L1::no_allocate.f32 %0, [%1];" : "=f"(x) : "l"(p));
    return x;
}
__device__ __forceinline__ Slot load_slot(const Slot *p)
{
    uint4 w;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w)
                 : "l"(p));
    return {(uint64_t)w.y << 32 | w.x, (int32_t)w.z, 0};
}
// The same as two loads, for the tensor-core kernels, whose L1 data path is
// their limit and does not carry the unused word so (8M visibilities in the
// BF16 form: 1094 us with one load, 1062 with two).
__device__ __forceinline__ Slot load_slot_split(const Slot *p)
{
    unsigned long long rec;
    int32_t vis;
    asm volatile("ld.global.L1::no_allocate.u64 %0, [%1];" : "=l"(rec) : "l"(&p->rec));
    asm volatile("ld.global.L1::no_allocate.s32 %0, [%1];" : "=r"(vis) : "l"(&p->vis));
    return {rec, vis, 0};
}
__device__ __forceinline__ void store_slot(Slot *p, uint64_t rec, int32_t vis)
{
    *reinterpret_cast<uint4 *>(p) =
        make_uint4((unsigned)rec, (unsigned)(rec >> 32), (unsigned)vis, 0u);
}

// One work item of the tiled kernels: a chunk of at most kChunk visibilities
// of one tile, stored contiguously in slot order.
struct WorkItem {
    int32_t tile;
    int32_t start;  // first slot
    int32_t count;  // number of slots
    int32_t pad;
};

// Checked build (nvcc -DSEPW_CHECKED=1, libsepw_checked.so): the scatter-
// form kernels check each work item and each plan record against the plan's
// bounds before use; a failed check records SEPW_EBOUNDS in the context's
// status word and the kernel skips the item or visibility.  The default build
// compiles every check to `true`.
#ifndef SEPW_CHECKED
#define SEPW_CHECKED 0
#endif

__device__ __forceinline__ bool check_ok(const DevParams &p, bool ok)
{
#if SEPW_CHECKED
    if (!ok && p.chk_status)
        atomicExch(p.chk_status, SEPW_EBOUNDS);
    return ok;
#else
    (void)p;
    (void)ok;
    return true;
#endif
}

// the item's tile and slot range lie inside the plan
__device__ __forceinline__ bool work_item_ok(const DevParams &p, const WorkItem &it)
{
    return check_ok(p, it.tile >= 0 && it.tile < p.chk_tiles && it.start >= 0 &&
                           it.count >= 0 && (int64_t)it.start + it.count <= p.chk_nvis);
}

// the slot's visibility index, table rows and footprint (inside the tile's
// window and the grid, the tile at grid origin (gy0, gx0)) are in range
__device__ __forceinline__ bool record_ok(const DevParams &p, uint64_t r, int i, int64_t gy0,
                                          int64_t gx0)
{
    return check_ok(p, i >= 0 && i < p.chk_nvis && rec_plane(r) < p.P && rec_ou(r) < p.OS &&
                           rec_ov(r) < p.OS && rec_lx(r) < p.T && rec_ly(r) < p.T &&
                           gx0 + rec_lx(r) + p.S <= p.N && gy0 + rec_ly(r) + p.S <= p.N);
}

// pdl_enter of the persistent kernels
__device__ __forceinline__ void pdl_enter(const DevParams &p)
{
    if (p.early)
        pdl_trigger();
    pdl_wait();
}
constexpr int64_t kEarlyVis = 128 << 10;  // most visibilities of a plan with p.early

constexpr int kChunk = 2048;      // largest work item (visibilities), the default
constexpr int kMaxWindow = 64;    // T + S - 1 <= kMaxWindow

// Binning below the tile: each tile's visibilities are grouped by the block
// of origins (edge 2^sub_log2) that holds their footprint origin before the
// tile is cut into work items.
//   kBinsWindow: edge 4, the window gridder's (its registers cover a block's
//     footprints); T <= 32, so at most 64 bins.
//   kBinsSorted: edge 8 (16 for T > 32) and conj apart, for plans whose items
//     are sorted by origin: an item then spans few bins and its runs of one
//     key are long.  Edge 4 made the scatter of 32M visibilities slower (535
//     against 438 us: its writes go to four times as many places) and the
//     runs no longer; without conj apart the S = 8 gridder took 190 us
//     against 181 us (4M visibilities).
//   kBinsFine: edge 4 (T > 32: as kBinsSorted), conj apart as far as 64 bins
//     go, for grids of few tiles: locate_bin_kernel sends an atomic per warp
//     and bin to the counters, and those of few bins lie in few L2 sectors,
//     where they queue.
//   kBinsTile: one bin, for the 16-bit tensor-core forms, which take any order.
// Which one: plan_bins.
enum PlanBins { kBinsWindow, kBinsSorted, kBinsFine, kBinsTile };
inline void set_bins(DevParams &d, PlanBins b)
{
    if (b == kBinsFine && d.T > 32)
        b = kBinsSorted;
    d.sub_log2 = b == kBinsWindow || b == kBinsFine ? 2
               : b == kBinsTile                     ? 6
               : d.T <= 32                          ? 3
                                                    : 4;
    d.sub_n = (d.T + (1 << d.sub_log2) - 1) >> d.sub_log2;
    d.sub_conj = b == kBinsSorted || (b == kBinsFine && d.sub_n * d.sub_n <= 32) ? 1 : 0;
    d.nsub = (d.sub_n * d.sub_n) << d.sub_conj;
}

// Bins of a plan that the window gridder does not take.
//
// Few tiles: the finer of the two block edges while the coarser one leaves few
// counters, at most 32768 for the tiled form, 12288 for the tensor-core forms
// (T = 26 of S = 6 has the same 32 bins either way, and with edge 4 none for
// conj).  Steps with edge 8 and edge 4, 4M visibilities in random order (d) or
// on tracks (t): tiled, S = 8, T = 32: 256^2 d 663 and 555 us, 1024^2 (32768
// counters) d 626 and 605, t 489 and 461, 2048^2 (131072) d 733 and 740, t 522
// and 525.  BF16: S = 16 256^2 d 693 and 557, S = 12 512^2 (12168) t 500 and
// 478, S = 6 512^2 (12800) d 536 and 532, t 459 and 482, S = 16 1024^2 (32768)
// d 578 and 568, t 469 and 477, S = 6 1024^2 (51200) t 453 and 473.
//
// One bin for the 16-bit tensor-core forms (their order within a tile is worth
// 2% to the kernels) where its counters are many, or the visibilities few
// enough that the scan of the bins counts for more than the queue at the
// counters.  Steps with one bin and edge 8, BF16: 16384 tiles 740 and 746 us
// (random order) and 512 and 516 (tracks), 65536 tiles 1718 and 1764, 579 and
// 618; but 6241 tiles 630 and 596, and 256 tiles 935 and 693 (557 with edge
// 4).  600k on 10404 tiles 306 and 314, 30k on 100 tiles 65 and 69 (tracks);
// 100k on 400 tiles 80 and 73.
//
// Not for FP16 hi + lo, whose error is that of the FP32 sums in tensor memory:
// an MMA adds its 16 visibilities to a cell at once, and in block order fewer MMAs
// reach a cell.  Error with one bin and edge 8, tracks: 30k on 700^2 at S = 8
// 1.4e-6 and 0.87e-6, 122k on 2162^2 at S = 6 8.1e-7 and 5.4e-7, 8M on 4096^2 at
// S = 16 2.3e-6 and 2.1e-6 (step 1648 and 1714 us).  (BF16 hi + lo: 4.5e-6 either
// way, by its operands.)
inline PlanBins plan_bins(const DevParams &p, int form, int64_t nvis, int64_t ntiles)
{
    const bool sorts = form == SEPW_FORM_TILED || form == SEPW_FORM_TC_TF32;
    if (!sorts && form != SEPW_FORM_TC_FP16X2 &&
        (ntiles >= 16384 || nvis < 64 * ntiles || nvis <= 32768))
        return kBinsTile;
    DevParams d = p;
    set_bins(d, kBinsSorted);
    return ntiles * d.nsub <= (form == SEPW_FORM_TILED ? 32768 : 12288) ? kBinsFine : kBinsSorted;
}
constexpr int kMaxSubBins = 64;

// the plan's bins follow a header that is cleared with them: the dropped
// count (8 bytes), then the tile passes' ticket and the mark of a plan whose
// items were sorted after it was made (launch_item_sort)
constexpr size_t kBinHeader = 64, kBinTicket = 8, kBinSortMark = 12;

// Bounds of locate_axis's integer path for grid size N and OS = 2^os_log2
// (os_log2 < 0: path off): |y OS| < 2^elim with 2^elim <= N OS / 2 and
// elim <= 21; margin (N OS) 2^-53 in units of 2^-32, rounded up, and 2 for the
// cut fraction.
inline void locate_fast_bounds(int N, int os_log2, int32_t &elim, int32_t &near)
{
    elim = INT32_MIN;
    near = 0;
    if (os_log2 < 0)
        return;
    const long long half_span = ((long long)N << os_log2) / 2;  // N OS / 2
    int e = 0;
    while (e < 21 && (1ll << (e + 1)) <= half_span)
        ++e;
    elim = e;
    near = (int32_t)((((long long)N << os_log2) >> 21) + 3);
}

// ceil(2^32 / T) for the tile edge T (8 <= T <= 64)
inline uint32_t tile_reciprocal(int T)
{
    return (uint32_t)((0x100000000ull + (uint64_t)T - 1) / (uint64_t)T);
}

// floor(n / T) for 0 <= n < 2^26 as one multiply-high.  With
// M = ceil(2^32 / T) = (2^32 + e) / T, 0 <= e < T, and n = q T + r
// (0 <= r <= T - 1): n M / 2^32 = q + (r + n e / 2^32) / T, whose fraction
// stays below 1 while n e < 2^32, true for n < 2^26 and T <= 64.
__device__ __forceinline__ int div_tile(int n, const DevParams &p)
{
    return (int)__umulhi((unsigned)n, p.t_inv);
}

// column-major: the blocks of one column are consecutive, downwards
__device__ __forceinline__ int sub_bin(int lx, int ly, bool conj, const DevParams &p)
{
    const int b = (lx >> p.sub_log2) * p.sub_n + (ly >> p.sub_log2);
    return p.sub_conj ? b << 1 | (conj ? 1 : 0) : b;
}

// Plan workspace (owned by the context).
struct Plan {
    int64_t nvis = 0;
    int64_t capacity = 0;       // allocated visibility slots
    int32_t ntiles = 0;
    int32_t tiles_capacity = 0;
    size_t bins_capacity = 0;   // bytes at d_bin_base
    int32_t items_capacity = 0;
    int32_t units_capacity = 0;
    int32_t unit = 256;         // most visibilities per unit
    int32_t unit_parts = 1;     // units are at most this part of their tile
    bool valid = false;
    bool sorted = true;         // items known to be sorted by (block, origin, conj)
    int64_t predictions = 0;    // degridding calls since the plan was made
    bool window = false;        // gridding by the window gridder
    int form = 0;
    // tiled forms
    int32_t *d_tile = nullptr;      // [nvis] bin id per visibility (-1 dropped)
    int32_t *d_rank = nullptr;      // [nvis] rank of the visibility inside its bin
                                    // (plan_splits: then visibility index, slot order)
    unsigned char *d_bin_base = nullptr;  // header, then [ntiles * nsub] counts, then slots
    uint64_t *d_rec0 = nullptr;     // [nvis] record, input order (plan_splits: then
                                    // in slot order)
    Slot *d_slots = nullptr;        // [nvis] records and visibility indices, slot order
    int32_t *d_tile_count = nullptr;   // [ntiles]
    void *d_blocks = nullptr;          // totals of the tile passes' blocks
    WorkItem *d_items = nullptr;       // [items_capacity]
    WorkItem *d_units = nullptr;       // [units_capacity], tiled form only
    int32_t *d_nitems = nullptr;       // [2]: items, units
    int32_t *d_nunits = nullptr;       // d_nitems + 1
    int32_t *d_item_counter = nullptr; // [2] persistent-kernel work counters
    unsigned long long *d_dropped = nullptr;  // in d_bin_base's header
    int64_t *dropped_out = nullptr;           // where the next gridding or degridding
                                              // call copies it, if anywhere
    int32_t *d_drop_list = nullptr;           // [nvis] indices of dropped visibilities
    int32_t ngrids = 1;                // batched plans: grids in the batch
    int64_t *d_offsets = nullptr;      // [ngrids + 1] visibility offsets per grid
    int32_t offsets_capacity = 0;
    std::vector<int64_t> h_offsets;    // plain form: per-grid ranges
    // plain form: the coordinates are read directly
    const double *u = nullptr, *v = nullptr, *w = nullptr;
};

// TF32 plans: the sort leaves the records and visibility indices of the slots in
// d_rec0 and d_rank as well, which the passes before it are done with.  The
// TF32 gridder is bound by L1 and lost 2 to 6% by slots of 16 bytes (16M
// visibilities on 1024^2: 1599 us with them, 1514 so; 32M on 4096^2 3249 and
// 3113); writing the arrays costs the sort 3 to 6% of the plan.
inline bool plan_splits(const Plan &plan) { return plan.form == SEPW_FORM_TC_TF32; }

// Device-side parameters of a checked sepw_params (sepw_api.cu): derived
// constants, and the tile edge resolved for the form when p->tile is 0.
DevParams make_dev_params(const sepw_params *p);

// ---- launchers (each .cu file implements its own) -------------------------

// sepw_taps.cu
cudaError_t launch_taper(const DevParams &p, double *taper64, float *taper32,
                         cudaStream_t s);
cudaError_t launch_twiddles(const DevParams &p, double2 *tw, cudaStream_t s);
cudaError_t launch_taps(const DevParams &p, const double *taper64, const double2 *tw,
                        double2 *out64, float2 *out32, cudaStream_t s);

// sepw_plain.cu
cudaError_t launch_count_dropped(const DevParams &p, int64_t nvis, const double *u,
                                 const double *v, const double *w,
                                 unsigned long long *dropped, cudaStream_t s);
cudaError_t launch_locate(const DevParams &p, int64_t nvis, const double *u,
                          const double *v, const double *w, int32_t *cu, int32_t *cv,
                          int32_t *ou, int32_t *ov, int32_t *plane, uint8_t *conj,
                          uint8_t *keep, cudaStream_t s);
cudaError_t launch_grid_plain(const DevParams &p, int64_t nvis, const double *u,
                              const double *v, const double *w, const float2 *vis,
                              const float *weight, const float2 *taps, float2 *grid,
                              unsigned long long *dropped, cudaStream_t s);
cudaError_t launch_degrid_plain(const DevParams &p, int64_t nvis, const double *u,
                                const double *v, const double *w, const float2 *grid,
                                const float *weight, const float2 *taps, float2 *vis,
                                unsigned long long *dropped, cudaStream_t s);

// sepw_bin.cu
// sizes of Plan::d_bin_base and Plan::d_blocks, and the units
size_t plan_bin_bytes(int64_t ntiles, const DevParams &p);
size_t plan_block_bytes(int64_t ntiles);
void set_units(const DevParams &p, int num_sms, Plan &plan);  // from nvis, ntiles, window
int64_t max_units(const Plan &plan);
bool plan_window(const DevParams &p, size_t table_bytes, int64_t nvis, int ngrids);
cudaError_t launch_plan(const DevParams &p, int64_t nvis, const double *u,
                        const double *v, const double *w, Plan &plan, int num_sms,
                        cudaStream_t s);
// sorts every item by (block, origin, conj); marked: unless an earlier such
// launch on the same plan has done it
cudaError_t launch_item_sort(const DevParams &p, const Plan &plan, int num_sms, bool marked,
                             cudaStream_t s);
// batched: plan.ngrids > 1 and plan.d_offsets hold the per-grid ranges
cudaError_t launch_zero_dropped(const Plan &plan, float2 *vis, cudaStream_t s);

// sepw_tiled.cu
// planar: workspace of 2 x (taps of both tables) floats for the lane-ordered
// planar copy of the tap table that the block gridder (S = 8, 16) builds and
// reads its v-taps from; null: the interleaved table is read directly
cudaError_t launch_grid_tiled(const DevParams &p, const Plan &plan, const float2 *vis,
                              const float *weight, const float2 *taps, float *planar,
                              float2 *grid, int num_sms, cudaStream_t s);
cudaError_t launch_degrid_tiled(const DevParams &p, const Plan &plan,
                                const float2 *grid, const float *weight,
                                const float2 *taps, float *tables, float2 *vis, int num_sms,
                                cudaStream_t s);

// sepw_window.cu: gridder of the tiled form for the supports the block gridder
// does not take (plan.window).  tables: window_tables_bytes(p) bytes for the
// per-call tap tables, 0 if it does not take these parameters.
size_t window_tables_bytes(const DevParams &p);
cudaError_t launch_grid_window(const DevParams &p, const Plan &plan, const float2 *vis,
                               const float *weight, const float2 *taps, float *tables,
                               float2 *grid, int num_sms, cudaStream_t s);

// degridder of the same plans for some supports (degrid_window_takes)
bool degrid_window_takes(const DevParams &p, const Plan &plan);
cudaError_t launch_degrid_window(const DevParams &p, const Plan &plan, const float2 *grid,
                                 const float *weight, const float2 *taps, float *tables,
                                 float2 *vis, int num_sms, cudaStream_t s);

// Control of the tensor-core kernels: the limit of every bounded mbarrier
// wait, and a test hook (stall != 0: the MMA thread issues and commits
// nothing, so the other roles' waits run out and the kernel reports
// SEPW_ETIMEOUT).
struct TcControl {
    unsigned long long wait_ns;
    int32_t stall;
};

// sepw_tc.cu: contraction-form degridder, prec 0 = BF16, 1 = FP16 (scaled
// per item), 2 = FP16 hi + lo (scaled), 3 = BF16 hi + lo; T + S - 1 <= 32,
// S <= 16.  tables: tc_degrid_tables_bytes(p,
// plan.items_capacity) bytes of device workspace for the per-call tap tables
// (the FP16 forms' per-item window scale is found in the kernel; the item
// count does not enter the size).
size_t tc_degrid_tables_bytes(const DevParams &p, int64_t items_capacity);
cudaError_t launch_degrid_tc(const DevParams &p, const Plan &plan, const float2 *grid,
                             const float *weight, const float2 *taps, void *tables, float2 *vis,
                             int num_sms, int prec, int32_t *status, TcControl ctl,
                             cudaStream_t s);

// sepw_tc_grid.cu: contraction-form gridder, T + S - 1 <= 32, S <= 16.
// prec: 0 = BF16, 1 = FP16 (scaled per item), 2 = FP16 hi + lo (scaled),
// 3 = BF16 hi + lo.  tables: tc2_tables_bytes(p, plan.items_capacity) bytes of
// device workspace for the per-call pre-shifted tap tables and the per-item
// scale exponents.
int tc2_tile_for_support(int S);
size_t tc2_tables_bytes(const DevParams &p, int64_t items_capacity);
cudaError_t launch_grid_tc2(const DevParams &p, const Plan &plan, const float2 *vis,
                            const float *weight, const float2 *taps, void *tables, float2 *grid,
                            int num_sms, int prec, int32_t *status, TcControl ctl,
                            cudaStream_t s);

// sepw_wstack.cu
cudaError_t launch_wstack_assign(int64_t nvis, const double *w, const double *c, int L,
                                 int32_t *slice, int32_t *count, cudaStream_t s);
cudaError_t launch_wstack_scatter(int64_t nvis, const double *u, const double *v,
                                  const double *w, const double *c, int L, const int32_t *slice,
                                  int32_t *cursor, int32_t *part, double *up, double *vp,
                                  double *wp, cudaStream_t s);
cudaError_t launch_wstack_compose(int64_t nvis, const Plan &plan, const int32_t *part,
                                  cudaStream_t s);
cudaError_t launch_wstack_sign(const DevParams &p, int L, float2 *g, cudaStream_t s);
cudaError_t launch_wstack_combine(const DevParams &p, int L, const float *taper,
                                  const float *wc, const float2 *g, float2 *image,
                                  cudaStream_t s);
cudaError_t launch_wstack_split(const DevParams &p, int L, const float *taper, const float *wc,
                                const float2 *image, float2 *g, cudaStream_t s);

// sepw_facet.cu (direction 0: into the facet, 1: back out)
cudaError_t launch_facet_shift(int64_t nvis, double l0, double m0, int direction,
                               const double *u, const double *v, const double *w,
                               const float2 *vin, double *uo, double *vo, float2 *vout,
                               cudaStream_t s);

// sepw_residual.cu (stored correction F_w - F~_w); work: residual_work_bytes
// bytes of device memory
size_t residual_work_bytes(const DevParams &p, int Sr, int OSr);
cudaError_t launch_residual_table(const DevParams &p, int Sr, int OSr, const double *taper64,
                                  const double2 *tw, const double2 *taps64, void *work,
                                  double2 *out64, float2 *out32, cudaStream_t s);
cudaError_t launch_grid_residual(const DevParams &p, int Sr, int OSr, const Plan &plan,
                                 const float2 *vis, const float *weight, const float2 *res,
                                 float2 *grid, int num_sms, cudaStream_t s);
cudaError_t launch_degrid_residual(const DevParams &p, int Sr, int OSr, const Plan &plan,
                                   const float2 *grid, const float *weight, const float2 *res,
                                   float2 *vis_out, int num_sms, cudaStream_t s);

// sepw_fft.cu: transforms of N x N grids for the N of rows_supported: columns
// in place on the grid side, before (to image) or after (to grid) the rows,
// which have the image side's passes folded in.  tab: rows_table_bytes(N) bytes
// filled by launch_rows_tables.  mode 1: n / (c c), 2: 1 / (n c c).  The column
// transforms and launch_slices_to_image want g 16-byte aligned.
bool rows_supported(int N);
size_t rows_table_bytes(int N);
cudaError_t launch_rows_tables(const DevParams &p, const double2 *tw, float2 *tab, cudaStream_t s);
cudaError_t launch_columns(const DevParams &p, bool inverse, int grids, const float2 *tab,
                           float2 *g, int num_sms, cudaStream_t s);
cudaError_t launch_rows_to_image(const DevParams &p, int mode, const float *taper,
                                 const float2 *tab, float2 *buf, cudaStream_t s);
cudaError_t launch_slices_to_image(const DevParams &p, int L, const float *taper, const float *wc,
                                   const float2 *tab, const float2 *g, float2 *image,
                                   cudaStream_t s);
cudaError_t launch_image_to_slices(const DevParams &p, int L, const float *taper, const float *wc,
                                   const float2 *tab, const float2 *image, float2 *g,
                                   cudaStream_t s);

// sepw_image.cu (other N, and towards the grid: around a 2-D transform)
cudaError_t launch_image_pre(const DevParams &p, int direction, const float *taper,
                             float2 *buf, cudaStream_t s);
cudaError_t launch_image_post(const DevParams &p, int direction, const float *taper,
                              float2 *buf, cudaStream_t s);

}  // namespace sepw
