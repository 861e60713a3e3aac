// Plan construction for the tiled forms: locate every visibility, bin it by
// the T x T tile that holds its footprint origin and, inside the tile, by the
// block of origins (set_bins; counting sort with warp-aggregated atomics), cut
// each tile into work items of at most kChunk visibilities (and into the smaller
// units of the tiled gridders), and, for the kernels that walk runs of one
// origin, sort each item by (footprint origin, conj).
//
// The update structure this serves is Sec. 5: every visibility adds a
// separable S x S block at its own offset; visibilities that share a tile
// share one shared-memory window, and visibilities that share an origin share
// one register block.
#include <algorithm>
#include <limits>

#include "sepw_internal.cuh"

namespace sepw {

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Pass 1: locate, record, bin histogram with each visibility's rank inside
// its bin (the order of arrival at the bin's counter), dropped count.
__global__ void __launch_bounds__(256) locate_bin_kernel(
    DevParams p, int64_t nvis, const double *u, const double *v,
    const double *w, int32_t *__restrict__ bin_of,
    int32_t *__restrict__ rank_of, uint64_t *__restrict__ rec0, int32_t *bin_count,
    unsigned long long *dropped, int32_t *__restrict__ drop_list, int ngrids,
    const int64_t *offsets)
{
    pdl_enter();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool active = i < nvis;
    int bin = -1;
    if (active) {
        Loc L = locate(u[i], v[i], w[i], p);
        if (L.keep) {
            int fx = L.cu - p.S / 2 + 1, fy = L.cv - p.S / 2 + 1;
            const int tx = div_tile(fx, p), ty = div_tile(fy, p);
            int g = 0;
            if (ngrids > 1) {  // grid of visibility i: offsets[g] <= i < offsets[g+1]
                int lo = 0, hi = ngrids - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (offsets[mid] <= i)
                        lo = mid;
                    else
                        hi = mid - 1;
                }
                g = lo;
            }
            const int lx = fx - tx * p.T, ly = fy - ty * p.T;
            bin = ((g * p.ntx + ty) * p.ntx + tx) * p.nsub + sub_bin(lx, ly, L.conj, p);
            rec0[i] = pack_rec(lx, ly, L.ou, L.ov, L.plane, L.conj);
        }
        bin_of[i] = bin;
    }
    unsigned act = __ballot_sync(0xffffffffu, active && bin >= 0);
    unsigned drop = __ballot_sync(0xffffffffu, active && bin < 0);
    int lane = threadIdx.x & 31;
    if (drop) {
        // append the dropped indices (degridding writes 0 there)
        int leader = __ffs(drop) - 1;
        unsigned long long base = 0;
        if (lane == leader)
            base = atomicAdd(dropped, (unsigned long long)__popc(drop));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (active && bin < 0)
            drop_list[base + __popc(drop & lanemask_lt())] = (int32_t)i;
    }
    if (active && bin >= 0) {
        const unsigned peers = __match_any_sync(act, bin);
        const int leader = __ffs(peers) - 1;
        int base = 0;
        if (lane == leader)
            base = atomicAdd(bin_count + bin, __popc(peers));
        base = __shfl_sync(act, base, leader);
        rank_of[i] = base + __popc(peers & lanemask_lt());
    }
}

// Passes 1b and 2: tile totals, then exclusive scans of the visibilities and
// of the items and units over all tiles.  Full pieces (`chunk` or `unit`
// visibilities) are listed before the partial ones, so that dynamically
// scheduled workers take the heavy ones first; within each list the pieces
// are in tile order.
//
// Pass 1b sums every tile's bins (a warp per tile) and every block's totals;
// the last block to finish scans the totals of all blocks, so pass 2 starts
// from its block's prefix with no launch in between.  The scan ran in a
// single block before and took 426 us for the 524,288 tiles of a 128-grid
// batch (now 20 us for its share of pass 2).
struct Totals {
    int32_t n, full_items, part_items, full_units, part_units;
};
__device__ __forceinline__ Totals operator+(const Totals &a, const Totals &b)
{
    return {a.n + b.n, a.full_items + b.full_items, a.part_items + b.part_items,
            a.full_units + b.full_units, a.part_units + b.part_units};
}
__device__ __forceinline__ Totals operator-(const Totals &a, const Totals &b)
{
    return {a.n - b.n, a.full_items - b.full_items, a.part_items - b.part_items,
            a.full_units - b.full_units, a.part_units - b.part_units};
}
// How tiles are cut: items of `chunk`; units of a `parts`-th of the tile, at
// most `unit` and a multiple of 32 (all of them `unit` when parts is 1).
//
// A cell's sum takes two steps, within a unit and over the units, and is the less
// exact the longer either of them is.  Units of a tile of kHeavyTile or more are
// no shorter than the root of its number, up to kLongUnit; windows from `dense`
// visibilities a tile on are no longer than kDenseUnit.  Error of grids on tracks
// with residuals that do not average out, units of 32, this rule, eighths of
// items, and the gridder's time with the first two: 35k visibilities on 240^2 at
// S = 6 1.8e-7, 1.3e-7, 1.4e-7 (15 and 32 us); 100k on 500^2 at S = 8 2.0e-7,
// 1.8e-7, 1.8e-7 (15 and 27); 300k on 300^2 at S = 8 3.4e-7, 2.4e-7, 2.7e-7 (19
// and 29).  Windows of 2048 at S = 6: 35k 5.7e-7, 1.5e-7 cut to 256; 300k on 700^2
// 5.3e-7 and 1.3e-7.  Lighter tiles are as exact with units of 32 (20k on 400^2 at
// S = 8 1.74e-7, 1.60e-7 with 64, 1.76e-7 with eighths), and faster (15 and 29 us).
constexpr int kHeavyTile = 4096, kLongUnit = 128, kDenseUnit = 256;
struct Cut {
    int32_t chunk, unit, parts, dense;
    __device__ __forceinline__ int unit_of(int n) const
    {
        const int u = parts > 1 ? max(32, min(unit, (n / parts + 31) & ~31)) : unit;
        if (n < min(dense, kHeavyTile))
            return u;
        const int root = n < kHeavyTile ? 0 : ((int)__fsqrt_rn((float)n) + 31) & ~31;
        return max(n >= dense ? min(u, kDenseUnit) : u, min(root, kLongUnit));
    }
};
__device__ __forceinline__ Totals tile_totals(int n, const Cut &cut)
{
    const int u = cut.unit_of(n), fi = n / cut.chunk, fu = n / u;
    return {n, fi, n != fi * cut.chunk, fu, n != fu * u};
}
__device__ __forceinline__ Totals shfl_up(const Totals &v, int d)
{
    return {__shfl_up_sync(0xffffffffu, v.n, d), __shfl_up_sync(0xffffffffu, v.full_items, d),
            __shfl_up_sync(0xffffffffu, v.part_items, d),
            __shfl_up_sync(0xffffffffu, v.full_units, d),
            __shfl_up_sync(0xffffffffu, v.part_units, d)};
}
__device__ __forceinline__ Totals warp_scan(Totals v, int lane)  // inclusive
{
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const Totals y = shfl_up(v, off);
        if (lane >= off)
            v = v + y;
    }
    return v;
}
// Inclusive scan over the block's threads; `total` gets the block's sum.
// warps: one entry per warp and one more (shared).
__device__ __forceinline__ Totals block_scan(Totals v, Totals *warps, Totals &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_scan(v, lane);
    __syncthreads();
    if (lane == 31)
        warps[warp] = v;
    __syncthreads();
    if (warp == 0) {
        const Totals w = lane < nw ? warps[lane] : Totals{0, 0, 0, 0, 0};
        const Totals x = warp_scan(w, lane);
        if (lane < nw)
            warps[lane] = x - w;
        if (lane == 31)
            warps[32] = x;
    }
    __syncthreads();
    total = warps[32];
    return v + warps[warp];
}

// Tiles a block of passes 1b and 2 takes: 32 (one per warp; 256 where a thread
// takes a tile) as long as that leaves at most 1024 blocks to scan, then more.
static int plan_block(int64_t ntiles, int nsub)
{
    int tb = nsub <= 4 ? 256 : 32;
    while (tb < 1024 && ntiles > 1024ll * tb)
        tb *= 2;
    return tb;
}
constexpr int kPlanThreads = 1024, kPlanWarps = kPlanThreads / 32;
constexpr int kOneBlockTiles = 256;  // up to here one block makes both passes

// s_n[k] = visibilities of tile t0 + k, k < tb
__device__ __forceinline__ void count_tiles(int t0, int tb, int ntiles, int nsub,
                                            const int32_t *bin, int32_t *s_n)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (nsub <= 4) {  // a thread per tile
        if ((int)threadIdx.x < tb) {
            int c = 0;
            if (t0 + (int)threadIdx.x < ntiles)
                for (int q = 0; q < nsub; ++q)
                    c += bin[(int64_t)(t0 + threadIdx.x) * nsub + q];
            s_n[threadIdx.x] = c;
        }
        return;
    }
#pragma unroll 2
    for (int k = warp; k < tb; k += kPlanWarps) {  // a warp per tile
        int c = 0;
        if (t0 + k < ntiles) {
            const int32_t *b = bin + (int64_t)(t0 + k) * nsub;
            if (lane < nsub)
                c = b[lane];
            if (lane + 32 < nsub)
                c += b[lane + 32];
        }
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0)
            s_n[k] = c;
    }
}

__global__ void __launch_bounds__(kPlanThreads) tile_count_kernel(
    int32_t ntiles, int32_t tb, int32_t nsub, Cut cut,
    const int32_t *bin, int32_t *__restrict__ tile_count,
    Totals *__restrict__ blocks, unsigned *ticket)
{
    __shared__ Totals s_warps[33];
    __shared__ int32_t s_n[1024];
    __shared__ bool s_last;
    pdl_enter();
    const int t0 = blockIdx.x * tb;
    count_tiles(t0, tb, ntiles, nsub, bin, s_n);
    __syncthreads();
    const int n = (int)threadIdx.x < tb ? s_n[threadIdx.x] : 0;
    if ((int)threadIdx.x < tb && t0 + (int)threadIdx.x < ntiles)
        tile_count[t0 + threadIdx.x] = n;
    Totals total;
    block_scan(tile_totals(n, cut), s_warps, total);
    if (threadIdx.x == 0) {
        blocks[blockIdx.x] = total;
        __threadfence();
        s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last)
        return;
    // exclusive prefixes of the blocks' totals, the sum of all at the end
    __threadfence();
    const int nb = gridDim.x;
    Totals run{0, 0, 0, 0, 0};
    for (int b0 = 0; b0 < nb; b0 += kPlanThreads) {
        const int b = b0 + threadIdx.x;
        Totals v{0, 0, 0, 0, 0};
        if (b < nb) {
            const volatile Totals *w = blocks + b;  // written by other blocks
            v = {w->n, w->full_items, w->part_items, w->full_units, w->part_units};
        }
        Totals sum;
        const Totals x = block_scan(v, s_warps, sum);
        if (b < nb)
            blocks[b] = run + x - v;
        run = run + sum;
    }
    if (threadIdx.x == 0)
        blocks[nb] = run;
}

// Lists the full pieces of the block's tb tiles (tile tile0 + k: those from
// piece pre[k] on, of size_of(k), the first at slot first[k]; total pieces),
// consecutive threads writing consecutive pieces.
template <typename F>
__device__ __forceinline__ void list_full(WorkItem *__restrict__ out, int tile0, int tb,
                                          int total, F size_of, const int32_t *pre,
                                          const int32_t *first)
{
    for (int e = threadIdx.x; e < total; e += kPlanThreads) {
        int k = 0;  // the last tile with pre[k] <= e
        for (int h = tb >> 1; h > 0; h >>= 1)
            if (pre[k + h] <= e)
                k += h;
        const int size = size_of(k);
        out[e] = {tile0 + k, first[k] + (e - pre[k]) * size, size, 0};
    }
}

// Pass 2: every bin's count replaced by its first slot; items and units.  ONE:
// the only block, which counts its tiles itself (no pass 1b).
template <bool ONE>
__global__ void __launch_bounds__(kPlanThreads) tile_items_kernel(
    int32_t ntiles, int32_t tb, int32_t nsub, Cut cut,
    const int32_t *tile_count, const Totals *blocks,
    int32_t *__restrict__ bin, WorkItem *__restrict__ items, int32_t *nitems,
    WorkItem *__restrict__ units, int32_t *nunits)
{
    __shared__ Totals s_warps[33];
    __shared__ int32_t s_n[1024], s_at[1024], s_items[1024], s_units[1024];
    pdl_enter();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t0 = blockIdx.x * tb, t = t0 + threadIdx.x;
    int n = 0;
    if constexpr (ONE) {
        count_tiles(0, tb, ntiles, nsub, bin, s_n);
        __syncthreads();
        n = (int)threadIdx.x < tb ? s_n[threadIdx.x] : 0;
    } else if ((int)threadIdx.x < tb && t < ntiles) {
        n = tile_count[t];
    }
    const Totals mine = tile_totals(n, cut);
    const int chunk = cut.chunk, unit = cut.unit_of(n);
    Totals sum;
    const Totals in = block_scan(mine, s_warps, sum) - mine;
    Totals before{0, 0, 0, 0, 0}, all = sum;  // exclusive prefix of the block, all blocks
    if constexpr (!ONE) {
        before = blocks[blockIdx.x];
        all = blocks[gridDim.x];
    }
    const Totals at = before + in;
    if (t == 0) {
        *nitems = all.full_items + all.part_items;
        if (units)
            *nunits = all.full_units + all.part_units;
    }
    if ((int)threadIdx.x < tb) {
        s_n[threadIdx.x] = n;
        s_at[threadIdx.x] = at.n;
        s_items[threadIdx.x] = in.full_items;
        s_units[threadIdx.x] = in.full_units;
        if (mine.part_items)
            items[all.full_items + at.part_items] = {t, at.n + mine.full_items * chunk,
                                                     n - mine.full_items * chunk, 0};
        if (units && mine.part_units)
            units[all.full_units + at.part_units] = {t, at.n + mine.full_units * unit,
                                                     n - mine.full_units * unit, 0};
    }
    __syncthreads();
    list_full(items + before.full_items, t0, tb, sum.full_items, [&](int) { return chunk; },
              s_items, s_at);
    if (units)
        list_full(units + before.full_units, t0, tb, sum.full_units,
                  [&](int k) { return cut.unit_of(s_n[k]); }, s_units, s_at);
    if (nsub <= 4) {  // a thread per tile
        if ((int)threadIdx.x < tb && n > 0) {
            int32_t *b = bin + (int64_t)t * nsub;
            for (int q = 0, run = at.n; q < nsub; ++q) {
                const int c = b[q];
                b[q] = run;
                run += c;
            }
        }
        return;
    }
#pragma unroll 2
    for (int k = warp; k < tb; k += kPlanWarps) {
        if (s_n[k] == 0)
            continue;  // nobody looks up the slots of an empty tile
        int32_t *b = bin + (int64_t)(t0 + k) * nsub;
        const int c0 = lane < nsub ? b[lane] : 0, c1 = lane + 32 < nsub ? b[lane + 32] : 0;
        int i0 = c0, i1 = c1;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y0 = __shfl_up_sync(0xffffffffu, i0, off);
            const int y1 = __shfl_up_sync(0xffffffffu, i1, off);
            if (lane >= off) {
                i0 += y0;
                i1 += y1;
            }
        }
        const int at0 = s_at[k], at1 = at0 + __shfl_sync(0xffffffffu, i0, 31);
        if (lane < nsub)
            b[lane] = at0 + i0 - c0;
        if (lane + 32 < nsub)
            b[lane + 32] = at1 + i1 - c1;
    }
}
static_assert(kMaxSubBins == 64, "two bins per lane");

// Pass 3: scatter records and visibility ids to their slots: first slot of the
// bin + rank inside the bin.  A slot is one 16-byte store: as an 8- and a
// 4-byte array the pass was bound by twice the partial sectors it sends to L2
// (32M visibilities 424 us; 331 us so).
__global__ void __launch_bounds__(256) scatter_kernel(
    int64_t nvis, const int32_t *bin_of, const int32_t *rank_of,
    const uint64_t *rec0, const int32_t *bin_first,
    Slot *__restrict__ slots)
{
    pdl_enter();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nvis)
        return;
    const int b = bin_of[i];
    if (b < 0)
        return;
    const int slot = bin_first[b] + rank_of[i];
    store_slot(slots + slot, rec0[i], (int32_t)i);
}

// Pass 4: inside each work item, counting sort by (footprint origin, conj),
// bin major: the key orders by the bin of pass 1 (block of origins and conj),
// then by the origin's row and column inside the block.  Visibilities that
// share a key share one register block in the tiled kernels, and the block
// never mixes conjugated and plain kernels; the bins stay contiguous inside an
// item, so a run of slots that starts and ends in one bin lies inside it.  One
// block of threads per item; the item's slots are rewritten in place.  The
// order among equal keys is arbitrary.  recs and ids (or null): the sorted records
// and visibility indices as two arrays, too (plan_splits).
constexpr int kSortThreads = 512;
constexpr int kMaxSortBins = 2 * 64 * 64;
constexpr int kMaxBinsPerThread = kMaxSortBins / kSortThreads;

__device__ __forceinline__ int sort_key(uint64_t r, const DevParams &p)
{
    const int lx = rec_lx(r), ly = rec_ly(r), lg = p.sub_log2, m = (1 << lg) - 1;
    const int k = (sub_bin(lx, ly, rec_conj(r), p) << lg | (ly & m)) << lg | (lx & m);
    return p.sub_conj ? k : k << 1 | (rec_conj(r) ? 1 : 0);
}
// keys of a tile: at most 2 x 64 x 64
static int sort_keys(const DevParams &p)
{
    return p.nsub << (2 * p.sub_log2 + (p.sub_conj ? 0 : 1));
}

__global__ void __launch_bounds__(kSortThreads) item_sort_kernel(
    DevParams p, const WorkItem *items, const int32_t *nitems, const int32_t *mark,
    Slot *__restrict__ slots, uint64_t *__restrict__ recs, int32_t *__restrict__ ids)
{
    extern __shared__ int32_t hist[];  // per * kSortThreads bins
    __shared__ uint64_t s_rec[kChunk];
    __shared__ int32_t s_perm[kChunk];
    __shared__ int32_t s_wsum[32];
    pdl_enter(p);
    if (mark && *mark)
        return;
    // blocks stride over the plan's items (sparse plans have far fewer items
    // than their capacity, so the grid is sized by the SM count, not by it)
    const int n_items = *nitems;
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
    const WorkItem it = items[item];
    const int n = it.count;
    const int nb = p.nsub << (2 * p.sub_log2 + (p.sub_conj ? 0 : 1));
    const int per = (nb + kSortThreads - 1) / kSortThreads;
    for (int b = threadIdx.x; b < per * kSortThreads; b += kSortThreads)
        hist[b] = 0;
    __syncthreads();
    // a warp's lanes hold consecutive slots, where runs of one key are
    // common: one shared-memory atomic per distinct key per warp
    const int lane_id = threadIdx.x & 31;
    for (int q0 = 0; q0 < n; q0 += kSortThreads) {
        const int q = q0 + (int)threadIdx.x;
        const bool act = q < n;
        int key = -1;
        if (act) {
            const uint4 w = *reinterpret_cast<const uint4 *>(slots + it.start + q);
            const uint64_t r = (uint64_t)w.y << 32 | w.x;
            s_rec[q] = r;
            s_perm[q] = (int32_t)w.z;
            key = sort_key(r, p);
        }
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        if (act && lane_id == __ffs(peers) - 1)
            atomicAdd(hist + key, __popc(peers));
    }
    __syncthreads();
    // exclusive scan: thread t owns bins [t*per, t*per + per)
    const int t = threadIdx.x;
    int local[kMaxBinsPerThread];
    int sum = 0;
#pragma unroll
    for (int q = 0; q < kMaxBinsPerThread; ++q) {
        local[q] = q < per ? hist[t * per + q] : 0;
        sum += local[q];
    }
    const int lane = t & 31, warp = t >> 5;
    int incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off)
            incl += y;
    }
    if (lane == 31)
        s_wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int nw = kSortThreads / 32;
        const int x = lane < nw ? s_wsum[lane] : 0;
        int y = x;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int z = __shfl_up_sync(0xffffffffu, y, off);
            if (lane >= off)
                y += z;
        }
        if (lane < nw)
            s_wsum[lane] = y - x;  // exclusive warp offsets
    }
    __syncthreads();
    int run = s_wsum[warp] + incl - sum;
#pragma unroll
    for (int q = 0; q < kMaxBinsPerThread; ++q) {
        if (q < per)
            hist[t * per + q] = run;
        run += local[q];
    }
    __syncthreads();
    for (int q0 = 0; q0 < n; q0 += kSortThreads) {
        const int q = q0 + (int)threadIdx.x;
        const bool act = q < n;
        uint64_t r = 0;
        int key = -1;
        if (act) {
            r = s_rec[q];
            key = sort_key(r, p);
        }
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        const int leader = __ffs(peers) - 1;
        int base = 0;
        if (act && lane_id == leader)
            base = atomicAdd(hist + key, __popc(peers));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (act) {
            const int dst = base + __popc(peers & lanemask_lt());
            store_slot(slots + it.start + dst, r, s_perm[q]);
            if (recs) {
                recs[it.start + dst] = r;
                ids[it.start + dst] = s_perm[q];
            }
        }
    }
    __syncthreads();  // shared memory is reused by the next item
    }
}

// Degridding writes 0 for every dropped visibility of the plan.  Also clears
// the degridder's work counter.
__global__ void zero_dropped_kernel(const int32_t *drop_list,
                                    const unsigned long long *ndrop,
                                    float2 *__restrict__ vis, int32_t *counter, int64_t *dropped)
{
    pdl_enter();
    const unsigned long long n = *ndrop;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *counter = 0;
        if (dropped)
            *dropped = (int64_t)n;
    }
    for (unsigned long long k = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
         k < n; k += (unsigned long long)gridDim.x * blockDim.x)
        vis[drop_list[k]] = make_float2(0.f, 0.f);
}

cudaError_t launch_zero_dropped(const Plan &plan, float2 *vis, cudaStream_t s)
{
    return launch_pdl(zero_dropped_kernel, 64, 256, 0, s, plan.d_drop_list, plan.d_dropped, vis,
                      plan.d_item_counter + 1, plan.dropped_out);
}

// The units of the tiled gridders: 32 to 256 (1024) visibilities, about two for each
// of the ~40 warps an SM holds; for the block gridders also an eighth of their
// tile, as long as that does not make more units than those warps can use
// (sparse tiles then weigh as little as dense ones at the end of the launch,
// and dense ones keep their runs).  Whole items of 2048 gave 524,288
// visibilities to 400 warps (S = 16, 758 us; 155 us so).  Above 256 the last
// warps work alone on 32M visibilities (2.13 ms for 256, 2.16 for 512, 2.24
// for 1024, 2.38 for 2048).  The window gridder adds whole windows at the ends
// of a unit: up to 1024 below one visibility per cell (63M visibilities over
// 128 grids of 2048^2 at S = 12: 5.96 ms for 256, 5.70 for 512, 5.58 for 1024
// and 2048; 20M over 40: 1.95 -> 1.82 ms), where no tile holds a large part of
// them; in dense data longer units only leave the end to few warps (32M on
// 4096^2: 2.14 ms for 256, 2.18 for 1024).
void set_units(const DevParams &p, int num_sms, Plan &plan)
{
    plan.unit_parts = 1;
    if (p.grid_parts > 0) {
        plan.unit = std::max(32, ((p.chunk + p.grid_parts - 1) / p.grid_parts + 31) & ~31);
        return;
    }
    const int64_t per = plan.window ? 320 : 80;
    const int64_t u = (plan.nvis / std::max<int64_t>(1, per * num_sms) + 31) & ~31ll;
    const bool sparse = plan.window && plan.nvis < (int64_t)plan.ntiles * p.T * p.T;
    plan.unit = (int32_t)std::min<int64_t>(sparse ? 1024 : 256, std::max<int64_t>(32, u));
    if (!plan.window)
        plan.unit_parts = (int32_t)std::min<int64_t>(
            8, std::max<int64_t>(1, 640ll * num_sms / std::max(1, plan.ntiles)));
}

// units of any plan that set_units cuts: a full one takes unit (kDenseUnit, where
// that is less) visibilities or more than a ninth of its tile
int64_t max_units(const Plan &plan)
{
    const int unit = std::min(plan.unit, kDenseUnit);
    const int64_t cut = plan.nvis / (plan.unit_parts > 1 ? 32 : unit);
    return std::min(cut, plan.nvis / unit + (int64_t)plan.unit_parts * plan.ntiles) +
           plan.ntiles + 1;
}

// Whether a plan of the tiled form is for the window gridder (table_bytes: what
// its tap tables take, 0 if it does not take the parameters, S = 8 among them):
// every support without a block gridder, and S = 16 below a visibility per four
// cells, where runs of one origin are short (524,288 visibilities on 2048^2:
// 155 us with the block gridder, 86 us with the window gridder; 4M: 355 and 468
// us).  At S = 8 the block gridder is the faster one (1M on 1024^2: 62 and 74
// us; 8M on 15 x 4096^2: 475 and 556 us).
//
// The tables are built in every call, about 2.3 us a MB, so calls of few
// visibilities with large tables are left to the column gridder.  Steps on
// 1000^2, random order (d) and tracks (t), window and column: 3k visibilities,
// 14 MB (S = 30) d 145 and 98 us, t 189 and 532, 24 MB (S = 12) d 75 and 57, t
// 79 and 136, 70 MB (S = 20) d 345 and 70, t 390 and 323; 20k, 24 MB (S = 12) d
// 95 and 70, t 86 and 599, 48 MB d 133 and 69, t 121 and 601; 100k, 48 MB d 134
// and 136, t 142 and 695.
bool plan_window(const DevParams &p, size_t table_bytes, int64_t nvis, int ngrids)
{
    if (table_bytes == 0 ||
        table_bytes > std::max<size_t>((size_t)16 << 20, 2048 * (size_t)nvis))
        return false;
    return p.S != 16 || 4 * nvis < (int64_t)ngrids * p.N * p.N;
}

size_t plan_bin_bytes(int64_t ntiles, const DevParams &p)
{
    return kBinHeader + sizeof(int32_t) * (size_t)p.nsub * (size_t)ntiles;
}
size_t plan_block_bytes(int64_t ntiles)
{
    const int tb = plan_block(ntiles, kMaxSubBins);  // the most blocks
    return sizeof(Totals) * (size_t)((ntiles + tb - 1) / tb + 1);
}

cudaError_t launch_plan(const DevParams &p, int64_t nvis, const double *u,
                        const double *v, const double *w, Plan &plan, int num_sms,
                        cudaStream_t s)
{
    cudaError_t e;
    // one clear for the dropped count, the ticket and the bins
    e = cudaMemsetAsync(plan.d_bin_base, 0, plan_bin_bytes(plan.ntiles, p), s);
    if (e != cudaSuccess)
        return e;
    int32_t *const bin = (int32_t *)(plan.d_bin_base + kBinHeader);
    if (nvis > 0 &&
        (e = launch_pdl(locate_bin_kernel, (nvis + 255) / 256, 256, 0, s, p, nvis, u, v, w,
                        plan.d_tile, plan.d_rank, plan.d_rec0, bin, plan.d_dropped,
                        plan.d_drop_list, plan.ngrids, plan.d_offsets)) != cudaSuccess)
        return e;
    const Cut cut{p.chunk, plan.unit, plan.unit_parts,
                  plan.window ? p.T * p.T : std::numeric_limits<int32_t>::max()};
    Totals *const blocks = (Totals *)plan.d_blocks;
    if (plan.ntiles <= kOneBlockTiles) {
        e = launch_pdl(tile_items_kernel<true>, 1, kPlanThreads, 0, s, plan.ntiles,
                       kOneBlockTiles, p.nsub, cut, plan.d_tile_count, blocks, bin, plan.d_items,
                       plan.d_nitems, plan.d_units, plan.d_nunits);
    } else {
        const int tb = plan_block(plan.ntiles, p.nsub), nblk = (plan.ntiles + tb - 1) / tb;
        e = launch_pdl(tile_count_kernel, nblk, kPlanThreads, 0, s, plan.ntiles, tb, p.nsub, cut,
                       bin, plan.d_tile_count, blocks,
                       (unsigned *)(plan.d_bin_base + kBinTicket));
        if (e == cudaSuccess)
            e = launch_pdl(tile_items_kernel<false>, nblk, kPlanThreads, 0, s, plan.ntiles, tb,
                           p.nsub, cut, plan.d_tile_count, blocks, bin, plan.d_items,
                           plan.d_nitems, plan.d_units, plan.d_nunits);
    }
    if (e != cudaSuccess)
        return e;
    if (nvis > 0) {
        e = launch_pdl(scatter_kernel, (nvis + 255) / 256, 256, 0, s, nvis, plan.d_tile,
                       plan.d_rank, plan.d_rec0, bin, plan.d_slots);
        if (e != cudaSuccess)
            return e;
        if (plan.sorted)
            return launch_item_sort(p, plan, num_sms, false, s);
    }
    return cudaSuccess;
}

// The per-item sort serves the kernels that walk runs of one origin; the
// 16-bit tensor-core forms and the window gridder take any order within a bin
// and leave it out until a call that gains by it.  That call may be captured
// into a graph, so whether the sort has run is known on the device alone: the
// mark makes every later one a launch that returns at once.
cudaError_t launch_item_sort(const DevParams &p, const Plan &plan, int num_sms, bool marked,
                             cudaStream_t s)
{
    const int nb = sort_keys(p);
    const size_t shm = sizeof(int32_t) * kSortThreads * ((nb + kSortThreads - 1) / kSortThreads);
    // the largest size, not this plan's: the limit belongs to the kernel, and
    // another thread's context may launch it with more in between
    cudaError_t e = cudaFuncSetAttribute(item_sort_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(int32_t) * kMaxSortBins);
    if (e != cudaSuccess)
        return e;
    int32_t *const mark = (int32_t *)(plan.d_bin_base + kBinSortMark);
    const int nblk = std::max(1, std::min(plan.items_capacity, 16 * num_sms));
    e = launch_pdl(item_sort_kernel, nblk, kSortThreads, shm, s, p, plan.d_items, plan.d_nitems,
                   marked ? mark : nullptr, plan.d_slots,
                   plan_splits(plan) ? plan.d_rec0 : nullptr, plan.d_rank);
    if (e == cudaSuccess && marked)
        e = cudaMemsetAsync(mark, 1, sizeof(*mark), s);
    return e;
}

}  // namespace sepw
