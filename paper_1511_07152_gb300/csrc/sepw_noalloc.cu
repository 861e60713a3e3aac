// sepw_grid_noalloc: tiled FP32 gridding that performs no device allocation.
//
// Some callers cannot let a library allocate device memory.  Examples: a
// real-time imaging pipeline that reserves all of its memory at start-up and
// must not block on cudaMalloc (which can synchronise the device) while it is
// observing, or a host framework that owns the device memory pool and forbids
// raw allocations from plugins.  This entry point serves them: instead of a
// context's workspace it uses one fixed scratch array compiled into the
// library as a file-scope __device__ variable, so every GPU that loads the
// library holds that array (kNoallocBytes, about 42 MB) until the process
// exits.
//
// The scratch holds the same plan as the context path (bin ids and ranks,
// packed records, slots, dropped-index list, per-tile counts and
// cursors, per-bin counts, work items and counters), and the existing plan
// and tiled-gridder launchers run on it unchanged.  Every call reuses the
// array: the plan launcher clears the bin counts and the dropped counter at
// the start of each call, the gridder clears its work counter, and
// everything else is overwritten before it is read.  Calls whose work
// overlaps on the GPU (other streams, other host threads) race on the array.
#include <mutex>

#include "sepw_internal.cuh"

namespace sepw {
namespace {

constexpr size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

constexpr int64_t kMaxVis = SEPW_NOALLOC_MAX_VIS;
constexpr int64_t kMaxTiles = SEPW_NOALLOC_MAX_TILES;
constexpr int64_t kMaxItems = kMaxTiles + kMaxVis / kChunk + 1;

// byte offsets of the plan arrays inside the scratch
constexpr size_t kOffTile = 0;
constexpr size_t kOffRank = align256(kOffTile + sizeof(int32_t) * kMaxVis);
constexpr size_t kOffRec0 = align256(kOffRank + sizeof(int32_t) * kMaxVis);
constexpr size_t kOffSlots = align256(kOffRec0 + sizeof(uint64_t) * kMaxVis);
constexpr size_t kOffDrop = align256(kOffSlots + sizeof(Slot) * kMaxVis);
constexpr int64_t kMaxUnits = kMaxTiles + kMaxVis / 32 + 1;
constexpr size_t kOffCount = align256(kOffDrop + sizeof(int32_t) * kMaxVis);
constexpr size_t kOffBlocks = align256(kOffCount + sizeof(int32_t) * kMaxTiles);
constexpr size_t kBlocksBytes = 64 * 1024;  // above plan_block_bytes(kMaxTiles): 1025 x 20 bytes
constexpr size_t kOffBin = align256(kOffBlocks + kBlocksBytes);
constexpr size_t kOffItems =
    align256(kOffBin + kBinHeader + sizeof(int32_t) * kMaxSubBins * kMaxTiles);
constexpr size_t kOffUnits = align256(kOffItems + sizeof(WorkItem) * kMaxItems);
constexpr size_t kOffNitems = align256(kOffUnits + sizeof(WorkItem) * kMaxUnits);
constexpr size_t kOffCounter = align256(kOffNitems + 2 * sizeof(int32_t));
// the gridder's copy of the tap table; callers with larger ones get the
// kernels that read theirs directly
constexpr size_t kTablesBytes = (size_t)4 << 20;
constexpr size_t kOffTables = align256(kOffCounter + 2 * sizeof(int32_t));
constexpr size_t kNoallocBytes = align256(kOffTables + kTablesBytes);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];

// Device address of g_noalloc_scratch per device.  In host code the name
// g_noalloc_scratch is only a host-side stand-in, so the address is looked up
// once per device (with that device current) and cached.
constexpr int kMaxDevices = 64;
std::mutex g_mu;
void *g_scratch_addr[kMaxDevices] = {};

int scratch_address(void **out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return SEPW_ECUDA;
    }
    if (dev < 0 || dev >= kMaxDevices)
        return SEPW_ENOTSUP;
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_scratch_addr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            cudaGetLastError();
            return SEPW_ECUDA;
        }
        g_scratch_addr[dev] = p;
    }
    *out = g_scratch_addr[dev];
    return SEPW_OK;
}

bool device_ptr_ok(const void *ptr, bool allow_null)
{
    if (!ptr)
        return allow_null;
    if (((uintptr_t)ptr) & 7)
        return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace
}  // namespace sepw

using namespace sepw;

extern "C" int sepw_grid_noalloc(const sepw_params *prm, const float *taps, int64_t nvis,
                                 const double *u, const double *v, const double *w,
                                 const float *vis, const float *weight, float *grid,
                                 int64_t *n_dropped, sepw_stream_t stream)
{
    if (!prm)
        return SEPW_EINVAL;
    // the tiled FP32 form runs whatever form the caller names: check (and
    // resolve the default tile of) that form, not the caller's
    sepw_params tp = *prm;
    tp.form = SEPW_FORM_TILED;
    int rc = sepw_check_params(&tp);
    if (rc != SEPW_OK)
        return rc;
    if (nvis < 0)
        return SEPW_EINVAL;
    if (nvis > kMaxVis)
        return SEPW_ETOOLARGE;

    DevParams dp = make_dev_params(&tp);
    const int64_t ntiles = (int64_t)dp.ntx * dp.ntx;
    if (ntiles > kMaxTiles)
        return SEPW_ETOOLARGE;

    if (!device_ptr_ok(taps, false) || !device_ptr_ok(grid, false) ||
        !device_ptr_ok(n_dropped, true))
        return SEPW_EINVAL;
    // the tiled gridder reads rows of taps as 16-byte vectors
    if (((uintptr_t)taps) & 15)
        return SEPW_EINVAL;
    if (nvis > 0 && (!device_ptr_ok(u, false) || !device_ptr_ok(v, false) ||
                     !device_ptr_ok(w, false) || !device_ptr_ok(vis, false) ||
                     !device_ptr_ok(weight, true)))
        return SEPW_EINVAL;

    void *base = nullptr;
    if ((rc = scratch_address(&base)) != SEPW_OK)
        return rc;
    int dev = 0, num_sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return SEPW_ECUDA;
    }

    unsigned char *b = (unsigned char *)base;
    Plan pl;
    pl.nvis = nvis;
    pl.capacity = kMaxVis;
    pl.ntiles = (int32_t)ntiles;
    pl.tiles_capacity = (int32_t)kMaxTiles;
    pl.items_capacity = (int32_t)(ntiles + nvis / kChunk + 1);
    pl.valid = true;
    pl.form = SEPW_FORM_TILED;
    pl.d_tile = (int32_t *)(b + kOffTile);
    pl.d_rank = (int32_t *)(b + kOffRank);
    pl.d_rec0 = (uint64_t *)(b + kOffRec0);
    pl.d_slots = (Slot *)(b + kOffSlots);
    pl.d_drop_list = (int32_t *)(b + kOffDrop);
    pl.d_tile_count = (int32_t *)(b + kOffCount);
    pl.d_blocks = b + kOffBlocks;
    pl.d_bin_base = b + kOffBin;
    pl.d_items = (WorkItem *)(b + kOffItems);
    pl.d_units = (WorkItem *)(b + kOffUnits);
    pl.d_nitems = (int32_t *)(b + kOffNitems);
    pl.d_nunits = pl.d_nitems + 1;
    pl.d_item_counter = (int32_t *)(b + kOffCounter);
    pl.d_dropped = (unsigned long long *)pl.d_bin_base;
    const size_t wbytes = window_tables_bytes(dp);
    pl.window = wbytes <= kTablesBytes && plan_window(dp, wbytes, nvis, 1);
    pl.sorted = !pl.window;
    set_units(dp, num_sms, pl);
    dp.early = nvis <= kEarlyVis ? 1 : 0;
    set_bins(dp, pl.window ? kBinsWindow : plan_bins(dp, SEPW_FORM_TILED, nvis, ntiles));
    float *tables = (float *)(b + kOffTables);
    if (!pl.window && sizeof(float2) * dp.P * dp.OS * (size_t)dp.S > kTablesBytes)
        tables = nullptr;

    pl.dropped_out = n_dropped;
    cudaStream_t s = (cudaStream_t)stream;
    if (launch_plan(dp, nvis, u, v, w, pl, num_sms, s) != cudaSuccess) {
        cudaGetLastError();
        return SEPW_ECUDA;
    }
    if (nvis > 0 && launch_grid_tiled(dp, pl, (const float2 *)vis, weight,
                                      (const float2 *)taps, tables, (float2 *)grid, num_sms,
                                      s) != cudaSuccess) {
        cudaGetLastError();
        return SEPW_ECUDA;
    }
    // with visibilities the gridder's launches have written it
    if (n_dropped && nvis == 0 &&
        cudaMemcpyAsync(n_dropped, pl.d_dropped, sizeof(int64_t), cudaMemcpyDeviceToDevice, s) !=
            cudaSuccess) {
        cudaGetLastError();
        return SEPW_ECUDA;
    }
    return SEPW_OK;
}
