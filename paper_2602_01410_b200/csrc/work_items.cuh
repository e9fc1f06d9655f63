// Work items of the persistent GEMM kernels: output tiles, and contraction slices of the tiles of the last, partial wave.
//
// Item w < split_first is tile w over the whole contraction; the tiles from split_first on are cut into nsplit slices each, item
// split_first + r * nsplit + j being slice j of tile split_first + r.  nsplit == 1: no slicing, num_items == number of tiles.  A
// slice's FP32 sums go to the workspace, and whoever delivers a sub-tile's last slice adds all of them in slice order; or the slices of a
// tile are the CTAs of a cluster (then split_first is 0) and each adds its share of the tile, in slice order too (gemm.cu).
#pragma once
#include "common.cuh"

namespace snip {

// at most kMaxSlices slices per tile; partial sums for kMaxSlicedItems of them fit the workspace
constexpr int kMaxSlices = 4, kMaxSlicedItems = 160;
constexpr int kSliceWarps = 8;   // epilogue warps of a CTA, each with a counter per sliced tile
constexpr size_t kSliceCountersOffset = 256, kSliceCountersBytes = 8192;   // counters: [sliced tile][epilogue warp], 32 bits each
static_assert((size_t)kMaxSlicedItems / 2 * kSliceWarps * 4 <= kSliceCountersBytes, "counter area");

struct WorkSplit {
    int32_t split_first, nsplit, num_items;
};

// The tiles of the last, partial wave (all tiles, if there are fewer than SMs) are cut along the contraction into as many slices as
// there are SMs to take them: at most kMaxSlices, none shorter than min_stages pipeline stages.  Whole if that saves fewer than
// min_saved stages, which the exchange of the slices' sums costs.
inline WorkSplit plan_work(int num_tiles, int num_stages, int sms, int min_stages, int min_saved, bool slice, int max_items = kMaxSlicedItems)
{
    WorkSplit s = {num_tiles, 1, num_tiles};
    if (!slice || sms <= 0) return s;
    const int full = (num_tiles / sms) * sms, rest = num_tiles - full;
    int ns = rest > 0 ? sms / rest : 1;
    if (ns > kMaxSlices) ns = kMaxSlices;
    while (ns > 1 && (num_stages / ns < min_stages || rest * ns > max_items)) --ns;
    if (num_stages - num_stages / ns < min_saved) return s;
    if (ns > 1) { s.split_first = full; s.nsplit = ns; s.num_items = full + rest * ns; }
    return s;
}

struct WorkItem {
    int t, ks0, ks1;       // tile, stage range of the contraction
    int tail, slice, nsl;  // index of a sliced tile among the sliced tiles, slice, number of slices (1: whole tile)
};
template <bool SLICED>   // false: every item is a whole tile (known at compile time)
__device__ __forceinline__ WorkItem work_item(const WorkSplit &g, int w, int num_kstages)
{
    WorkItem wi;
    if (!SLICED || w < g.split_first) {
        wi.t = w; wi.ks0 = 0; wi.ks1 = num_kstages; wi.tail = 0; wi.slice = 0; wi.nsl = 1;
    } else {
        const int i = w - g.split_first;
        wi.tail = i / g.nsplit;
        wi.slice = i - wi.tail * g.nsplit;
        wi.nsl = g.nsplit;
        wi.t = g.split_first + wi.tail;
        wi.ks0 = (int)((int64_t)wi.slice * num_kstages / g.nsplit);
        wi.ks1 = (int)((int64_t)(wi.slice + 1) * num_kstages / g.nsplit);
    }
    return wi;
}

// Tile coordinates: groups of 16 row-tiles share their B panels in L2 while they are resident together.
__device__ __forceinline__ void tile_coords(int t, int num_m, int num_n, int &m_idx, int &n_idx)
{
    constexpr int kGroupM = 16;
    const int group_size = kGroupM * num_n;
    const int g = t / group_size;
    const int first_m = g * kGroupM;
    const int gm = min(num_m - first_m, kGroupM);
    const int r = t - g * group_size;
    m_idx = first_m + r % gm;
    n_idx = r / gm;
}

}  // namespace snip
