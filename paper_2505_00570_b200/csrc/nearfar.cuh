// The compression Y = P X in one pass over the cache: near rows exactly, far rows through a few values per tile.
#pragma once
#include <vector>

#include "common.cuh"
#include "gemm.cuh"

namespace freqkv {

constexpr int32_t NEARFAR_ERR_WAIT = 0x1000;  // status-word bit: a wait of the kernel ran out

// How the compression of one (n_in, n_keep) is cut up (host only).
struct NearFarShape {
    int32_t tiles;         // output tiles of 128 rows
    int32_t rank;          // far values per tile
    int32_t slices;        // 64-column slices of a tile's near block; its last 16 columns hold the far weights
    int32_t margin;        // near rows on either side of the rows under a tile
    int32_t k_slices;      // 64-row slices of the input
    int32_t part_slices;   // slices of one far job
    int32_t parts;         // far jobs per 128 far rows
    int32_t far_tiles;     // blocks of 128 far rows
    size_t near_bytes, far_bytes, bytes;  // of the near blocks, the far blocks, the whole plan
};
NearFarShape nearfar_shape(int32_t n_in, int32_t n_keep);

// Fills the `shape.bytes` at `out` (near blocks, far blocks, tables); two launches.
cudaError_t launch_build_nearfar(void* out, int32_t n_in, int32_t n_keep, cudaStream_t stream);

// One or several sequences of the cache (a uniform call: one item that covers every sequence).
struct NearFarItem {
    int32_t batch0, batch_count;  // sequences, relative to the view
    int32_t n_in, n_keep;
    const void* plan;
};
// Everything a launch needs that is not a stream operation; launch_nearfar calls it itself, a caller that must not
// allocate later (stream capture) calls it first.
cudaError_t nearfar_prepare(GemmState* state, const CacheView& view, const std::vector<NearFarItem>& items);
// The work area of any uniform call of these lengths with up to some 15000 groups of 16 tiles (about 15 MB for each block of 128 far
// rows), so that the calls after a plan allocate nothing.
cudaError_t nearfar_reserve(GemmState* state, int32_t n_in, int32_t n_keep);
cudaError_t launch_nearfar(GemmState* state, const CacheView& view, const std::vector<NearFarItem>& items, int32_t sink,
                           int32_t* status_dev, int sm_count, const LaunchHooks& hooks, cudaStream_t stream);

}  // namespace freqkv
