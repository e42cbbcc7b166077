// vr_modes.cuh -- launch helpers shared by the other uses of the ray march
// (vr_modes.cu, vr_sortlast.cu).
#pragma once

#include "vr_device.cuh"

namespace vr {

constexpr int kModeThreads = 256;

// Pixel of a lane's ray: its warp's 8 x 4 tile, or (GROUPS) 2 x 2 tile with
// eight lanes to a ray.  These kernels march in groups for the views that
// vr_render does (march_in_groups): 150 x 100 views of a 200 x 220 x 190 float
// cube, maximum 207 -> 35 us, sigma clipping with its mini-map 378 -> 88, six
// sub-boxes and their composite 842 -> 240 (bound by the host's calls).
template <bool GROUPS> __device__ __forceinline__ int2 mode_pixel(unsigned tile, int tiles_x)
{
    if (GROUPS) return group_pixel(tile, tiles_x);
    const int2 at = tile_pixel(threadIdx.x & 31, 3);
    return make_int2((int)(tile % tiles_x) * 8 + at.x, (int)(tile / tiles_x) * 4 + at.y);
}

// Tiles of an image, across and in all.
inline unsigned mode_tiles(const CamDev &c, bool groups, int &tiles_x)
{
    tiles_x = groups ? (c.W + 1) / 2 : (c.W + 7) / 8;
    return (unsigned)tiles_x * (unsigned)(groups ? (c.H + 1) / 2 : (c.H + 3) / 4);
}

// Persistent grid of a kernel over its tiles.
template <typename K>
unsigned persistent_grid(K fn, unsigned ntiles, int threads = kModeThreads)
{
    const int per_sm = occupancy_blocks((const void *)fn, threads, 0);
    unsigned grid = (unsigned)(per_sm * sm_count());
    const unsigned useful = (ntiles + threads / 32 - 1) / (threads / 32);
    if (grid > useful) grid = useful;
    return grid < 1 ? 1 : grid;
}

}  // namespace vr
