// vr_modes.cuh -- launch helpers shared by the other uses of the ray march
// (vr_modes.cu, vr_sortlast.cu).
#pragma once

#include "vr_device.cuh"

namespace vr {

constexpr int kModeThreads = 256;

// These kernels march in groups for the views that vr_render does: 150 x 100
// views of a 200 x 220 x 190 float cube, maximum 207 -> 35 us, sigma clipping
// with its mini-map 378 -> 88, six sub-boxes and their composite 842 -> 240
// (bound by the host's calls).

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
