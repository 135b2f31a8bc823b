// Blocks of the plan kernel (host code).
#pragma once

namespace sipf {

constexpr int kPlanNT = 512;
constexpr int kPlanCluster = 8;   // blocks of the plan kernel on large grids

// One block of 16 warps, at most two strips of 32 tiles each, up to 1024 tiles (H = 80);
// beyond, a cluster of eight blocks, if the GPU that the process sees can hold one
// (`clusters` at a time), else one block with more strips per warp.
inline int plan_blocks(int ntiles, int clusters) {
    return ntiles > 2 * kPlanNT && clusters > 0 ? kPlanCluster : 1;
}

}  // namespace sipf
