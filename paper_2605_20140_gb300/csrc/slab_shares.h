// How the slab path of the allocation-free deposit cuts a grid into slabs of z-planes,
// and how many blocks it launches (host and device code).
#pragma once

#ifdef __CUDACC__
#define SIPF_HD __host__ __device__
#else
#define SIPF_HD
#endif

namespace sipf {

constexpr int kSlabBytes = 200 * 1024;   // a slab's node sums at most, eight bytes each

SIPF_HD inline int slab_planes(int H) {   // planes per slab, one more is held
    const int p = kSlabBytes / (H * H * 8) - 1;
    return p < H ? p : H;
}

SIPF_HD inline int slab_count(int H) { return (H + slab_planes(H) - 1) / slab_planes(H); }

// One block per SM, but never fewer than slabs: the kernel gives every slab a block
// and shares out the rest (64^3 has 13 slabs; a process may see fewer SMs than that).
inline int slab_grid(int sms, int H) { return sms > slab_count(H) ? sms : slab_count(H); }

}  // namespace sipf
