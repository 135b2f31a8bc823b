// Allocation-free particle-to-grid deposit.
//
// Some callers cannot allocate device memory at the moment they need a
// density: code that runs while another framework owns the device memory
// budget (a caching allocator that must not see foreign cudaMalloc calls,
// which also synchronise the device), real-time loops that may not block
// or fail on allocation, or plug-ins handed only pre-allocated buffers.
// sipf_deposit_noalloc serves them: it computes the same deposit as the
// context path (sipf_fields with SIPF_FIELD_U) but keeps its integer
// accumulator in a fixed file-scope device array instead of context
// memory, so it never calls cudaMalloc, cudaFree or any allocating
// routine.  The array holds at most kNoAllocMaxNodes grid nodes; every GPU
// that loads the library keeps it until the process exits.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "sipf_internal.cuh"
#include "slab_shares.h"

namespace {

constexpr int kNoAllocMaxH = 64;
constexpr int kNoAllocMaxNodes = kNoAllocMaxH * kNoAllocMaxH * kNoAllocMaxH;
constexpr int kMaxParts = 1024;     // largest number of blocks of the first pass
constexpr int kPlanes = kMaxParts;  // first of the particle counts per z-plane (slab path)
constexpr int kCtl = kMaxParts + kNoAllocMaxH;   // words in front of the node sums
constexpr int kMaxDevices = 64;

// [0, kMaxParts): bits of each first-pass block's largest mass;
// [kPlanes, kCtl): particles per z-plane; [kCtl, kCtl + H^3): fixed-point node
// sums.  Shared by every call.
static __device__ __align__(256) unsigned long long g_noalloc_scratch[kCtl + kNoAllocMaxNodes];

// Particles from which the slab path is taken (figures at k_na_slab).
int64_t slab_min(int H) { return H <= 32 ? int64_t{1} << 18 : int64_t{1} << 19; }

std::mutex g_mutex;
unsigned long long* g_scratch_ptr[kMaxDevices] = {nullptr};

constexpr int kNaNT = 256;

// A particle contributes only if its mass is finite and positive: an
// infinite or NaN mass is skipped (it would otherwise fix the scale of every
// node), a zero mass adds nothing anyway.
__device__ __forceinline__ bool na_counts(double m) { return isfinite(m) && m > 0.0; }

// Largest of a block's values (non-negative int64), given to every thread.
__device__ __forceinline__ long long na_block_max(long long v) {
    __shared__ long long part[kNaNT / 32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const long long o = __shfl_xor_sync(0xffffffffu, v, off);
        v = o > v ? o : v;
    }
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    v = part[0];
#pragma unroll
    for (int k = 1; k < kNaNT / 32; ++k) v = part[k] > v ? part[k] : v;
    return v;
}

// A coordinate in grid units, wrapped into [0, H) (a result rounding to H
// becomes 0), split into its cell and the fraction.
__device__ __forceinline__ int na_cell(float x, float o, float h, int H, float& frac) {
    const float Hf = __int2float_rn(H);
    float v = __fdiv_rn(__fsub_rn(x, o), h);
    if (!(v >= 0.0f && v < Hf)) {
        v = __fsub_rn(v, __fmul_rn(Hf, floorf(__fdiv_rn(v, Hf))));
        if (v < 0.0f) v = __fadd_rn(v, Hf);
        if (!(v < Hf)) v = 0.0f;
    }
    const int c = min(max(static_cast<int>(v), 0), H - 1);
    frac = __fsub_rn(v, __int2float_rn(c));
    return c;
}

// First pass: clears the node sums and finds the largest mass; with z not null
// it also counts the particles per z-plane (into counters cleared before).
// Bound by reading the masses (8 B each) and by launch latency; each block
// leaves one maximum in a slot of its own, which the next passes reduce
// themselves (an atomic on one word for every particle took 0.5 of the 0.83 ms
// of a call with 10^6 particles, and a slot that is always written needs no
// clearing launch before it).
__global__ void __launch_bounds__(kNaNT)
    k_na_begin(const double* __restrict__ mass, int64_t N, int nodes, const float* __restrict__ z,
               int H, float o2, float h, unsigned long long* s) {
    __shared__ int planes[kNoAllocMaxH];
    if (z) {
        if (threadIdx.x < kNoAllocMaxH) planes[threadIdx.x] = 0;
        __syncthreads();
    }
    // waits first: the next pass reads the caller's arrays as soon as every
    // block of this one has passed the trigger
    sipf::pdl_wait();
    sipf::pdl_trigger();
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kNaNT;
    const int64_t t = static_cast<int64_t>(blockIdx.x) * kNaNT + threadIdx.x;
    for (int64_t i = t; i < nodes; i += stride) s[kCtl + i] = 0ull;
    long long mx = 0;   // non-negative doubles order like int64
    for (int64_t i = t; i < N; i += stride) {
        const double m = mass[i];
        const long long b = __double_as_longlong(m);
        if (!na_counts(m)) continue;
        if (b > mx) mx = b;
        if (z) {
            float f;
            atomicAdd(planes + na_cell(z[i], o2, h, H, f), 1);
        }
    }
    mx = na_block_max(mx);
    if (threadIdx.x == 0) s[blockIdx.x] = static_cast<unsigned long long>(mx);
    if (z && threadIdx.x < H && planes[threadIdx.x])
        atomicAdd(s + kPlanes + threadIdx.x, static_cast<unsigned long long>(planes[threadIdx.x]));
}

// 2^S with S chosen so that the largest mass times 2^S stays below 2^30.
// Called by whole blocks.
__device__ __forceinline__ int na_shift(const unsigned long long* s, int parts) {
    long long mx = 0;
    for (int k = threadIdx.x; k < parts; k += kNaNT) {
        const long long b = static_cast<long long>(s[k]);
        mx = b > mx ? b : mx;
    }
    const double mmax = __longlong_as_double(na_block_max(mx));
    if (!(mmax > 0.0)) return 0;
    int e;
    frexp(mmax, &e);    // mmax < 2^e
    return 30 - e;
}

// The eight contributions of a particle of mass a (in units of 2^-S) with
// fractions f to the corners of its cell.
__device__ __forceinline__ void na_corners(float a, const float (&f)[3], uint32_t (&q)[8]) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float wx = (k & 1) ? f[0] : __fsub_rn(1.0f, f[0]);
        const float wy = ((k >> 1) & 1) ? f[1] : __fsub_rn(1.0f, f[1]);
        const float wz = (k >> 2) ? f[2] : __fsub_rn(1.0f, f[2]);
        q[k] = __float2uint_rn(__fmul_rn(__fmul_rn(a, wz), __fmul_rn(wx, wy)));
    }
}

// Second pass: eight 64-bit sums per particle in L2, exact in any order.
// Bound by the L2's atomic throughput (8 N additions, which in a clustered cloud
// meet in a few lines); the positions and masses are read before the wait for
// the first pass.
__global__ void __launch_bounds__(kNaNT)
    k_na_deposit(const float* __restrict__ x, const double* __restrict__ mass, int64_t N, int H,
                 float o0, float o1, float o2, float h, int parts, unsigned long long* s) {
    sipf::pdl_trigger();
    const int64_t i = static_cast<int64_t>(blockIdx.x) * kNaNT + threadIdx.x;
    const bool in = i < N;
    const double m = in ? mass[i] : 0.0;
    const float o[3] = {o0, o1, o2};
    int c[3], c1[3];
    float f[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        c[d] = na_cell(in ? x[static_cast<int64_t>(d) * N + i] : o[d], o[d], h, H, f[d]);
        c1[d] = c[d] + 1 < H ? c[d] + 1 : 0;
    }
    sipf::pdl_wait();   // the first pass's maxima and cleared sums
    const int shift = na_shift(s, parts);
    if (!na_counts(m)) return;
    uint32_t q[8];
    na_corners(static_cast<float>(ldexp(m, shift)), f, q);
    unsigned long long* acc = s + kCtl;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int node = (((k >> 2) ? c1[2] : c[2]) * H + (((k >> 1) & 1) ? c1[1] : c[1])) * H +
                         ((k & 1) ? c1[0] : c[0]);
        if (q[k]) atomicAdd(acc + node, static_cast<unsigned long long>(q[k]));
    }
}

// Second pass for many particles: a block sums the particles of a slab of
// z-planes in shared memory (a low and a high 32-bit word per node, the carry
// taken from the old low word, so the sums are as exact as 64-bit ones) and adds
// its nodes to the grid once.  Every slab's blocks read all z; the blocks are shared
// out over the slabs by their particle counts, so that a clustered cloud does not
// leave one block with most of it, and a warp gathers the particles that fall
// into its slab until it has 32.  Against the path above, us per call (three
// clusters / uniform): 32^3 with 2^18 particles 34 / 35 against 69 / 28, with 2^22 279 / 166
// against 797 / 250; 48^3 with 10^6 84 / 67 against 193 / 55; 64^3 with 10^6 123 / 97
// against 128 / 54, and 126 against 166 (three clusters) with inputs not in L2 on the default
// stream; 32^3 with 2^17 26 / 31 against 34 / 18.  Clusters are the method's usual
// state, so it is taken from 2^18 particles on up to 32^3 and from 2^19 on beyond,
// where the reading of z by every slab weighs more.
constexpr int kSlabNT = 512;
constexpr int kScan = 4;        // z read per thread and round

__global__ void __launch_bounds__(kSlabNT)
    k_na_slab(const float* __restrict__ x, const double* __restrict__ mass, int64_t N, int H,
              float o0, float o1, float o2, float h, int parts, unsigned long long* s) {
    extern __shared__ uint32_t sm[];
    __shared__ int mine[3];                       // slab, part of it, its parts
    __shared__ int queue[kSlabNT / 32][32 * (kScan + 1)];
    sipf::pdl_trigger();
    const int P = sipf::slab_planes(H), slabs = (H + P - 1) / P, plane = H * H;
    const int nodes = (P + 1) * plane;
    uint32_t* lo = sm;
    uint32_t* hi = sm + nodes;
    for (int i = threadIdx.x; i < 2 * nodes; i += kSlabNT) sm[i] = 0u;
    sipf::pdl_wait();
    // largest mass (as na_shift, for this block size)
    long long mx = 0;
    for (int k = threadIdx.x; k < parts; k += kSlabNT) {
        const long long b = static_cast<long long>(s[k]);
        mx = b > mx ? b : mx;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const long long o = __shfl_xor_sync(0xffffffffu, mx, off);
        mx = o > mx ? o : mx;
    }
    __shared__ long long warp_max[kSlabNT / 32];
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = mx;
    if (threadIdx.x == 0) {
        // blocks per slab: in proportion to its particles plus the reading of all z
        // (about a 24th of a particle each), at least one (the grid has that many)
        double all = 0.0;
        for (int k = 0; k < H; ++k) all += static_cast<double>(s[kPlanes + k]);
        const double scan = static_cast<double>(N) / 24.0, total = all + scan * slabs;
        int first = 0;
        mine[0] = -1;
        for (int b = 0; b < slabs; ++b) {
            double n = scan;
            for (int k = b * P; k < min(H, (b + 1) * P); ++k) n += static_cast<double>(s[kPlanes + k]);
            const int r = 1 + static_cast<int>((static_cast<int>(gridDim.x) - slabs) * (n / total));
            const int id = static_cast<int>(blockIdx.x) - first;
            if (id >= 0 && id < r) {
                mine[0] = b;
                mine[1] = id;
                mine[2] = r;
            }
            first += r;
        }
    }
    __syncthreads();
    const int slab = mine[0];
    if (slab < 0) return;
    mx = warp_max[0];
    for (int k = 1; k < kSlabNT / 32; ++k) mx = warp_max[k] > mx ? warp_max[k] : mx;
    int shift = 0;
    const double mmax = __longlong_as_double(mx);
    if (mmax > 0.0) {
        int e;
        frexp(mmax, &e);
        shift = 30 - e;
    }
    const int z0 = slab * P, z1 = min(H, z0 + P), lane = threadIdx.x & 31;
    const int64_t beg = N * mine[1] / mine[2], end = N * (mine[1] + 1) / mine[2];
    int* q_mine = queue[threadIdx.x >> 5];
    int held = 0;
    auto take = [&](int first, int n) {   // n (at most 32) particles of the queue
        if (lane < n) {
            const int64_t i = beg + q_mine[first + lane];
            const double m = mass[i];
            float f[3];
            const int cx = na_cell(x[i], o0, h, H, f[0]), cy = na_cell(x[N + i], o1, h, H, f[1]);
            const int cz = na_cell(x[2 * N + i], o2, h, H, f[2]) - z0;
            const int x1 = cx + 1 < H ? cx + 1 : 0, y1 = cy + 1 < H ? cy + 1 : 0;
            if (na_counts(m)) {
                uint32_t q[8];
                na_corners(static_cast<float>(ldexp(m, shift)), f, q);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int node = (cz + (k >> 2)) * plane + (((k >> 1) & 1) ? y1 : cy) * H +
                                     ((k & 1) ? x1 : cx);
                    const uint32_t old = atomicAdd(lo + node, q[k]);
                    if (old + q[k] < old) atomicAdd(hi + node, 1u);
                }
            }
        }
    };
    for (int64_t i0 = beg; i0 < end; i0 += kScan * kSlabNT) {
        float zr[kScan];
#pragma unroll
        for (int k = 0; k < kScan; ++k) {
            const int64_t i = i0 + k * kSlabNT + threadIdx.x;
            zr[k] = i < end ? x[2 * N + i] : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < kScan; ++k) {
            const int64_t i = i0 + k * kSlabNT + threadIdx.x;
            float f;
            const int cz = na_cell(zr[k], o2, h, H, f);
            const bool in = i < end && cz >= z0 && cz < z1;
            const unsigned sel = __ballot_sync(0xffffffffu, in);
            if (in) q_mine[held + __popc(sel & ((1u << lane) - 1u))] = static_cast<int>(i - beg);
            held += __popc(sel);
        }
        __syncwarp();
        int done = 0;
        for (; held - done >= 32; done += 32) take(done, 32);
        if (done) {
            const int rest = lane < held - done ? q_mine[done + lane] : 0;
            __syncwarp();
            q_mine[lane] = rest;
            held -= done;
        }
        __syncwarp();
    }
    take(0, held);
    __syncthreads();
    unsigned long long* acc = s + kCtl;
    for (int i = threadIdx.x; i < (z1 - z0 + 1) * plane; i += kSlabNT) {
        const unsigned long long q = (static_cast<unsigned long long>(hi[i]) << 32) | lo[i];
        if (!q) continue;
        const int zz = z0 + i / plane;
        atomicAdd(acc + (zz < H ? zz : zz - H) * plane + i % plane, q);
    }
}

__global__ void __launch_bounds__(kNaNT)
    k_na_finish(const unsigned long long* s, int nodes, int parts, double inv_h3,
                float* __restrict__ u) {
    sipf::pdl_trigger();
    sipf::pdl_wait();
    const int shift = na_shift(s, parts);
    const int i = blockIdx.x * kNaNT + threadIdx.x;
    if (i >= nodes) return;
    const double scale = ldexp(inv_h3, -shift);
    u[i] = static_cast<float>(static_cast<double>(s[kCtl + i]) * scale);
}

// Device address of the scratch array on the current device (looked up
// once per device; host code only sees a host-side stand-in otherwise).
// The address is kept for the life of the process, so the entry point must
// not be used on a device after cudaDeviceReset in the same process.
int scratch_for_current_device(unsigned long long** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SIPF_ECUDA;
    std::lock_guard<std::mutex> lock(g_mutex);
    if (!g_scratch_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return SIPF_ECUDA;
        g_scratch_ptr[dev] = static_cast<unsigned long long*>(p);
    }
    *out = g_scratch_ptr[dev];
    return SIPF_OK;
}

}  // namespace

extern "C" int sipf_deposit_noalloc(const sipf_grid* grid, const float* x, const double* mass,
                                    int64_t N, float* u, void* stream) {
    if (!grid || !x || !mass || !u) return SIPF_EINVAL;
    const int H = grid->H;
    if (H < 1 || H > kNoAllocMaxH) return SIPF_EINVAL;   // scratch holds at most 64^3 nodes
    if (N < 1 || N >= (int64_t{1} << 31)) return SIPF_EINVAL;
    if (!(isfinite(grid->L) && grid->L > 0.0)) return SIPF_EINVAL;
    for (int k = 0; k < 3; ++k)
        if (!isfinite(grid->origin[k])) return SIPF_EINVAL;
    unsigned long long* s = nullptr;
    const int r = scratch_for_current_device(&s);
    if (r != SIPF_OK) return r;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int nodes = H * H * H;
    const double h = grid->L / H;
    const float o0 = static_cast<float>(grid->origin[0]), o1 = static_cast<float>(grid->origin[1]);
    const float o2 = static_cast<float>(grid->origin[2]), hf = static_cast<float>(h);
    const int64_t pblocks = (N + kNaNT - 1) / kNaNT;   // N < 2^31: fits a grid
    const int nblocks = (nodes + kNaNT - 1) / kNaNT;
    // first pass: two values per thread, at most kMaxParts blocks
    const int64_t want = (std::max<int64_t>(N, nodes) + 2 * kNaNT - 1) / (2 * kNaNT);
    const int parts = static_cast<int>(std::min<int64_t>(want, kMaxParts));
    const float* none = nullptr;
    cudaError_t e = cudaSuccess;
    if (N < slab_min(H)) {
        e = sipf::launch_pdl(k_na_begin, dim3(parts), dim3(kNaNT), 0, st, mass, N, nodes, none, H,
                             o2, hf, s);
        if (e == cudaSuccess)
            e = sipf::launch_pdl(k_na_deposit, dim3(static_cast<unsigned>(pblocks)), dim3(kNaNT), 0,
                                 st, x, mass, N, H, o0, o1, o2, hf, parts, s);
    } else {
        int dev = 0, nsm = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess)
            e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        const size_t smem =
            static_cast<size_t>(sipf::slab_planes(H) + 1) * H * H * 2 * sizeof(uint32_t);
        if (e == cudaSuccess)
            // the limit belongs to the kernel, not to this call: the same for every H
            e = cudaFuncSetAttribute(k_na_slab, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     sipf::kSlabBytes);
        if (e == cudaSuccess)
            e = cudaMemsetAsync(s + kPlanes, 0, kNoAllocMaxH * sizeof(unsigned long long), st);
        if (e == cudaSuccess)
            e = sipf::launch_pdl(k_na_begin, dim3(parts), dim3(kNaNT), 0, st, mass, N, nodes,
                                 x + 2 * N, H, o2, hf, s);
        if (e == cudaSuccess)
            e = sipf::launch_pdl(k_na_slab, dim3(sipf::slab_grid(nsm, H)), dim3(kSlabNT), smem, st,
                                 x, mass, N, H, o0, o1, o2, hf, parts, s);
    }
    if (e == cudaSuccess)
        e = sipf::launch_pdl(k_na_finish, dim3(nblocks), dim3(kNaNT), 0, st,
                             static_cast<const unsigned long long*>(s), nodes, parts,
                             1.0 / (h * h * h), u);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return SIPF_ECUDA;
    }
    if (cudaGetLastError() != cudaSuccess) return SIPF_ECUDA;
    return SIPF_OK;
}
