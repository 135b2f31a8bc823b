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

namespace {

constexpr int kNoAllocMaxH = 64;
constexpr int kNoAllocMaxNodes = kNoAllocMaxH * kNoAllocMaxH * kNoAllocMaxH;
constexpr int kMaxParts = 1024;     // largest number of blocks of the first pass
constexpr int kCtl = kMaxParts;     // words in front of the node sums: per-block largest masses
constexpr int kMaxDevices = 64;

// [0, kMaxParts): bits of each first-pass block's largest mass;
// [kCtl, kCtl + H^3): fixed-point node sums.  Shared by every call.
static __device__ __align__(256) unsigned long long g_noalloc_scratch[kCtl + kNoAllocMaxNodes];

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

// First pass: clears the node sums and finds the largest mass.  Bound by
// reading the masses (8 B each) and by launch latency; each block leaves one
// maximum in a slot of its own, which the next passes reduce themselves (an
// atomic on one word for every particle took 0.5 of the 0.83 ms of a call
// with 10^6 particles, and a slot that is always written needs no clearing
// launch before it).
__global__ void __launch_bounds__(kNaNT)
    k_na_begin(const double* __restrict__ mass, int64_t N, int nodes, unsigned long long* s) {
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
        if (na_counts(m) && b > mx) mx = b;
    }
    mx = na_block_max(mx);
    if (threadIdx.x == 0) s[blockIdx.x] = static_cast<unsigned long long>(mx);
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

// Second pass: eight 64-bit sums per particle in L2, exact in any order.
// Bound by the L2's atomic throughput (8 N additions); the positions and
// masses are read before the wait for the first pass.
__global__ void __launch_bounds__(kNaNT)
    k_na_deposit(const float* __restrict__ x, const double* __restrict__ mass, int64_t N, int H,
                 float o0, float o1, float o2, float h, int parts, unsigned long long* s) {
    sipf::pdl_trigger();
    const int64_t i = static_cast<int64_t>(blockIdx.x) * kNaNT + threadIdx.x;
    const bool in = i < N;
    const double m = in ? mass[i] : 0.0;
    const float Hf = __int2float_rn(H);
    const float o[3] = {o0, o1, o2};
    int c[3], c1[3];
    float f[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        // grid units, wrapped into [0, H) (a result rounding to H becomes 0)
        const float xd = in ? x[static_cast<int64_t>(d) * N + i] : 0.0f;
        float v = __fdiv_rn(__fsub_rn(xd, o[d]), h);
        if (!(v >= 0.0f && v < Hf)) {
            v = __fsub_rn(v, __fmul_rn(Hf, floorf(__fdiv_rn(v, Hf))));
            if (v < 0.0f) v = __fadd_rn(v, Hf);
            if (!(v < Hf)) v = 0.0f;
        }
        c[d] = min(max(static_cast<int>(v), 0), H - 1);
        c1[d] = c[d] + 1 < H ? c[d] + 1 : 0;
        f[d] = __fsub_rn(v, __int2float_rn(c[d]));
    }
    sipf::pdl_wait();   // the first pass's maxima and cleared sums
    const int shift = na_shift(s, parts);
    if (!na_counts(m)) return;
    const float a = static_cast<float>(ldexp(m, shift));
    unsigned long long* acc = s + kCtl;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int dx = k & 1, dy = (k >> 1) & 1, dz = k >> 2;
        const float wx = dx ? f[0] : __fsub_rn(1.0f, f[0]);
        const float wy = dy ? f[1] : __fsub_rn(1.0f, f[1]);
        const float wz = dz ? f[2] : __fsub_rn(1.0f, f[2]);
        const uint32_t q = __float2uint_rn(__fmul_rn(__fmul_rn(a, wz), __fmul_rn(wx, wy)));
        const int node = ((dz ? c1[2] : c[2]) * H + (dy ? c1[1] : c[1])) * H + (dx ? c1[0] : c[0]);
        if (q) atomicAdd(acc + node, static_cast<unsigned long long>(q));
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
    cudaError_t e = sipf::launch_pdl(k_na_begin, dim3(parts), dim3(kNaNT), 0, st, mass, N, nodes, s);
    if (e == cudaSuccess)
        e = sipf::launch_pdl(k_na_deposit, dim3(static_cast<unsigned>(pblocks)), dim3(kNaNT), 0, st,
                             x, mass, N, H, o0, o1, o2, hf, parts, s);
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
