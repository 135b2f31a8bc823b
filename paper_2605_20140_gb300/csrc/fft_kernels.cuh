// Kernel templates of the spectral passes (see fft.cu for the pass
// structure): the two plane passes for H <= 128, the line passes along z and
// y, the row passes for H > 128, and their launch templates.  Each translation unit that
// launches them includes this header (internal linkage) and instantiates the
// grid sizes and radix plans it serves, so that the instantiations compile in
// parallel.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "fft_stages.cuh"
#include "sipf_internal.cuh"

namespace sipf {
namespace {


using namespace fftk;

// (H - k) mod H for 0 <= k <= H: the index of the mode -k.
template <int H>
__device__ __forceinline__ int neg_mod(int k) {
    if constexpr ((H & (H - 1)) == 0) return (H - k) & (H - 1);
    else return k == 0 ? 0 : H - k;
}

// Threads of the plane passes, chosen so that the radix-16 or radix-8 stages
// hold at most two butterflies per thread.
template <int H> struct Cfg;
template <> struct Cfg<8> { static constexpr int NT1 = 64, NT3 = 64; };
template <> struct Cfg<16> { static constexpr int NT1 = 256, NT3 = 256; };
template <> struct Cfg<24> { static constexpr int NT1 = 256, NT3 = 256; };
template <> struct Cfg<32> { static constexpr int NT1 = 256, NT3 = 256; };
template <> struct Cfg<48> { static constexpr int NT1 = 256, NT3 = 256; };
template <> struct Cfg<64> { static constexpr int NT1 = 512, NT3 = 512; };
template <> struct Cfg<72> { static constexpr int NT1 = 512, NT3 = 512; };
template <> struct Cfg<96> { static constexpr int NT1 = 768, NT3 = 768; };
template <> struct Cfg<128> { static constexpr int NT1 = 1024, NT3 = 1024; };

// Threads of the line passes (kCols lines per block) and of the row passes
// (H > 128 and radix plan 2: kRows complex rows per block).
template <int H> struct LineCfg;
template <> struct LineCfg<8> { static constexpr int NT = 64, NTX = 32; };
template <> struct LineCfg<16> { static constexpr int NT = 64, NTX = 32; };
template <> struct LineCfg<24> { static constexpr int NT = 128, NTX = 64; };
template <> struct LineCfg<32> { static constexpr int NT = 128, NTX = 64; };
template <> struct LineCfg<48> { static constexpr int NT = 192, NTX = 64; };
template <> struct LineCfg<64> { static constexpr int NT = 128, NTX = 64; };
template <> struct LineCfg<72> { static constexpr int NT = 192, NTX = 96; };
template <> struct LineCfg<96> { static constexpr int NT = 192, NTX = 96; };
template <> struct LineCfg<128> { static constexpr int NT = 128, NTX = 64; };
template <> struct LineCfg<144> { static constexpr int NT = 192, NTX = 96; };
template <> struct LineCfg<192> { static constexpr int NT = 256, NTX = 128; };
template <> struct LineCfg<216> { static constexpr int NT = 288, NTX = 160; };
template <> struct LineCfg<256> { static constexpr int NT = 256, NTX = 128; };
template <> struct LineCfg<288> { static constexpr int NT = 384, NTX = 160; };
template <> struct LineCfg<384> { static constexpr int NT = 384, NTX = 192; };
template <> struct LineCfg<432> { static constexpr int NT = 384, NTX = 224; };
template <> struct LineCfg<512> { static constexpr int NT = 512, NTX = 256; };

// Blocks per SM the registers of the row and line passes are set for: 64 registers a
// thread, 56 at 288 and 384, where a third block of 384 threads then shares the SM.  The rule
// stands as measured at these sizes; 432 has 384 threads too, but its z pass wants 80 registers
// (two blocks, 88 bytes spilled in plan 0) and has not been measured with fewer.  The caps
// spill 96 to 120 bytes in k_rows_forward at 144 (plan 0), 192, 288 and 384, 36 at 256 and
// in k_lines_z at 288.
template <int H> constexpr int line_blocks() {
    return 65536 / ((H == 288 || H == 384 ? 56 : 64) * LineCfg<H>::NT);
}

template <int H> constexpr int row_blocks() { return 65536 / (64 * LineCfg<H>::NTX); }

constexpr int kCols = 16;   // lines per block of the line passes: 128 bytes of neighbours
constexpr int kRows = 8;    // rows per block of the row passes

template <int H> constexpr int kxp() { return H / 2 + 2; }
// shared-memory pitch (float2) of half-spectrum rows in the inverse pass: odd,
// so that lanes reading one element of consecutive rows hit distinct banks
template <int H> constexpr int kxs() { return H / 2 + 1; }
// shared-memory pitch (float2) of rows that are transformed along the row
template <int H> constexpr int rowp() { return H + 1; }

__device__ __forceinline__ int signed_mode(int k, int H) { return k < H / 2 ? k : k - H; }

// Row layout in shared memory for lines transformed along x: position p of
// line t at t PITCH + p + p / R1.  The first stage's lanes write R1 apart (its
// outputs j R1 + r over lanes j), which the pad spreads over the banks; the
// stages whose lanes take consecutive lines (eight, or eight and a few more,
// so two butterflies per 16 lanes) want a pitch of 2 mod 16.
template <int H, int R1> struct RowAt8 {
    static constexpr int LEN = H + H / R1;
    static constexpr int PITCH = LEN + (18 - LEN % 16) % 16;
    __device__ __forceinline__ int operator()(int t, int p) const { return t * PITCH + p + p / R1; }
};

// ---------------------------------------------------------------- pointwise
// int64 (two's complement) deposit accumulator -> float, via the signed high
// and the unsigned low 32-bit halves (the single 64-bit conversion would run
// on the FP64 pipe).
__device__ __forceinline__ float acc_to_float(unsigned long long q) {
    const float hi = __int2float_rn(static_cast<int>(static_cast<unsigned>(q >> 32)));
    const float lo = __uint2float_rn(static_cast<unsigned>(q));
    return fmaf(hi, 4294967296.0f, lo);
}

// R_tau at one node (explicit Euler of S = (-alpha m v; u; gamma v - eta(u) w),
// eta(u) = 2u/(1+u)): m*, w* and v^n.  um is the u of the m source: u itself,
// or K_sigma * u (Eq. m_reg).  The quotients use the hardware reciprocal
// (within 2 ulp): the denominators are at least 1.
__device__ __forceinline__ float react_m(const SpectralArgs& a, float mm, float um) {
    return mm + a.tau * um;
}
__device__ __forceinline__ float react_w(const SpectralArgs& a, float vv, float ww, float u) {
    const float eta = __fdividef(2.0f * u, 1.0f + u);
    return ww + a.tau * (a.gamma * vv - eta * ww);
}
__device__ __forceinline__ float react_v(const SpectralArgs& a, float vv, float mm) {
    return (a.v_update == SIPF_V_IMPLICIT) ? __fdividef(vv, 1.0f + a.alpha * a.tau * mm)
                                           : vv * (1.0f - a.alpha * a.tau * mm);
}

__device__ __forceinline__ void react(const SpectralArgs& a, float vv, float mm, float ww, float u,
                                      float um, float& ms, float& ws, float& vn) {
    ms = mm;
    ws = ww;
    if (a.do_mw) {
        ms = react_m(a, mm, um);
        ws = react_w(a, vv, ww, u);
    }
    vn = react_v(a, vv, mm);
}

// The factor of mode (qx, qy, qz) on the m (field 0) or w (field 1) spectrum.
__device__ __forceinline__ float2 diffuse_mode(const SpectralArgs& a, int field, float q2,
                                               float2 val) {
    const float c = field == 0 ? a.m_c : a.w_c;
    float f = a.diffusion == SIPF_DIFFUSION_IMPLICIT ? __fdividef(1.0f, 1.0f + c * q2)
                                                     : expf(-c * q2);
    if (a.filter) f *= expf(-a.inv_H0sq_2pi2 * q2);
    val = make_float2(f * val.x, f * val.y);
    // times r0 = hi + lo: the float32 rounding of r0 itself is compensated
    const float hi = field == 0 ? a.m_r0_hi : a.w_r0_hi;
    const float lo = field == 0 ? a.m_r0_lo : a.w_r0_lo;
    return make_float2(fmaf(val.x, lo, val.x * hi), fmaf(val.y, lo, val.y * hi));
}

// i k val, zero at the Nyquist mode (q = -H/2 or H/2).
template <int H>
__device__ __forceinline__ float2 times_ik(float scale, int q, float2 val) {
    const float k = (q == H / 2 || q == -H / 2) ? 0.0f : scale * static_cast<float>(q);
    return make_float2(-k * val.y, k * val.x);
}

// The modes of two real signals x1 + i x2 from z(k) and z(-k):
// X1(k) = (z(k) + conj z(-k))/2, X2(k) = (z(k) - conj z(-k))/(2i).
__device__ __forceinline__ void split_modes(float2 zk, float2 zc, float2& x1, float2& x2) {
    x1 = make_float2(0.5f * (zk.x + zc.x), 0.5f * (zk.y - zc.y));
    x2 = make_float2(0.5f * (zk.y + zc.y), -0.5f * (zk.x - zc.x));
}

// ---------------------------------------------------------------- plane pass, forward
// Launch-parameter batches: NB = 1 for one context's step, kMaxBatch for an
// ensemble's runs of one grid size (the run index is a grid dimension).
template <int H, int NB, int V>
__global__ void __launch_bounds__(Cfg<H>::NT1)
    k_forward_xy(const __grid_constant__ SpecBatch<NB> batch) {
    const SpecRun& R = batch.run[NB == 1 ? 0 : blockIdx.y];
    const SpectralArgs& a = R.a;
    const float* v = R.v;
    const float* __restrict__ m = R.m;
    const float* __restrict__ w = R.w;
    unsigned long long* __restrict__ acc = R.acc;
    float* v_out = R.v_out;
    float2* __restrict__ gM = R.specM;
    float2* __restrict__ gW = R.specW;
    float2* __restrict__ gV = R.specV;
    const float2* __restrict__ twg = R.twiddle;
    const float* __restrict__ voff = R.voff;
    const StepScalars* __restrict__ sc = R.sc;
    const float* __restrict__ us = R.us;
    constexpr int NT = Cfg<H>::NT1, KXP = kxp<H>(), HK = H / 2 + 1, RP = rowp<H>();
    pdl_trigger();
    extern __shared__ float2 sm[];
    float2* Z = sm;               // [H][RP]: m* + i w*
    float2* Vb = Z + H * RP;      // v^n: [H/2][RP] row pairs, then [H][KXP] half rows
    float2* tw = Vb + H * KXP;    // [H]
    const int z = blockIdx.x;
    for (int i = threadIdx.x; i < H; i += NT) tw[i] = twg[i];
    pdl_wait();   // the deposit, fields and step scalars of the kernels before
    const float u_scale = sc->u_scale;   // u_bar per accumulator unit
    const size_t plane = static_cast<size_t>(z) * H * H;
    const float c0 = *voff;   // the v spectrum only feeds derivatives: remove a constant
    {
        // node pairs (p, x), (p + H/2, x): consecutive lanes take consecutive x,
        // so the rows of Z and the row pairs of Vb are written without bank
        // conflicts; all loads of a batch are issued first
        constexpr int HH = H / 2, NPR = HH * H, ITER = (NPR + NT - 1) / NT;
        constexpr int CH = ITER < 2 ? ITER : 2;
        const float* vp = v + plane;
        const float* mp = m + plane;
        const float* wp = w + plane;
        unsigned long long* ap = acc + plane;
        float* vo = v_out + plane;
#pragma unroll 1
        for (int i0 = 0; i0 < ITER; i0 += CH) {
            float rv[CH][2], rm[CH][2], rw[CH][2], ru[CH][2];
            unsigned long long ra[CH][2];
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int q = threadIdx.x + (i0 + c) * NT;
                if (i0 + c < ITER && q < NPR) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int o = q + h * NPR;   // (p + h H/2) H + x
                        rv[c][h] = vp[o];
                        rm[c][h] = mp[o];
                        rw[c][h] = wp[o];
                        ra[c][h] = ap[o];
                        ru[c][h] = us ? us[plane + o] : 0.f;
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int q = threadIdx.x + (i0 + c) * NT;
                if (!(i0 + c < ITER && q < NPR)) continue;
                const int pr = q / H, x = q % H;
                float vn[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int o = q + h * NPR;
                    ap[o] = 0ull;
                    float ms, ws;
                    const float u = acc_to_float(ra[c][h]) * u_scale;
                    react(a, rv[c][h], rm[c][h], rw[c][h], u, us ? ru[c][h] : u, ms, ws, vn[h]);
                    Z[(pr + h * HH) * RP + x] = make_float2(ms, ws);
                    if (a.write_v) vo[o] = vn[h];
                }
                Vb[pr * RP + x] = make_float2(vn[0] - c0, vn[1] - c0);
            }
        }
    }
    __syncthreads();
    if (a.do_mw) fft_axis<H, V, H, 1, RP, NT, -1>(Z, tw);
    fft_axis<H, V, H / 2, 1, RP, NT, -1>(Vb, tw);
    {
        // split each transformed row pair z = x1 + i x2 (rows p, p + H/2) into
        // the half rows X1, X2 (kx <= H/2).  X(0) and X(H/2) of a real row are
        // real: column 0 holds X(0) + i X(H/2), so H/2 columns remain
        constexpr int HH = H / 2, NS = HH * HH, SPT = (NS + NT - 1) / NT;
        float2 x1[SPT], x2[SPT];
#pragma unroll
        for (int s = 0; s < SPT; ++s) {
            const int idx = threadIdx.x + s * NT;
            if (idx < NS) {
                const int p = idx / HH, k = idx % HH;
                const float2 zp = Vb[p * RP + k];
                const float2 zm = Vb[p * RP + (k == 0 ? HH : H - k)];
                if (k == 0) {
                    // zm is z(H/2) here: X1(0) = Re z(0), X1(H/2) = Re z(H/2), X2 from Im
                    x1[s] = make_float2(zp.x, zm.x);
                    x2[s] = make_float2(zp.y, zm.y);
                } else {
                    x1[s] = make_float2(0.5f * (zp.x + zm.x), 0.5f * (zp.y - zm.y));
                    x2[s] = make_float2(0.5f * (zp.y + zm.y), -0.5f * (zp.x - zm.x));
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < SPT; ++s) {
            const int idx = threadIdx.x + s * NT;
            if (idx < NS) {
                const int p = idx / HH, k = idx % HH;
                Vb[p * KXP + k] = x1[s];
                Vb[(p + HH) * KXP + k] = x2[s];
            }
        }
        __syncthreads();
    }
    if (a.do_mw) fft_axis<H, V, H, RP, 1, NT, -1>(Z, tw);
    fft_axis<H, V, H / 2, KXP, 1, NT, -1>(Vb, tw);
    // half spectra, rows of KXP (the last slot, kx = H/2 + 1, is zero); M, W
    // separated from the 2D spectrum of m* + i w*; one mode per thread
    constexpr int NP = H * KXP;
    const size_t sbase = static_cast<size_t>(z) * H * KXP;
    for (int idx = threadIdx.x; idx < NP; idx += NT) {
        const int ky = idx / KXP, k = idx % KXP;
        float2 M = make_float2(0.f, 0.f), W = M, Vk = M;
        if (k < HK) {
            const float2 zk = Z[ky * RP + k];
            const float2 zc = Z[neg_mod<H>(ky) * RP + neg_mod<H>(k)];
            M = make_float2(0.5f * (zk.x + zc.x), 0.5f * (zk.y - zc.y));
            W = make_float2(0.5f * (zk.y + zc.y), -0.5f * (zk.x - zc.x));
            if (k == 0 || k == H / 2) {
                // the packed column P = V(0, .) + i V(H/2, .): V(0, ky) =
                // (P(ky) + conj P(-ky))/2, V(H/2, ky) = (P(ky) - conj P(-ky))/(2i)
                const float2 pk = Vb[ky * KXP], pc = Vb[neg_mod<H>(ky) * KXP];
                Vk = k == 0 ? make_float2(0.5f * (pk.x + pc.x), 0.5f * (pk.y - pc.y))
                            : make_float2(0.5f * (pk.y + pc.y), -0.5f * (pk.x - pc.x));
            } else {
                Vk = Vb[ky * KXP + k];
            }
        }
        if (a.do_mw) {
            gM[sbase + idx] = M;
            gW[sbase + idx] = W;
        }
        gV[sbase + idx] = Vk;
    }
}

// ---------------------------------------------------------------- line pass (z)
// Block (tile, field): kCols neighbouring columns (ky, kx) of a half spectrum,
// in flat order over the plane: forward DFT along z, the factor, inverse DFT.
// Field 0 M, 1 W: the implicit (or exponential) diffusion factor; 2: i k_z V
// -> B; 3 (with the low-pass filter) the filtered V -> A.  A tile's rows are whole
// 128-byte lines (a plane has H (H/2 + 2) columns, a multiple of 16, whatever
// the row pitch), its 16 H complex numbers take 16 KB at H = 128, so many
// small blocks share an SM, their loads, exchanges and stores overlap, and
// the last wave is short.  Bound by the latency of the loads and the
// exchanges.  One block per ky row and field of 544 threads and 68 KB before:
// 22.9 -> 18.3 us per pass at 128^3, 152 -> 91 us at 256^3.
template <int H> struct LineShape {
    static constexpr int TC = H * kxp<H>() / kCols;        // tiles of one half spectrum
    static constexpr size_t bytes = (static_cast<size_t>(H) * kCols + H) * sizeof(float2);
    static_assert(H * kxp<H>() % kCols == 0, "whole tiles");
};

template <int H, int NB, int V>
__global__ void __launch_bounds__(LineCfg<H>::NT, line_blocks<H>())
    k_lines_z(const __grid_constant__ SpecBatch<NB> batch, int field0) {
    const SpecRun& R = batch.run[NB == 1 ? 0 : blockIdx.z];
    const SpectralArgs& a = R.a;
    constexpr int NT = LineCfg<H>::NT, KXP = kxp<H>();
    extern __shared__ float2 sm[];
    float2* buf = sm;                          // [H][kCols]
    float2* tw = buf + H * kCols;              // [H]
    pdl_trigger();
    for (int i = threadIdx.x; i < H; i += NT) tw[i] = R.twiddle[i];
    __syncthreads();
    pdl_wait();   // the forward pass's spectra
    const int field = field0 + blockIdx.y;
    const int col = blockIdx.x * kCols + threadIdx.x % kCols;
    const int ky = col / KXP, qx = col % KXP, qy = signed_mode(ky, H);
    const float2* src = (field == 0 ? R.specM : field == 1 ? R.specW : R.specV) + col;
    float2* dst = (field == 0 ? R.specM : field == 1 ? R.specW
                  : field == 2 ? R.specB : R.specA) + col;
    const int q2xy = qx * qx + qy * qy;
    float* voff = R.voff;
    round_trip<H, V, kCols, NT>(
        buf, tw, Strided<1, kCols>{},
        [=](int, int zz) { return src[static_cast<size_t>(zz) * (H * KXP)]; },
        [=](int, int kz, float2 val) {
            const int qz = signed_mode(kz, H);
            const float q2 = static_cast<float>(q2xy + qz * qz);
            if (field < 2) return diffuse_mode(a, field, q2, val);
            if (field == 2) {
                // DC of (v^n - c0): move the offset to the mean of v^n for the next step
                if (col == 0 && kz == 0) *voff = *voff + val.x * a.out_scale;
                val = times_ik<H>(a.two_pi_over_L, qz, val);
            }
            if (a.filter) {
                const float f = expf(-a.inv_H0sq_2pi2 * q2);
                val = make_float2(f * val.x, f * val.y);
            }
            return val;
        },
        [=](int, int zz, float2 val) { dst[static_cast<size_t>(zz) * (H * KXP)] = val; });
}

// ---------------------------------------------------------------- plane pass, inverse
// Build the full-length complex row Z[kx] = X1[kx] + i X2[kx] of two real
// signals from their half spectra (Hermitian extension, C2R semantics at
// kx = 0 and kx = H/2).
template <int H>
__device__ __forceinline__ float2 pack_two(const float2* r1, const float2* r2, int kx) {
    float2 a, b;
    if (kx <= H / 2) {
        a = r1[kx];
        b = r2[kx];
        if (kx == 0 || kx == H / 2) {
            a.y = 0.f;
            b.y = 0.f;
        }
    } else {
        a = conjf2(r1[H - kx]);
        b = conjf2(r2[H - kx]);
    }
    return make_float2(a.x - b.y, a.y + b.x);
}

// Loaders for the fused first stages of the inverse pass.
struct PlaneLoad {      // half-spectrum plane from global memory, optionally times i k
    const float2* p;
    int kxp;
    float kx_scale, ky_scale;   // 2 pi / L, or 0 for "no multiplier"
    int H, dir;                 // dir 0: plain, 1: i k_x, 2: i k_y
    __device__ __forceinline__ float2 operator()(int kx, int ky) const {
        const float2 val = __ldg(p + static_cast<size_t>(ky) * kxp + kx);
        if (dir == 0) return val;
        float k;
        if (dir == 1) {
            k = (kx >= H / 2) ? 0.0f : kx_scale * static_cast<float>(kx);
        } else {
            const int qy = ky < H / 2 ? ky : ky - H;
            k = (qy == -H / 2) ? 0.0f : ky_scale * static_cast<float>(qy);
        }
        return make_float2(-k * val.y, k * val.x);
    }
};

template <int H>
struct PackLoad {       // complex row of two real signals from their half spectra
    const float2* r1;
    const float2* r2;
    int pitch1, pitch2;         // row pitch (float2) of the two sources
    __device__ __forceinline__ float2 operator()(int row, int kx) const {
        return pack_two<H>(r1 + row * pitch1, r2 + row * pitch2, kx);
    }
};

// group 1: (i k_x V, i k_y V, B) -> grad v^n; group 0: (m, w) -> m^n, w^n.
// The first inverse-y stage reads the planes straight from global memory and
// the first inverse-x stage reads the packed rows straight from the y output.
template <int H, int NB, int V>
__global__ void __launch_bounds__(Cfg<H>::NT3)
    k_inverse_xy(const __grid_constant__ SpecBatch<NB> batch) {
    const SpecRun& R = batch.run[NB == 1 ? 0 : blockIdx.z];
    const SpectralArgs& a = R.a;
    const float2* __restrict__ gM = R.specM;
    const float2* __restrict__ gW = R.specW;
    const float2* __restrict__ gV = a.filter ? R.specA : R.specV;
    const float2* __restrict__ gB = R.specB;
    float* __restrict__ m_out = R.m_out;
    float* __restrict__ w_out = R.w_out;
    float* __restrict__ G = R.G;
    const float2* __restrict__ twg = R.twiddle;
    constexpr int NT = Cfg<H>::NT3, KXP = kxp<H>(), KXS = kxs<H>(), HK = H / 2 + 1;
    constexpr int RP = rowp<H>(), R1 = Radix<H, V>::R1;
    static_assert(H * RP <= 2 * H * KXS, "packed rows must fit in B0/B1");
    static_assert((H / 2) * RP <= H * KXS, "packed row pairs must fit in B2");
    extern __shared__ float2 sm[];
    float2* B0 = sm;              // [H][KXS]
    float2* B1 = B0 + H * KXS;    // [H][KXS]
    float2* B2 = B1 + H * KXS;    // [H][KXS] (group 1)
    float2* tw = B2 + H * KXS;
    float2* Z = sm;               // [H][RP] packed rows (aliases B0/B1)
    float2* Z2 = B2;              // [H/2][RP] rows y, y + H/2 of B2 packed (aliases B2)
    // the two groups of a plane are neighbouring blocks: their partial writes
    // of the gather array's nodes (x, y, z components, then w) follow each
    // other closely, while the lines are still in L2
    const int z = blockIdx.x >> 1, group = 1 - static_cast<int>(blockIdx.x & 1);
    pdl_trigger();
    if (group == 0 && !a.do_mw) return;
    for (int i = threadIdx.x; i < H; i += NT) tw[i] = twg[i];
    __syncthreads();
    pdl_wait();   // the z pass's spectra
    const size_t pbase = static_cast<size_t>(z) * H * KXP;
    // inverse y: first stage from global, second in shared memory
    if (group == 0) {
        stage1_from<H, R1, HK, KXS, 1, NT, +1>(B0, PlaneLoad{gM + pbase, KXP, 0.f, 0.f, H, 0});
        stage1_from<H, R1, HK, KXS, 1, NT, +1>(B1, PlaneLoad{gW + pbase, KXP, 0.f, 0.f, H, 0});
    } else {
        const float k = a.two_pi_over_L;
        stage1_from<H, R1, HK, KXS, 1, NT, +1>(B0, PlaneLoad{gV + pbase, KXP, k, k, H, 1});
        stage1_from<H, R1, HK, KXS, 1, NT, +1>(B1, PlaneLoad{gV + pbase, KXP, k, k, H, 2});
        stage1_from<H, R1, HK, KXS, 1, NT, +1>(B2, PlaneLoad{gB + pbase, KXP, 0.f, 0.f, H, 0});
    }
    fft_rest<H, V, HK, KXS, 1, NT, +1>(B0, tw);
    fft_rest<H, V, HK, KXS, 1, NT, +1>(B1, tw);
    if (group == 1) fft_rest<H, V, HK, KXS, 1, NT, +1>(B2, tw);
    // inverse x: first stage from the packed half spectra (in place), second stage
    if (group == 1) {
        // B2's rows y and y + H/2 as one complex row -> Z2 (B2's own space); done
        // first, B0/B1 are still intact
        stage1_from<H, R1, H / 2, 1, RP, NT, +1>(Z2,
                                                  PackLoad<H>{B2, B2 + (H / 2) * KXS, KXS, KXS});
    }
    stage1_from<H, R1, H, 1, RP, NT, +1>(Z, PackLoad<H>{B0, B1, KXS, KXS});
    fft_rest<H, V, H, 1, RP, NT, +1>(Z, tw);
    if (group == 1) fft_rest<H, V, H / 2, 1, RP, NT, +1>(Z2, tw);
    const size_t plane = static_cast<size_t>(z) * H * H;
    float* Gp = G + 4 * plane;
    if (group == 0) {
        // m^n, w^n, and w^n again as the fourth component of the gather array
        // (consecutive lanes read consecutive x: no bank conflicts)
        const float sc = a.out_scale;
        float* p1 = m_out + plane;
        float* p2 = w_out + plane;
        for (int i = threadIdx.x; i < H * H; i += NT) {
            const int y = i / H, x = i % H;
            const float2 e = Z[y * RP + x];
            const float wv = e.y * sc;
            p1[i] = e.x * sc;
            p2[i] = wv;
            Gp[4 * i + 3] = wv;
        }
    } else {
        // (dv/dx, dv/dy, dv/dz) into components 0..2 of the gather array
        const float sxy = a.out_scale_xy, sz_ = a.out_scale;
        for (int i = threadIdx.x; i < H * H; i += NT) {
            const int y = i / H, x = i % H;
            const float2 e = Z[y * RP + x];
            const bool upper = y >= H / 2;
            const float2 f = Z2[(upper ? y - H / 2 : y) * RP + x];
            *reinterpret_cast<float2*>(Gp + 4 * i) = make_float2(e.x * sxy, e.y * sxy);
            Gp[4 * i + 2] = (upper ? f.y : f.x) * sz_;
        }
    }
}

// X1 + i X2 of two real signals at mode k from their half spectra a(k') and
// b(k') at k' = min(k, H - k) (C2R semantics at k = 0 and k = H/2).
template <int H>
__device__ __forceinline__ float2 pack_modes(float2 a, float2 b, int k) {
    if (k > H / 2) {
        a.y = -a.y;
        b.y = -b.y;
    } else if (k == 0 || k == H / 2) {
        a.y = 0.f;
        b.y = 0.f;
    }
    return make_float2(a.x - b.y, a.y + b.x);
}

// ---------------------------------------------------------------- line pass (y)
// For the per-axis pipeline: y DFT of kCols lines of the half spectra.  Tiles
// of kCols neighbouring columns kx < H/2 of one plane, then tiles of the kx =
// H/2 columns of kCols planes (which would otherwise cost every plane a tile
// of one column).  SIGN -1: families 0 M, 1 W, 2 V in place.  SIGN +1: 0
// M, 1 W, 2 B in place, V (or its filtered copy) -> 3 i k_x V, 4 i k_y V.
template <int H> struct YTiles {
    static constexpr int PER = (H / 2 + kCols - 1) / kCols;             // per plane
    static constexpr int ALL = H * PER + (H + kCols - 1) / kCols;
};

template <int H, int SIGN, int V>
__global__ void __launch_bounds__(LineCfg<H>::NT)
    k_lines_y(const __grid_constant__ SpecBatch<1> batch, int family0) {
    const SpecRun& R = batch.run[0];
    const SpectralArgs& a = R.a;
    constexpr int NT = LineCfg<H>::NT, KXP = kxp<H>(), HH = H / 2, PER = YTiles<H>::PER;
    extern __shared__ float2 sm[];
    float2* buf = sm;
    float2* tw = buf + H * kCols;
    for (int i = threadIdx.x; i < H; i += NT) tw[i] = R.twiddle[i];
    __syncthreads();
    const int tile = blockIdx.x, t0 = threadIdx.x % kCols;
    int z, k;
    bool in;
    if (tile < H * PER) {
        z = tile / PER;
        k = (tile % PER) * kCols + t0;
        in = k < HH;
    } else {
        z = (tile - H * PER) * kCols + t0;
        k = HH;
        in = z < H;
    }
    const int family = family0 + blockIdx.y;
    const size_t base = static_cast<size_t>(z) * H * KXP + k;
    const float2* src = (family == 0 ? R.specM : family == 1 ? R.specW
                        : family == 2 ? (SIGN < 0 ? R.specV : R.specB)
                        : a.filter ? R.specA : R.specV) + base;
    float2* dst = (family == 0 ? R.specM : family == 1 ? R.specW
                  : family == 2 ? (SIGN < 0 ? R.specV : R.specB)
                  : family == 3 ? R.specDx : R.specDy) + base;
    const float ks = a.two_pi_over_L;
    one_way<H, V, kCols, NT, SIGN>(
        buf, tw, Strided<1, kCols>{},
        [=](int, int y) {
            if (!in) return make_float2(0.f, 0.f);
            float2 x = src[y * KXP];
            if (SIGN > 0 && family >= 3)
                x = times_ik<H>(ks, family == 3 ? k : signed_mode(y, H), x);
            return x;
        },
        [=](int, int y, float2 val) {
            if (in) dst[y * KXP] = val;
        });
}

// ---------------------------------------------------------------- row passes
// x transforms of kRows complex rows for the per-axis pipeline.  Forward, by
// MODE: 0 (radix plan 2) m* + i w* of kRows rows; 1 pairs of neighbouring rows
// (2p, 2p + 1) of m*, then of w*; 2, 3 pairs of rows of v^n - c0, (2p, 2p + 1) or
// (radix plan 2) (y, y + H/2).  Modes 0 and 1 store v^n and clear the deposit
// accumulator; 2 and 3 follow them in a launch of their own, which reads v^n
// again but keeps every thread busy (v^n within the first launch left half
// the threads idle: 207 us against 128 + 24 at 256^3).  Out: the half rows (kx <= H/2)
// of M and W, or of V.  The loads feed the first stage in registers.  Bound by
// DRAM (60 bytes per node and 12 per mode at 256^3 and above).
template <int H, int V> struct RowShape {
    static constexpr int R1 = Radix<H, V>::R1;
    using At = RowAt8<H, R1>;
    static constexpr int Z = kRows * At::PITCH;
    static constexpr size_t bytes = (static_cast<size_t>(Z) + H) * sizeof(float2);
};

template <int H, int V, int MODE>
__global__ void __launch_bounds__(LineCfg<H>::NTX, row_blocks<H>())
    k_rows_forward(const __grid_constant__ SpecBatch<1> batch) {
    const SpecRun& R = batch.run[0];
    const SpectralArgs& a = R.a;
    using S = RowShape<H, V>;
    constexpr int NT = LineCfg<H>::NTX, KXP = kxp<H>(), HH = H / 2, R1 = S::R1, NJ = H / R1;
    constexpr int KP = kRows / 2;
    extern __shared__ float2 sm[];
    float2* Z = sm;                              // [kRows][PITCH]
    float2* tw = Z + S::Z;
    for (int i = threadIdx.x; i < H; i += NT) tw[i] = R.twiddle[i];
    // first row, flat over (z, y); the V modes take kRows row pairs
    constexpr bool VV = MODE >= 2;
    constexpr int PAIR = MODE == 3 ? HH : 1;     // distance of the two rows of a pair
    constexpr int STEP = MODE == 0 || MODE == 3 ? 1 : 2;   // rows from one complex row to the next
    constexpr int VB = HH / kRows;               // mode 3: blocks per plane
    const size_t row0 = MODE == 3 ? static_cast<size_t>(blockIdx.x / VB) * H + (blockIdx.x % VB) * kRows
                                  : static_cast<size_t>(blockIdx.x) * (MODE == 2 ? 2 * kRows : kRows);
    const float u_scale = R.sc->u_scale;
    const float c0 = VV ? *R.voff : 0.0f;   // that spectrum only feeds derivatives
    const float* v = R.v + row0 * H;
    const float* m = R.m + row0 * H;
    const float* w = R.w + row0 * H;
    unsigned long long* acc = R.acc + row0 * H;
    const float* us = R.us ? R.us + row0 * H : nullptr;
    float* vo = R.v_out + row0 * H;
    constexpr int CH = MODE == 0 ? (R1 % 4 == 0 ? 4 : 2) : 2;
    static_assert(R1 % CH == 0, "whole chunks");
    constexpr int NR = MODE == 0 ? 1 : 2;        // real rows per complex row
#pragma unroll 1
    for (int b = threadIdx.x; b < kRows * NJ; b += NT) {
        const int t = b / NJ, j = b % NJ;
        const int row = STEP * (MODE == 1 ? t % KP : t);
        const bool want_w = MODE == 0 || (MODE == 1 && t >= KP);   // w* and v^n
        float2 val[R1];
#pragma unroll
        for (int r0 = 0; r0 < R1; r0 += CH) {
            // all loads of a chunk before its stores
            float rv[CH][NR], rm[CH][NR], rw[CH][NR], ru[CH][NR];
            unsigned long long ra[CH][NR];
#pragma unroll
            for (int c = 0; c < CH; ++c) {
#pragma unroll
                for (int h = 0; h < NR; ++h) {
                    const int o = (row + h * PAIR) * H + j + (r0 + c) * NJ;
                    rv[c][h] = rm[c][h] = rw[c][h] = ru[c][h] = 0.f;
                    ra[c][h] = 0ull;
                    if (VV) {
                        rv[c][h] = vo[o];
                    } else {
                        rm[c][h] = m[o];
                        ra[c][h] = acc[o];
                        if (us) ru[c][h] = us[o];
                        if (want_w) {
                            rv[c][h] = v[o];
                            rw[c][h] = w[o];
                        }
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                float out[2];
#pragma unroll
                for (int h = 0; h < NR; ++h) {
                    const int o = (row + h * PAIR) * H + j + (r0 + c) * NJ;
                    const float u = acc_to_float(ra[c][h]) * u_scale;
                    const float um = us ? ru[c][h] : u;
                    if (MODE == 0) {
                        out[0] = react_m(a, rm[c][h], um);
                        out[1] = react_w(a, rv[c][h], rw[c][h], u);
                    } else if (MODE == 1) {
                        out[h] = want_w ? react_w(a, rv[c][h], rw[c][h], u)
                                        : react_m(a, rm[c][h], um);
                    } else {
                        out[h] = rv[c][h] - c0;
                    }
                    if (!VV && want_w) vo[o] = react_v(a, rv[c][h], rm[c][h]);
                }
                val[r0 + c] = make_float2(out[0], out[1]);
            }
        }
        dft<R1, -1>(val);
#pragma unroll
        for (int r = 0; r < R1; ++r) Z[t * S::At::PITCH + j * (R1 + 1) + r] = val[r];
    }
    __syncthreads();
    if (!VV) {
        ulonglong2* q = reinterpret_cast<ulonglong2*>(acc);
        for (int i = threadIdx.x; i < kRows * H / 2; i += NT) q[i] = make_ulonglong2(0ull, 0ull);
    }
    const typename S::At at{};
    fft_rest_at<H, V, kRows, NT, -1>(Z, tw, at);
    for (int q = threadIdx.x; q < kRows * HH; q += NT) {
        const int t = q / HH, k = q % HH;
        float2* d1;
        float2* d2;
        if (MODE == 0) {
            d1 = R.specM + (row0 + t) * KXP;
            d2 = R.specW + (row0 + t) * KXP;
        } else {
            d1 = (VV ? R.specV + (row0 + STEP * t) * KXP
                     : (t < KP ? R.specM : R.specW) + (row0 + STEP * (t % KP)) * KXP);
            d2 = d1 + PAIR * KXP;
        }
        float2 x1, x2;
        split_modes(Z[at(t, k)], Z[at(t, k == 0 ? 0 : H - k)], x1, x2);
        d1[k] = x1;
        d2[k] = x2;
        if (k == 0) {
            const float2 zn = Z[at(t, HH)];
            split_modes(zn, zn, x1, x2);
            d1[HH] = x1;
            d2[HH] = x2;
        }
    }
}

// Inverse: two half rows to two real rows per complex transform, kRows
// transforms per block.  Five neighbouring blocks cover 2 kRows rows: two take
// (m, w) rows, two (dv/dx, dv/dy) rows, one dv/dz row pairs, so that the components of
// a node of the gather array are written close together in time, while its
// line is in L2.  PAIRH: the 2 kRows rows are y0 .. y0 + 7 and the same + H/2,
// paired across (radix plan 2); else consecutive, paired (2p, 2p + 1).  Half
// rows feed the first stage in registers and the last stage, its lanes along x,
// stores to global memory.  (One block for all 20 transforms of 8 rows, storing whole
// nodes from shared memory, took 234 us at 256^3
// and 976 us at 384^3, against 169 and 523.)
template <int H, int V, bool PAIRH>
__global__ void __launch_bounds__(LineCfg<H>::NTX, row_blocks<H>())
    k_rows_inverse(const __grid_constant__ SpecBatch<1> batch) {
    const SpecRun& R = batch.run[0];
    const SpectralArgs& a = R.a;
    using S = RowShape<H, V>;
    using P = Radix<H, V>;
    constexpr int NT = LineCfg<H>::NTX, KXP = kxp<H>(), HH = H / 2;
    extern __shared__ float2 sm[];
    float2* Z = sm;                              // [kRows][PITCH]
    float2* tw = Z + S::Z;
    const int group = blockIdx.x / 5, part = blockIdx.x % 5;
    const int kind = part < 2 ? 0 : part < 4 ? 1 : 2;
    if (kind == 0 && !a.do_mw) return;           // a state's initial gradient: no m, w
    for (int i = threadIdx.x; i < H; i += NT) tw[i] = R.twiddle[i];
    __syncthreads();
    constexpr int VB = HH / kRows;
    const size_t g0 = PAIRH ? static_cast<size_t>(group / VB) * H + (group % VB) * kRows
                            : static_cast<size_t>(group) * (2 * kRows);   // flat over (z, y)
    const size_t row0 = g0 + (kind == 2 ? 0 : (part & 1) * (PAIRH ? HH : kRows));
    constexpr int PAIR = PAIRH ? HH : 1;
    const int step = kind == 2 && !PAIRH ? 2 : 1;        // rows from one transform to the next
    const float2* s1 = (kind == 0 ? R.specM : kind == 1 ? R.specDx : R.specB) + row0 * KXP;
    const float2* s2 = kind == 0 ? R.specW + row0 * KXP
                     : kind == 1 ? R.specDy + row0 * KXP : s1 + PAIR * KXP;
    const typename S::At at{};
    auto sload = [=](int t, int p) { return Z[at(t, p)]; };
    auto sstore = [=](int t, int p, float2 val) { Z[at(t, p)] = val; };
    stage_ls<H, S::R1, 1, kRows, NT, +1, true, false>(
        tw,
        [=](int t, int kx) {
            const int k = kx <= HH ? kx : H - kx;
            return pack_modes<H>(s1[t * step * KXP + k], s2[t * step * KXP + k], kx);
        },
        sstore);
    __syncthreads();
    if constexpr (P::R3 > 1) {
        stage_ls<H, P::R2, S::R1, kRows, NT, +1, false, true>(tw, sload, sstore);
        __syncthreads();
    }
    if constexpr (P::R4 > 1) {
        stage_ls<H, P::R3, S::R1 * P::R2, kRows, NT, +1, false, true>(tw, sload, sstore);
        __syncthreads();
    }
    constexpr int RL = P::R4 > 1 ? P::R4 : P::R3 > 1 ? P::R3 : P::R2;
    const float sc = a.out_scale, sxy = a.out_scale_xy;
    float* m_out = R.m_out + row0 * H;
    float* w_out = R.w_out + row0 * H;
    float* G = R.G + 4 * row0 * H;
    stage_ls<H, RL, H / RL, kRows, NT, +1, true, false>(
        tw, sload, [=](int t, int x, float2 val) {
            const int o = t * step * H + x;
            if (kind == 0) {
                const float wv = val.y * sc;
                m_out[o] = val.x * sc;
                w_out[o] = wv;
                G[4 * o + 3] = wv;
            } else if (kind == 1) {
                *reinterpret_cast<float2*>(G + 4 * o) = make_float2(val.x * sxy, val.y * sxy);
            } else {
                G[4 * o + 2] = val.x * sc;
                G[4 * (o + PAIR * H) + 2] = val.y * sc;
            }
        });
}

// ---------------------------------------------------------------- launches
template <class K>
void allow_smem(K kernel, size_t bytes) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         static_cast<int>(bytes));
}

// Shared memory of the plane passes.
template <int H> struct FusedSmem {
    static constexpr size_t fwd = (static_cast<size_t>(H) * rowp<H>() + H * kxp<H>() + H) * sizeof(float2);
    static constexpr size_t inv = (3 * static_cast<size_t>(H) * kxs<H>() + H) * sizeof(float2);
};

// One fused pass over a batch of nb runs of grid size H <= 128: 0 forward
// planes, 1 z lines, 2 inverse planes.
template <int H, int NB, int V>
cudaError_t fused_pass(const SpecBatch<NB>& batch, int nb, int pass, int device, cudaStream_t s) {
    static int configured_device = -1;   // attributes are set once per process and device
    if (configured_device != device) {
        allow_smem(k_forward_xy<H, NB, V>, FusedSmem<H>::fwd);
        allow_smem(k_lines_z<H, NB, V>, LineShape<H>::bytes);
        allow_smem(k_inverse_xy<H, NB, V>, FusedSmem<H>::inv);
        configured_device = device;
    }
    const SpectralArgs& a = batch.run[0].a;   // a batch of several: full steps without the filter
    if (pass == 0)
        return launch_pdl(k_forward_xy<H, NB, V>, dim3(H, nb), dim3(Cfg<H>::NT1),
                          FusedSmem<H>::fwd, s, batch);
    if (pass == 1) {
        const int f0 = a.do_mw ? 0 : 2, f1 = a.filter ? 4 : 3;
        return launch_pdl(k_lines_z<H, NB, V>, dim3(LineShape<H>::TC, f1 - f0, nb),
                          dim3(LineCfg<H>::NT), LineShape<H>::bytes, s, batch, f0);
    }
    return launch_pdl(k_inverse_xy<H, NB, V>, dim3(2 * H, 1, nb), dim3(Cfg<H>::NT3),
                      FusedSmem<H>::inv, s, batch);
}

// One fused pass over n runs (n = 1: the batch-of-one instantiation).
template <int H, int V>
cudaError_t fused_runs(const SpecRun* runs, int n, int pass, int device, cudaStream_t s) {
    if (n == 1) {
        SpecBatch<1> one;
        one.run[0] = runs[0];
        return fused_pass<H, 1, V>(one, 1, pass, device, s);
    }
    SpecBatch<kMaxBatch> batch;
    for (int i = 0; i < n; ++i) batch.run[i] = runs[i];
    return fused_pass<H, kMaxBatch, V>(batch, n, pass, device, s);
}

// Passes of the per-axis pipeline, grouped like the fused ones: 0 forward
// (x, y), 1 z, 2 inverse (y, x).  PLAN2: how rows are packed and paired.  Ordinary
// launches: with programmatic ones the plan kernel on the second stream kept
// the passes waiting (256^3: 1.49 against 1.31 ms per step).
template <int H, int V, bool PLAN2>
cudaError_t axis_pass(const SpecRun& run, int pass, int device, cudaStream_t s) {
    using L = LineShape<H>;
    using X = RowShape<H, V>;
    constexpr int MW = PLAN2 ? 0 : 1, VV = PLAN2 ? 3 : 2;
    static int configured_device = -1;
    if (configured_device != device) {
        allow_smem(k_rows_forward<H, V, MW>, X::bytes);
        allow_smem(k_rows_forward<H, V, VV>, X::bytes);
        allow_smem(k_rows_inverse<H, V, PLAN2>, X::bytes);
        allow_smem(k_lines_y<H, -1, V>, L::bytes);
        allow_smem(k_lines_y<H, +1, V>, L::bytes);
        allow_smem(k_lines_z<H, 1, V>, L::bytes);
        configured_device = device;
    }
    SpecBatch<1> one;
    one.run[0] = run;
    const SpectralArgs& a = run.a;
    const dim3 nx(LineCfg<H>::NTX), nl(LineCfg<H>::NT);
    const unsigned rows = H * H / kRows;
    const int f0 = a.do_mw ? 0 : 2;
    if (pass == 0) {
        if (a.do_mw) k_rows_forward<H, V, MW><<<rows, nx, X::bytes, s>>>(one);
        k_rows_forward<H, V, VV><<<rows / 2, nx, X::bytes, s>>>(one);
        k_lines_y<H, -1, V><<<dim3(YTiles<H>::ALL, 3 - f0), nl, L::bytes, s>>>(one, f0);
    } else if (pass == 1) {
        const int f1 = a.filter ? 4 : 3;
        k_lines_z<H, 1, V><<<dim3(L::TC, f1 - f0), nl, L::bytes, s>>>(one, f0);
    } else {
        k_lines_y<H, +1, V><<<dim3(YTiles<H>::ALL, 5 - f0), nl, L::bytes, s>>>(one, f0);
        k_rows_inverse<H, V, PLAN2><<<rows / 2 * 5, nx, X::bytes, s>>>(one);
    }
    return cudaGetLastError();
}

}  // namespace
}  // namespace sipf
