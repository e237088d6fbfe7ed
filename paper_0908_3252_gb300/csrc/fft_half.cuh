// fft_half.cuh -- transforms of M = 256 and 512 points with at most M / 2 nonzero
// inputs or kept outputs, as 256-point DFTs of half a warp each: a sequence a
// half-warp at M = 256; at M = 512 a warp, which half the even and which the odd
// frequencies.  Lane l of half h of a warp, 16 values a lane.
#pragma once

#include "fft_reg.cuh"
#include "phase.cuh"

namespace spirec {
namespace fftd {

constexpr int kHalfArea = 16 * 17;   // exchange area of a half-warp
constexpr int kHalfTables = 512;     // T256[k1][l] = w256^(l k1), then w512^n (M = 512)

template <int MC>
__host__ __device__ constexpr bool half_warp_size() { return MC == 256 || MC == 512; }

// The tables from tw (w_M^k), by the whole block; the caller synchronises.
template <int MC>
__device__ __forceinline__ void half_tables(float2* t, const float2* __restrict__ tw)
{
    for (int e = threadIdx.x; e < 256; e += blockDim.x) {
        t[e] = __ldg(tw + (MC / 256) * (e & 15) * (e >> 4));
        if (MC == 512) t[256 + e] = __ldg(tw + e);
    }
}

// The 256-point DFT (conjugate twiddles when INV) of the sequence whose element
// l + 16 j is in x[j] of lane l of a half-warp, both halves of the warp a
// sequence each: DFT16 over the registers, twiddles w256^(l k1) from t, an
// exchange through the half-warp's area (16 x 17), DFT16 over the registers.
// Element l + 16 k of the result ends in x[k].  HALF_IN: x[8 ..] is zero.
template <bool INV, bool HALF_IN>
__device__ __forceinline__ void fft256(float2 (&x)[16], float2* area, const float2* t, int l)
{
    freg::dft16_dif<INV, HALF_IN>(x);
#pragma unroll
    for (int k1 = 0; k1 < 16; ++k1) {
        const float2 w = t[k1 * 16 + l];
        area[k1 * 17 + l] = cmul(x[freg::bitrev4(k1)], INV ? conjf2(w) : w);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = area[l * 17 + i];
    __syncwarp();
    freg::dft16_dif<INV>(x);
#pragma unroll
    for (int k = 0; k < 16; ++k) {  // bit-reversed order to the natural one (a renaming)
        const int b = freg::bitrev4(k);
        if (k < b) {
            const float2 v = x[k];
            x[k] = x[b];
            x[b] = v;
        }
    }
}

// Forward transform of a sequence of M = MC points whose elements n < N <= M / 2
// are load(n) (zero beyond, and all when N = 0): frequency half_freq(k) = l + 16 k
// (M = 256) or 2 (l + 16 k) + h (M = 512, half h: DFT256 of x w512^(h n)) in x[k].
template <int MC, typename F>
__device__ __forceinline__ void half_fwd(float2 (&x)[16], F&& load, int N, float2* area, const float2* t, int l, int h)
{
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        if (MC == 256 && j >= 8) break;
        const int n = l + 16 * j;
        x[j] = n < N ? load(n) : make_float2(0.f, 0.f);
    }
    __syncwarp();  // the exchange areas may lie where the inputs do
    if (MC == 512 && h)
#pragma unroll
        for (int j = 0; j < 16; ++j) x[j] = cmul(x[j], t[256 + l + 16 * j]);
    fft256<false, MC == 256>(x, area, t, l);
}

template <int MC>
__device__ __forceinline__ int half_freq(int l, int h, int k)
{
    return MC == 512 ? 2 * (l + 16 * k) + h : l + 16 * k;
}

// The inverse of half_fwd's order: out[i], i < 8, is element l + 16 i (M = 256) or
// l + 16 (8 h + i) (M = 512: u_0 + w512^(-n) u_1, the halves of the warp handing
// each other what the other needs) of the transform, n < M / 2.
template <int MC>
__device__ __forceinline__ void half_inv(float2 (&x)[16], float2 (&out)[8], float2* area, const float2* t, int l, int h)
{
    fft256<true, false>(x, area, t, l);
    if constexpr (MC == 256) {
#pragma unroll
        for (int i = 0; i < 8; ++i) out[i] = x[i];
    } else {
        if (h)
#pragma unroll
            for (int k = 0; k < 16; ++k) x[k] = cmul(x[k], conjf2(t[256 + l + 16 * k]));
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 give = h ? x[i] : x[8 + i], keep = h ? x[8 + i] : x[i];
            const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, give.x, 16), __shfl_xor_sync(0xffffffffu, give.y, 16));
            out[i] = freg::add(keep, got);
        }
    }
}

template <int MC>
__device__ __forceinline__ int half_elem(int l, int h, int i)
{
    return l + 16 * (MC == 512 ? 8 * h + i : i);
}

}  // namespace fftd
}  // namespace spirec
