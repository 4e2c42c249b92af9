// Warp sums of several values per lane, in a fixed order, shared by the moments
// (assign.cu) and the binning (spectra.cu).
#pragma once

#include <cuda_runtime.h>

namespace pkmom {

// (hi, lo) += (bh, bl) for unevaluated float pairs: a two-sum of the high parts, then
// the low parts and the rounding error added and renormalised.
__device__ __forceinline__ void pair_add(float &hi, float &lo, float bh, float bl)
{
    const float sh = __fadd_rn(hi, bh);
    const float bb = __fsub_rn(sh, hi);
    const float se = __fadd_rn(__fsub_rn(hi, __fsub_rn(sh, bb)), __fsub_rn(bh, bb));
    const float t = __fadd_rn(se, __fadd_rn(lo, bl));
    hi = __fadd_rn(sh, t);
    lo = __fsub_rn(t, __fsub_rn(hi, sh));
}
__device__ __forceinline__ void pair_add(double &hi, double &lo, double bh, double bl)
{
    hi = (hi + lo) + (bh + bl);  // FP64: plain adds
    lo = 0.0;
}

// Warp sums of 8 values per lane (value k as the pair hi[k] + lo[k]) by reduce-scatter:
// at the steps across lanes 16, 8 and 4 apart each lane keeps half of the values it
// still holds and adds its partner's copy of them, then the lanes 2 and 1 apart add their
// single values. Lane L ends with the sum of value ((L >> 2) & 7) over the warp, the
// same in lanes 4k..4k+3; 9 pair additions per lane instead of 40 for eight butterflies.
// Returned as FP64; fixed order.
template <typename T>
__device__ __forceinline__ double warp_scatter_sum8(T (&hi)[8], T (&lo)[8])
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int half = 4, o = 16; half >= 1; half >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;  // keeps the upper half of its values
#pragma unroll
        for (int j = 0; j < half; ++j) {
            const T mh = up ? hi[j + half] : hi[j], ml = up ? lo[j + half] : lo[j];
            const T sh = up ? hi[j] : hi[j + half], sl = up ? lo[j] : lo[j + half];
            const T rh = __shfl_xor_sync(full, sh, o), rl = __shfl_xor_sync(full, sl, o);
            hi[j] = mh, lo[j] = ml;
            pair_add(hi[j], lo[j], rh, rl);
        }
    }
#pragma unroll
    for (int o = 2; o >= 1; o >>= 1) {
        const T rh = __shfl_xor_sync(full, hi[0], o), rl = __shfl_xor_sync(full, lo[0], o);
        pair_add(hi[0], lo[0], rh, rl);
    }
    return static_cast<double>(hi[0]) + static_cast<double>(lo[0]);
}

// The same for plain FP64 values: 9 FP64 adds a lane (FP64 is rare on this part).
__device__ __forceinline__ double warp_scatter_sum8(double (&v)[8])
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int half = 4, o = 16; half >= 1; half >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int j = 0; j < half; ++j) {
            const double mine = up ? v[j + half] : v[j], send = up ? v[j] : v[j + half];
            v[j] = mine + __shfl_xor_sync(full, send, o);
        }
    }
#pragma unroll
    for (int o = 2; o >= 1; o >>= 1) v[0] += __shfl_xor_sync(full, v[0], o);
    return v[0];
}

}  // namespace pkmom
