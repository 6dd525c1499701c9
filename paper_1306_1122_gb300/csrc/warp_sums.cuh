// warp_sums.cuh -- sums of float pairs over the lanes of a warp.
#pragma once
#include "ff_math.cuh"

namespace dbie {

// Sums v[0..NSUM) over the warp by halving: each step hands half of the sums to the partner lane,
// so NP - 1 pair additions and a few more reduce NSUM <= NP sums (a butterfly per sum takes 5 NSUM).
// Lane l ends with sum l / (32 / NP), NP = NSUM rounded up to a power of two; returns it.
template <int NSUM>
struct WarpSums {
  static constexpr int NP = NSUM > 16 ? 32 : NSUM > 8 ? 16 : NSUM > 4 ? 8 : 4;
  static constexpr int GL = 32 / NP;   // lanes that end with the same sum
  static_assert(NSUM <= 32, "one sum per lane at most");

  __device__ static __forceinline__ ff::ds plus(ff::ds a, ff::ds b) {
    const ff::ds s = ff::two_sum(a.hi, b.hi);
    return ff::ds{s.hi, __fadd_rn(__fadd_rn(a.lo, b.lo), s.lo)};
  }
  __device__ static __forceinline__ ff::ds reduce(const ff::ds (&in)[NSUM], int lane) {
    ff::ds v[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) v[i] = i < NSUM ? in[i < NSUM ? i : 0] : ff::ds{0.f, 0.f};
    int off = 16;
#pragma unroll
    for (int half = NP / 2; half >= 1; half >>= 1, off >>= 1) {
      const bool up = (lane & off) != 0;
#pragma unroll
      for (int i = 0; i < half; ++i) {
        const ff::ds give = up ? v[i] : v[i + half];
        const ff::ds keep = up ? v[i + half] : v[i];
        v[i] = plus(keep, ff::ds{__shfl_xor_sync(0xffffffffu, give.hi, off),
                                 __shfl_xor_sync(0xffffffffu, give.lo, off)});
      }
    }
#pragma unroll
    for (; off >= 1; off >>= 1)
      v[0] = plus(v[0], ff::ds{__shfl_xor_sync(0xffffffffu, v[0].hi, off),
                               __shfl_xor_sync(0xffffffffu, v[0].lo, off)});
    return v[0];
  }
};

}  // namespace dbie
