// few_sums.cuh -- FP32 pair sums of one query over strips of pixels, by the lanes of a warp.
#pragma once
#include "kernels.h"
#include "pairsum.cuh"
#include "warp_sums.cuh"

namespace dbie {

constexpr int STRIP = 128;   // pixels per warp step: 32 lanes x 4
static_assert(TILE / STRIP == FEW_STRIPS_PER_TILE, "strips tile the tile");

// A lane's four pixels of one strip: two f32x2 pixel pairs.
template <int VAR, bool TIED, bool SPLIT, int NS>
__device__ __forceinline__ void strip_step(const float* T, int k, const Query<f32x2, TIED>& q2,
                                           f32x2* acc2) {
  auto ld = [&](int f) { return __ldg(reinterpret_cast<const float4*>(T + f * TILE + k)); };
  const float4 X = ld(0), Y = ld(1), BX = ld(2), BY = ld(3), BZ = ld(4);
  float4 XL = make_float4(0.f, 0.f, 0.f, 0.f), YL = XL;
  if constexpr (SPLIT) {
    XL = ld(5);
    YL = ld(6);
  }
  const f32x2 px2[2] = {pack2(X.x, X.y), pack2(X.z, X.w)};
  const f32x2 py2[2] = {pack2(Y.x, Y.y), pack2(Y.z, Y.w)};
  const f32x2 b2[2][3] = {{pack2(BX.x, BX.y), pack2(BY.x, BY.y), pack2(BZ.x, BZ.y)},
                          {pack2(BX.z, BX.w), pack2(BY.z, BY.w), pack2(BZ.z, BZ.w)}};
  auto pair = [&](auto half) {
    constexpr int h = decltype(half)::value;
    f32x2 dx = vsub(q2.x, px2[h]), dy = vsub(q2.y, py2[h]);
    if constexpr (SPLIT) {
      dx = vsub(dx, h == 0 ? pack2(XL.x, XL.y) : pack2(XL.z, XL.w));
      dy = vsub(dy, h == 0 ? pack2(YL.x, YL.y) : pack2(YL.z, YL.w));
    }
    TermsV<f32x2, VAR, TIED> tm;
    pair_angularv<f32x2, VAR, TIED, h>(q2, pair_geomv_d<f32x2, TIED>(q2, dx, dy), b2[h], tm);
    accumulatev<f32x2, VAR, TIED, NS>(acc2, tm, b2[h]);
  };
  pair(Half<0>{});
  pair(Half<1>{});
}

// Sums of a query over strips [s0, s1) of its problem; lane l returns sum l / WarpSums<NSUM>::GL.
template <int VAR, bool TIED, bool SPLIT>
__device__ __forceinline__ ff::ds strip_sums(const ProbDesc& pd, const Query<f32x2, TIED>& q2,
                                             int s0, int s1, int lane) {
  constexpr int NS = nsum_per_comp(VAR);
  constexpr int NSUM = 3 * NS;
  constexpr int NF = SPLIT ? NFIELD_SPLIT : NFIELD;
  constexpr int FOLD = SUB / 4;   // strips between folds: SUB pixels of a lane
  f32x2 acc2[NSUM], hi2[NSUM];
#pragma unroll
  for (int s = 0; s < NSUM; ++s) acc2[s] = hi2[s] = vconst<f32x2>(0.f);
#pragma unroll 1
  for (int b0 = s0; b0 < s1; b0 += FOLD) {
    const int b1 = b0 + FOLD < s1 ? b0 + FOLD : s1;
#pragma unroll 2
    for (int st = b0; st < b1; ++st)
      strip_step<VAR, TIED, SPLIT, NS>(
          pd.tiles32 + (int64_t)(st / FEW_STRIPS_PER_TILE) * (NF * TILE),
          (st % FEW_STRIPS_PER_TILE) * STRIP + lane * 4, q2, acc2);
#pragma unroll
    for (int s = 0; s < NSUM; ++s) fold2(hi2[s], acc2[s]);
  }
  ff::ds v[NSUM];
#pragma unroll
  for (int s = 0; s < NSUM; ++s) {
    float h0, h1, e0, e1;
    unpack2(hi2[s], h0, h1);
    unpack2(acc2[s], e0, e1);   // the folds' rounding errors
    const ff::ds t = ff::two_sum(h0, h1);
    v[s] = ff::ds{t.hi, __fadd_rn(t.lo, __fadd_rn(e0, e1))};
  }
  return WarpSums<NSUM>::reduce(v, lane);
}

}  // namespace dbie
