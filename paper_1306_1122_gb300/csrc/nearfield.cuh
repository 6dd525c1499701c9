// nearfield.cuh -- the FP64 near field of one query, shared out over lanes.
#pragma once
#include "ff_math.cuh"
#include "kernels.h"

namespace dbie {

// Near-field correction (mixed precision, points with z <= near_z): over the (2W+1)^2 pixels
// around the point, replace the FP32 pair terms that the pair-sum kernel added by FP64 ones.
// The FP32 terms are recomputed with the same explicitly rounded code (pair_terms32), so the
// correction sum_k (t64 - t32) removes exactly what was added.  The correction is added in place
// to the query's split-0 partial sums (a dense pass: run after the pair sums) or is the query's
// last record (a pass of few queries: in any order with it).
// Index (along one axis) of the quadrature point nearest to coordinate x: the pixel for the
// midpoint rule; for nine-node elements of width 2h with g Gauss points, element e and the
// nearest abscissa a give e * g + a.
__device__ __forceinline__ long near_index(double x, double x0, double h, int nq,
                                           const ProbDesc& pd) {
  if (pd.quad_g == 0) return lrint((x - x0) / h);
  const int g = pd.quad_g;
  const long ne = nq / g;
  long e = (long)floor((x - x0) / (2.0 * h));
  e = e < 0 ? 0 : (e > ne - 1 ? ne - 1 : e);
  const double xi = (x - x0) / h - (double)(2 * e + 1);
  int best = 0;
  double bd = fabs(xi - pd.gx[0]);
  for (int a = 1; a < g; ++a) {
    const double d = fabs(xi - pd.gx[a]);
    if (d < bd) { bd = d; best = a; }
  }
  return e * g + best;
}

// Number of values per lane after near_window (NP in use, LEFT valid) and of lanes that hold the
// same ones: lane `sub` of a group of GL ends with sums sub / SAME * LEFT + i, i < LEFT.
template <int NSUM, int GL>
struct NearLanes {
  static constexpr int NP = NSUM > 16 ? 32 : NSUM > 8 ? 16 : NSUM > 4 ? 8 : 4;
  static constexpr int LEFT = NP / GL > 0 ? NP / GL : 1;
  static constexpr int SAME = NP < GL ? GL / NP : 1;
};

// Correction sums of one query over GL lanes (a divisor of 32; every lane of the warp calls it).
template <int VAR, bool TIED, int GL>
__device__ __forceinline__ void near_window(
    const ProbDesc& pd, float4 pos, Lam4 lam, bool valid, const float4* s_tab, int sub,
    double (&v)[NearLanes<3 * nsum_per_comp(VAR), GL>::NP]) {
  constexpr int NS = nsum_per_comp(VAR);
  constexpr int NSUM = 3 * NS;
  constexpr int NP = NearLanes<NSUM, GL>::NP;
  // sin and cos of lambda r in float-float on the FP32 pipe (absolute error ~1e-13 + 5e-15 |lambda
  // r|, far below the FP32 terms' error that the correction removes) instead of FP64 sincos,
  // which cost most of this kernel's FP64-pipe time
  auto sincos_ff = [&](double th, double& s, double& c) {
    ff::ds S, C;
    ff::sincos_ds_any(ff::from_double(th), s_tab, S, C);
    s = ff::to_double(S);
    c = ff::to_double(C);
  };
  const Query<float, TIED> q32 = make_query<float, TIED>(pos, lam);
  const Query<double, TIED> q64 = make_query<double, TIED>(pos, lam);
  const int W = pd.near_w > 0 ? pd.near_w : NEAR_W;
  const long ix = near_index((double)pos.x, pd.x0, pd.hx, pd.nx, pd);
  const long iy = near_index((double)pos.y, pd.y0, pd.hy, pd.ny, pd);
  const long i0 = ix - W < 0 ? 0 : ix - W;
  const long i1 = ix + W > pd.nx - 1 ? pd.nx - 1 : ix + W;
  const long j0 = iy - W < 0 ? 0 : iy - W;
  const long j1 = iy + W > pd.ny - 1 ? pd.ny - 1 : iy + W;
  const long wi = i1 - i0 + 1, wj = j1 - j0 + 1;
  double c[NSUM];
#pragma unroll
  for (int s = 0; s < NSUM; ++s) c[s] = 0.0;
  if (valid && wi > 0 && wj > 0 && wi <= 2 * W + 1 && wj <= 2 * W + 1) {
    const int nwin = (int)(wi * wj), wx = (int)wi;
    for (int e = sub; e < nwin; e += GL) {
      const int64_t k = (j0 + e / wx) * (int64_t)pd.nx + (i0 + e % wx);
      const int nf = pd.nf32 > 0 ? pd.nf32 : NFIELD;
      const float b32[3] = {*tile_field(pd.tiles32, k, 2, nf), *tile_field(pd.tiles32, k, 3, nf),
                            *tile_field(pd.tiles32, k, 4, nf)};
      const double b64[3] = {*tile_field(pd.tiles64, k, 2), *tile_field(pd.tiles64, k, 3),
                             *tile_field(pd.tiles64, k, 4)};
      Terms32<VAR, TIED> t32;
      Terms64<VAR, TIED> t64;
      if (nf == NFIELD_SPLIT)
        pair_terms32_split<VAR, TIED>(q32, *tile_field(pd.tiles32, k, 0, nf),
                                      *tile_field(pd.tiles32, k, 1, nf),
                                      *tile_field(pd.tiles32, k, 5, nf),
                                      *tile_field(pd.tiles32, k, 6, nf), b32, k & 2, t32);
      else
        pair_terms32<VAR, TIED>(q32, *tile_field(pd.tiles32, k, 0), *tile_field(pd.tiles32, k, 1),
                                b32, k & 2, t32);
      pair_terms64_sc<VAR, TIED>(q64, *tile_field(pd.tiles64, k, 0),
                                 *tile_field(pd.tiles64, k, 1), b64, t64, sincos_ff);
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        const int lp = TIED ? 0 : p;
        // FP32 contributions as the scalar FP32 code computes them (products of two FP32
        // factors, exact in FP64; the packed kernel's can differ by a rounding of a factor),
        // replaced by the FP64 terms.
        if constexpr (has_hess(VAR)) c[p * NS] += t64.t0[p] - (double)t32.t0[p];
        else if constexpr (has_value(VAR)) c[p * NS] += t64.t0[p] - (double)t32.u[lp] * (double)t32.rb[p];
        if constexpr (has_grad(VAR)) {
          c[p * NS + 1] += t64.t1[p] - (double)t32.t1[p];
          c[p * NS + 2] += t64.t1[p] * t64.dx - (double)t32.t1[p] * (double)t32.dx;
          c[p * NS + 3] += t64.t1[p] * t64.dy - (double)t32.t1[p] * (double)t32.dy;
        }
        if constexpr (has_hess(VAR))
          c[p * NS + idx_sl(VAR)] += t64.tl[p] - (double)t32.tl[p];
        else if constexpr (has_dlam(VAR))
          c[p * NS + idx_sl(VAR)] += t64.tl[p] - (double)t32.cr[lp] * (double)b32[p];
        if constexpr (has_newton(VAR)) {
          c[p * NS + IDX_TX] += t64.t0[p] * t64.dx - (double)t32.t0[p] * (double)t32.dx;
          c[p * NS + IDX_TY] += t64.t0[p] * t64.dy - (double)t32.t0[p] * (double)t32.dy;
        }
        if constexpr (has_hess(VAR)) {
          c[p * NS + IDX_Q] += t64.tq[p] - (double)t32.sn[lp] * (double)b32[p];
          c[p * NS + IDX_UX] += t64.tl[p] * t64.dx - (double)t32.tl[p] * (double)t32.dx;
          c[p * NS + IDX_UY] += t64.tl[p] * t64.dy - (double)t32.tl[p] * (double)t32.dy;
        }
      }
    }
  }
  // the lanes' sums, by halving: each step hands half of the sums to the partner lane (16 FP64
  // additions for 12 sums over 32 lanes instead of 60)
#pragma unroll
  for (int s = 0; s < NP; ++s) v[s] = s < NSUM ? c[s < NSUM ? s : 0] : 0.0;
  int half = NP / 2;
#pragma unroll
  for (int off = GL / 2; off > 0; off >>= 1, half >>= 1) {
    if (half >= 1) {
      const bool up = (sub & off) != 0;
#pragma unroll
      for (int s = 0; s < half; ++s) {
        const double give = up ? v[s] : v[s + half];
        const double keep = up ? v[s + half] : v[s];
        v[s] = keep + __shfl_xor_sync(0xffffffffu, give, off);
      }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
    }
  }
}

}  // namespace dbie
