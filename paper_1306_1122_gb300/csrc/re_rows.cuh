// re_rows.cuh -- float-float sums and difference sums of one query over rows of pixels, one pixel
// per thread and row (pairsum_re.cu says what they are).
#pragma once
#include "ff_math.cuh"
#include "kernels.h"

namespace dbie {

constexpr int RE_NF = 2 * NFIELD;    // floats per pixel in a float-float tile
constexpr int DIF_BLK = 8;           // pixels per FP32 block sum of the differences

// The query of an item, prepared by the CTA's first threads (FP64 issues at 1/64 of the FP32
// rate here: once per CTA, not once per thread).
struct ReQuery {
  float x, y, z;
  float lh[3], ll[3];      // lambda (hi, lo)
  float hs[3], hd[3], pq[3], qq[3];   // differences: (la + l0) / 2, (la - l0) / 2, la^2 -+ l0^2
  int slow;                // lambda r may leave the range of the float-float reduction
};

// Whether lambda r may leave the range of sincos_ds for some pixel: |lambda| times the largest
// distance to the quadrature grid's box (pixel centres, or Gauss points of elements two node
// spacings wide, all inside [x0 - |hx|, x0 + 2 nx |hx|] with nx quadrature points per row); such a
// query (rare: a far-out or infinite trial lambda) takes the path with the FP64 fallback, so the
// common path stays branch-free.  (A NaN lambda gives NaN on either path and reads no table entry
// past the last.)
__device__ __forceinline__ bool beyond_reduction(const ProbDesc& pd, float4 pos, float lmax) {
  const float x0 = (float)pd.x0, y0 = (float)pd.y0;
  const float ax = (float)fabs(pd.hx), ay = (float)fabs(pd.hy);
  const float ex = fmaxf(fabsf(pos.x - (x0 - ax)), fabsf(pos.x - (x0 + 2.0f * pd.nx * ax)));
  const float ey = fmaxf(fabsf(pos.y - (y0 - ay)), fabsf(pos.y - (y0 + 2.0f * pd.ny * ay)));
  const float rmax = sqrtf(ex * ex + ey * ey + pos.z * pos.z);
  return !(lmax * rmax < 0.9f * ff::SC_MAX_ARG);
}

// Lambda l of a query, and with l0 the factors of its difference from l0 (formed in FP64).
__device__ __forceinline__ void set_lambda(ReQuery& q, int i, double l) {
  const ff::ds h = ff::from_double(l);
  q.lh[i] = h.hi;
  q.ll[i] = h.lo;
}
__device__ __forceinline__ void set_difference(ReQuery& q, int i, double l, double l0) {
  q.hs[i] = (float)(0.5 * (l + l0));
  q.hd[i] = (float)(0.5 * (l - l0));
  q.pq[i] = (float)((l - l0) * (l + l0));
  q.qq[i] = (float)(l * l + l0 * l0);
}

__device__ __forceinline__ float re_load(const float* tile, int f, int part, int e) {
  return __ldg(tile + f * 2 * TILE + part * TILE + e);
}

// A query's float-float factors.
template <bool TIED>
struct FfQuery {
  static constexpr int NL = TIED ? 1 : 3;
  ff::ds x, y, z2, lam[NL], lam2[NL];
  __device__ __forceinline__ explicit FfQuery(const ReQuery& q)
      : x{q.x, 0.f}, y{q.y, 0.f}, z2(ff::two_prod(q.z, q.z)) {
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      lam[l] = ff::ds{q.lh[l], q.ll[l]};
      lam2[l] = ff::mul(lam[l], lam[l]);
    }
  }
};

// Adds one pixel's float-float terms (re_points_kernel); ld(f, part): the pixel's field f, part 0 (hi)
// or 1 (lo).
template <int VAR, bool TIED, bool ANY, typename Load>
__device__ __forceinline__ void ff_pixel(const FfQuery<TIED>& q, const float4* tab, Load ld,
                                         ff::ds (&acc)[3 * nsum_per_comp(VAR)]) {
  using D = ff::ds;
  constexpr int NS = nsum_per_comp(VAR);
  constexpr int NL = FfQuery<TIED>::NL;
  const D X = D{ld(0, 0), ld(0, 1)};
  const D Y = D{ld(1, 0), ld(1, 1)};
  const D dx = ff::sub(q.x, X);
  const D dy = ff::sub(q.y, Y);
  // (products that feed a further float-float operation stay unnormalised: mul_nr)
  const D r2 = ff::add(ff::add(ff::mul_nr(dx, dx), ff::mul_nr(dy, dy)), q.z2);
  D r, ri;
  ff::sqrt_rsqrt(r2, r, ri);
  const D ri2 = ff::mul_nr(ri, ri);
  const D ri3 = ff::mul_nr(ri2, ri);
  D u[NL], c[NL];
#pragma unroll
  for (int l = 0; l < NL; ++l) {
    const D th = ff::mul_nr(q.lam[l], r);
    D s;
    if constexpr (ANY) ff::sincos_ds_any(th, tab, s, c[l]);
    else ff::sincos_ds<float>(th, tab, s, c[l]);
    u[l] = ff::add(ff::mul_nr(th, s), c[l]);
  }
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const int lp = TIED ? 0 : p;
    const D rb = ff::mul_nr(ri3, D{ld(2 + p, 0), ld(2 + p, 1)});
    ff::acc_add(acc[p * NS], ff::mul_nr(u[lp], rb));
    if constexpr (has_grad(VAR)) {
      // psi b = (lambda^2 cos(lambda r) - 3 u / r^2) b / r^3
      const D w = ff::sub(ff::mul_nr(q.lam2[lp], c[lp]),
                          ff::mul_f_nr(ff::mul_nr(u[lp], ri2), 3.0f));
      const D t1 = ff::mul_nr(w, rb);
      ff::acc_add(acc[p * NS + 1], t1);
      ff::acc_add(acc[p * NS + 2], ff::mul_nr(t1, dx));
      ff::acc_add(acc[p * NS + 3], ff::mul_nr(t1, dy));
    }
  }
}

// Float-float sums of pixel t of each row of ROW pixels in [r0, r1).  (ff_pixel's operations in
// ff_pixel's order, written out: through that function the loop is scheduled worse, 4,096 points with
// gradient over 128 x 128 pixels 1.62 -> 1.65 ms.)
template <int VAR, bool TIED, bool ANY, int ROW>
__device__ __forceinline__ void ff_rows(const float* tiles, int r0, int r1, int t, const ReQuery& q,
                                        const float4* tab, ff::ds (&acc)[3 * nsum_per_comp(VAR)]) {
  using D = ff::ds;
  constexpr int NS = nsum_per_comp(VAR);
  constexpr int NL = TIED ? 1 : 3;
  const D xq = D{q.x, 0.f}, yq = D{q.y, 0.f};
  const D z2 = ff::two_prod(q.z, q.z);
  D lam[NL], lam2[NL];
#pragma unroll
  for (int l = 0; l < NL; ++l) {
    lam[l] = D{q.lh[l], q.ll[l]};
    lam2[l] = ff::mul(lam[l], lam[l]);
  }
#pragma unroll 1
  for (int row = r0; row < r1; ++row) {
    const float* T = tiles + (int64_t)(row / (TILE / ROW)) * (RE_NF * TILE);
    const int e = (row % (TILE / ROW)) * ROW + t;
    const D X = D{re_load(T, 0, 0, e), re_load(T, 0, 1, e)};
    const D Y = D{re_load(T, 1, 0, e), re_load(T, 1, 1, e)};
    const D dx = ff::sub(xq, X);
    const D dy = ff::sub(yq, Y);
    // (products that feed a further float-float operation stay unnormalised: mul_nr)
    const D r2 = ff::add(ff::add(ff::mul_nr(dx, dx), ff::mul_nr(dy, dy)), z2);
    D r, ri;
    ff::sqrt_rsqrt(r2, r, ri);
    const D ri2 = ff::mul_nr(ri, ri);
    const D ri3 = ff::mul_nr(ri2, ri);
    D u[NL], c[NL];
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      const D th = ff::mul_nr(lam[l], r);
      D s;
      if constexpr (ANY) ff::sincos_ds_any(th, tab, s, c[l]);
      else ff::sincos_ds<float>(th, tab, s, c[l]);
      u[l] = ff::add(ff::mul_nr(th, s), c[l]);
    }
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const int lp = TIED ? 0 : p;
      const D rb = ff::mul_nr(ri3, D{re_load(T, 2 + p, 0, e), re_load(T, 2 + p, 1, e)});
      ff::acc_add(acc[p * NS], ff::mul_nr(u[lp], rb));
      if constexpr (has_grad(VAR)) {
        // psi b = (lambda^2 cos(lambda r) - 3 u / r^2) b / r^3
        const D w = ff::sub(ff::mul_nr(lam2[lp], c[lp]),
                            ff::mul_f_nr(ff::mul_nr(u[lp], ri2), 3.0f));
        const D t1 = ff::mul_nr(w, rb);
        ff::acc_add(acc[p * NS + 1], t1);
        ff::acc_add(acc[p * NS + 2], ff::mul_nr(t1, dx));
        ff::acc_add(acc[p * NS + 3], ff::mul_nr(t1, dy));
      }
    }
  }
}

// sin(d), cos(d): Taylor polynomials through d^9 and d^10 for |d| <= 1 (truncation below 3e-8
// relative), the SFU beyond.
__device__ __forceinline__ void sincos_delta(float d, float& s, float& c) {
  if (fabsf(d) <= 1.0f) {
    const float d2 = d * d;
    s = d * fmaf(d2, fmaf(d2, fmaf(d2, fmaf(d2, 1.0f / 362880.0f, -1.0f / 5040.0f),
                                   1.0f / 120.0f), -1.0f / 6.0f), 1.0f);
    c = fmaf(d2, fmaf(d2, fmaf(d2, fmaf(d2, fmaf(d2, -1.0f / 3628800.0f, 1.0f / 40320.0f),
                                        -1.0f / 720.0f), 1.0f / 24.0f), -0.5f), 1.0f);
  } else {
    s = sin_mufu(d);
    c = cos_mufu(d);
  }
}

// Adds one pixel's difference terms to the FP32 block sums bs (ld as above; z2 = z^2).
template <bool TIED, typename Load>
__device__ __forceinline__ void dif_pixel(const ReQuery& q, float z2, Load ld, float (&bs)[12]) {
  constexpr int NL = TIED ? 1 : 3;
  const float dx = (q.x - ld(0, 0)) - ld(0, 1);
  const float dy = (q.y - ld(1, 0)) - ld(1, 1);
  const float r2 = fmaf(dx, dx, fmaf(dy, dy, z2));
  const float ri = rsqrt_mufu(r2);
  const float r = r2 * ri;
  const float ri2 = ri * ri;
  const float ri3 = ri2 * ri;
  float du[NL], dw[NL];
#pragma unroll
  for (int l = 0; l < NL; ++l) {
    const float sg = q.hs[l] * r, dl = q.hd[l] * r;
    const float ss = sin_mufu(sg), cs = cos_mufu(sg);
    float sd, cd;
    sincos_delta(dl, sd, cd);
    const float cs_sd = cs * sd, ss_sd = ss * sd;
    du[l] = 2.0f * (fmaf(dl, ss * cd, sg * cs_sd) - ss_sd);
    dw[l] = fmaf(q.pq[l], cs * cd, fmaf(-q.qq[l], ss_sd, -3.0f * du[l] * ri2));
  }
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const int lp = TIED ? 0 : p;
    const float rb = ri3 * ld(2 + p, 0);
    const float t1 = dw[lp] * rb;
    bs[4 * p + 0] = fmaf(du[lp], rb, bs[4 * p + 0]);
    bs[4 * p + 1] += t1;
    bs[4 * p + 2] = fmaf(t1, dx, bs[4 * p + 2]);
    bs[4 * p + 3] = fmaf(t1, dy, bs[4 * p + 3]);
  }
}
__device__ __forceinline__ void dif_fold(ff::ds (&acc)[12], const float (&bs)[12]) {
#pragma unroll
  for (int s = 0; s < 12; ++s) {
    const ff::ds f = ff::two_sum(acc[s].hi, bs[s]);
    acc[s] = ff::ds{f.hi, __fadd_rn(acc[s].lo, f.lo)};
  }
}

// Difference sums: FP32 over blocks of DIF_BLK pixels of a thread, the block sums in float-float.
template <bool TIED, int ROW>
__device__ __forceinline__ void dif_rows(const float* tiles, int r0, int r1, int t, const ReQuery& q,
                                         ff::ds (&acc)[12]) {
  const float z2 = q.z * q.z;
#pragma unroll 1
  for (int b0 = r0; b0 < r1; b0 += DIF_BLK) {
    float bs[12];
#pragma unroll
    for (int s = 0; s < 12; ++s) bs[s] = 0.f;
    const int b1 = b0 + DIF_BLK < r1 ? b0 + DIF_BLK : r1;
#pragma unroll 2
    for (int row = b0; row < b1; ++row) {
      const float* T = tiles + (int64_t)(row / (TILE / ROW)) * (RE_NF * TILE);
      const int e = (row % (TILE / ROW)) * ROW + t;
      dif_pixel<TIED>(q, z2, [&](int f, int part) { return re_load(T, f, part, e); }, bs);
    }
    dif_fold(acc, bs);
  }
}

}  // namespace dbie
