// solve_step.cuh -- the per-point objective, its error bounds and one simplex step, as device code.
//
// Compiled with -fmad=false: the simplex arithmetic and the objective are evaluated with
// separately rounded operations, as written.
#pragma once
#include "kernels.h"
#include "solve.cuh"

namespace dbie {

struct Eval {
  double B[3];
  double f, g, phi;
  double nJ, nB;   // |J|, |B|
  float s;         // signed tie radius of phi (certified decisions; see TieLog)
};

__device__ __forceinline__ void objective(const double B[3], const double G[9], double g_scale,
                                          double w_g, double& f, double& g, double& phi,
                                          double* norms = nullptr) {
  const double Jx = G[3 * 2 + 1] - G[3 * 1 + 2];
  const double Jy = G[3 * 0 + 2] - G[3 * 2 + 0];
  const double Jz = G[3 * 1 + 0] - G[3 * 0 + 1];
  const double div = G[0] + G[4] + G[8];
  const double cx = Jy * B[2] - Jz * B[1];
  const double cy = Jz * B[0] - Jx * B[2];
  const double cz = Jx * B[1] - Jy * B[0];
  const double nJ = sqrt(Jx * Jx + Jy * Jy + Jz * Jz);
  const double nB = sqrt(B[0] * B[0] + B[1] * B[1] + B[2] * B[2]);
  const double nC = sqrt(cx * cx + cy * cy + cz * cz);
  f = (nJ * nB > 0.0) ? nC / (nJ * nB) : 0.0;
  g = (nB > 0.0) ? fabs(div) * g_scale / nB : 0.0;
  phi = f + w_g * g;
  if (norms) {
    norms[0] = nJ;
    norms[1] = nB;
  }
}

// Pixel-exact near field: add the point's lambda-independent correction of B and grad B
// (corr: dB_p at p, d(dB_p/dx_j) at 3 + 3 p + j).
__device__ __forceinline__ void add_corr(const double* corr, double B[3], double G[9]) {
  if (!corr) return;
  for (int p = 0; p < 3; ++p) B[p] += corr[p];
  for (int j = 0; j < 9; ++j) G[j] += corr[3 + j];
}

// B, gradient and objective from the 12 objective sums of one query (corr: see add_corr).
__device__ __forceinline__ void assemble_obj(const double S[12], double z, double g_scale,
                                             double w_g, Eval& e, double G[9],
                                             const double* corr) {
  for (int p = 0; p < 3; ++p) {
    const double S0 = S[p * 4 + 0], S1 = S[p * 4 + 1], Sx = S[p * 4 + 2], Sy = S[p * 4 + 3];
    e.B[p] = z * S0;
    G[3 * p + 0] = z * Sx;
    G[3 * p + 1] = z * Sy;
    G[3 * p + 2] = S0 + z * z * S1;
  }
  add_corr(corr, e.B, G);
  double norms[2];
  objective(e.B, G, g_scale, w_g, e.f, e.g, e.phi, norms);
  e.nJ = norms[0];
  e.nB = norms[1];
}

// ------------------------------------------------------------------ simplex state ----
// (blocks of 32 points: coalesced over neighbouring points, and every field of a point is at a
// constant offset from its first, so an access needs no address arithmetic)
__device__ __forceinline__ double& SD(const SolveArgs& a, int f, int64_t g) {
  return a.sd[(g >> 5) * (int64_t)(D_NFIELDS * 32) + (g & 31) + f * 32];
}
__device__ __forceinline__ int32_t& SI(const SolveArgs& a, int f, int64_t g) {
  return a.si[(g >> 5) * (int64_t)(I_NFIELDS * 32) + (g & 31) + f * 32];
}

// First query slot of a point's problem: the problem's own range, or one queue for all.
__device__ __forceinline__ int64_t queue_base(const SolveArgs& a, const ProbDesc& pd) {
  return a.one_queue ? 0 : pd.q_off;
}

// Field f of value record id (vertex slot, VID_R, VID_E) of point g.
__device__ __forceinline__ double& SV(const SolveArgs& a, int id, int f, int64_t g) {
  return SD(a, id * VREC + f, g);
}
// A float as a double, without a conversion (which would run at the FP64 rate); subnormals to 0.
__device__ __forceinline__ double f64_of(float x) {
  const unsigned b = __float_as_uint(x), e = (b >> 23) & 0xffu;
  const unsigned hi = e == 0u ? 0u : (e == 255u ? 0x7ff00000u : (e + 896u) << 20);
  const unsigned m = e == 0u ? 0u : b & 0x7fffffu;
  return __hiloint2double((int)((b & 0x80000000u) | hi | (m >> 3)), (int)(m << 29));
}
__device__ __forceinline__ void store_value(const SolveArgs& a, int id, int64_t g, const Eval& e) {
  for (int p = 0; p < 3; ++p) SV(a, id, V_B + p, g) = e.B[p];
  SV(a, id, V_F, g) = e.f;
  SV(a, id, V_G, g) = e.g;
  SV(a, id, V_PHI, g) = e.phi;
  SV(a, id, V_S, g) = f64_of(e.s);
}
__device__ __forceinline__ void copy_value(const SolveArgs& a, int from, int to, int64_t g) {
  double v[VREC];
#pragma unroll
  for (int f = 0; f < VREC; ++f) v[f] = SV(a, from, f, g);
#pragma unroll
  for (int f = 0; f < VREC; ++f) SV(a, to, f, g) = v[f];
}

// What a step compares: Phi, its signed tie radius, the vertex's storage slot and the record that
// holds the value (the slot, or VID_R / VID_E for a value that is about to take the slot's place).
struct Vert {
  double phi;
  float s;
  int slot, id;
};

// The pixel-exact correction of point g, or null (none, or the point is above its height).
__device__ __forceinline__ const double* corr_of(const SolveArgs& a, const ProbDesc& pd,
                                                 int64_t g, double z) {
  return (a.corr && pd.pxe_z > 0.0 && z <= pd.pxe_z) ? a.corr + 12 * g : nullptr;
}

// ------------------------------------------------------------- certified decisions ----
// Error bound of Phi computed from the mixed form's sums (FP32 pair terms).  Per pair term the
// error of the FP32 evaluation is bounded by the measured accuracy of its operations on GB300:
// SFU sine and cosine within 3.3e-7 absolute on [0, pi] and about 1.1e-7 |theta| beyond (the
// unit's own scaling of the argument), reciprocal square root within 1.25e-7 relative, plus
// FP32 rounding.  With theta = lambda r and u = theta sin(theta) + cos(theta) that gives, for a
// pixel of component p,
//   |d(u b / r^3)|   <= (A0 + A1 theta + A2 theta^2) |b| / r^3,
//   |d(psi b)|       <= [lambda^2 (A0 + A2 theta) + 3 (A3 + A4 theta + A2 theta^2) / r^2] |b| / r^3
// (psi r^3 = lambda^2 cos(theta) - 3 u / r^2; Sx and Sy carry |dx|, |dy| <= r more), and the sum
// over pixels turns these into polynomials in |lambda_p| whose coefficients are the point's
// lambda-independent sums M_j = sum_k |b_pk| / r^j, j = 1..5.  The bounds of B and grad B are
// carried to J = curl B, div B, f (Eq. 8) and g (Eq. 9) to first order:
//   |df| <= |dJ| / |J| + |dB| / |B|  (at most 1),   |dg| <= g_scale |d div B| / |B| + g |dB| / |B|.
// It is a worst case: on the Low & Lou and active-region workloads the measured error of Phi
// stays below 5 % of it.
constexpr double BND_A0 = 9.5e-7, BND_A1 = 1.06e-6, BND_A2 = 1.1e-7, BND_A3 = 1.45e-6,
                 BND_A4 = 1.56e-6;

// The bounds are evaluated in FP32: an FP64 warp instruction takes 64 cycles here, the bound
// took two thirds of a value's time, and a worst case whose coefficients have two or three
// digits (and M_j, summed from FP32 terms) does not need more.  Nor does it need more range: the
// polynomials are nested, so no power of lambda stands alone and a part underflows only where the
// pair terms that it bounds (FP32 too) have done so, and a bound that overflows counts as infinite:
// its value ties with every other and is re-evaluated (radius_of).
// A double's value in FP32, truncated (FP64 conversions run at the FP64 rate).
__device__ __forceinline__ float f32_of(double x) {
  const int hi = __double2hiint(x);
  const int e = ((hi >> 20) & 0x7ff) - 896;   // FP32 exponent field
  const unsigned m = ((unsigned)hi << 3 & 0x7fffffu) | ((unsigned)__double2loint(x) >> 29);
  const unsigned sg = (unsigned)hi & 0x80000000u;
  if (e <= 0) return __uint_as_float(sg);                              // below FP32's range: 0
  if (e >= 255) return __uint_as_float(sg | 0x7f800000u | (e == 1151 ? m : 0u));   // inf, NaN
  return __uint_as_float(sg | (unsigned)e << 23 | m);
}
// Norm without overflow or underflow of the squares (of infinite elements infinite, NaN stays).
__device__ __forceinline__ float norm3f(float x, float y, float z) {
  const float m = fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z)));
  if (!(m > 0.f && m <= 3.4e38f)) return fabsf(x) + fabsf(y) + fabsf(z);   // 0, infinite or NaN
  const float i = 1.0f / m;
  x *= i;
  y *= i;
  z *= i;
  return m * sqrtf(x * x + y * y + z * z);
}

// First-order bound of Phi's error from the bounds dB (3) and dG (9) of B and grad B.
__device__ __forceinline__ float propagate_bound(const float dB[3], const float dG[9],
                                                 const Eval& e, double g_scale, double w_g) {
  const float nJ = f32_of(e.nJ), nB = f32_of(e.nB);
  if (!(e.nB > 0.0)) return 2.0f;
  const float ndJ = norm3f(dG[7] + dG[5], dG[2] + dG[6], dG[3] + dG[1]);
  const float rB = norm3f(dB[0], dB[1], dB[2]) / nB;
  float sf = nJ > 0.f ? ndJ / nJ + rB : 1.0f;
  if (!(sf <= 1.0f)) sf = 1.0f;
  const float sg = f32_of(g_scale) * (dG[0] + dG[4] + dG[8]) / nB + f32_of(e.g) * rB;
  return sf + f32_of(w_g) * sg;
}

// Bounds of S0, S1 and of Sx, Sy of one component at |lambda| = L (m: its M_1..M_5).
__device__ __forceinline__ void mixed_component(const float* m, float L, float& s0, float& s1,
                                                float& sx) {
  constexpr float A0 = BND_A0, A1 = BND_A1, A2 = BND_A2, A3 = BND_A3, A4 = BND_A4;
  s0 = A0 * m[2] + L * (A1 * m[1] + A2 * (L * m[0]));
  sx = L * (L * (A0 * m[1] + A2 * (L * m[0]))) +
       3.0f * (A3 * m[3] + L * (A4 * m[2] + A2 * (L * m[1])));
  s1 = L * (L * (A0 * m[2] + A2 * (L * m[1]))) +
       3.0f * (A3 * m[4] + L * (A4 * m[3] + A2 * (L * m[2])));
}

__device__ __forceinline__ float mixed_phi_bound(const float* M, const double lam[3], int dim,
                                                 float z, const Eval& e, double g_scale,
                                                 double w_g) {
  float dB[3], dG[9];
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    float s0, s1, sx;
    mixed_component(M + 5 * p, fabsf(f32_of(dim == 1 ? lam[0] : lam[p])), s0, s1, sx);
    dB[p] = z * s0;
    dG[3 * p + 0] = z * sx;
    dG[3 * p + 1] = z * sx;
    dG[3 * p + 2] = s0 + z * z * s1;
  }
  return propagate_bound(dB, dG, e, g_scale, w_g);
}

// Error bounds of the difference sums (re_rows.cuh) that take a point's float-float
// reference sums at lambda_0 to lambda_a, per component p, with dl = |lambda_a - lambda_0| and
// L = |lambda_a| + |lambda_0|.  Every product of a pixel's difference terms carries a factor
// |delta| = dl r / 2 (or dl).  With the operation accuracies of mixed_phi_bound (SFU sine and
// cosine of sigma within 3.3e-7 + 1.1e-7 |sigma| absolute, sigma, delta and r within 3.2e-7
// relative, the Taylor sine and cosine of delta within 3e-8, FP32 rounding, and sums over blocks
// of 8 pixels in FP32) the changes du of u and dw of psi r^3 are in error by at most
//   dl (2.1e-6 r + 2.6e-6 L r^2 + 1.1e-7 L^2 r^3)                   (du, b / r^3 included)
//   dl (6.3e-6 / r + 1.22e-5 L + 2.6e-6 L^2 r + 1.1e-7 L^3 r^2)     (dw)
// (|du| <= dl L r^2 and |dw| <= dl (5 L + L^2 r) bound the relative roundings), and summed with
// |b| / r^3 they become polynomials in dl and L over the point's sums M_j = sum_k |b_pk| / r^j,
// j = 0..5.  The coefficients below are twice those.  The float-float reference sums add 1e-12
// of their absolute-value sums (their measured error is at most 1.4e-13 of them).
constexpr double DIF_C00 = 4.2e-6, DIF_C01 = 5.2e-6, DIF_C02 = 2.2e-7;
constexpr double DIF_C10 = 1.3e-5, DIF_C11 = 2.4e-5, DIF_C12 = 5.2e-6, DIF_C13 = 2.2e-7;
constexpr double DIF_FF = 1e-12;

// Bounds of S0, S1 and of Sx, Sy of one component (m[j - 1]: its M_j, m0: M_0) from
// dl = |lambda_a - lambda_0|, L = |lambda_a| + |lambda_0| and R = |lambda_0|.
template <typename T>
__device__ __forceinline__ void dif_component(const T* m, T m0, T dl, T L, T R, T& e0, T& e1, T& ex) {
  constexpr T C00 = DIF_C00, C01 = DIF_C01, C02 = DIF_C02, C10 = DIF_C10, C11 = DIF_C11,
              C12 = DIF_C12, C13 = DIF_C13, FF = DIF_FF;
  e0 = dl * (C00 * m[1] + L * (C01 * m[0] + C02 * (L * m0))) + FF * (m[2] + R * m[1]);
  e1 = dl * (C10 * m[3] + L * (C11 * m[2] + L * (C12 * m[1] + C13 * (L * m[0])))) +
       FF * (T(3) * m[4] + R * (T(3) * m[3] + R * m[2]));
  ex = dl * (C10 * m[2] + L * (C11 * m[1] + L * (C12 * m[0] + C13 * (L * m0)))) +
       FF * (T(3) * m[3] + R * (T(3) * m[2] + R * m[1]));
}

// e[4 p + s]: bounds of S0, S1, Sx, Sy of component p (dl, L, R per free lambda).
template <typename T>
__device__ __forceinline__ void dif_sum_bounds(const T* M, const T* M0, const T dl[3], const T L[3],
                                               const T R[3], int dim, T e[12]) {
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const int q = dim == 1 ? 0 : p;
    dif_component(M + 5 * p, M0[p], dl[q], L[q], R[q], e[4 * p], e[4 * p + 1], e[4 * p + 2]);
    e[4 * p + 3] = e[4 * p + 2];
  }
}

// Phi bound of a value assembled from reference plus difference sums with sum bounds eb.
__device__ __forceinline__ float dif_phi_bound(const float eb[12], float z, const Eval& e,
                                               double g_scale, double w_g) {
  float dB[3], dG[9];
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    dB[p] = z * eb[4 * p];
    dG[3 * p + 0] = z * eb[4 * p + 2];
    dG[3 * p + 1] = z * eb[4 * p + 3];
    dG[3 * p + 2] = eb[4 * p] + z * z * eb[4 * p + 1];
  }
  return propagate_bound(dB, dG, e, g_scale, w_g);
}

// Comparisons of doubles on the integer pipe, with the results of <, <= on doubles (NaN false).
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  return (b << 1) == 0 ? 0 : b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ bool not_nan(double x) {
  return (__double_as_longlong(x) & 0x7fffffffffffffffll) <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool less(double x, double y) {
  return not_nan(x) && not_nan(y) && order_key(x) < order_key(y);
}
__device__ __forceinline__ bool less_eq(double x, double y) {
  return not_nan(x) && not_nan(y) && order_key(x) <= order_key(y);
}

// Tie radius of a value: `band` times its bound (never 0, which marks a value without one; infinite,
// a tie with any value, where the bound is not a number because its parts overflowed).
__device__ __forceinline__ float radius_of(double band, float bound) {
  const float r = f32_of(band) * bound;
  return r != r ? __int_as_float(0x7f800000) : (r < 1e-37f ? 1e-37f : r);
}

// The first near tie of a step: a comparison whose two values differ by no more than the sum of
// their tie radii.  A mixed-form value carries the radius band x bound (certify), a value
// re-evaluated by difference certify_ref x bound, stored negated, and one re-evaluated in
// float-float 0.  (No value carries one when decisions are not certified.)
struct TieLog {
  int a, b;        // ids of the first near-tied values (-1: none)
  // Values ia, ib with signed radii ra, rb whose Phis (or Phi and threshold) are x and y.  Most are
  // far from a tie, which FP32 tells: the FP64 difference is taken only within its rounding.
  __device__ __forceinline__ void note(int ia, float ra, int ib, float rb, double x, double y) {
    if (a < 0 && (ra != 0.f || rb != 0.f)) {
      const float r = fabsf(ra) + fabsf(rb), fx = f32_of(x), fy = f32_of(y);
      if (fabsf(fx - fy) > r + 4e-7f * (fabsf(fx) + fabsf(fy))) return;
      if (less_eq(fabs(x - y), f64_of(r))) {
        a = ra != 0.f ? ia : -1;
        b = rb != 0.f ? ib : -1;
        if (a < 0) { a = b; b = -1; }
      }
    }
  }
  __device__ __forceinline__ void note(const Vert& v, double x, double y) {
    note(v.id, v.s, -1, 0.f, x, y);
  }
  __device__ __forceinline__ bool lt(const Vert& x, const Vert& y) {
    note(x.id, x.s, y.id, y.s, x.phi, y.phi);
    return less(x.phi, y.phi);
  }
  __device__ __forceinline__ bool le(const Vert& x, const Vert& y) {
    note(x.id, x.s, y.id, y.s, x.phi, y.phi);
    return less_eq(x.phi, y.phi);
  }
};

// Records to leave out of a query's sums: of a pass of few queries the last one is the near field's,
// zero above near_z.
__device__ __forceinline__ int near_skip(const SolveArgs& a, const ProbDesc& pd, double z) {
  return a.one_queue && a.o.near_on && !less_eq(z, pd.near_z) ? 1 : 0;
}

// Objective of the k-th pending query of point g; its error bound when decisions are certified.
__device__ __forceinline__ void read_eval(const SolveArgs& a, const PlanHdr& h, int pidx,
                                          int64_t slot, double z, Eval& e, int64_t g,
                                          const double lam[3]) {
  const ProbDesc& pd = a.probs[pidx];
  double S[12], G[9];
  gather_sums<12>(a.out, h, a.item_off, pidx, slot - queue_base(a, pd), S, near_skip(a, pd, z));
  assemble_obj(S, z, pd.g_scale, a.o.w_g, e, G, corr_of(a, pd, g, z));
  e.s = 0.f;
  if (a.o.tie > 0.0 && a.msc)
    e.s = radius_of(a.o.tie, mixed_phi_bound(a.msc + 15 * g, lam, a.o.dim, (float)z, e, pd.g_scale,
                                             a.o.w_g));
}

// Objective of a re-evaluated value of point g at lambda lt and its 12 sums: float-float sums
// (bound 0), or (dif) the point's float-float reference sums plus difference sums, with the bound
// stored negated (a difference value).  One site for both kinds: lanes of a warp whose values
// are of different kinds run the FP64 objective together.
__device__ __forceinline__ void read_reeval(const SolveArgs& a, bool dif, int pidx, int64_t slot,
                                            double z, Eval& e, int64_t g, const double lt[3],
                                            double S[12]) {
  const ProbDesc& pd = a.probs[pidx];
  const double* out = dif ? a.dout : a.fout;
  const PlanHdr h = dif ? *a.dplan : *a.fplan;
  double G[9];
  gather_sums<12>(out, h, nullptr, 0, slot, S);
  if (dif) {
#pragma unroll
    for (int s = 0; s < 12; ++s) S[s] = SD(a, D_REFS + s, g) + S[s];
  }
  assemble_obj(S, z, pd.g_scale, a.o.w_g, e, G, corr_of(a, pd, g, z));
  e.s = 0.f;
  if (dif) {
    float dl[3], L[3], R[3], eb[12];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double l0 = SD(a, D_REFL + d, g);
      dl[d] = fabsf(f32_of(lt[d] - l0));
      R[d] = fabsf(f32_of(l0));
      L[d] = fabsf(f32_of(lt[d])) + R[d];
    }
    dif_sum_bounds<float>(a.msc + 15 * g, a.msc0 + 3 * g, dl, L, R, a.o.dim, eb);
    e.s = -radius_of(a.o.tie_dif, dif_phi_bound(eb, (float)z, e, pd.g_scale, a.o.w_g));
  }
}

// One value by four lanes (all 32 lanes call it; `on`: the quad has a value).  Lane c < 3 of the quad
// works on component c, and independent square roots and divisions sit in different lanes, so
// that the warp issues about 45 FP64 instructions for eight values where one lane per value issues
// about 120 for up to 32.  The operations are those of assemble_obj and objective, in their order.
// vid: the value's record; sums of a pass (out, h, slot, without the last `skip` records); dif: a
// re-evaluation by difference; S: lane c's sums S0, S1, Sx, Sy on return.
__device__ __forceinline__ void value_quad(const SolveArgs& a, bool on, bool reeval, bool dif,
                                           const double* out, const PlanHdr& h, int64_t j, int skip,
                                           const ProbDesc& pd, const int32_t* item_off, int pidx,
                                           int vid, int64_t g, float zf, double (&S)[4]) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, c = lane & 3, quad = lane & ~3;
  const int p = c < 3 ? c : 2;               // (lane 3 repeats component 2)
  const int c1 = p == 2 ? 0 : p + 1, c2 = p == 0 ? 2 : p - 1;
  const double z = (double)zf;
  double B = 0.0, G[3] = {0.0, 0.0, 0.0};
  if (on) {
    const double* src = out + out_index(h, item_off, pidx, j, 0, 4 * p, 12);
    const int64_t step = (int64_t)12 * h.qper;
#pragma unroll
    for (int s = 0; s < 4; ++s) S[s] = src[(int64_t)s * h.qper];
    for (int sp = 1; sp < h.nsplit - skip; ++sp) {
      src += step;
#pragma unroll
      for (int s = 0; s < 4; ++s) S[s] += src[(int64_t)s * h.qper];
    }
    if (dif) {
#pragma unroll
      for (int s = 0; s < 4; ++s) S[s] = SD(a, D_REFS + 4 * p + s, g) + S[s];
    }
    B = z * S[0];
    G[0] = z * S[2];
    G[1] = z * S[3];
    G[2] = S[0] + z * z * S[1];
    if (const double* corr = corr_of(a, pd, g, z)) {
      B += corr[p];
#pragma unroll
      for (int i = 0; i < 3; ++i) G[i] += corr[3 + 3 * p + i];
    }
  }
  auto pick = [](const double (&v)[3], int i) { return i == 0 ? v[0] : (i == 1 ? v[1] : v[2]); };
  // J_p = d_c1 B_c2 - d_c2 B_c1: lane c2 hands its G[c1 of p], lane c1 its G[c2 of p]
  const double J = __shfl_sync(FULL, pick(G, c2), quad + c2) - __shfl_sync(FULL, pick(G, c1), quad + c1);
  const double diag = pick(G, p);
  const double div = __shfl_sync(FULL, diag, quad) + __shfl_sync(FULL, diag, quad + 1) +
                     __shfl_sync(FULL, diag, quad + 2);
  const double C = __shfl_sync(FULL, J, quad + c1) * __shfl_sync(FULL, B, quad + c2) -
                   __shfl_sync(FULL, J, quad + c2) * __shfl_sync(FULL, B, quad + c1);
  // lane 0: |J|, lane 1: |B|, lane 2: |J x B|
  double v[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double vj = __shfl_sync(FULL, J, quad + i), vb = __shfl_sync(FULL, B, quad + i),
                 vc = __shfl_sync(FULL, C, quad + i);
    v[i] = c == 0 ? vj : (c == 1 ? vb : vc);
  }
  const double norm = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
  const double nJ = __shfl_sync(FULL, norm, quad), nB = __shfl_sync(FULL, norm, quad + 1),
               nC = __shfl_sync(FULL, norm, quad + 2);
  // lane 0: f = |J x B| / (|J| |B|), lane 1: g = |div B| g_scale / |B|
  const double den = c == 0 ? nJ * nB : nB;
  const double num = c == 0 ? nC : fabs(div) * pd.g_scale;
  const double ratio = less(0.0, den) ? num / den : 0.0;
  Eval e;
  e.f = __shfl_sync(FULL, ratio, quad);
  e.g = __shfl_sync(FULL, ratio, quad + 1);
  e.phi = e.f + a.o.w_g * e.g;
  e.nJ = nJ;
  e.nB = nB;
  e.s = 0.f;
  if (a.o.tie > 0.0 && a.msc && __any_sync(FULL, on && (!reeval || dif))) {
    // the bound: component p's parts per lane, put together in all
    const float* M = a.msc + 15 * g;
    const float l = on ? f32_of(SV(a, vid, V_L + (a.o.dim == 1 ? 0 : p), g)) : 0.f;
    float s0 = 0.f, sx = 0.f, s1 = 0.f;
    if (on && dif) {
      const double ld = SV(a, vid, V_L + (a.o.dim == 1 ? 0 : p), g);
      const double l0 = SD(a, D_REFL + (a.o.dim == 1 ? 0 : p), g);
      const float rf = fabsf(f32_of(l0));
      dif_component(M + 5 * p, a.msc0[3 * g + p], fabsf(f32_of(ld - l0)), fabsf(l) + rf, rf, s0, s1, sx);
    } else if (on && !reeval) {
      mixed_component(M + 5 * p, fabsf(l), s0, s1, sx);
    }
    const float db = zf * s0, dxy = zf * sx, dz = s0 + zf * zf * s1;
    float dB[3], dG[9];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      dB[i] = __shfl_sync(FULL, db, quad + i);
      dG[3 * i] = dG[3 * i + 1] = __shfl_sync(FULL, dxy, quad + i);
      dG[3 * i + 2] = __shfl_sync(FULL, dz, quad + i);
    }
    if (!reeval || dif) {
      const float r = radius_of(dif ? a.o.tie_dif : a.o.tie,
                                propagate_bound(dB, dG, e, pd.g_scale, a.o.w_g));
      e.s = dif ? -r : r;
    }
  }
  if (on) {
    if (c < 3) SV(a, vid, V_B + c, g) = B;
    // lane 0: f, lane 1: g, lane 2: Phi, lane 3: tie radius
    SV(a, vid, V_F + c, g) = c == 0 ? e.f : (c == 1 ? e.g : (c == 2 ? e.phi : f64_of(e.s)));
  }
}

// atomicAdd(ctr, v) for the lanes of a warp that reach it together (whatever branch they are
// in): lanes with the same counter add their total with one atomic and take consecutive ranges
// in lane order.  Every simplex or quasi-Newton point emits its trial queries through these
// counters each round, so one atomic per lane would serialise N updates of one address.
__device__ __forceinline__ int atomic_add_warp(int* ctr, int v) {
  const unsigned active = __activemask();
  const unsigned peers = __match_any_sync(active, reinterpret_cast<unsigned long long>(ctr));
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(peers) - 1;
  const unsigned below = peers & ((1u << lane) - 1u);
  int same = 0;
  __match_all_sync(peers, v, &same);
  int prefix = 0, total = 0;
  if (same) {
    prefix = v * __popc(below);
    total = v * __popc(peers);
  } else {
    for (unsigned m = peers; m; m &= m - 1u) {
      const int l = __ffs(m) - 1;
      const int vl = __shfl_sync(peers, v, l);
      if (l < lane) prefix += vl;
      total += vl;
    }
  }
  int base = 0;
  if (lane == leader) base = atomicAdd(ctr, total);
  base = __shfl_sync(peers, base, leader);
  return base + prefix;
}

// Queue K trial points (lambda rows) of point g for the next round (K fixed at compile time, so
// the rows stay in registers).
template <int K>
__device__ __forceinline__ void emit(const SolveArgs& a, int64_t g, const float4& pos, int pidx,
                                     const double (*lam)[3]) {
  const ProbDesc& pd = a.probs[pidx];
  const int base = atomic_add_warp(a.nxt.q_cnt + (a.one_queue ? 0 : pidx), K);
  const int64_t slot0 = queue_base(a, pd) + base;
#pragma unroll
  for (int j = 0; j < K; ++j) {
    a.nxt.qpos[slot0 + j] = pos;
    if (a.o.dim == 1) a.nxt.qlam[slot0 + j] = make_lam4(lam[j][0], lam[j][0], lam[j][0]);
    else a.nxt.qlam[slot0 + j] = make_lam4(lam[j][0], lam[j][1], lam[j][2]);
  }
  if (a.o.near_on && (double)pos.z <= pd.near_z) {
    const int nb = atomic_add_warp(a.nxt.near_cnt, K);
#pragma unroll
    for (int j = 0; j < K; ++j) a.nxt.near[nb + j] = (int32_t)(slot0 + j);
  }
  SI(a, I_QSLOT, g) = (int32_t)slot0;
  a.nxt.act[atomic_add_warp(a.nxt.act_cnt, 1)] = (int32_t)g;
}

// Queue the re-evaluation of k (1 or 2) values of point g on side `sd` and put the point on that
// side's waiting list: value j in float-float, or (dif[j]) as the difference from the point's
// float-float reference at lambda lref.  The value ids go to I_RTGT, one per byte (| RT_DIF for
// differences), and the first slot of each kind to I_RSLOT, I_DSLOT.
__device__ __forceinline__ void emit_reeval(const SolveArgs& a, const RoundBuf& sd, int64_t g,
                                            const float4& pos, int k,
                                            const double (&l)[2][3], int id0, int id1,
                                            const bool (&dif)[2], const double lref[3]) {
  const int nd = (dif[0] ? 1 : 0) + (k > 1 && dif[1] ? 1 : 0);
  const int nf = k - nd;
  auto lam4 = [&](const double* x) {
    return a.o.dim == 1 ? make_lam4(x[0], x[0], x[0]) : make_lam4(x[0], x[1], x[2]);
  };
  int64_t fs = 0, ds = 0;
  if (nf > 0) fs = atomic_add_warp(sd.fq_cnt, nf);
  if (nd > 0) ds = atomic_add_warp(sd.dq_cnt, nd);
  SI(a, I_RSLOT, g) = (int32_t)fs;
  SI(a, I_DSLOT, g) = (int32_t)ds;
  int tg = 0xffff, nt = 0;
#pragma unroll
  for (int it = 0; it < 4; ++it) {   // differences first
    const int j = it & 1;
    if (j >= k || dif[j] != (it < 2)) continue;
    const int id = j == 0 ? id0 : id1;
    if (dif[j]) {
      sd.dpos[ds] = pos;
      sd.dlam[ds] = lam4(l[j]);
      sd.dlam0[ds] = lam4(lref);
      ++ds;
    } else {
      sd.fpos[fs] = pos;
      sd.flam[fs] = lam4(l[j]);
      ++fs;
    }
    const int sh = 8 * nt++;
    tg = (tg & ~(0xff << sh)) | (((id | (dif[j] ? RT_DIF : 0)) & 0xff) << sh);
  }
  SI(a, I_RTGT, g) = tg;
  sd.ref[atomic_add_warp(sd.ref_cnt, 1)] = (int32_t)g;
  if (a.stat_ties) atomicAdd(a.stat_ties, 1ull);
  if (nd > 0 && a.stat_difs) atomicAdd(a.stat_difs, (unsigned long long)nd);
}

// The initial simplex of point g (lambda_init, or 0, plus one edge per free lambda) and its queries.
// N: the number of free lambdas (3, or 1 when the components share one).
template <int N>
__device__ __forceinline__ void init_point(const SolveArgs& a, const double* lam_init, int64_t g) {
  const float4 pos = a.ppos[g];
  const int pidx = __float_as_int(pos.w);
  constexpr int n = N;
  double lam[N + 1][3];
#pragma unroll
  for (int v = 0; v <= n; ++v)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double l0 = lam_init ? lam_init[3 * g + d] : 0.0;
      lam[v][d] = (d < n) ? l0 + ((v == d + 1) ? a.probs[pidx].step : 0.0) : 0.0;
    }
#pragma unroll
  for (int v = 0; v <= n; ++v)
#pragma unroll
    for (int d = 0; d < 3; ++d) SV(a, v, V_L + d, g) = lam[v][d];
  SI(a, I_STAGE, g) = ST_INIT;
  SI(a, I_ITERS, g) = 0;
  SI(a, I_NFEV, g) = 0;
  SI(a, I_STATUS, g) = PT_RUNNING;
  SI(a, I_ORDER, g) = 0x3210;
  if (a.o.tie_dif > 0.0) SD(a, D_REFS, g) = __longlong_as_double(0x7ff8000000000000LL);  // NaN
  emit<N + 1>(a, g, pos, pidx, lam);
}

// Stable insertion sort of the N+1 vertices by Phi (ties keep their order), unrolled into
// adjacent compare-exchanges so their keys stay in registers.  Without the early exit of the
// textbook loop the result is the same: after inserting each vertex no adjacent pair of the
// sorted prefix is out of order (v[j].phi < v[j-1].phi false), so the comparisons below the
// insertion point never swap.  The insertion's own comparisons (those down to the insertion
// point) go through the tie log; the ones below it decide nothing.
template <int N>
__device__ __forceinline__ void sort_verts(Vert* v, TieLog& tl) {
#pragma unroll
  for (int i = 1; i <= N; ++i) {
    bool moving = true;
#pragma unroll
    for (int j = i; j > 0; --j) {
      const bool sw = moving ? tl.lt(v[j], v[j - 1]) : v[j].phi < v[j - 1].phi;
      if (sw) {
        const Vert t = v[j];
        v[j] = v[j - 1];
        v[j - 1] = t;
      } else {
        moving = false;
      }
    }
  }
}

constexpr int QUAD_POINTS = 8;   // points of a warp up to which four lanes compute a value

// x / n, correctly rounded.  x / 3 in two operations: with zh + zl = 1/3 to 107 bits, x zh + x zl
// is x / 3 to about 2^-105, and x / 3 is never nearer than 1/6 ulp to the middle between two
// doubles (a third of an integer is no nearer than 1/6 to a half-integer), so rounding the one sum
// in fma rounds x / 3.  (Away from underflow of x zl.)
template <int n>
__device__ __forceinline__ double over(double x) {
  static_assert(n == 1 || n == 3, "simplex of one or three lambdas");
  if (n == 1) return x;
  const double zh = 0x1.5555555555555p-2, zl = 0x1.5555555555555p-56;
  if (!less(fabs(x), 1e-250)) return __fma_rn(x, zh, __dmul_rn(x, zl));
  return x / 3.0;
}

// One simplex step per waiting point.  REF = false: the points whose queries the mixed pass of
// this round evaluated (their results are read and their bounds computed); REF = true: the
// points whose near-tied values this round's re-evaluation pass computed (the values are
// replaced, and the step is decided again).  A step is taken only when none of its comparisons is
// a near tie (TieLog); otherwise the near-tied values are queued for re-evaluation and the state
// stays as it is, so every decision is the one that sums accurate to the float-float level would
// take.  With a.o.tie == 0 every step is taken as evaluated.
//
// What bounds it: one warp's chain of instructions, its FP64 instructions above all (64 cycles
// each), so the time is the instruction count of the longest warp.  Hence FP64 only where the
// values and lambdas are formed (comparisons on the integer pipe, bounds in FP32), and three
// phases.  First the lanes share out the values to compute, whatever the points' stages (a shrink
// has 3, the start 4; taken in turn by the point's own lane they set the length for the whole
// warp): one FP64 objective and bound per lane, or per four lanes where the warp has few points.
// Then each lane decides its point's step on Phi and tie radius alone; vertices stay in their slots,
// and a step writes one record, not four.  Then the lanes share out the trial points' lambdas.  On
// 2,048 points a step took 63 us and the waiting points' 112 us with one lane per point evaluating
// and sorting whole vertices, in CTAs of 128 threads; now 28 and 15.
// Warp `warp` of `nwarps` takes ppw points at a time.
template <int N, bool REF>
__device__ __forceinline__ void step_points(const SolveArgs& a, int warp, int nwarps, int ppw) {
  const double rho = 1.0, chi = 2.0, psi = 0.5, sigma = 0.5;
  const unsigned FULL = 0xffffffffu;
  const int nact = REF ? *a.cur.ref_cnt : *a.cur.act_cnt;
  const int32_t* list = REF ? a.cur.ref : a.cur.act;
  constexpr int n = N;
  const PlanHdr h = *a.plan;
  const int lane = threadIdx.x & 31;
  for (int base = warp * ppw; base < nact; base += nwarps * ppw) {
    const bool on = lane < ppw && base + lane < nact;
    const int gi = on ? list[base + lane] : 0;
    const int64_t g = gi;
    int stage = ST_DONE, order = 0, targets = 0xffff, nev = 0;
    int slot0 = 0, slot1 = 0;   // first query slot (REF: float-float and difference slot)
    if (on) {
      stage = SI(a, I_STAGE, g);
      order = SI(a, I_ORDER, g);
      if (REF) {
        targets = SI(a, I_RTGT, g);
        slot0 = SI(a, I_RSLOT, g);
        slot1 = SI(a, I_DSLOT, g);
        nev = (targets >> 8) == 0xff ? 1 : 2;
      } else {
        slot0 = SI(a, I_QSLOT, g);
        nev = stage == ST_INIT ? n + 1 : (stage == ST_SHRINK ? n : 1);
      }
    }

    // ---- phase 1: value q of the warp's points, by lane q
    int incl = nev;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int t = __shfl_up_sync(FULL, incl, off);
      if (lane >= off) incl += t;
    }
    const int total = __shfl_sync(FULL, incl, 31);
    // (few points of this warp: four lanes per value, see value_quad)
    const bool quads = ppw <= QUAD_POINTS;
    const int per = quads ? 8 : 32;
    for (int q0 = 0; q0 < total; q0 += per) {
      const int q = q0 + (quads ? lane >> 2 : lane);
      int o = 0;   // the point (lane) that owns value q: the first with incl > q
#pragma unroll
      for (int st = 16; st > 0; st >>= 1)
        if (__shfl_sync(FULL, incl, o + st - 1) <= q) o += st;
      const int k = q - (__shfl_sync(FULL, incl, o) - __shfl_sync(FULL, nev, o));
      const int64_t og = __shfl_sync(FULL, gi, o);
      const int ostage = __shfl_sync(FULL, stage, o), oorder = __shfl_sync(FULL, order, o);
      const int otg = __shfl_sync(FULL, targets, o);
      const int os0 = __shfl_sync(FULL, slot0, o), os1 = __shfl_sync(FULL, slot1, o);
      const bool mine = q < total;
      const float4 pos = mine ? a.ppos[og] : make_float4(0.f, 0.f, 1.f, 0.f);
      const int pidx = __float_as_int(pos.w);
      int id = 0;
      bool dif = false;
      int64_t slot = 0;
      if (mine) {
        if (REF) {
          const int code = (otg >> (8 * k)) & 0xff;
          dif = (code & RT_DIF) != 0;
          id = code & ~RT_DIF;
          // (targets: differences first, each kind in consecutive slots)
          const int nd = ((otg & RT_DIF) ? 1 : 0) + ((otg >> 8) != 0xff && (otg & (RT_DIF << 8)) ? 1 : 0);
          slot = dif ? os1 + k : os0 + (k - nd);
        } else {
          id = ostage == ST_INIT ? k : (ostage == ST_SHRINK ? (oorder >> (4 * (k + 1))) & 15 : VID_E);
          slot = os0 + k;
        }
      }
      // the last float-float value becomes the point's reference
      const bool newref = REF && mine && !dif && a.o.tie_dif > 0.0 && (k == 1 || (otg >> 8) == 0xff);
      double S[12];
      if (quads) {
        const ProbDesc& pd = a.probs[pidx];
        double Sq[4];
        if (REF) {
          value_quad(a, mine, true, dif, dif ? a.dout : a.fout, dif ? *a.dplan : *a.fplan, slot, 0, pd,
                     nullptr, 0, id, og, pos.z, Sq);
        } else {
          value_quad(a, mine, false, false, a.out, h, slot - queue_base(a, pd),
                     near_skip(a, pd, (double)pos.z), pd, a.item_off, pidx, id, og, pos.z, Sq);
        }
        __syncwarp();   // the differences have read the old reference sums
        if (newref && (lane & 3) < 3) {
          SD(a, D_REFL + (lane & 3), og) = SV(a, id, V_L + (lane & 3), og);
#pragma unroll
          for (int s = 0; s < 4; ++s) SD(a, D_REFS + 4 * (lane & 3) + s, og) = Sq[s];
        }
      } else {
        if (mine) {
          Eval ev;
          const double lq[3] = {SV(a, id, V_L, og), SV(a, id, V_L + 1, og), SV(a, id, V_L + 2, og)};
          if (REF) read_reeval(a, dif, pidx, slot, (double)pos.z, ev, og, lq, S);
          else read_eval(a, h, pidx, slot, (double)pos.z, ev, og, lq);
          store_value(a, id, og, ev);
        }
        __syncwarp();
        if (newref) {
          for (int d = 0; d < 3; ++d) SD(a, D_REFL + d, og) = SV(a, id, V_L + d, og);
          for (int s = 0; s < 12; ++s) SD(a, D_REFS + s, og) = S[s];
        }
      }
    }
    __syncwarp();     // values are in the state

    // ---- phase 2: the step of the lane's point
    bool emit_trial = false;
    double coef_c = 0.0, coef_w = 0.0;   // next trial point: coef_c centroid + coef_w worst
    float4 pos = make_float4(0.f, 0.f, 1.f, 0.f);
    auto decide = [&]() {
    pos = a.ppos[g];
    const int pidx = __float_as_int(pos.w);
    int iters = SI(a, I_ITERS, g);
    int nfev = SI(a, I_NFEV, g) + (REF ? 0 : nev);
    const bool single = stage != ST_INIT && stage != ST_SHRINK;
    TieLog tl{-1, -1};
    auto vert = [&](int id, int slot) {
      return Vert{SV(a, id, V_PHI, g), f32_of(SV(a, id, V_S, g)), slot, id};
    };
    Vert w[N + 1], e{}, R{};
#pragma unroll
    for (int k = 0; k <= n; ++k) {
      const int sl = (order >> (4 * k)) & 15;
      w[k] = vert(sl, sl);
    }
    if (single) e = vert(VID_E, 0);
    if (stage == ST_EXPAND || stage == ST_OCONTRACT) R = vert(VID_R, 0);
    bool to_check = false, store_R = false, emit_shrink = false;
    bool mirror = false;
    int next_stage = stage;
    int taken = -1;                      // record that takes the worst vertex's slot
    char code = 0;
    int fin = -1;
    auto trial = [&](double cc, double cw) {
      coef_c = cc;
      coef_w = cw;
      emit_trial = true;
    };
    auto take = [&](const Vert& x, char c) {
      w[n].phi = x.phi;
      w[n].s = x.s;
      w[n].id = taken = x.id;
      code = c;
      to_check = true;
    };

    if (stage == ST_INIT) {
      to_check = true;
    } else if (stage == ST_REFLECT) {
      if (tl.lt(e, w[0])) {
        store_R = true;
        trial(1.0 + rho * chi, -(rho * chi));
        next_stage = ST_EXPAND;
      } else if (tl.lt(e, w[n - 1])) {
        take(e, 'R');
      } else if (tl.lt(e, w[n])) {
        store_R = true;
        trial(1.0 + psi * rho, -(psi * rho));
        next_stage = ST_OCONTRACT;
      } else {
        trial(1.0 - psi, psi);
        next_stage = ST_ICONTRACT;
      }
    } else if (stage == ST_EXPAND) {
      if (tl.lt(e, R)) take(e, 'E');
      else take(R, 'R');
    } else if (stage == ST_OCONTRACT || stage == ST_ICONTRACT) {
      const bool ok = (stage == ST_OCONTRACT) ? tl.le(e, R) : tl.lt(e, w[n]);
      if (ok) {
        take(e, (stage == ST_OCONTRACT) ? 'O' : 'I');
      } else {
        next_stage = ST_SHRINK;
        emit_shrink = true;
      }
    } else if (stage == ST_SHRINK) {
      code = 'S';
      to_check = true;
    }
    if (to_check) {
      sort_verts<N>(w, tl);
      // Eq. 12 at the best vertex, then the value spread, then the iteration count
      const double f0 = SV(a, w[0].id, V_F, g), g0 = SV(a, w[0].id, V_G, g);
      const bool f_met = less_eq(f0, a.o.eps_f), g_met = less_eq(g0, a.o.eps_g);
      tl.note(w[0], f0, a.o.eps_f);
      if (f_met) tl.note(w[0], g0, a.o.eps_g);
      if (f_met && g_met) {
        fin = PT_CONVERGED;
      } else {
        const double spread = w[n].phi - w[0].phi;
        tl.note(w[n].id, w[n].s, w[0].id, w[0].s, spread, a.o.tol);
        if (less_eq(spread, a.o.tol)) fin = PT_CONVERGED;
        else if (iters >= a.o.max_iter) fin = PT_MAXITER;
      }
      if (fin < 0) {
        if (n == 1 && SV(a, w[0].id, V_L, g) == 0.0) {
          // Mirror step: with the best vertex at lambda = 0 the reflection is -w[1], where Phi
          // (even in lambda, Eq. 6) takes w[1]'s value exactly.  Its comparisons are settled
          // (not below w[0], by the sort just done; not below w[1], by equality), so the step
          // goes straight to the inside contraction, and the reflection is counted as the
          // evaluation the search makes.  Every form then decides these exact ties as exact
          // arithmetic does, instead of by the rounding of two sums.
          trial(1.0 - psi, psi);
          next_stage = ST_ICONTRACT;
          mirror = true;
        } else {
          trial(1.0 + rho, -rho);
          next_stage = ST_REFLECT;
        }
      }
    }

    if (tl.a >= 0) {
      // near tie: keep the state and re-evaluate the near-tied values (tl.a >= 0 always;
      // tl.b >= 0 when both values carry a bound)
      double lt[2][3];
      const int ida = tl.a, idb = tl.b;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        lt[0][d] = SV(a, ida, V_L + d, g);
        lt[1][d] = idb < 0 ? 0.0 : SV(a, idb, V_L + d, g);
      }
      // A value goes to the difference pass when the point has a float-float reference, the
      // value still carries its mixed-form bound and it lies near the reference (the difference
      // bound, relative to the mixed one, grows as |lambda - lambda_ref| times the point's mean
      // pixel distance sum |b| / sum |b| / r: estimated below about 0.5 here); otherwise to
      // float-float.  Without a reference only the value with the larger bound goes to
      // float-float: it becomes the reference, and the other value, if still near-tied, goes
      // to the difference pass in the next round.
      int k = idb >= 0 ? 2 : 1;
      int id0 = ida, id1 = idb;
      bool dif[2] = {false, false};
      double lref[3] = {0.0, 0.0, 0.0};
      if (a.o.tie_dif > 0.0) {
        const float sv[2] = {f32_of(SV(a, ida, V_S, g)), idb < 0 ? 0.f : f32_of(SV(a, idb, V_S, g))};
        if (!isnan(SD(a, D_REFS, g))) {
#pragma unroll
          for (int d = 0; d < 3; ++d) lref[d] = SD(a, D_REFL + d, g);
          bool near[2] = {sv[0] > 0.f, k > 1 && sv[1] > 0.f};
#pragma unroll
          for (int p = 0; p < 3; ++p) {
            const int q = n == 1 ? 0 : p;
            const float m1 = a.msc[15 * g + 5 * p];
            const float reach = m1 > 0.f ? a.msc0[3 * g + p] / m1 : 0.f;
#pragma unroll
            for (int j = 0; j < 2; ++j)
              near[j] = near[j] && fabsf(f32_of(lt[j][q]) - f32_of(lref[q])) * reach < 0.25f;
          }
          dif[0] = near[0];
          dif[1] = near[1];
        } else if (k == 2 && sv[0] > 0.f && sv[1] > 0.f) {
          k = 1;
          if (sv[1] > sv[0]) {
            id0 = idb;
#pragma unroll
            for (int d = 0; d < 3; ++d) lt[0][d] = lt[1][d];
          }
        }
      }
      emit_reeval(a, REF ? a.nxt : a.cur, g, pos, k, lt, id0, id1, dif, lref);
      SI(a, I_NFEV, g) = nfev;
      emit_trial = false;
      return;
    }

    // ---- the step is certain: take it
    if (code && a.codes && iters >= 1 && iters <= a.codes_stride)
      a.codes[g * a.codes_stride + (iters - 1)] = code;
    if (fin >= 0) {
      for (int p = 0; p < 3; ++p) {
        a.res_B[3 * g + p] = SV(a, w[0].id, V_B + p, g);
        a.res_lam[3 * g + p] = fabs(SV(a, w[0].id, V_L + (n == 1 ? 0 : p), g));
      }
      a.res_f[g] = SV(a, w[0].id, V_F, g);
      a.res_g[g] = SV(a, w[0].id, V_G, g);
      a.res_iters[g] = iters;
      a.res_status[g] = fin;
      a.res_nfev[g] = nfev;
      stage = ST_DONE;
      SI(a, I_STATUS, g) = fin;
    } else {
      if (store_R || taken >= 0) {
        int to = VID_R;
        if (taken >= 0) {
#pragma unroll
          for (int k = 0; k <= n; ++k)
            if (w[k].id == taken) to = w[k].slot;
        }
        copy_value(a, taken >= 0 ? taken : VID_E, to, g);
      }
      if (to_check) {
        iters += 1;
        int ord = 0;
#pragma unroll
        for (int k = 0; k <= n; ++k) ord |= w[k].slot << (4 * k);
        SI(a, I_ORDER, g) = order = ord;
      }
      if (mirror) nfev += 1;
      if (emit_shrink) {
        double rows[N][3], l0[3];
        for (int d = 0; d < 3; ++d) l0[d] = SV(a, w[0].slot, V_L + d, g);
#pragma unroll
        for (int k = 1; k <= n; ++k)
          for (int d = 0; d < 3; ++d) {
            const double l = SV(a, w[k].slot, V_L + d, g);
            rows[k - 1][d] = (d < n) ? l0[d] + sigma * (l - l0[d]) : 0.0;
            SV(a, w[k].slot, V_L + d, g) = rows[k - 1][d];
          }
        emit<N>(a, g, pos, pidx, rows);
      }
      stage = next_stage;
    }
    SI(a, I_STAGE, g) = stage;
    SI(a, I_ITERS, g) = iters;
    SI(a, I_NFEV, g) = nfev;
    };
    if (on) decide();
    // The lanes of phase 3 read vertices that other lanes have just stored (copy_value), and
    // overwrite the lambdas of trial records that other lanes have just copied from.  (The votes and
    // shuffles below order no memory.)
    __syncwarp();

    // ---- phase 3: the trial points, a lane per lambda of a point (seven FP64 instructions a pass)
    const unsigned trials = __ballot_sync(FULL, emit_trial);
    for (unsigned left = trials; left;) {
      constexpr int PER = 32 / n;                      // points per pass
      const int k = lane / n, d = lane - k * n;
      unsigned m = left;
      for (int i = 0; i < k && m; ++i) m &= m - 1u;    // the k-th point of this pass
      const bool act = k < PER && m != 0;
      const int o = act ? __ffs(m) - 1 : 0;
      const int64_t og = __shfl_sync(FULL, gi, o);
      const int oord = __shfl_sync(FULL, order, o);
      const double cc = __shfl_sync(FULL, coef_c, o), cw = __shfl_sync(FULL, coef_w, o);
      double row = 0.0;
      if (act) {
        double c = 0.0;
#pragma unroll
        for (int i = 0; i < n; ++i) c += SV(a, (oord >> (4 * i)) & 15, V_L + d, og);
        // (cw is a power of two: its product is exact, the fma rounds as the sum does)
        row = __fma_rn(cw, SV(a, (oord >> (4 * n)) & 15, V_L + d, og), cc * over<n>(c));
        SV(a, VID_E, V_L + d, og) = row;
        if (n == 1) SV(a, VID_E, V_L + 1, og) = SV(a, VID_E, V_L + 2, og) = 0.0;
      }
      // back to the owners
      const int rank = __popc(left & ((1u << lane) - 1u));
      const bool done = ((left >> lane) & 1u) && rank < PER;
      double rows[1][3] = {{0.0, 0.0, 0.0}};
#pragma unroll
      for (int i = 0; i < n; ++i) rows[0][i] = __shfl_sync(FULL, row, done ? rank * n + i : 0);
      if (done) emit<1>(a, g, pos, __float_as_int(pos.w), rows);
      left &= ~__ballot_sync(FULL, done);
    }
    __syncwarp();
  }
}

}  // namespace dbie
