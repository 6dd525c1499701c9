// solve.cu -- per-point objective and the on-device Downhill Simplex search for lambda.
//
// Compiled with -fmad=false: the simplex arithmetic and the objective are evaluated with
// separately rounded operations, as written.
//
//  * objective: B_p = z S0_p, dB_p/dx = z Sx_p, dB_p/dy = z Sy_p, dB_p/dz = S0_p + z^2 S1_p
//    (the fixed-lambda derivatives of Eq. 13), J = curl B (Eq. 14), f = |J x B| / (|J||B|)
//    (Eq. 8), g = |div B| dV/dSigma / |B| (Eq. 9), Phi = f + w_g g.
//  * simplex (Sect. 2.1; Nelder & Mead 1965, reflection 1, expansion 2, contraction 1/2,
//    shrink 1/2, outside/inside contraction as in Lagarias et al. 1998): one thread per active
//    point advances a state machine by one step per round; every round evaluates all pending
//    trial points of all active points in one pair-sum pass.
#include "kernels.h"
#include "solve.cuh"
#include "warp_sums.cuh"

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

// ----------------------------------------------------------------- eval finalize ----
template <int VAR>
__global__ void finalize_eval_kernel(int64_t n, const PlanHdr* __restrict__ plan,
                                     const int32_t* __restrict__ item_off,
                                     const double* __restrict__ out,
                                     const float4* __restrict__ qpos,
                                     const Lam4* __restrict__ qlam, double g_scale, double w_g,
                                     double* B, double* gradB, double* dBdl, const double* gB,
                                     double* fgphi, const double* corr) {
  constexpr int NS = nsum_per_comp(VAR);
  constexpr int NSUM = 3 * NS;
  const PlanHdr h = *plan;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float4 pos = qpos[i];
    const double z = (double)pos.z;
    double S[NSUM];
    gather_sums<NSUM>(out, h, item_off, 0, i, S);
    double Bv[3], G[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int p = 0; p < 3; ++p) Bv[p] = z * S[p * NS];
    if constexpr (has_grad(VAR)) {
      for (int p = 0; p < 3; ++p) {
        G[3 * p + 0] = z * S[p * NS + 2];
        G[3 * p + 1] = z * S[p * NS + 3];
        G[3 * p + 2] = S[p * NS] + z * z * S[p * NS + 1];
      }
    }
    add_corr(corr ? corr + 12 * i : nullptr, Bv, G);
    if (B)
      for (int p = 0; p < 3; ++p) B[3 * i + p] = Bv[p];
    if constexpr (has_grad(VAR)) {
      if (gradB)
        for (int j = 0; j < 9; ++j) gradB[9 * i + j] = G[j];
      if (fgphi) {
        double f, g, phi;
        objective(Bv, G, g_scale, w_g, f, g, phi);
        fgphi[3 * i + 0] = f;
        fgphi[3 * i + 1] = g;
        fgphi[3 * i + 2] = phi;
      }
    }
    if constexpr (has_dlam(VAR)) {
      const Lam4 l = qlam[i];
      const double lam[3] = {l.x, l.y, l.z};
      for (int p = 0; p < 3; ++p) {
        const double d = z * lam[p] * S[p * NS + idx_sl(VAR)];
        if (gB) {
          if (dBdl) dBdl[3 * i + p] = gB[3 * i + p] * d;
        } else if (dBdl) {
          dBdl[3 * i + p] = d;
        }
      }
    }
  }
}

void launch_finalize_eval(int var, int64_t n, const PlanHdr* plan, const int32_t* item_off,
                          const double* out, const float4* qpos, const Lam4* qlam, double g_scale,
                          double w_g, double* B, double* gradB, double* dBdl, const double* gB,
                          double* fgphi, const double* corr, cudaStream_t s) {
  if (n <= 0) return;
  const PerPoint L(n);
#define FIN(V)                                                                                \
  finalize_eval_kernel<V><<<L.grid, L.nt, 0, s>>>(n, plan, item_off, out, qpos, qlam, g_scale, \
                                                  w_g, B, gradB, dBdl, gB, fgphi, corr)
  switch (var) {
    case VAR_V: FIN(VAR_V); break;
    case VAR_VL: FIN(VAR_VL); break;
    case VAR_OBJ: FIN(VAR_OBJ); break;
    default: FIN(VAR_OBJL); break;
  }
#undef FIN
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

// The bounds are evaluated in FP32: a dependent FP64 instruction takes 70 cycles and more here, the
// bound took two thirds of a value's time, and a worst case whose coefficients have two or three
// digits (and M_j, summed from FP32 terms) does not need more.
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
// Norm without overflow or underflow of the squares.
__device__ __forceinline__ float norm3f(float x, float y, float z) {
  const float m = fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z)));
  if (!(m > 0.f)) return m;
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
  if (sf > 1.0f) sf = 1.0f;
  const float sg = f32_of(g_scale) * (dG[0] + dG[4] + dG[8]) / nB + f32_of(e.g) * rB;
  return sf + f32_of(w_g) * sg;
}

__device__ __forceinline__ float mixed_phi_bound(const float* M, const double lam[3], int dim,
                                                 float z, const Eval& e, double g_scale,
                                                 double w_g) {
  constexpr float A0 = BND_A0, A1 = BND_A1, A2 = BND_A2, A3 = BND_A3, A4 = BND_A4;
  float dB[3], dG[9];
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const float L = fabsf(f32_of(dim == 1 ? lam[0] : lam[p]));
    const float* m = M + 5 * p;
    const float L2 = L * L, L3 = L2 * L;
    const float s0 = A0 * m[2] + A1 * L * m[1] + A2 * L2 * m[0];
    const float sx = A0 * L2 * m[1] + A2 * L3 * m[0] +
                     3.0f * (A3 * m[3] + A4 * L * m[2] + A2 * L2 * m[1]);
    const float s1 = A0 * L2 * m[2] + A2 * L3 * m[1] +
                     3.0f * (A3 * m[4] + A4 * L * m[3] + A2 * L2 * m[2]);
    dB[p] = z * s0;
    dG[3 * p + 0] = z * sx;
    dG[3 * p + 1] = z * sx;
    dG[3 * p + 2] = s0 + z * z * s1;
  }
  return propagate_bound(dB, dG, e, g_scale, w_g);
}

// Error bounds of the difference sums (pairsum_dif.cu) that take a point's float-float
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

// e[4 p + s]: bounds of S0, S1, Sx, Sy of component p (M: M_1..M_5 per component, M0: M_0; per free
// lambda, dl = |lambda_a - lambda_0|, L = |lambda_a| + |lambda_0| and R = |lambda_0|).
template <typename T>
__device__ __forceinline__ void dif_sum_bounds(const T* M, const T* M0, const T dl_[3],
                                               const T L_[3], const T R_[3], int dim, T e[12]) {
  constexpr T C00 = DIF_C00, C01 = DIF_C01, C02 = DIF_C02, C10 = DIF_C10, C11 = DIF_C11,
              C12 = DIF_C12, C13 = DIF_C13, FF = DIF_FF;
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const int q = dim == 1 ? 0 : p;
    const T dl = dl_[q], L = L_[q], L2 = L * L, L3 = L2 * L;
    const T R = R_[q], R2 = R * R;
    const T* m = M + 5 * p;   // m[j - 1] = M_j
    const T m0 = M0[p];
    const T e0 = dl * (C00 * m[1] + C01 * L * m[0] + C02 * L2 * m0) + FF * (m[2] + R * m[1]);
    const T e1 = dl * (C10 * m[3] + C11 * L * m[2] + C12 * L2 * m[1] + C13 * L3 * m[0]) +
                 FF * (T(3) * m[4] + T(3) * R * m[3] + R2 * m[2]);
    const T ex = dl * (C10 * m[2] + C11 * L * m[1] + C12 * L2 * m[0] + C13 * L3 * m0) +
                 FF * (T(3) * m[3] + T(3) * R * m[2] + R2 * m[1]);
    e[4 * p + 0] = e0;
    e[4 * p + 1] = e1;
    e[4 * p + 2] = ex;
    e[4 * p + 3] = ex;
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

// Tie radius of a value: `band` times its bound (never 0, which marks a value without one).
__device__ __forceinline__ float radius_of(double band, float bound) {
  const float r = f32_of(band) * bound;
  return r < 1e-37f ? 1e-37f : r;
}

// The first near tie of a step: a comparison whose two values differ by no more than the sum of
// their tie radii.  A mixed-form value carries the radius band x bound (certify), a value
// re-evaluated by difference certify_ref x bound, stored negated, and one re-evaluated in
// float-float 0.  (No value carries one when decisions are not certified.)
struct TieLog {
  int a, b;        // ids of the first near-tied values (-1: none)
  // values ia, ib with signed radii ra, rb
  __device__ __forceinline__ void note(int ia, float ra, int ib, float rb, double gap) {
    if (a < 0 && (ra != 0.f || rb != 0.f)) {
      const float r = fabsf(ra) + fabsf(rb);
      if (less_eq(fabs(gap), f64_of(r))) {
        a = ra != 0.f ? ia : -1;
        b = rb != 0.f ? ib : -1;
        if (a < 0) { a = b; b = -1; }
      }
    }
  }
  __device__ __forceinline__ void note(const Vert& x, double gap) { note(x.id, x.s, -1, 0.f, gap); }
  __device__ __forceinline__ void note(const Vert& x, const Vert& y, double gap) {
    note(x.id, x.s, y.id, y.s, gap);
  }
  __device__ __forceinline__ bool lt(const Vert& x, const Vert& y) {
    note(x, y, x.phi - y.phi);
    return less(x.phi, y.phi);
  }
  __device__ __forceinline__ bool le(const Vert& x, const Vert& y) {
    note(x, y, x.phi - y.phi);
    return less_eq(x.phi, y.phi);
  }
};

// Objective of the k-th pending query of point g; its error bound when decisions are certified.
__device__ __forceinline__ void read_eval(const SolveArgs& a, const PlanHdr& h, int pidx,
                                          int64_t slot, double z, Eval& e, int64_t g,
                                          const double lam[3]) {
  const ProbDesc& pd = a.probs[pidx];
  double S[12], G[9];
  // (of a pass of few queries the last record is the near field's: zero above near_z)
  const int skip = a.one_queue && a.o.near_on && !less_eq(z, pd.near_z) ? 1 : 0;
  gather_sums<12>(a.out, h, a.item_off, pidx, slot - queue_base(a, pd), S, skip);
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

// N: the number of free lambdas (3, or 1 when the components share one).
template <int N>
__global__ void solve_init_kernel(const SolveArgs a, const double* __restrict__ lam_init) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < a.N;
       g += (int64_t)gridDim.x * blockDim.x) {
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
}

void launch_solve_init(const SolveArgs& a, const double* lam_init, int grid, cudaStream_t s) {
  if (a.o.dim == 1) solve_init_kernel<1><<<grid, 256, 0, s>>>(a, lam_init);
  else solve_init_kernel<3><<<grid, 256, 0, s>>>(a, lam_init);
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

// Points of one warp of a step kernel.  A warp's time is its chain of dependent FP64 instructions
// (70 to 150 cycles each), not the FP64 rate, so a few points are spread over all SMs and their
// sub-partitions, one warp each, with as few lanes (fewer of them in different stages) as that
// needs; full warps come when there are more than 128 points per SM.  (2,048 points in warps of
// 14, 7, 4 and 2: 8.6, 8.2, 8.0 and 8.2 ms per search.)
constexpr int STEP_NT = 128;
__device__ __forceinline__ int points_per_warp(int n, int nsm) {
  const int p = (n + 4 * nsm - 1) / (4 * nsm);
  return p < 1 ? 1 : (p > 32 ? 32 : p);
}

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
// What bounds it: one warp's chain of instructions, its FP64 instructions above all (70 to 150
// cycles each), so the time is the instruction count of the longest warp.  Hence FP64 only where the
// values and lambdas are formed (comparisons on the integer pipe, bounds in FP32), and two
// phases.  First the lanes share out the values to compute, one FP64 objective and bound per lane
// whatever the points' stages (a shrink has 3, the start 4; taken in turn by the point's own lane
// they set the length for the whole warp).  Then each lane decides its point's step on Phi and
// bound alone; vertices stay in their slots, and a step writes one record, not four.  On 2,048
// points a step took 63 us (the waiting points' 112 us) with one lane per point evaluating and
// sorting whole vertices, in CTAs of 128 threads.
template <int N, bool REF>
__global__ void __launch_bounds__(STEP_NT) nm_step_kernel(const SolveArgs a) {
  const double rho = 1.0, chi = 2.0, psi = 0.5, sigma = 0.5;
  const unsigned FULL = 0xffffffffu;
  const int nact = REF ? *a.cur.ref_cnt : *a.cur.act_cnt;
  const int32_t* list = REF ? a.cur.ref : a.cur.act;
  constexpr int n = N;
  const PlanHdr h = *a.plan;
  if (!REF && a.rework && blockIdx.x == 0 && threadIdx.x == 0) a.rework[0] = a.rework[1] = 0;
  const int ppw = points_per_warp(nact, a.nsm);
  const int lane = threadIdx.x & 31;
  const int warp = blockIdx.x * (STEP_NT / 32) + (threadIdx.x >> 5);
  const int nwarps = gridDim.x * (STEP_NT / 32);
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
    for (int q0 = 0; q0 < total; q0 += 32) {
      const int q = q0 + lane;
      int o = 0;   // the point (lane) that owns value q: the first with incl > q
#pragma unroll
      for (int st = 16; st > 0; st >>= 1)
        if (__shfl_sync(FULL, incl, o + st - 1) <= q) o += st;
      const int k = q - (__shfl_sync(FULL, incl, o) - __shfl_sync(FULL, nev, o));
      const int64_t og = __shfl_sync(FULL, gi, o);
      const int ostage = __shfl_sync(FULL, stage, o), oorder = __shfl_sync(FULL, order, o);
      const int otg = __shfl_sync(FULL, targets, o);
      const int os0 = __shfl_sync(FULL, slot0, o), os1 = __shfl_sync(FULL, slot1, o);
      double S[12];
      bool newref = false;
      if (q < total) {
        const float4 pos = a.ppos[og];
        const int pidx = __float_as_int(pos.w);
        Eval ev;
        int id;
        bool dif = false;
        if (REF) {
          const int code = (otg >> (8 * k)) & 0xff;
          dif = (code & RT_DIF) != 0;
          id = code & ~RT_DIF;
        } else {
          id = ostage == ST_INIT ? k : (ostage == ST_SHRINK ? (oorder >> (4 * (k + 1))) & 15 : VID_E);
        }
        const double lq[3] = {SV(a, id, V_L, og), SV(a, id, V_L + 1, og), SV(a, id, V_L + 2, og)};
        if (REF) {
          // (targets: differences first, each kind in consecutive slots)
          const int nd = ((otg & RT_DIF) ? 1 : 0) + ((otg >> 8) != 0xff && (otg & (RT_DIF << 8)) ? 1 : 0);
          read_reeval(a, dif, pidx, dif ? os1 + k : os0 + (k - nd), (double)pos.z, ev, og, lq, S);
          // the last float-float value becomes the point's reference
          newref = !dif && a.o.tie_dif > 0.0 && (k == 1 || (otg >> 8) == 0xff);
        } else {
          read_eval(a, h, pidx, os0 + k, (double)pos.z, ev, og, lq);
        }
        store_value(a, id, og, ev);
        if (newref)
          for (int d = 0; d < 3; ++d) SD(a, D_REFL + d, og) = lq[d];
      }
      __syncwarp();   // the differences have read the old reference sums
      if (newref)
        for (int s = 0; s < 12; ++s) SD(a, D_REFS + s, og) = S[s];
    }
    __syncwarp();     // values are in the state
    if (!on) continue;

    // ---- phase 2: the step of the lane's point
    const float4 pos = a.ppos[g];
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
    bool to_check = false, store_R = false, emit_shrink = false, emit_trial = false;
    bool mirror = false;
    int next_stage = stage;
    int taken = -1;                      // record that takes the worst vertex's slot
    double coef_c = 0.0, coef_w = 0.0;   // next trial point: coef_c centroid + coef_w worst
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
      tl.note(w[0], f0 - a.o.eps_f);
      if (f_met) tl.note(w[0], g0 - a.o.eps_g);
      if (f_met && g_met) {
        fin = PT_CONVERGED;
      } else {
        const double spread = w[n].phi - w[0].phi;
        tl.note(w[n], w[0], spread - a.o.tol);
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
              near[j] = near[j] && fabsf(f32_of(lt[j][q] - lref[q])) * reach < 0.25f;
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
      continue;
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
        SI(a, I_ORDER, g) = ord;
      }
      if (mirror) nfev += 1;
      if (emit_trial) {
        // one site for every kind of step: its divisions are run once per warp
        double rows[1][3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          double s = 0.0;
          if (d < n) {
#pragma unroll
            for (int k = 0; k < n; ++k) s += SV(a, w[k].slot, V_L + d, g);
            // (coef_w is a power of two: its product is exact, the fma rounds as the sum does)
            rows[0][d] = __fma_rn(coef_w, SV(a, w[n].slot, V_L + d, g), coef_c * over<n>(s));
          } else {
            rows[0][d] = 0.0;
          }
        }
        for (int d = 0; d < 3; ++d) SV(a, VID_E, V_L + d, g) = rows[0][d];
        emit<1>(a, g, pos, pidx, rows);
      } else if (emit_shrink) {
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
  }
}

void launch_nm_step(const SolveArgs& a, int grid, cudaStream_t s) {
  if (a.o.dim == 1) nm_step_kernel<1, false><<<grid, STEP_NT, 0, s>>>(a);
  else nm_step_kernel<3, false><<<grid, STEP_NT, 0, s>>>(a);
}
void launch_nm_refine(const SolveArgs& a, int grid, cudaStream_t s) {
  if (a.o.dim == 1) nm_step_kernel<1, true><<<grid, STEP_NT, 0, s>>>(a);
  else nm_step_kernel<3, true><<<grid, STEP_NT, 0, s>>>(a);
}

// --------------------------------------------------------------- per-round plan ----
__global__ void plan_round_kernel(const PlanArgs a) {
  __shared__ long long s_blocks;
  __shared__ int s_minTiles;
  if (threadIdx.x == 0) {
    s_blocks = 0;
    s_minTiles = 1 << 30;
  }
  __syncthreads();
  for (int p = threadIdx.x; p < a.nprob; p += blockDim.x) {
    const int q = a.q_cnt_cur[p];
    a.q_cnt_pass[p] = q;
    if (q > 0) {
      atomicAdd((unsigned long long*)&s_blocks, (unsigned long long)((q + a.qper - 1) / a.qper));
      atomicMin(&s_minTiles, a.probs[p].ntiles);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const long long blocks = s_blocks;
    int nsplit = 1;
    if (blocks > 0 && blocks < a.target_items) {
      nsplit = (int)((a.target_items + blocks - 1) / blocks);
      if (nsplit > a.nsplit_cap) nsplit = a.nsplit_cap;
      if (nsplit > s_minTiles) nsplit = s_minTiles;
      if (nsplit < 1) nsplit = 1;
    }
    int acc = 0;
    double pairs = 0.0;
    unsigned long long queries = 0;
    for (int p = 0; p < a.nprob; ++p) {
      a.item_off[p] = acc;
      const int q = a.q_cnt_pass[p];
      acc += ((q + a.qper - 1) / a.qper) * nsplit;
      pairs += (double)q * (double)(a.probs[p].nx) * (double)(a.probs[p].ny);
      queries += (unsigned long long)q;
    }
    a.item_off[a.nprob] = acc;
    PlanHdr h;
    h.nitems = acc;
    h.nsplit = nsplit;
    h.qper = a.qper;
    h.pad0 = 0;
    *a.plan = h;
    *a.work = 0;
    *a.act_cnt_nxt = 0;
    *a.near_cnt_nxt = 0;
    if (a.fq_cnt_nxt) *a.fq_cnt_nxt = 0;
    if (a.dq_cnt_nxt) *a.dq_cnt_nxt = 0;
    if (a.ref_cnt_nxt) *a.ref_cnt_nxt = 0;
    *a.round_ctr += 1;
    *a.stat_queries += queries;
    *a.stat_pairs += pairs;
  }
  for (int p = threadIdx.x; p < a.nprob; p += blockDim.x) {
    if (a.q_cnt_nxt) a.q_cnt_nxt[p] = 0;
  }
}

void launch_plan_round(const PlanArgs& a, cudaStream_t s) { plan_round_kernel<<<1, 256, 0, s>>>(a); }

// The lambda-independent absolute-value sums of every point, the coefficients of the mixed
// form's error bound: msc[15 g + 5 p + j - 1] = sum_k |b_pk| / r_gk^j, j = 1..5, and msc0[3 g + p] =
// sum_k |b_pk|, over the quadrature points of the point's problem.  FP32 terms summed per 256
// pixels of a thread, those in float pairs (relative error below 1e-4: a scale, not a result).
// FP32 issue bounds it (about 30 instructions per pair); a point per CTA, its lanes taking four
// pixels each, keeps a search of few points from walking the boundary pixel by pixel (2,048 points
// over 32 x 32 pixels: 100 us with a thread per point).
constexpr int MSC_NT = 128;
template <typename T>
__global__ void __launch_bounds__(MSC_NT) msc_kernel(const ProbDesc* __restrict__ probs, int64_t N,
                                                     const float4* __restrict__ ppos,
                                                     T* __restrict__ msc, T* __restrict__ msc0) {
  constexpr int NSUM = 18;
  __shared__ double s_red[MSC_NT / 32][NSUM];
  const int lane = threadIdx.x & 31;
  for (int64_t g = blockIdx.x; g < N; g += gridDim.x) {
    const float4 pos = ppos[g];
    const ProbDesc& pd = probs[__float_as_int(pos.w)];
    const float z2 = __fmul_rn(pos.z, pos.z);
    const int groups = pd.ntiles * (TILE / 4);
    ff::ds tot[NSUM];
#pragma unroll
    for (int i = 0; i < NSUM; ++i) tot[i] = ff::ds{0.f, 0.f};
    for (int q0 = threadIdx.x; q0 < groups; q0 += 64 * MSC_NT) {
      float acc[NSUM];
#pragma unroll
      for (int i = 0; i < NSUM; ++i) acc[i] = 0.f;
      const int q1 = q0 + 64 * MSC_NT < groups ? q0 + 64 * MSC_NT : groups;
      for (int q = q0; q < q1; q += MSC_NT) {
        const float* T32 = pd.tiles32 + (int64_t)(q / (TILE / 4)) * pd.nf32 * TILE +
                           (q % (TILE / 4)) * 4;
        auto ld = [&](int f) { return __ldg(reinterpret_cast<const float4*>(T32 + f * TILE)); };
        const float4 X = ld(0), Y = ld(1), B[3] = {ld(2), ld(3), ld(4)};
        const float x[4] = {X.x, X.y, X.z, X.w}, y[4] = {Y.x, Y.y, Y.z, Y.w};
        const float b[3][4] = {{B[0].x, B[0].y, B[0].z, B[0].w},
                               {B[1].x, B[1].y, B[1].z, B[1].w},
                               {B[2].x, B[2].y, B[2].z, B[2].w}};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float dx = pos.x - x[e], dy = pos.y - y[e];
          const float ri = rsqrtf(__fmaf_rn(dx, dx, __fmaf_rn(dy, dy, z2)));
          float wj = 1.f;
#pragma unroll
          for (int j = 0; j < 6; ++j) {   // acc[3 j + p]: M_j of component p
#pragma unroll
            for (int p = 0; p < 3; ++p) acc[3 * j + p] = __fmaf_rn(fabsf(b[p][e]), wj, acc[3 * j + p]);
            wj *= ri;
          }
        }
      }
#pragma unroll
      for (int i = 0; i < NSUM; ++i) ff::acc_add(tot[i], ff::ds{acc[i], 0.f});
    }
    const ff::ds r = WarpSums<NSUM>::reduce(tot, lane);
    __syncthreads();   // the previous point's sums are read
    if (lane < NSUM) s_red[threadIdx.x >> 5][lane] = ff::to_double(r);
    __syncthreads();
    if (threadIdx.x < NSUM) {
      double t = s_red[0][threadIdx.x];
#pragma unroll
      for (int w = 1; w < MSC_NT / 32; ++w) t += s_red[w][threadIdx.x];
      const int j = threadIdx.x / 3, p = threadIdx.x % 3;
      if (j > 0) msc[15 * g + 5 * p + j - 1] = (T)t;
      else msc0[3 * g + p] = (T)t;
    }
  }
}

template <typename T>
static void launch_msc_t(const ProbDesc* probs, int64_t N, const float4* ppos, T* msc, T* msc0,
                         int sm_count, cudaStream_t s) {
  const int64_t most = 16LL * sm_count;
  if (N > 0) msc_kernel<T><<<(int)(N < most ? N : most), MSC_NT, 0, s>>>(probs, N, ppos, msc, msc0);
}
void launch_msc(const ProbDesc* probs, int64_t N, const float4* ppos, float* msc, float* msc0,
                int sm_count, cudaStream_t s) {
  launch_msc_t(probs, N, ppos, msc, msc0, sm_count, s);
}
void launch_msc(const ProbDesc* probs, int64_t N, const float4* ppos, double* msc, double* msc0,
                int sm_count, cudaStream_t s) {
  launch_msc_t(probs, N, ppos, msc, msc0, sm_count, s);
}

// Difference sums of n queries of one problem (slots 0..n-1) and their bounds (debug entry).
__global__ void dif_debug_kernel(int64_t n, const PlanHdr* __restrict__ plan,
                                 const double* __restrict__ out, const Lam4* __restrict__ qlam,
                                 const Lam4* __restrict__ qlam0, const double* __restrict__ msc,
                                 const double* __restrict__ msc0, int dim, double* dS,
                                 double* dS_bound) {
  const PlanHdr h = *plan;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    gather_sums<12>(out, h, nullptr, 0, i, dS + 12 * i);
    if (dS_bound) {
      const double la[3] = {qlam[i].x, qlam[i].y, qlam[i].z};
      const double l0[3] = {qlam0[i].x, qlam0[i].y, qlam0[i].z};
      double dl[3], L[3], R[3], e[12];
      for (int d = 0; d < 3; ++d) {
        dl[d] = fabs(la[d] - l0[d]);
        R[d] = fabs(l0[d]);
        L[d] = fabs(la[d]) + R[d];
      }
      dif_sum_bounds<double>(msc + 15 * i, msc0 + 3 * i, dl, L, R, dim, e);
      for (int s = 0; s < 12; ++s) dS_bound[12 * i + s] = e[s];
    }
  }
}

void launch_dif_debug(int64_t n, const PlanHdr* plan, const double* out, const Lam4* qlam,
                      const Lam4* qlam0, const double* msc, const double* msc0,
                      int dim, double* dS, double* dS_bound, cudaStream_t s) {
  const int64_t nb = (n + 127) / 128;
  if (n > 0)
    dif_debug_kernel<<<(int)(nb < 1024 ? nb : 1024), 128, 0, s>>>(
        n, plan, out, qlam, qlam0, msc, msc0, dim, dS, dS_bound);
}

// ------------------------------------------------------------------ certified B ----
// Worst-case error of the mixed form's B at lambda (the B part of mixed_phi_bound): per
// component z (A0 M3 + A1 |lambda| M2 + A2 lambda^2 M1); returns the Euclidean norm.
__device__ __forceinline__ double mixed_b_bound(const float* M, const double lam[3], int dim,
                                                double z) {
  double s = 0.0;
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const double L = fabs(dim == 1 ? lam[0] : lam[p]);
    const float* m = M + 5 * p;
    const double d = z * (BND_A0 * m[2] + BND_A1 * L * m[1] + BND_A2 * L * L * m[0]);
    s += d * d;
  }
  return sqrt(s);
}

// After a certified search: every point whose final B the bound does not certify to `rel`
// relative (the cancellation-dominated points) queues a float-float value query at lambda* on
// side cur and joins cur's waiting list.
__global__ void certb_flag_kernel(const SolveArgs a, double rel) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < a.N;
       g += (int64_t)gridDim.x * blockDim.x) {
    const float4 pos = a.ppos[g];
    const double lam[3] = {a.res_lam[3 * g], a.res_lam[3 * g + 1], a.res_lam[3 * g + 2]};
    const double* B = a.res_B + 3 * g;
    const double nB = sqrt(B[0] * B[0] + B[1] * B[1] + B[2] * B[2]);
    if (!(mixed_b_bound(a.msc + 15 * g, lam, a.o.dim, (double)pos.z) > rel * nB)) continue;
    const int64_t slot = atomic_add_warp(a.cur.fq_cnt, 1);
    a.cur.fpos[slot] = pos;
    a.cur.flam[slot] = make_lam4(lam[0], lam[1], lam[2]);
    SI(a, I_RSLOT, g) = (int32_t)slot;
    a.cur.ref[atomic_add_warp(a.cur.ref_cnt, 1)] = (int32_t)g;
  }
}

// B of the queued points from the float-float value sums (3 per query).
__global__ void certb_apply_kernel(const SolveArgs a) {
  const int n = *a.cur.ref_cnt;
  const PlanHdr hf = *a.fplan;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int64_t g = a.cur.ref[i];
    const float4 pos = a.ppos[g];
    const int pidx = __float_as_int(pos.w);
    const ProbDesc& pd = a.probs[pidx];
    const double z = (double)pos.z;
    const int64_t slot = SI(a, I_RSLOT, g);
    const double* corr = corr_of(a, pd, g, z);
    double S[3];
    gather_sums<3>(a.fout, hf, nullptr, 0, slot, S);
    for (int p = 0; p < 3; ++p) a.res_B[3 * g + p] = z * S[p] + (corr ? corr[p] : 0.0);
  }
}

void launch_certb_flag(const SolveArgs& a, double rel, int grid, cudaStream_t s) {
  certb_flag_kernel<<<grid, 128, 0, s>>>(a, rel);
}
void launch_certb_apply(const SolveArgs& a, int grid, cudaStream_t s) {
  certb_apply_kernel<<<grid, 128, 0, s>>>(a);
}

}  // namespace dbie

// ======================================================= objective gradient, quasi-Newton ----
namespace dbie {

// Phi and dPhi/dlambda_q from the 21 sums of VAR_OBJN (per component: S0, S1, Sx, Sy, Sl, Tx, Ty).
// lambda_q moves only component q: dB_q = z lambda Sl, d(dB_q/dx) = -z lambda Tx,
// d(dB_q/dy) = -z lambda Ty, d(dB_q/dz) = lambda Sl - z^2 lambda S0; the rest is the chain rule
// through J = curl B, div B and the norms (kinks of f and g contribute 0).
__device__ void objective_grad(const double* S, double z, const double lam[3], double g_scale,
                               double w_g, Eval& e, double dphi[3], const double* corr) {
  double G[9], dBdl[3], dGdl[9];
  for (int p = 0; p < 3; ++p) {
    const double* s = S + 7 * p;
    e.B[p] = z * s[0];
    G[3 * p + 0] = z * s[2];
    G[3 * p + 1] = z * s[3];
    G[3 * p + 2] = s[0] + z * z * s[1];
    dBdl[p] = z * lam[p] * s[4];
    dGdl[3 * p + 0] = -(z * lam[p] * s[5]);
    dGdl[3 * p + 1] = -(z * lam[p] * s[6]);
    dGdl[3 * p + 2] = lam[p] * s[4] - z * z * lam[p] * s[0];
  }
  add_corr(corr, e.B, G);
  objective(e.B, G, g_scale, w_g, e.f, e.g, e.phi);
  const double* B = e.B;
  const double J[3] = {G[3 * 2 + 1] - G[3 * 1 + 2], G[3 * 0 + 2] - G[3 * 2 + 0],
                       G[3 * 1 + 0] - G[3 * 0 + 1]};
  const double D = G[0] + G[4] + G[8];
  const double C[3] = {J[1] * B[2] - J[2] * B[1], J[2] * B[0] - J[0] * B[2],
                       J[0] * B[1] - J[1] * B[0]};
  const double nJ = sqrt(J[0] * J[0] + J[1] * J[1] + J[2] * J[2]);
  const double nB = sqrt(B[0] * B[0] + B[1] * B[1] + B[2] * B[2]);
  const double nC = sqrt(C[0] * C[0] + C[1] * C[1] + C[2] * C[2]);
  for (int q = 0; q < 3; ++q) {
    double dB[3] = {0, 0, 0}, dG[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    dB[q] = dBdl[q];
    for (int j = 0; j < 3; ++j) dG[3 * q + j] = dGdl[3 * q + j];
    const double dJ[3] = {dG[3 * 2 + 1] - dG[3 * 1 + 2], dG[3 * 0 + 2] - dG[3 * 2 + 0],
                          dG[3 * 1 + 0] - dG[3 * 0 + 1]};
    const double dD = dG[0] + dG[4] + dG[8];
    const double dC[3] = {dJ[1] * B[2] - dJ[2] * B[1] + J[1] * dB[2] - J[2] * dB[1],
                          dJ[2] * B[0] - dJ[0] * B[2] + J[2] * dB[0] - J[0] * dB[2],
                          dJ[0] * B[1] - dJ[1] * B[0] + J[0] * dB[1] - J[1] * dB[0]};
    double df = 0.0, dg = 0.0;
    if (nJ * nB > 0.0) {
      const double JdJ = J[0] * dJ[0] + J[1] * dJ[1] + J[2] * dJ[2];
      const double BdB = B[0] * dB[0] + B[1] * dB[1] + B[2] * dB[2];
      const double CdC = C[0] * dC[0] + C[1] * dC[1] + C[2] * dC[2];
      df = (nC > 0.0 ? CdC / (nC * nJ * nB) : 0.0) - e.f * (JdJ / (nJ * nJ) + BdB / (nB * nB));
    }
    if (nB > 0.0) {
      const double BdB = B[0] * dB[0] + B[1] * dB[1] + B[2] * dB[2];
      const double sgn = D > 0.0 ? 1.0 : (D < 0.0 ? -1.0 : 0.0);
      dg = g_scale * (sgn * dD / nB - fabs(D) * BdB / (nB * nB * nB));
    }
    dphi[q] = df + w_g * dg;
  }
}

__global__ void finalize_objective_kernel(int64_t n, const PlanHdr* __restrict__ plan,
                                          const int32_t* __restrict__ item_off,
                                          const double* __restrict__ out,
                                          const float4* __restrict__ qpos,
                                          const Lam4* __restrict__ qlam, double g_scale,
                                          double w_g, double* fgphi, double* dphi, double* B,
                                          const double* corr) {
  const PlanHdr h = *plan;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double S[21];
    gather_sums<21>(out, h, item_off, 0, i, S);
    const Lam4 l = qlam[i];
    const double lam[3] = {l.x, l.y, l.z};
    Eval e;
    double dp[3];
    objective_grad(S, (double)qpos[i].z, lam, g_scale, w_g, e, dp, corr ? corr + 12 * i : nullptr);
    if (fgphi) {
      fgphi[3 * i] = e.f;
      fgphi[3 * i + 1] = e.g;
      fgphi[3 * i + 2] = e.phi;
    }
    if (dphi)
      for (int q = 0; q < 3; ++q) dphi[3 * i + q] = dp[q];
    if (B)
      for (int p = 0; p < 3; ++p) B[3 * i + p] = e.B[p];
  }
}

void launch_finalize_objective(int64_t n, const PlanHdr* plan, const int32_t* item_off,
                               const double* out, const float4* qpos, const Lam4* qlam,
                               double g_scale, double w_g, double* fgphi, double* dphi, double* B,
                               const double* corr, cudaStream_t s) {
  if (n <= 0) return;
  const PerPoint L(n);
  finalize_objective_kernel<<<L.grid, L.nt, 0, s>>>(n, plan, item_off, out, qpos, qlam, g_scale,
                                                    w_g, fgphi, dphi, B, corr);
}

// ----------------------------------------------------------------------- quasi-Newton ----
// Same algorithm, same order of operations as the oracle's orc_bfgs (this file is compiled
// without FMA contraction): one line-search trial per point per round.

__global__ void bfgs_init_kernel(const SolveArgs a, const double* __restrict__ lam_init) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < a.N;
       g += (int64_t)gridDim.x * blockDim.x) {
    const float4 pos = a.ppos[g];
    const int pidx = __float_as_int(pos.w);
    const int n = a.o.dim;
    // Phi is even in every lambda_p, so lambda = 0 is a stationary point: start one step away
    // from the initial lambda along (1, 1, 1).
    double x[1][3];
    for (int d = 0; d < 3; ++d) {
      x[0][d] = d < n ? (lam_init ? lam_init[3 * g + d] : 0.0) + a.probs[pidx].step : 0.0;
      SD(a, B_X + d, g) = x[0][d];
    }
    SI(a, I_STAGE, g) = ST_BF_INIT;
    SI(a, I_ITERS, g) = 0;
    SI(a, I_NFEV, g) = 0;
    SI(a, I_STATUS, g) = PT_RUNNING;
    emit<1>(a, g, pos, pidx, x);
  }
}

void launch_bfgs_init(const SolveArgs& a, const double* lam_init, int grid, cudaStream_t s) {
  bfgs_init_kernel<<<grid, 256, 0, s>>>(a, lam_init);
}

// N: the number of free lambdas (3, or 1 when the components share one); fixed at compile time
// so the per-point state stays in registers.
template <int N>
__global__ void bfgs_step_kernel(const SolveArgs a) {
  const int nact = *a.cur.act_cnt;
  constexpr int n = N;
  const PlanHdr h = *a.plan;
  const int ppw = points_per_warp(nact, a.nsm);
  const int lane = threadIdx.x & 31;
  if (lane >= ppw) return;
  const int warp = blockIdx.x * (STEP_NT / 32) + (threadIdx.x >> 5);
  const int nwarps = gridDim.x * (STEP_NT / 32);
  for (int ia = warp * ppw + lane; ia < nact; ia += nwarps * ppw) {
    const int64_t g = a.cur.act[ia];
    const float4 pos = a.ppos[g];
    const int pidx = __float_as_int(pos.w);
    const ProbDesc& pd = a.probs[pidx];
    const double z = (double)pos.z;
    const int stage = SI(a, I_STAGE, g);
    int iters = SI(a, I_ITERS, g);
    int nfev = SI(a, I_NFEV, g) + 1;
    double x[3], gr[3], H[9], dv[3], B[3];
    for (int i = 0; i < 3; ++i) {
      x[i] = SD(a, B_X + i, g);
      gr[i] = SD(a, B_GR + i, g);
      dv[i] = SD(a, B_D + i, g);
      B[i] = SD(a, B_B + i, g);
    }
    for (int i = 0; i < 9; ++i) H[i] = SD(a, B_H + i, g);
    double F = SD(a, B_PHI, g), fv = SD(a, B_F, g), gv = SD(a, B_G, g);
    double alpha = SD(a, B_ALPHA, g), gd = SD(a, B_GD, g), gn = SD(a, B_GN, g);

    // the pending trial's objective and gradient
    double xt[3] = {0, 0, 0};
    if (stage == ST_BF_INIT) {
      for (int i = 0; i < n; ++i) xt[i] = x[i];
    } else {
      for (int i = 0; i < n; ++i) xt[i] = x[i] + alpha * dv[i];
    }
    const double lamt[3] = {xt[0], n == 1 ? xt[0] : xt[1], n == 1 ? xt[0] : xt[2]};
    double S[21];
    gather_sums<21>(a.out, h, a.item_off, pidx, (int64_t)SI(a, I_QSLOT, g) - queue_base(a, pd), S);
    Eval e;
    double dp[3], gt[3] = {0, 0, 0};
    objective_grad(S, z, lamt, pd.g_scale, a.o.w_g, e, dp, corr_of(a, pd, g, z));
    if (n == 1) gt[0] = dp[0] + dp[1] + dp[2];
    else { gt[0] = dp[0]; gt[1] = dp[1]; gt[2] = dp[2]; }
    const bool flagt = e.f <= a.o.eps_f && e.g <= a.o.eps_g;

    int fin = -1;  // final status, or -1 to continue
    bool flag = false;
    bool need_dir = false;
    if (stage == ST_BF_INIT) {
      for (int i = 0; i < 3; ++i) { gr[i] = gt[i]; B[i] = e.B[i]; }
      F = e.phi; fv = e.f; gv = e.g; flag = flagt;
      gn = 0.0;
      for (int i = 0; i < n; ++i) gn += gr[i] * gr[i];
      gn = sqrt(gn);
      for (int i = 0; i < 9; ++i) H[i] = 0.0;
      if (gn > 0.0)
        for (int i = 0; i < n; ++i) H[3 * i + i] = pd.step / gn;
      need_dir = true;
    } else if (e.phi <= F + 1e-4 * alpha * gd) {  // Armijo: accept the trial
      iters += 1;
      double sv[3] = {0, 0, 0}, yv[3] = {0, 0, 0}, sy = 0.0, ss = 0.0, yy = 0.0;
      for (int i = 0; i < n; ++i) {
        sv[i] = xt[i] - x[i];
        yv[i] = gt[i] - gr[i];
        sy += sv[i] * yv[i];
        ss += sv[i] * sv[i];
        yy += yv[i] * yv[i];
      }
      if (sy > 1e-12 * sqrt(ss) * sqrt(yy)) {
        const double rho = 1.0 / sy;
        double Hy[3] = {0, 0, 0}, yHy = 0.0;
        for (int i = 0; i < n; ++i) {
          double t = 0.0;
          for (int k = 0; k < n; ++k) t += H[3 * i + k] * yv[k];
          Hy[i] = t;
        }
        for (int i = 0; i < n; ++i) yHy += yv[i] * Hy[i];
        const double c2 = rho * rho * yHy + rho;
        for (int i = 0; i < n; ++i)
          for (int k = 0; k < n; ++k)
            H[3 * i + k] = H[3 * i + k] - rho * (sv[i] * Hy[k] + Hy[i] * sv[k]) + c2 * sv[i] * sv[k];
      }
      const double dec = F - e.phi;
      for (int i = 0; i < n; ++i) { x[i] = xt[i]; gr[i] = gt[i]; }
      for (int i = 0; i < 3; ++i) B[i] = e.B[i];
      F = e.phi; fv = e.f; gv = e.g; flag = flagt;
      gn = 0.0;
      for (int i = 0; i < n; ++i) gn += gr[i] * gr[i];
      gn = sqrt(gn);
      if (dec <= a.o.tol) fin = PT_CONVERGED;
      else need_dir = true;
    } else {  // reject: halve the step (at most 31 trials per line search)
      alpha = 0.5 * alpha;
      if (alpha < 9.313225746154785e-10) fin = PT_CONVERGED;  // 2^-30
      else {
        double row[1][3] = {{0, 0, 0}};
        for (int i = 0; i < n; ++i) row[0][i] = x[i] + alpha * dv[i];
        SD(a, B_ALPHA, g) = alpha;
        SI(a, I_NFEV, g) = nfev;
        emit<1>(a, g, pos, pidx, row);
        continue;
      }
    }
    if (need_dir) {
      if (flag) fin = PT_CONVERGED;
      else if (!(gn > 0.0)) fin = PT_CONVERGED;
      else if (iters >= a.o.max_iter) fin = PT_MAXITER;
      else {
        for (int i = 0; i < n; ++i) {
          double s = 0.0;
          for (int k = 0; k < n; ++k) s += H[3 * i + k] * gr[k];
          dv[i] = -s;
        }
        gd = 0.0;
        for (int i = 0; i < n; ++i) gd += gr[i] * dv[i];
        if (!(gd < 0.0)) {
          for (int i = 0; i < 9; ++i) H[i] = 0.0;
          for (int i = 0; i < n; ++i) H[3 * i + i] = pd.step / gn;
          gd = 0.0;
          for (int i = 0; i < n; ++i) { dv[i] = -(H[3 * i + i] * gr[i]); gd += gr[i] * dv[i]; }
        }
        alpha = 1.0;
        double row[1][3] = {{0, 0, 0}};
        for (int i = 0; i < n; ++i) row[0][i] = x[i] + alpha * dv[i];
        emit<1>(a, g, pos, pidx, row);
      }
    }
    if (fin >= 0) {
      for (int p = 0; p < 3; ++p) {
        a.res_B[3 * g + p] = B[p];
        a.res_lam[3 * g + p] = fabs(n == 1 ? x[0] : x[p]);
      }
      a.res_f[g] = fv;
      a.res_g[g] = gv;
      a.res_iters[g] = iters;
      a.res_status[g] = fin;
      a.res_nfev[g] = nfev;
      SI(a, I_STATUS, g) = fin;
    }
    for (int i = 0; i < 3; ++i) {
      SD(a, B_X + i, g) = x[i];
      SD(a, B_GR + i, g) = gr[i];
      SD(a, B_D + i, g) = dv[i];
      SD(a, B_B + i, g) = B[i];
    }
    for (int i = 0; i < 9; ++i) SD(a, B_H + i, g) = H[i];
    SD(a, B_PHI, g) = F;
    SD(a, B_F, g) = fv;
    SD(a, B_G, g) = gv;
    SD(a, B_ALPHA, g) = alpha;
    SD(a, B_GD, g) = gd;
    SD(a, B_GN, g) = gn;
    SI(a, I_STAGE, g) = fin >= 0 ? ST_DONE : ST_BF_LS;
    SI(a, I_ITERS, g) = iters;
    SI(a, I_NFEV, g) = nfev;
  }
}

void launch_bfgs_step(const SolveArgs& a, int grid, cudaStream_t s) {
  if (a.o.dim == 1) bfgs_step_kernel<1><<<grid, STEP_NT, 0, s>>>(a);
  else bfgs_step_kernel<3><<<grid, STEP_NT, 0, s>>>(a);
}

}  // namespace dbie
