// solve.cu -- per-point objective and the on-device Downhill Simplex search for lambda.
//
// Compiled with -fmad=false: the simplex arithmetic and the objective are evaluated with
// separately rounded operations, as written.
//
//  * objective: B_p = z S0_p, dB_p/dx = z Sx_p, dB_p/dy = z Sy_p, dB_p/dz = S0_p + z^2 S1_p
//    (the fixed-lambda derivatives of Eq. 13), J = curl B (Eq. 14), f = |J x B| / (|J||B|)
//    (Eq. 8), g = |div B| dV/dSigma / |B| (Eq. 9), Phi = f + w_g g.
//  * simplex (Sect. 2.1; Nelder & Mead 1965, reflection 1, expansion 2, contraction 1/2,
//    shrink 1/2, outside/inside contraction as in Lagarias et al. 1998): every active point is a
//    state machine that advances by one step per round, the lanes of its warp sharing out the
//    values and trial points of all its points (solve_step.cuh); every round evaluates all pending
//    trial points of all active points in one pair-sum pass.  Few points on few pixels run all of
//    it in one kernel (search.cu).
#include "kernels.h"
#include "solve_step.cuh"
#include "warp_sums.cuh"

namespace dbie {

// ----------------------------------------------------------------- eval finalize ----
// WIDE: CTAs of GATHER_WARPS warps, 32 points each; else a thread per point.
template <int VAR, bool WIDE>
__global__ void finalize_eval_kernel(int64_t n, const PlanHdr* __restrict__ plan,
                                     const int32_t* __restrict__ item_off,
                                     const double* __restrict__ out,
                                     const float4* __restrict__ qpos,
                                     const Lam4* __restrict__ qlam, double g_scale, double w_g,
                                     double* B, double* gradB, double* dBdl, const double* gB,
                                     double* fgphi, const double* corr) {
  constexpr int NS = nsum_per_comp(VAR);
  constexpr int NSUM = 3 * NS;
  __shared__ double sh[WIDE ? NSUM * 32 * GATHER_WARPS : 1];
  const PlanHdr h = *plan;
  const int per = WIDE ? 32 : blockDim.x;
  for (int64_t i0 = blockIdx.x * (int64_t)per; i0 < n; i0 += (int64_t)gridDim.x * per) {
    const int64_t i = i0 + (WIDE ? threadIdx.x & 31 : threadIdx.x);
    double S[NSUM];
    if constexpr (WIDE) gather_by_warps<NSUM>(out, h, item_off, i, i < n, S, sh);
    if (i >= n || (WIDE && threadIdx.x >= 32)) continue;
    const float4 pos = qpos[i];
    const double z = (double)pos.z;
    if constexpr (!WIDE) gather_sums<NSUM>(out, h, item_off, 0, i, S);
    double Bv[3], G[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int p = 0; p < 3; ++p) Bv[p] = has_value(VAR) ? z * S[p * NS] : 0.0;
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
        double d = z * lam[p] * S[p * NS + idx_sl(VAR)];
        // an angle without a cosine: see half_turns
        if (isinf(lam[p]) || (has_value(VAR) && isnan(S[p * NS]))) d = __longlong_as_double(0x7ff8000000000000LL);
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
                          double* fgphi, const double* corr, int64_t nsplit, cudaStream_t s) {
  if (n <= 0) return;
  const PerPoint L(n);
#define FIN(V)                                                                                  \
  if (gather_wide(n, nsplit))                                                                           \
    finalize_eval_kernel<V, true><<<gather_grid(n), 32 * GATHER_WARPS, 0, s>>>(                 \
        n, plan, item_off, out, qpos, qlam, g_scale, w_g, B, gradB, dBdl, gB, fgphi, corr);     \
  else                                                                                          \
    finalize_eval_kernel<V, false><<<L.grid, L.nt, 0, s>>>(                                     \
        n, plan, item_off, out, qpos, qlam, g_scale, w_g, B, gradB, dBdl, gB, fgphi, corr)
  switch (var) {
    case VAR_V: FIN(VAR_V); break;
    case VAR_VL: FIN(VAR_VL); break;
    case VAR_L: FIN(VAR_L); break;
    case VAR_OBJ: FIN(VAR_OBJ); break;
    default: FIN(VAR_OBJL); break;
  }
#undef FIN
}

// -------------------------------------------------------------------- simplex rounds ----
template <int N>
__global__ void solve_init_kernel(const SolveArgs a, const double* __restrict__ lam_init) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < a.N;
       g += (int64_t)gridDim.x * blockDim.x)
    init_point<N>(a, lam_init, g);
}

void launch_solve_init(const SolveArgs& a, const double* lam_init, int grid, cudaStream_t s) {
  if (a.o.dim == 1) solve_init_kernel<1><<<grid, 256, 0, s>>>(a, lam_init);
  else solve_init_kernel<3><<<grid, 256, 0, s>>>(a, lam_init);
}

// Points of one warp of a step kernel.  An FP64 warp instruction occupies its SM sub-partition for
// 64 cycles whatever its lanes, so a warp's time is its number of FP64 instructions and few points
// are spread over all SMs and their sub-partitions, one warp each, with as few lanes (fewer of them
// in different stages) as that needs; full warps come when there are more than 128 points per SM.
// (2,048 points in warps of 14, 7, 4 and 2: 8.6, 8.2, 8.0 and 8.2 ms per search.)
constexpr int STEP_NT = 128;
__device__ __forceinline__ int points_per_warp(int n, int nsm) {
  const int p = (n + 4 * nsm - 1) / (4 * nsm);
  return p < 1 ? 1 : (p > 32 ? 32 : p);
}

template <int N, bool REF>
__global__ void __launch_bounds__(STEP_NT) nm_step_kernel(const SolveArgs a) {
  if (!REF && a.rework && blockIdx.x == 0 && threadIdx.x == 0) a.rework[0] = a.rework[1] = 0;
  step_points<N, REF>(a, blockIdx.x * (STEP_NT / 32) + (threadIdx.x >> 5),
                      gridDim.x * (STEP_NT / 32),
                      points_per_warp(REF ? *a.cur.ref_cnt : *a.cur.act_cnt, a.nsm));
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
      if (nsplit > s_minTiles * a.parts) nsplit = s_minTiles * a.parts;
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

// The same by a thread per point, for many points over few pixels, where the combination of a CTA's
// sums outweighs the terms.  Measured (us, CTA / thread per point): 12,000 points over 16 x 16 pixels
// 40 / 23, 400,000 1,330 / 250; 25,000 over 32 x 32 118 / 112; 50,000 over 64 x 48 (12 tiles) 339 / 343,
// 100,000 672 / 502; 100,000 over 128 x 64 (32 tiles) 1,242 / 1,274, 200,000 2,471 / 2,243.
template <typename T>
__global__ void __launch_bounds__(MSC_NT) msc_points_kernel(const ProbDesc* __restrict__ probs,
                                                            int64_t N,
                                                            const float4* __restrict__ ppos,
                                                            T* __restrict__ msc,
                                                            T* __restrict__ msc0) {
  for (int64_t g = blockIdx.x * (int64_t)MSC_NT + threadIdx.x; g < N;
       g += (int64_t)gridDim.x * MSC_NT) {
    const float4 pos = ppos[g];
    const ProbDesc& pd = probs[__float_as_int(pos.w)];
    const float z2 = __fmul_rn(pos.z, pos.z);
    ff::ds tot[18];
#pragma unroll
    for (int i = 0; i < 18; ++i) tot[i] = ff::ds{0.f, 0.f};
    for (int t = 0; t < pd.ntiles; ++t) {
      const float* T32 = pd.tiles32 + (int64_t)t * pd.nf32 * TILE;
      float acc[18];
#pragma unroll
      for (int i = 0; i < 18; ++i) acc[i] = 0.f;
      for (int e = 0; e < TILE; ++e) {
        const float dx = pos.x - __ldg(T32 + e), dy = pos.y - __ldg(T32 + TILE + e);
        const float ri = rsqrtf(__fmaf_rn(dx, dx, __fmaf_rn(dy, dy, z2)));
        float wj = 1.f;
#pragma unroll
        for (int j = 0; j < 6; ++j) {   // acc[3 j + p]: M_j of component p
#pragma unroll
          for (int p = 0; p < 3; ++p)
            acc[3 * j + p] = __fmaf_rn(fabsf(__ldg(T32 + (2 + p) * TILE + e)), wj, acc[3 * j + p]);
          wj *= ri;
        }
      }
#pragma unroll
      for (int i = 0; i < 18; ++i) ff::acc_add(tot[i], ff::ds{acc[i], 0.f});
    }
#pragma unroll
    for (int j = 0; j < 6; ++j)
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        const T v = (T)ff::to_double(tot[3 * j + p]);
        if (j > 0) msc[15 * g + 5 * p + j - 1] = v;
        else msc0[3 * g + p] = v;
      }
  }
}

// ntiles: of the largest problem.
template <typename T>
static void launch_msc_t(const ProbDesc* probs, int64_t N, const float4* ppos, T* msc, T* msc0,
                         int ntiles, int sm_count, cudaStream_t s) {
  if (N <= 0) return;
  if (N >= 6000LL * ntiles) {
    const int64_t nb = (N + MSC_NT - 1) / MSC_NT, most = 32LL * sm_count;
    msc_points_kernel<T><<<(int)(nb < most ? nb : most), MSC_NT, 0, s>>>(probs, N, ppos, msc, msc0);
    return;
  }
  const int64_t most = 16LL * sm_count;
  msc_kernel<T><<<(int)(N < most ? N : most), MSC_NT, 0, s>>>(probs, N, ppos, msc, msc0);
}
void launch_msc(const ProbDesc* probs, int64_t N, const float4* ppos, float* msc, float* msc0,
                int ntiles, int sm_count, cudaStream_t s) {
  launch_msc_t(probs, N, ppos, msc, msc0, ntiles, sm_count, s);
}
void launch_msc(const ProbDesc* probs, int64_t N, const float4* ppos, double* msc, double* msc0,
                int ntiles, int sm_count, cudaStream_t s) {
  launch_msc_t(probs, N, ppos, msc, msc0, ntiles, sm_count, s);
}

// Difference sums of n queries of one problem (slots 0..n-1) and their bounds (debug entry).
__global__ void dif_debug_kernel(int64_t n, const PlanHdr* __restrict__ plan,
                                 const int32_t* __restrict__ item_off,
                                 const double* __restrict__ out, const Lam4* __restrict__ qlam,
                                 const Lam4* __restrict__ qlam0, const double* __restrict__ msc,
                                 const double* __restrict__ msc0, int dim, double* dS,
                                 double* dS_bound) {
  const PlanHdr h = *plan;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    gather_sums<12>(out, h, item_off, 0, i, dS + 12 * i);
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

void launch_dif_debug(int64_t n, const PlanHdr* plan, const int32_t* item_off, const double* out,
                      const Lam4* qlam, const Lam4* qlam0, const double* msc, const double* msc0,
                      int dim, double* dS, double* dS_bound, cudaStream_t s) {
  const int64_t nb = (n + 127) / 128;
  if (n > 0)
    dif_debug_kernel<<<(int)(nb < 1024 ? nb : 1024), 128, 0, s>>>(
        n, plan, item_off, out, qlam, qlam0, msc, msc0, dim, dS, dS_bound);
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

template <bool WIDE>
__global__ void finalize_objective_kernel(int64_t n, const PlanHdr* __restrict__ plan,
                                          const int32_t* __restrict__ item_off,
                                          const double* __restrict__ out,
                                          const float4* __restrict__ qpos,
                                          const Lam4* __restrict__ qlam, double g_scale,
                                          double w_g, double* fgphi, double* dphi, double* B,
                                          const double* corr) {
  __shared__ double sh[WIDE ? 21 * 32 * GATHER_WARPS : 1];
  const PlanHdr h = *plan;
  const int per = WIDE ? 32 : blockDim.x;
  for (int64_t i0 = blockIdx.x * (int64_t)per; i0 < n; i0 += (int64_t)gridDim.x * per) {
    const int64_t i = i0 + (WIDE ? threadIdx.x & 31 : threadIdx.x);
    double S[21];
    if constexpr (WIDE) gather_by_warps<21>(out, h, item_off, i, i < n, S, sh);
    if (i >= n || (WIDE && threadIdx.x >= 32)) continue;
    if constexpr (!WIDE) gather_sums<21>(out, h, item_off, 0, i, S);
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
                               const double* corr, int64_t nsplit, cudaStream_t s) {
  if (n <= 0) return;
  const PerPoint L(n);
  if (gather_wide(n, nsplit, 8192))
    finalize_objective_kernel<true><<<gather_grid(n), 32 * GATHER_WARPS, 0, s>>>(
        n, plan, item_off, out, qpos, qlam, g_scale, w_g, fgphi, dphi, B, corr);
  else
    finalize_objective_kernel<false><<<L.grid, L.nt, 0, s>>>(
        n, plan, item_off, out, qpos, qlam, g_scale, w_g, fgphi, dphi, B, corr);
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
