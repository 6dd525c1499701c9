// kernels.h -- host-side interface to the device kernels (launch wrappers and kernel lookup).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "solve.cuh"

namespace dbie {

// Launch configurations of the pair-sum kernels: points (or pixels) per thread, CTA size, and a
// minimum number of resident CTAs per SM (a register cap; 1 = none).  The autotuner picks one.
// The two capped shapes depend on the variant: the Hessian pass (30 compensated sums, ~250
// registers uncapped) is capped at 3 or 4 CTAs of 128 threads (168 or 128 registers), the others
// at 6 or 7 (80 or 72 registers).
constexpr int NCFG = 6;
constexpr int NSTAGE = 3;
struct LaunchCfg { int p, nt, minb; };
__host__ __device__ constexpr LaunchCfg cfg_of(int c, int var = -1) {
  return c == 0 ? LaunchCfg{1, 128, 1}
       : c == 1 ? LaunchCfg{2, 128, 1}
       : c == 2 ? LaunchCfg{1, 256, 1}
       : c == 3 ? LaunchCfg{1, 128, var == VAR_HESS ? 3 : 6}
       : c == 4 ? LaunchCfg{1, 64, 1}
                : LaunchCfg{1, 128, var == VAR_HESS ? 4 : 7};
}

// Launch shape of kernels with one thread per point or pixel (gathering of partial sums, FP64
// objective): their length is one thread's latency, so few points go to small CTAs on all 152 SMs
// instead of filling some of them (4,096 points: 66 us in 16 CTAs of 256 threads).
struct PerPoint {
  int grid, nt;
  explicit PerPoint(int64_t n, int nt_many = 256) {
    const int64_t warps = (n + 32 * 152 - 1) / (32 * 152);   // per SM
    nt = warps >= nt_many / 32 ? nt_many : (warps < 1 ? 32 : 32 * (int)warps);
    const int64_t g = (n + nt - 1) / nt;
    grid = (int)(g < 1 ? 1 : (g < 4096 ? g : 4096));
  }
};

// Launch shape of those kernels where a query has many splits, gathered by the eight warps of a CTA
// (gather_by_warps; otherwise one thread's serial chain of loads and FP64 additions: a call with
// 4,096 points over 36,864 quadrature points, 76 splits, 466 -> 399 us).  Fewer than eight
// splits are not worth the exchange, nor are many points, whose threads fill the chip (us per
// call, thread / warps, at 32 x 32 pixels and at most four splits: field and gradient of 20,000
// points 100 / 103, 65,536 points 200 / 215; adjoint of 65,536 points, 53 splits, 159 / 120; at 300 x
// 300 pixels the same of 4,096 points 777 / 712, B of 64 points 48 / 41).  `most`: the points up to
// which it pays; the objective's gradient, long after its sums are there, runs on one warp in eight
// (20,000 points over 128 x 128 pixels 897 / 926, 4,096 points over 300 x 300 1,020 / 978).
constexpr int GATHER_WARPS = 8;
inline bool gather_wide(int64_t n, int64_t nsplit, int64_t most = 65536) {
  return nsplit >= GATHER_WARPS && n <= most;
}
inline int gather_grid(int64_t n) {
  const int64_t g = (n + 31) / 32;
  return (int)(g < 8192 ? g : 8192);
}

struct KernelRef {
  const void* fn;     // __global__ function
  int nt;             // threads per CTA
  int qper;           // queries (or pixels) per CTA = nt * points per thread
  size_t smem;        // dynamic shared memory bytes
};

// rows: every aligned group of 4 quadrature points lies on one row (row length % 4 == 0)
KernelRef g1_ref_f32(int var, bool tied, int cfg, bool rows);   // pairsum_f32_*.cu
KernelRef g1_ref_f64(int var, bool tied);            // pairsum_f64.cu

// pairsum_few.cu: FP32 sums of few queries, the lanes of a warp taking pixels.
constexpr int FEW_STRIPS_PER_TILE = TILE / 128;   // strips: 128 pixels, 4 per lane
// Counters of the next side that a search round's pass clears (null outside a search).
struct NextSide {
  int32_t *q_cnt, *act_cnt, *near_cnt, *fq_cnt, *dq_cnt, *ref_cnt;   // the last three nullable
};
struct FewArgs {
  const ProbDesc* probs;
  const int32_t* cnt;       // queries (device), or null: n
  int32_t n;
  int32_t near_on;          // a record per query for the near field (after the ranges)
  double near_z;            // near field for z <= near_z (< 0: the problem's own near_z)
  float4* qpos;             // [slot] x, y, z, problem
  Lam4* qlam;               // [slot] lambda
  const float* xyz;         // a call's points (n, 3) and lambda (float or double), packed into
  const float* lam_f;       // qpos, qlam by the kernel; null: qpos, qlam hold the queries
  const double* lam_d;
  double* out;              // [slot][record][sums]
  PlanHdr* plan;            // written by the kernel: records per query (items of one query)
  int32_t strips;           // strips of the largest problem
  int32_t pad0;
  NextSide next;
  int32_t* round_ctr;       // statistics of a search (or null)
  unsigned long long* stat_queries;
  double* stat_pairs;
};
KernelRef few_ref(int var, bool tied, bool split);
// records that a launch of `grid` CTAs writes at most for up to this many queries
int64_t few_records(int64_t queries, int grid);

// Strip ranges per query of a pass of nq queries on `warps` warps.  Short passes are one wave
// (rounded down: an item too many would be a wave of its own); with more than 32 strips for every
// warp about four items each even out the end, of at least 8 strips, which pay for their
// combination.  At most 32 ranges: a thread of a step kernel adds them up.
__host__ __device__ inline int few_split(int nq, int strips, int warps) {
  if (nq <= 0) return 1;
  const bool large = (int64_t)nq * strips > (int64_t)32 * warps;
  const int64_t ns = large ? (4 * (int64_t)warps + nq - 1) / nq : warps / nq;
  int64_t most = large ? strips / 8 : strips;
  most = most > 32 ? 32 : most;
  return (int)(ns > most ? (most < 1 ? 1 : most) : (ns < 1 ? 1 : ns));
}

// search.cu: the simplex search of few points, whole in one kernel.
struct ResidentArgs {
  SolveArgs a;              // state, results and options (its round buffers are not used)
  const double* lam_init;   // (N, 3) or null
  const float4* sctab;
  int32_t* next;            // queue position, zero before the launch
  int32_t points;           // points of a CTA at a time, at most KernelRef::qper
  int32_t strips;           // strips of 128 pixels of the largest problem
  int32_t max_rounds;       // rounds a point can take
  int32_t pad0;
  int32_t* rounds;          // statistics
  unsigned long long* stat_queries;
  double *stat_pairs, *stat_ff_pairs, *stat_dif_pairs;
};
KernelRef search_ref(bool tied, bool split);

// pairsum_re.cu: float-float sums (VAR_V, VAR_OBJ) and difference sums (objective) of queued
// queries, one CTA per query and row range.
struct ReList {
  const int32_t* cnt;       // queries
  const float4* pos;        // [slot] x, y, z, problem index (int bits)
  const Lam4* lam;          // [slot] lambda
  const Lam4* lam0;         // [slot] reference lambda (differences)
  double* out;              // [slot][split][sums]
  PlanHdr* plan;            // written by the kernel: the split count (items of one query each)
};
struct ReArgs {
  const ProbDesc* probs;
  ReList f, d;              // float-float queries, difference queries
  int32_t* work;            // item counter, zero before the launch
  const float4* sctab;      // sine and cosine table (launch_fill_sincos)
  double* stat_ff_pairs;    // pairs of this pass are added (or null)
  double* stat_dif_pairs;
  int32_t rows;             // rows of 128 pixels of the largest problem
  int32_t pad0;
};
constexpr int RE_ROWS_PER_TILE = TILE / 128;
constexpr int SINCOS_TABLE = 52;   // ff::SC_TABLE
KernelRef reeval_ref(int var, bool tied, bool dif);
// The same of one problem's queries, one per thread (plan, item_off and out as a dense pass).
struct RePointsArgs {
  G1Args g;
  const Lam4* qlam0;        // [slot] reference lambda (differences)
  const float4* sctab;
};
KernelRef re_points_ref(int var, bool tied, bool dif);
// items that a launch of `grid` CTAs writes at most for up to this many queries
int64_t reeval_items(int64_t queries, int grid);
void launch_stage_ff(const double* t64, int ntiles, float* tff, cudaStream_t s);
void launch_fill_sincos(float4* tab, cudaStream_t s);   // ff::SC_TABLE entries
KernelRef vjp_ref(bool fp64, bool tied, int cfg);    // vjp.cu
KernelRef vjp7_ref(bool fp64, bool tied);            // vjp.cu (seven-weight adjoint)
// FP32 form over element Gauss points with float-pair positions (pairsum_f32_split.cu)
KernelRef g1_ref_f32_split(int var, bool tied, bool rows);
KernelRef vjp_ref_split(bool tied);
KernelRef vjp7_ref_split(bool tied);

// Gauss rule of the nine-node elements (Eq. 15): g points per side, abscissae and weights.
struct QuadInfo {
  int g;
  double gx[MAX_GAUSS], gw[MAX_GAUSS];
};

// aux.cu
void launch_stage_q9(const float* B0, int nx, int ny, double x0, double y0, double hx, double hy,
                     const QuadInfo& qi, int ntiles, float* t32, double* t64, cudaStream_t s);
void launch_q9_gather(const double* T, int nx, int ny, double hx, double hy, const QuadInfo& qi,
                      double* gB0, int accumulate, cudaStream_t s);
void launch_stage_boundary(const float* Bx, const float* By, const float* Bz, int nx, int ny,
                           double x0, double y0, double hx, double hy, double scale,
                           int ntiles, float* t32, double* t64, cudaStream_t s);
void launch_pack_eval(int64_t n, const float* xyz, const float* lam_f, const double* lam_d,
                      float4* qpos, Lam4* qlam, int32_t* near_list, int32_t* near_cnt,
                      int near_on, double near_z, cudaStream_t s);
void launch_plan_single(PlanHdr* plan, int32_t* item_off, int32_t* q_cnt, int32_t* work,
                        int nitems, int nsplit, int qper, int qcount, cudaStream_t s);
// Near-field correction of the queries of a pass: added to the partial sums of a dense pass
// (plan, item_off), or written as the last record of a pass of few queries (warps > 0).
struct NearArgs {
  const ProbDesc* probs;
  const int32_t* list;      // near query slots; null: all of n queries, those with z <= near_z
  const int32_t* cnt;       // entries of list (device)
  int32_t n;
  int32_t warps, strips;    // the pass of few queries: its warps and strips (0: a dense pass)
  const int32_t* q_cnt;     // and its query count (device), or null: n
  double near_z;
  const float4* qpos;
  const Lam4* qlam;
  const PlanHdr* plan;      // dense pass
  const int32_t* item_off;
  const float4* sctab;      // sine and cosine table, or null: made by every CTA
  double* out;
};
void launch_nearfield(int var, bool tied, const NearArgs& a, int sm_count, cudaStream_t s);
void launch_pack_vjp(int64_t n, const float* xyz, const double* lam, const double* gB, int tied,
                     int nptiles, float* p32, double* p64, int fp64, cudaStream_t s);
void launch_finalize_vjp(int64_t npix, const PlanHdr* plan, const double* out, double scale,
                         double* gB0, int accumulate, int64_t nsplit, cudaStream_t s);

// pxe.cu (pixel-exact near field)
void launch_pxe_corr(bool fp64, const ProbDesc* probs, int64_t n, const float4* pos, double zmax,
                     double* corr, int grid, cudaStream_t s);
// chunks of near points per pixel; the partial buffer holds (nchunk + 1) * npix * 3 doubles (the
// extra part: the window pairs of the mixed form), the bin buffer 3 * pxe_bins + 1 + n int32
int pxe_adjoint_chunks(int64_t n, int64_t npix, int sm_count);
int64_t pxe_bins(int nx, int ny);
cudaError_t launch_pxe_adjoint(bool fp64, bool full, const ProbDesc* prob, int64_t n, int nx,
                               int ny, const float4* pos, double zmax, const double* w,
                               int32_t* list, int32_t* cnt, int32_t* bins, int nchunk,
                               double* part, double* gB0, cudaStream_t s);

void launch_count_bad(const float* a, int64_t n, int mode, int32_t* cnt, cudaStream_t s);
void launch_pack_points(int64_t n, const float* xyz, int pidx, float4* ppos, cudaStream_t s);

// solve.cu
// corr (nullable): per query the pixel-exact correction of B (3) and grad B (9), added after the
// sums are assembled.
void launch_finalize_eval(int var, int64_t n, const PlanHdr* plan, const int32_t* item_off,
                          const double* out, const float4* qpos, const Lam4* qlam, double g_scale,
                          double w_g, double* B, double* gradB, double* dBdl,
                          const double* gB_for_glam, double* fgphi, const double* corr,
                          int64_t nsplit, cudaStream_t s);
void launch_finalize_objective(int64_t n, const PlanHdr* plan, const int32_t* item_off,
                               const double* out, const float4* qpos, const Lam4* qlam,
                               double g_scale, double w_g, double* fgphi, double* dphi, double* B,
                               const double* corr, int64_t nsplit, cudaStream_t s);
// second_order.cu
void launch_finalize_hessian(int64_t n, const PlanHdr* plan, const int32_t* item_off,
                             const double* out, const float4* qpos, const Lam4* qlam, int dim,
                             double g_scale, double w_g, double* phi, double* grad, double* hess,
                             const double* corr, cudaStream_t s);
// corr as above; pxe_w (nullable, with corr): per point the 12 weights of the transposed
// correction, gB_p - dW/dB_p and -dW/d(dB_p/dx_j) with W = v . grad_lambda Phi (at 4 p + m).
void launch_implicit_weights(int64_t n, int nptiles, const PlanHdr* plan, const int32_t* item_off,
                             const double* out, const float4* qpos, const Lam4* qlam,
                             const double* gB, int dim, double g_scale, double w_g, float* p32,
                             double* p64, int fp64, double* v_out, int32_t* flags,
                             const double* corr, double* pxe_w, cudaStream_t s);
void launch_finalize_nv(int64_t n, const PlanHdr* plan, const int32_t* item_off, const double* out,
                        const float4* qpos, double* var, cudaStream_t s);
void launch_stage_variance(const float* sx, const float* sy, const float* sz, double sigma0,
                           int nx, int ny, double x0, double y0, double hx, double hy, double w,
                           int ntiles, float* t32, double* t64, cudaStream_t s);

void launch_bfgs_init(const SolveArgs& a, const double* lam_init, int grid, cudaStream_t s);
void launch_bfgs_step(const SolveArgs& a, int grid, cudaStream_t s);
void launch_solve_init(const SolveArgs& a, const double* lam_init, int grid, cudaStream_t s);
void launch_plan_round(const PlanArgs& a, cudaStream_t s);
void launch_nm_step(const SolveArgs& a, int grid, cudaStream_t s);
void launch_nm_refine(const SolveArgs& a, int grid, cudaStream_t s);
void launch_msc(const ProbDesc* probs, int64_t N, const float4* ppos, float* msc, float* msc0,
                int ntiles, int sm_count, cudaStream_t s);
void launch_msc(const ProbDesc* probs, int64_t N, const float4* ppos, double* msc, double* msc0,
                int ntiles, int sm_count, cudaStream_t s);
void launch_dif_debug(int64_t n, const PlanHdr* plan, const int32_t* item_off, const double* out,
                      const Lam4* qlam, const Lam4* qlam0, const double* msc, const double* msc0,
                      int dim, double* dS, double* dS_bound, cudaStream_t s);
void launch_certb_flag(const SolveArgs& a, double rel, int grid, cudaStream_t s);
void launch_certb_apply(const SolveArgs& a, int grid, cudaStream_t s);

}  // namespace dbie
