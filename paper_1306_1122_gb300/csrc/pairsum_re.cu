// pairsum_re.cu -- the accurate pair sums: float-float sums, and difference sums between two
// lambdas of a point.
//
// Float-float sums.  Every pair term of Eq. 16 (and of the fixed-lambda derivatives of Eq. 13) is
// carried as hi + lo float pairs (ff_math.cuh): the point-pixel offsets, r and 1/r from the SFU
// reciprocal square root with Newton corrections, sin and cos of lambda r by a Cody-Waite
// reduction and a table, the products of the terms and the running sums.  The result agrees with
// the FP64 sums to about 1e-13 of the absolute-value sum, at the FP32 pipe's issue rate: on GB300
// about ten times faster than the same sweep in native FP64.
//
// Difference sums: the change of the objective sums between lambda_0 and lambda_a of one point,
// from FP32 terms whose error is proportional to the change.  Per pixel and component, with
// theta = lambda r, sigma = (lambda_a + lambda_0) r / 2 and delta = (lambda_a - lambda_0) r / 2,
//   cos(theta_a) - cos(theta_0)                     = -2 sin(sigma) sin(delta)
//   theta_a sin(theta_a) - theta_0 sin(theta_0)     =  2 [delta sin(sigma) cos(delta)
//                                                         + sigma cos(sigma) sin(delta)]
//   lambda_a^2 cos(theta_a) - lambda_0^2 cos(theta_0) = (lambda_a^2 - lambda_0^2) cos(sigma) cos(delta)
//                                                     - (lambda_a^2 + lambda_0^2) sin(sigma) sin(delta)
// so the change of u = theta sin(theta) + cos(theta) and of w = lambda^2 cos(theta) - 3 u / r^2
// is a sum of products that each carry a factor delta (or lambda_a - lambda_0).  Evaluated in FP32
// (SFU sine and cosine of sigma; sin and cos of delta by their Taylor polynomials for |delta| <= 1),
// every rounding and every SFU error is relative to that factor: the error of a difference sum is
// a bound times |lambda_a - lambda_0|, where the error of the plain FP32 sums is a bound times 1.
// Added to float-float sums at lambda_0, the differences give the sums at lambda_a with an error
// that shrinks with the distance between the two lambdas.
//
// The lambda search re-evaluates with both the queries whose simplex decision the FP32-term sums
// cannot certify; dbie_eval offers the float-float sums as DBIE_PREC_FLOAT_FLOAT and
// dbie_eval_difference the difference sums.
//
// Work distribution.  Both are bound by FP32 issue (838 and 183 instructions per pair, with the
// combination of the threads' sums), and their
// queries are few and scattered: a search round queues tens to thousands of them, over all
// problems.  So the lanes of a CTA take pixels, not queries: an item is one query and a range of
// rows of 128 pixels, one pixel per thread, and no lane idles whatever the number of queries
// (a block of one query per thread kept 128 lanes for the last few queries of every problem, and
// one thread's 256 dependent pixels of a tile were the length of a round's pass: on a
// 32 x 32-pixel search of 2,048 points 166 us float-float and 53 us differences per round).
// Measured against that layout: 4,096 queries over 128 x 128 pixels, float-float, 2.06 -> 1.71 ms
// (3.3e10 -> 3.9e10 pairs/s); the whole search above 45.6 -> 24.4 ms; 16 magnetograms of 32 to
// 128 pixels with up to 300 points each, searched in one call, 237 -> 59 ms.
// Queries of all problems share one queue; one launch takes the float-float items first and the
// cheaper difference items after them, which fill its tail.  Terms need 40 bytes of tile data
// per 153 or more instructions, which plain coalesced loads through L1 sustain; nothing is staged.
#include <type_traits>

#include "pairsum.cuh"
#include "re_rows.cuh"
#include "warp_sums.cuh"

namespace dbie {

using ff::ds;

constexpr int RE_NT = 128;           // threads per CTA = pixels per row of an item
constexpr int RE_MAX_SPLIT = 64;     // row ranges per query: the reader adds them one by one
constexpr int RE_WAVES = 8;          // items per CTA at most (the tail is then 1/8 of a pass)
static_assert(TILE / RE_NT == RE_ROWS_PER_TILE && TILE % RE_NT == 0, "rows tile the tile");

// Float-float tiles: per field (x, y, bx, by, bz) TILE hi parts, then TILE lo parts.
__global__ void stage_ff_kernel(const double* __restrict__ t64, int ntiles,
                                float* __restrict__ tff) {
  const int64_t total = (int64_t)ntiles * TILE;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t tile = k / TILE;
    const int e = (int)(k % TILE);
    for (int f = 0; f < NFIELD; ++f) {
      const ds d = ff::from_double(t64[tile * (NFIELD * TILE) + f * TILE + e]);
      float* dst = tff + tile * (int64_t)(RE_NF * TILE) + f * 2 * TILE + e;
      dst[0] = d.hi;
      dst[TILE] = d.lo;
    }
  }
}

void launch_stage_ff(const double* t64, int ntiles, float* tff, cudaStream_t s) {
  const int64_t total = (int64_t)ntiles * TILE;
  const int grid = (int)((total + 255) / 256 < 8192 ? (total + 255) / 256 : 8192);
  stage_ff_kernel<<<grid, 256, 0, s>>>(t64, ntiles, tff);
}

__global__ void fill_sincos_kernel(float4* tab) { ff::fill_sincos_table(tab, threadIdx.x); }

void launch_fill_sincos(float4* tab, cudaStream_t s) {
  static_assert(ff::SC_TABLE == SINCOS_TABLE && SINCOS_TABLE <= 64, "one thread per table entry");
  fill_sincos_kernel<<<1, 64, 0, s>>>(tab);
}

// Row ranges per query.  While a pass is short (at most 4 rows for every CTA) one wave of items
// spreads it over the chip; a longer pass takes up to RE_WAVES items per CTA, so that the uneven
// end is a fraction of it.  Rounded down: an item too many would be a wave of its own.
__device__ __forceinline__ int re_split(int cnt, int rows, int ctas) {
  if (cnt <= 0) return 1;
  const int64_t waves = (int64_t)cnt * rows / (4 * (int64_t)ctas);
  const int64_t target = (int64_t)ctas * (waves < 1 ? 1 : (waves > RE_WAVES ? RE_WAVES : waves));
  const int most = rows < RE_MAX_SPLIT ? rows : RE_MAX_SPLIT;
  const int64_t ns = target / cnt;
  return ns < 1 ? 1 : (ns > most ? most : (int)ns);
}

// Sums over the CTA's threads: over the lanes of each warp, then the warps' sums in FP64.
// `red` holds 4 * NSUM doubles.  Writes NSUM values to dst; callers synchronise before red is
// written again.
template <int NSUM>
__device__ __forceinline__ void reduce_store(const ds (&acc)[NSUM], double* red, double* dst) {
  constexpr int GL = WarpSums<NSUM>::GL;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const ds r = WarpSums<NSUM>::reduce(acc, lane);
  if (lane % GL == 0 && lane / GL < NSUM) red[warp * NSUM + lane / GL] = ff::to_double(r);
  __syncthreads();
  if (threadIdx.x < NSUM) {
    double t = red[threadIdx.x];
#pragma unroll
    for (int w = 1; w < RE_NT / 32; ++w) t += red[w * NSUM + threadIdx.x];
    dst[threadIdx.x] = t;
  }
}

// Float-float sums of a.f and, with DIF, difference sums of a.d (objective sums).
template <int VAR, bool TIED, bool DIF>
__global__ void __launch_bounds__(RE_NT) reeval_kernel(const ReArgs a) {
  static_assert(VAR == VAR_V || VAR == VAR_OBJ, "float-float form: value and objective sums");
  static_assert(!DIF || VAR == VAR_OBJ, "differences: objective sums");
  constexpr int NSUM = 3 * nsum_per_comp(VAR);
  __shared__ float4 s_tab[ff::SC_TABLE];
  __shared__ double s_red[RE_NT / 32 * NSUM];
  __shared__ ReQuery s_q;
  __shared__ int s_item;
  const int tid = threadIdx.x;
  if (tid < ff::SC_TABLE) s_tab[tid] = __ldg(a.sctab + tid);
  const int nf = *a.f.cnt;
  const int nd = DIF ? *a.d.cnt : 0;
  const int fs = re_split(nf, a.rows, gridDim.x);
  const int dsp = DIF ? re_split(nd, a.rows, gridDim.x) : 1;
  const int fitems = nf * fs, items = fitems + nd * dsp;
  if (blockIdx.x == 0 && tid == 0) {
    *a.f.plan = PlanHdr{fitems, fs, 1, 0};
    if (DIF) *a.d.plan = PlanHdr{nd * dsp, dsp, 1, 0};
  }
  bool first = true;   // (a CTA's first item is its own number: see pairsum.cuh)
  long long pf = 0, pd_ = 0;   // thread 32: pairs of the queries whose first range it set up

  for (;;) {
    if (tid == 0) s_item = first ? (int)blockIdx.x : (int)gridDim.x + atomicAdd(a.work, 1);
    first = false;
    __syncthreads();   // (also: the previous item's readers of s_red and s_q are done)
    const int it = s_item;
    if (it >= items) break;
    const bool dif = DIF && it >= fitems;
    const int ns = dif ? dsp : fs;
    const int local = dif ? it - fitems : it;
    const int slot = local / ns, sp = local - slot * ns;
    const ReList& L = dif ? a.d : a.f;
    const float4 pos = L.pos[slot];
    const ProbDesc& pd = a.probs[__float_as_int(pos.w)];
    if (tid < (TIED ? 1 : 3)) {
      const Lam4 l4 = L.lam[slot];
      const double la = tid == 0 ? l4.x : (tid == 1 ? l4.y : l4.z);
      set_lambda(s_q, tid, la);
      if (DIF && dif) {
        const Lam4 r4 = L.lam0[slot];
        set_difference(s_q, tid, la, tid == 0 ? r4.x : (tid == 1 ? r4.y : r4.z));
      }
    } else if (tid == 32) {
      s_q.x = pos.x;
      s_q.y = pos.y;
      s_q.z = pos.z;
      const Lam4 l4 = L.lam[slot];
      const float lx = fabsf((float)l4.x);
      s_q.slow = beyond_reduction(pd, pos, TIED ? lx : fmaxf(fmaxf(lx, fabsf((float)l4.y)),
                                                             fabsf((float)l4.z)));
      if (sp == 0) {
        const long long px = (long long)pd.nx * pd.ny;
        if (dif) pd_ += px;
        else pf += px;
      }
    }
    __syncthreads();
    const int rows = pd.ntiles * (TILE / RE_NT);
    const int r0 = (int)((int64_t)sp * rows / ns), r1 = (int)((int64_t)(sp + 1) * rows / ns);
    ds acc[NSUM];
#pragma unroll
    for (int s = 0; s < NSUM; ++s) acc[s] = ds{0.f, 0.f};
    if constexpr (DIF) {
      if (dif) dif_rows<TIED, RE_NT>(pd.tilesff, r0, r1, tid, s_q, acc);
      else if (s_q.slow) ff_rows<VAR, TIED, true, RE_NT>(pd.tilesff, r0, r1, tid, s_q, s_tab, acc);
      else ff_rows<VAR, TIED, false, RE_NT>(pd.tilesff, r0, r1, tid, s_q, s_tab, acc);
    } else {
      if (s_q.slow) ff_rows<VAR, TIED, true, RE_NT>(pd.tilesff, r0, r1, tid, s_q, s_tab, acc);
      else ff_rows<VAR, TIED, false, RE_NT>(pd.tilesff, r0, r1, tid, s_q, s_tab, acc);
    }
    reduce_store<NSUM>(acc, s_red, L.out + (int64_t)local * NSUM);
  }
  if (tid == 32) {
    if (pf && a.stat_ff_pairs) atomicAdd(a.stat_ff_pairs, (double)pf);
    if (DIF && pd_ && a.stat_dif_pairs) atomicAdd(a.stat_dif_pairs, (double)pd_);
  }
}

// The same sums with one query per thread, for calls of many queries on few pixels (reeval_dense in
// capi.cu): where an item above is a few rows, its set-up and the combination of its threads' sums
// outweigh the terms.  Items are blocks of 128 queries and a tile range, tiles come through the ring of
// pairsum.cuh, read by all threads at once.  FP32 issue bounds it as it does the other form.
// Measured, an item per query and pixel range / this form (ms): differences of 300,000 points over
// 33 x 20 pixels 2.14 / 1.12, 100,000 over 128 x 128 9.0 / 7.7 (tied 6.1 / 4.1), 30,000 over 300 x 257
// 12.5 / 11.9; float-float B of 400,000 points over 16 x 16 pixels 2.27 / 1.85.
template <int VAR, bool TIED, bool DIF>
__global__ void __launch_bounds__(RE_NT) re_points_kernel(const RePointsArgs a) {
  constexpr int NSUM = 3 * nsum_per_comp(VAR);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[NSTAGE];
  __shared__ __align__(8) uint64_t empty_bar[NSTAGE];
  __shared__ int s_item;
  __shared__ volatile int s_abort;
  __shared__ float4 s_tab[ff::SC_TABLE];
  const int tid = threadIdx.x;
  TileRing<float, NSTAGE, RE_NT / 32> ring{reinterpret_cast<float*>(smem_raw), full_bar, empty_bar,
                                           &s_abort, a.g.err, (uint32_t)(RE_NF * TILE), 0u, 0u};
  if (tid < ff::SC_TABLE) s_tab[tid] = __ldg(a.sctab + tid);
  if (tid == 0) {
    ring.init_barriers();
    s_abort = 0;
  }
  __syncthreads();
  const PlanHdr plan = *a.g.plan;
  const ProbDesc& pd = a.g.probs[0];
  const int n = *a.g.q_cnt;
  // (items by the counter alone: with the first-item rule of pairsum.cuh the difference sums schedule
  // worse, 30,000 points over 300 x 257 pixels 11.9 -> 13.1 ms)
  for (;;) {
    if (tid == 0) s_item = s_abort ? plan.nitems : atomicAdd(a.g.work, 1);
    __syncthreads();
    const int it = s_item;
    __syncthreads();
    if (it >= plan.nitems) break;
    const int blk = it / plan.nsplit, sp = it - blk * plan.nsplit;
    const int t0 = (int)(((int64_t)sp * pd.ntiles) / plan.nsplit);
    const int t1 = (int)(((int64_t)(sp + 1) * pd.ntiles) / plan.nsplit);
    const int64_t j = (int64_t)blk * RE_NT + tid;
    const bool valid = j < n;
    const float4 pos = valid ? a.g.qpos[j] : make_float4(0.f, 0.f, 1.f, 0.f);
    const Lam4 l4 = valid ? a.g.qlam[j] : make_lam4(0.0, 0.0, 0.0);
    ReQuery q;
    q.x = pos.x;
    q.y = pos.y;
    q.z = pos.z;
    const double la[3] = {l4.x, l4.y, l4.z};
    if constexpr (DIF) {
      const Lam4 r4 = valid ? a.qlam0[j] : l4;
      const double l0[3] = {r4.x, r4.y, r4.z};
#pragma unroll
      for (int i = 0; i < (TIED ? 1 : 3); ++i) set_difference(q, i, la[i], l0[i]);
    } else {
#pragma unroll
      for (int i = 0; i < (TIED ? 1 : 3); ++i) set_lambda(q, i, la[i]);
    }
    ds acc[NSUM];
#pragma unroll
    for (int s = 0; s < NSUM; ++s) acc[s] = ds{0.f, 0.f};
    // (a warp without a query only keeps the ring's protocol)
    const bool busy = __any_sync(0xffffffffu, valid);
    if constexpr (DIF) {
      const float z2 = q.z * q.z;
      sweep_tiles(ring, pd.tilesff, t0, t1, tid, [&](const float* sx) {
        if (!busy) return;
#pragma unroll 1
        for (int k0 = 0; k0 < TILE; k0 += DIF_BLK) {
          float bs[12];
#pragma unroll
          for (int s = 0; s < 12; ++s) bs[s] = 0.f;
#pragma unroll 2
          for (int k = k0; k < k0 + DIF_BLK; ++k)
            dif_pixel<TIED>(q, z2, [&](int f, int part) { return sx[(2 * f + part) * TILE + k]; }, bs);
          dif_fold(acc, bs);
        }
      });
    } else {
      const float lx = fabsf(q.lh[0]);
      const bool slow = __any_sync(
          0xffffffffu,
          valid && beyond_reduction(pd, pos, TIED ? lx : fmaxf(fmaxf(lx, fabsf(q.lh[1])),
                                                               fabsf(q.lh[2]))));
      const FfQuery<TIED> fq(q);
      auto tile = [&](const float* sx, auto any) {
#pragma unroll 1
        for (int k = 0; k < TILE; ++k)
          ff_pixel<VAR, TIED, decltype(any)::value>(
              fq, s_tab, [&](int f, int part) { return sx[(2 * f + part) * TILE + k]; }, acc);
      };
      sweep_tiles(ring, pd.tilesff, t0, t1, tid, [&](const float* sx) {
        if (!busy) return;
        if (slow) tile(sx, std::true_type{});
        else tile(sx, std::false_type{});
      });
    }
    if (valid) {
#pragma unroll
      for (int s = 0; s < NSUM; ++s)
        a.g.out[((int64_t)it * NSUM + s) * RE_NT + tid] = ff::to_double(acc[s]);
    }
  }
  if (tid == 0) ring.drain();
}

template <int VAR, bool TIED, bool DIF>
static KernelRef re_points_t() {
  return KernelRef{(const void*)&re_points_kernel<VAR, TIED, DIF>, RE_NT, RE_NT,
                   (size_t)NSTAGE * RE_NF * TILE * sizeof(float)};
}

KernelRef re_points_ref(int var, bool tied, bool dif) {
  if (dif) return tied ? re_points_t<VAR_OBJ, true, true>() : re_points_t<VAR_OBJ, false, true>();
  if (var == VAR_V) return tied ? re_points_t<VAR_V, true, false>() : re_points_t<VAR_V, false, false>();
  return tied ? re_points_t<VAR_OBJ, true, false>() : re_points_t<VAR_OBJ, false, false>();
}

template <int VAR, bool TIED, bool DIF>
static KernelRef re_ref_t() {
  return KernelRef{(const void*)&reeval_kernel<VAR, TIED, DIF>, RE_NT, 1, 0};
}

KernelRef reeval_ref(int var, bool tied, bool dif) {
  if (var == VAR_V) return tied ? re_ref_t<VAR_V, true, false>() : re_ref_t<VAR_V, false, false>();
  if (!dif) return tied ? re_ref_t<VAR_OBJ, true, false>() : re_ref_t<VAR_OBJ, false, false>();
  return tied ? re_ref_t<VAR_OBJ, true, true>() : re_ref_t<VAR_OBJ, false, true>();
}

int64_t reeval_items(int64_t queries, int grid) {
  return queries > (int64_t)RE_WAVES * grid ? queries : (int64_t)RE_WAVES * grid;
}

}  // namespace dbie
