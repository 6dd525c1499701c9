// search.cu -- the Downhill Simplex search of few points, whole in one kernel.
//
// A search round by launches (solve_impl's graph) costs the latency of five dependent kernels over
// all points, however few queries it has (60 us where the sums take 3), and as many rounds as the
// slowest point of all takes.  Points do not depend on each other, so here a CTA takes up to
// RS_POINTS of them and runs their rounds by itself: the pair sums and the near field of their
// queries (its warps share out items of queries and pixel strips), the steps, the re-evaluation of
// near ties when it has any, and points from the queue in the place of finished ones.  Queues, sums
// and counters live in shared memory, the simplex state in global memory; no CTA waits for another.
// The arithmetic is that of the separate kernels (few_sums.cuh, nearfield.cuh, re_rows.cuh,
// solve_step.cuh).
// A round of one point here is about 40 us, and one of seven 100: more points or pixels per CTA are
// better off spread over the chip by launches (figures and the rule: use_resident in capi.cu).
//
// Compiled with -fmad=false for the steps.
#include "few_sums.cuh"
#include "nearfield.cuh"
#include "re_rows.cuh"
#include "solve_step.cuh"

namespace dbie {

namespace {

constexpr int RS_NT = 256;
constexpr int RS_WARPS = RS_NT / 32;
constexpr int RS_STEP_WARPS = 2;      // warps that step (1 to 8 measure the same)
constexpr int RS_POINTS = 32;        // points of a CTA at a time, at most
constexpr int RS_RECORDS = 256;      // records of a round's sums (query and range, or near field)
constexpr int RS_RE_RECORDS = 128;   // records of re-evaluated sums, of either kind
constexpr int RE_ROW = 32;           // pixels per row of a warp's re-evaluation item

struct RsSide {   // one side of the round buffers (RoundBuf)
  float4 qpos[4 * RS_POINTS];
  Lam4 qlam[4 * RS_POINTS];
  float4 fpos[2 * RS_POINTS], dpos[2 * RS_POINTS];
  Lam4 flam[2 * RS_POINTS], dlam[2 * RS_POINTS], dlam0[2 * RS_POINTS];
  int32_t near[4 * RS_POINTS], act[RS_POINTS], ref[RS_POINTS];
  int32_t q_cnt, act_cnt, near_cnt, fq_cnt, dq_cnt, ref_cnt;
};

struct RsShared {
  SolveArgs args[2];   // the steps' arguments with side i current
  RsSide side[2];
  float4 tab[ff::SC_TABLE];
  double out[RS_RECORDS * 12];
  double fout[RS_RE_RECORDS * 12], dout[RS_RE_RECORDS * 12];
  PlanHdr plan, fplan, dplan;
  int item;
};

// Ranges per query so that about four items per warp share out `cnt` queries, within `most`.
__device__ __forceinline__ int rs_split(int cnt, int most) {
  if (cnt <= 0) return 1;
  const int ns = (4 * RS_WARPS + cnt - 1) / cnt;
  return ns < 1 ? 1 : (ns > most ? (most < 1 ? 1 : most) : ns);
}

// The FP32 sums of query j over strip range sp of ns -> record (j, sp).
template <bool TIED, bool SPLIT>
__device__ __noinline__ long long rs_mixed(RsShared& S, const SolveArgs& a, int j, int sp, int ns,
                                           int nrec) {
  const int lane = threadIdx.x & 31;
  const float4 pos = a.cur.qpos[j];
  const ProbDesc& pd = a.probs[__float_as_int(pos.w)];
  const Query<f32x2, TIED> q2 = splat_query<TIED>(make_query<float, TIED>(pos, a.cur.qlam[j]));
  const int strips = pd.ntiles * FEW_STRIPS_PER_TILE;
  const int s0 = (int)((int64_t)sp * strips / ns), s1 = (int)((int64_t)(sp + 1) * strips / ns);
  const ff::ds r = strip_sums<VAR_OBJ, TIED, SPLIT>(pd, q2, s0, s1, lane);
  constexpr int GL = WarpSums<12>::GL;
  const int s = lane / GL;
  if (lane % GL == 0 && s < 12) S.out[(j * nrec + sp) * 12 + s] = ff::to_double(r);
  return sp == 0 && lane == 0 ? (long long)pd.nx * pd.ny : 0;
}

// The near field of query j -> its last record.
template <bool TIED>
__device__ __noinline__ void rs_near(RsShared& S, const SolveArgs& a, int j, int nrec) {
  using Lanes = NearLanes<12, 32>;
  const int lane = threadIdx.x & 31;
  const float4 pos = a.cur.qpos[j];
  double v[Lanes::NP];
  near_window<VAR_OBJ, TIED, 32>(a.probs[__float_as_int(pos.w)], pos, a.cur.qlam[j], true, S.tab,
                                 lane, v);
  const int s = lane / Lanes::SAME;
  if (lane % Lanes::SAME == 0 && s < 12) S.out[(j * nrec + nrec - 1) * 12 + s] = v[0];
}

// Float-float sums, or with DIF difference sums, of queued value j over row range sp of ns.
template <bool TIED, bool DIF>
__device__ __noinline__ long long rs_reeval(RsShared& S, const SolveArgs& a, int j, int sp, int ns) {
  const int lane = threadIdx.x & 31;
  const float4 pos = DIF ? a.cur.dpos[j] : a.cur.fpos[j];
  const Lam4 lam = DIF ? a.cur.dlam[j] : a.cur.flam[j];
  const ProbDesc& pd = a.probs[__float_as_int(pos.w)];
  constexpr int NL = TIED ? 1 : 3;
  ReQuery q;
  q.x = pos.x;
  q.y = pos.y;
  q.z = pos.z;
  {   // lane i prepares lambda i (its FP64 once, not per lambda)
    ReQuery m;
    const double l = lane == 0 ? lam.x : (lane == 1 ? lam.y : lam.z);
    set_lambda(m, 0, l);
    if constexpr (DIF) {
      const Lam4 l0 = a.cur.dlam0[j];
      set_difference(m, 0, l, lane == 0 ? l0.x : (lane == 1 ? l0.y : l0.z));
    }
    float lmax = 0.f;
#pragma unroll
    for (int i = 0; i < NL; ++i) {
      q.lh[i] = __shfl_sync(0xffffffffu, m.lh[0], i);
      q.ll[i] = __shfl_sync(0xffffffffu, m.ll[0], i);
      lmax = fmaxf(lmax, fabsf(q.lh[i]));   // (of NaN the others: its sums are NaN on either path)
      if constexpr (DIF) {
        q.hs[i] = __shfl_sync(0xffffffffu, m.hs[0], i);
        q.hd[i] = __shfl_sync(0xffffffffu, m.hd[0], i);
        q.pq[i] = __shfl_sync(0xffffffffu, m.pq[0], i);
        q.qq[i] = __shfl_sync(0xffffffffu, m.qq[0], i);
      }
    }
    q.slow = DIF ? 0 : beyond_reduction(pd, pos, lmax);
  }
  const int rows = pd.ntiles * (TILE / RE_ROW);
  const int r0 = (int)((int64_t)sp * rows / ns), r1 = (int)((int64_t)(sp + 1) * rows / ns);
  ff::ds acc[12];
#pragma unroll
  for (int s = 0; s < 12; ++s) acc[s] = ff::ds{0.f, 0.f};
  if constexpr (DIF) {
    dif_rows<TIED, RE_ROW>(pd.tilesff, r0, r1, lane, q, acc);
  } else {
    if (q.slow) ff_rows<VAR_OBJ, TIED, true, RE_ROW>(pd.tilesff, r0, r1, lane, q, S.tab, acc);
    else ff_rows<VAR_OBJ, TIED, false, RE_ROW>(pd.tilesff, r0, r1, lane, q, S.tab, acc);
  }
  const ff::ds r = WarpSums<12>::reduce(acc, lane);
  constexpr int GL = WarpSums<12>::GL;
  const int s = lane / GL;
  if (lane % GL == 0 && s < 12) (DIF ? S.dout : S.fout)[(j * ns + sp) * 12 + s] = ff::to_double(r);
  return sp == 0 && lane == 0 ? (long long)pd.nx * pd.ny : 0;
}

// The steps of n points, by RS_STEP_WARPS warps.
template <int N, bool REF>
__device__ __noinline__ void rs_step(const SolveArgs& a, int n) {
  const int warp = threadIdx.x >> 5, ppw = (n + RS_STEP_WARPS - 1) / RS_STEP_WARPS;
  if (warp < RS_STEP_WARPS) step_points<N, REF>(a, warp, RS_STEP_WARPS, ppw < 1 ? 1 : ppw);
}

// Point number i of the queue: the problems in descriptor order (largest work first).
__device__ __forceinline__ int64_t queued_point(const SolveArgs& a, int64_t i) {
  int p = 0;
  while (p < a.nprob - 1 && i >= a.probs[p].npts) i -= a.probs[p++].npts;
  return a.probs[p].pt_off + i;
}

// Fills side nxt of `a` up to `points` points from the queue (warp 0).
template <int N>
__device__ __noinline__ void rs_refill(const SolveArgs& a, const ResidentArgs& r, int points) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  const int want = points - *a.nxt.act_cnt - *a.nxt.ref_cnt;
  __syncwarp();   // every lane has read the counts that init_point adds to
  int64_t first = 0;
  if (lane == 0 && want > 0) first = atomicAdd(r.next, want);
  first = __shfl_sync(0xffffffffu, first, 0);
  if (lane < want && first + lane < a.N) init_point<N>(a, r.lam_init, queued_point(a, first + lane));
  __syncwarp();
}

}  // namespace

template <bool TIED, bool SPLIT>
__global__ void __launch_bounds__(RS_NT, 2) search_kernel(const ResidentArgs r) {
  extern __shared__ __align__(16) unsigned char rs_raw[];
  RsShared& S = *reinterpret_cast<RsShared*>(rs_raw);
  constexpr int N = TIED ? 1 : 3;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < ff::SC_TABLE) S.tab[tid] = __ldg(r.sctab + tid);
  if (tid < 2) {
    RsSide& c = S.side[tid];
    c.q_cnt = c.act_cnt = c.near_cnt = c.fq_cnt = c.dq_cnt = c.ref_cnt = 0;
    auto buf = [&](RsSide& x) {
      return RoundBuf{x.qpos, x.qlam, &x.q_cnt, x.act,  &x.act_cnt, x.near,  &x.near_cnt, x.fpos,
                      x.flam, &x.fq_cnt, x.ref, &x.ref_cnt, x.dpos, x.dlam, x.dlam0, &x.dq_cnt};
    };
    SolveArgs& a = S.args[tid];
    a = r.a;
    a.cur = buf(S.side[tid]);
    a.nxt = buf(S.side[tid ^ 1]);
    a.out = S.out;
    a.plan = &S.plan;
    a.fout = S.fout;
    a.fplan = &S.fplan;
    a.dout = S.dout;
    a.dplan = &S.dplan;
    a.one_queue = 1;
  }
  __syncthreads();
  if (warp == 0) rs_refill<N>(S.args[1], r, r.points);

  long long pairs = 0, ff_pairs = 0, dif_pairs = 0, queries = 0;
  int rounds = 0, stalled = 0, last = 0;
  const int near1 = r.a.o.near_on ? 1 : 0;
  for (int cur = 0;; cur ^= 1) {
    __syncthreads();   // the side's queries are queued
    const SolveArgs& a = S.args[cur];
    RsSide& c = S.side[cur];
    const int nq = c.q_cnt, nnear = c.near_cnt, busy = c.act_cnt + c.ref_cnt;
    if (busy == 0) break;
    // every point ends within max_rounds rounds
    stalled = busy < last ? 0 : stalled + 1;
    last = busy;
    if (stalled > r.max_rounds) {
      if (tid == 0) atomicOr(r.a.err, ERR_BAD_PLAN);
      break;
    }
    ++rounds;
    const int most = nq > 0 ? RS_RECORDS / nq - near1 : 1;
    const int ns = rs_split(nq, most < r.strips ? most : r.strips), nrec = ns + near1;
    __syncthreads();
    if (tid == 0) {
      RsSide& x = S.side[cur ^ 1];
      x.q_cnt = x.act_cnt = x.near_cnt = x.fq_cnt = x.dq_cnt = x.ref_cnt = 0;
      S.plan = PlanHdr{nq * ns, nrec, 1, 0};
      S.item = 0;
      queries += nq;
    }
    __syncthreads();
    // near-field items (the longest) first
    const int items = nnear + nq * ns;
    for (;;) {
      int it = 0;
      if (lane == 0) it = atomicAdd(&S.item, 1);
      it = __shfl_sync(0xffffffffu, it, 0);
      if (it >= items) break;
      if (it < nnear) {
        rs_near<TIED>(S, a, c.near[it], nrec);
      } else {
        const int k = it - nnear;
        pairs += rs_mixed<TIED, SPLIT>(S, a, k % nq, k / nq, ns, nrec);
      }
    }
    __syncthreads();
    rs_step<N, false>(a, c.act_cnt);
    __syncthreads();
    if (c.ref_cnt > 0) {
      const int nf = c.fq_cnt, nd = c.dq_cnt;
      const int rows = r.strips * (128 / RE_ROW);
      const int fcap = nf > 0 ? RS_RE_RECORDS / nf : 1, dcap = nd > 0 ? RS_RE_RECORDS / nd : 1;
      const int fs = rs_split(nf, fcap < rows ? fcap : rows);
      const int dsp = rs_split(nd, dcap < rows ? dcap : rows);
      if (tid == 0) {
        S.fplan = PlanHdr{nf * fs, fs, 1, 0};
        S.dplan = PlanHdr{nd * dsp, dsp, 1, 0};
        S.item = 0;
      }
      __syncthreads();
      const int re_items = nf * fs + nd * dsp;
      for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(&S.item, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= re_items) break;
        const int k = it - nf * fs;
        if (k < 0) ff_pairs += rs_reeval<TIED, false>(S, a, it / fs, it % fs, fs);
        else dif_pairs += rs_reeval<TIED, true>(S, a, k / dsp, k % dsp, dsp);
      }
      __syncthreads();
      rs_step<N, true>(a, c.ref_cnt);
    }
    __syncthreads();
    if (warp == 0) rs_refill<N>(a, r, r.points);
  }
  if (lane == 0) {
    if (pairs) atomicAdd(r.stat_pairs, (double)pairs);
    if (ff_pairs) atomicAdd(r.stat_ff_pairs, (double)ff_pairs);
    if (dif_pairs) atomicAdd(r.stat_dif_pairs, (double)dif_pairs);
  }
  if (tid == 0) {
    atomicAdd(r.stat_queries, (unsigned long long)queries);
    atomicMax(r.rounds, rounds);
  }
}

KernelRef search_ref(bool tied, bool split) {
  const void* fn = tied ? (split ? (const void*)&search_kernel<true, true>
                                 : (const void*)&search_kernel<true, false>)
                        : (split ? (const void*)&search_kernel<false, true>
                                 : (const void*)&search_kernel<false, false>);
  return KernelRef{fn, RS_NT, RS_POINTS, sizeof(RsShared)};
}

}  // namespace dbie
