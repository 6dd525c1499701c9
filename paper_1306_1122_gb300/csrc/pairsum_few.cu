// pairsum_few.cu -- the FP32 pair sums of Eq. 16 for few queries.
//
// pairsum.cuh's kernels give a query to a thread and stream boundary tiles past blocks of 128 of
// them: right when the queries fill the chip.  A call with tens to a few thousand points does not
// (300 points over 129 x 70 pixels are 108 items of 256 dependent pixels, on 152 SMs), and the
// thread that then adds up a query's dozens of tile-range partials is another serial chain.
// Here the lanes of a warp take pixels: an item is one query and a range of strips of 128 pixels,
// four pixels per lane and load (five or seven 128-bit loads, from L1: the warps of an SM work on
// neighbouring queries of the same range), the arithmetic is the other kernels' (f32x2 pixel
// pairs, folded every 64 pixels of a lane), and the lanes' sums are combined in the warp.  The SFU
// bounds it as it does the dense kernels (7 operations per pair); a warp's combination costs about
// as much issue time as 10 pixels per lane, but no SFU time.
// Measured, dense kernels and their reduction against this one: B at 64 points over 128 x 128
// pixels 113 -> 50 us per call (the kernels 107 -> about 15 us), B, gradient and objective at 300
// points over 129 x 70 pixels 167 -> 112 us; a search of 2,048 points over 32 x 32 pixels 20.7 ->
// 11.1 ms.
#include "kernels.h"
#include "pairsum.cuh"
#include "warp_sums.cuh"

namespace dbie {

constexpr int FEW_NT = 128;
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
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    f32x2 dx = vsub(q2.x, px2[h]), dy = vsub(q2.y, py2[h]);
    if constexpr (SPLIT) {
      dx = vsub(dx, h == 0 ? pack2(XL.x, XL.y) : pack2(XL.z, XL.w));
      dy = vsub(dy, h == 0 ? pack2(YL.x, YL.y) : pack2(YL.z, YL.w));
    }
    TermsV<f32x2, VAR, TIED> tm;
    pair_angularv<f32x2, VAR, TIED>(q2, pair_geomv_d<f32x2, TIED>(q2, dx, dy), b2[h], tm);
    accumulatev<f32x2, VAR, TIED, NS>(acc2, tm, b2[h]);
  }
}

template <int VAR, bool TIED, bool SPLIT>
__global__ void __launch_bounds__(FEW_NT) g1_few_kernel(const FewArgs a) {
  constexpr int NS = nsum_per_comp(VAR);
  constexpr int NSUM = 3 * NS;
  constexpr int NF = SPLIT ? NFIELD_SPLIT : NFIELD;
  constexpr int FOLD = SUB / 4;   // strips between folds: SUB pixels of a lane
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * FEW_NT + threadIdx.x) >> 5;
  const int nwarps = gridDim.x * (FEW_NT / 32);
  const int nq = a.cnt ? *a.cnt : a.n;
  const int ns = few_split(nq, a.strips, nwarps);
  const int nrec = ns + (a.near_on ? 1 : 0);   // partials per query: ranges, then the near field
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *a.plan = PlanHdr{nq * ns, nrec, 1, 0};
    if (a.next.act_cnt) {   // a search round: the next side's counters
      *a.next.act_cnt = 0;
      *a.next.near_cnt = 0;
      *a.next.q_cnt = 0;
      if (a.next.fq_cnt) *a.next.fq_cnt = 0;
      if (a.next.dq_cnt) *a.next.dq_cnt = 0;
      if (a.next.ref_cnt) *a.next.ref_cnt = 0;
      *a.round_ctr += 1;
      *a.stat_queries += (unsigned long long)nq;
    }
  }
  long long pairs = 0;
  // neighbouring warps take neighbouring queries of the same pixel range
  for (int64_t it = warp; it < (int64_t)nq * ns; it += nwarps) {
    const int sp = (int)(it / nq), j = (int)(it - (int64_t)sp * nq);
    float4 pos;
    Lam4 lam;
    if (a.xyz) {   // a call's arrays, packed here for the kernels that follow
      pos = make_float4(a.xyz[3 * j], a.xyz[3 * j + 1], a.xyz[3 * j + 2], __int_as_float(0));
      if (a.lam_d) lam = make_lam4(a.lam_d[3 * j], a.lam_d[3 * j + 1], a.lam_d[3 * j + 2]);
      else lam = make_lam4((double)a.lam_f[3 * j], (double)a.lam_f[3 * j + 1],
                           (double)a.lam_f[3 * j + 2]);
      if (sp == 0 && lane == 0) {
        a.qpos[j] = pos;
        a.qlam[j] = lam;
      }
    } else {
      pos = a.qpos[j];
      lam = a.qlam[j];
    }
    const ProbDesc& pd = a.probs[__float_as_int(pos.w)];
    const Query<f32x2, TIED> q2 = splat_query<TIED>(make_query<float, TIED>(pos, lam));
    const int strips = pd.ntiles * FEW_STRIPS_PER_TILE;
    const int s0 = (int)((int64_t)sp * strips / ns), s1 = (int)((int64_t)(sp + 1) * strips / ns);
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
    const ff::ds r = WarpSums<NSUM>::reduce(v, lane);
    const int s = lane / WarpSums<NSUM>::GL;
    if (lane % WarpSums<NSUM>::GL == 0 && s < NSUM) {
      double* rec = a.out + ((int64_t)j * nrec + sp) * NSUM + s;
      *rec = ff::to_double(r);
      // no near field for this query: its record is zero
      const double near_z = a.near_z < 0.0 ? pd.near_z : a.near_z;
      if (a.near_on && sp == 0 && !((double)pos.z <= near_z)) rec[ns * NSUM] = 0.0;
    }
    if (sp == 0) pairs += (long long)pd.nx * pd.ny;
  }
  if (pairs && lane == 0 && a.stat_pairs) atomicAdd(a.stat_pairs, (double)pairs);
}

template <int VAR, bool TIED>
static KernelRef few_ref_t(bool split) {
  return KernelRef{split ? (const void*)&g1_few_kernel<VAR, TIED, true>
                         : (const void*)&g1_few_kernel<VAR, TIED, false>,
                   FEW_NT, 1, 0};
}

KernelRef few_ref(int var, bool tied, bool split) {
  switch (var) {
    case VAR_V: return few_ref_t<VAR_V, false>(split);
    case VAR_VL: return few_ref_t<VAR_VL, false>(split);
    case VAR_OBJ: return tied ? few_ref_t<VAR_OBJ, true>(split) : few_ref_t<VAR_OBJ, false>(split);
    case VAR_OBJL: return few_ref_t<VAR_OBJL, false>(split);
    default: return tied ? few_ref_t<VAR_OBJN, true>(split) : few_ref_t<VAR_OBJN, false>(split);
  }
}

int64_t few_records(int64_t queries, int grid) {
  const int64_t warps = (int64_t)grid * (FEW_NT / 32);
  return 2 * queries + 4 * warps;
}

}  // namespace dbie
