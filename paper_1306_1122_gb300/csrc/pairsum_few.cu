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
// bounds it as it does the dense kernels (5 or 7 operations per pair); a warp's combination costs about
// as much issue time as 10 pixels per lane, but no SFU time.
// Measured, dense kernels and their reduction against this one: B at 64 points over 128 x 128
// pixels 113 -> 50 us per call (the kernels 107 -> about 15 us; 31 us per call since with a shorter
// front end and gathering by warps), B, gradient and objective at 300 points over 129 x 70 pixels
// 167 -> 112 us (81 us since); a search of 2,048 points over 32 x 32 pixels 20.7 ->
// 11.1 ms.
#include "few_sums.cuh"

namespace dbie {

constexpr int FEW_NT = 128;
template <int VAR, bool TIED, bool SPLIT>
__global__ void __launch_bounds__(FEW_NT) g1_few_kernel(const FewArgs a) {
  constexpr int NSUM = 3 * nsum_per_comp(VAR);
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
    const ff::ds r = strip_sums<VAR, TIED, SPLIT>(pd, q2, s0, s1, lane);
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
    case VAR_L: return few_ref_t<VAR_L, false>(split);
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
