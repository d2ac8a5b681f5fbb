// One-kernel banded passes of small problems: window plan and window sums of a row group in one CTA.
//
// Such a pass is latency: launch, a trip to L2 for the rows, the plan, its way through L2 to the next
// kernel, the rows again, one window.  Here a CTA stages its rows once (one bulk copy per row),
// plans their windows (fot_plan.cuh) and sums them from shared memory (fot_window.cuh).  The arithmetic is that
// of the two-kernel passes.  Products: 8 rows and up to 8 tiles per CTA, one per warp (a loop over a warp's
// tiles kept its state on the stack across the call of the uncommon units: 7.0 against 5.2 us at 256^2,
// eps 64).  Exact sums: 2 rows (the group sizes of the window units) and all their tiles, at every size: the
// windows are a few blocks long, so that plan and staging are much of the work.  band_pass (fot_band.cu)
// has both sides' times.
#pragma once

#include "fot_plan.cuh"

namespace fot {

constexpr int kSmallWarps = 16;      // of a CTA, at most

// dynamic shared memory: four -inf (padded), the rows, their plan staging, the plan itself
__host__ __device__ inline size_t small_smem(int rr, int pitch, int row_floats, int tiles) {
  return (size_t)(16 + rr * (pitch + row_floats) + 3 * rr * tiles) * sizeof(float);
}

template <int MODE, int FORM, int RR, int MAXP>
__global__ void __launch_bounds__(RR == 8 ? 256 : 32 * kSmallWarps, 2) small_pass_kernel(const __grid_constant__ BandTable<MAXP> tab) {
  extern __shared__ __align__(128) float s_x[];
  __shared__ __align__(8) uint64_t s_bar;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const BandArgs& a = tab.p[find_prob<MAXP, 0>(tab, (int)blockIdx.x)];
  // products: a.parts CTAs share a row group's tiles, each has T of them from t_first on
  const int local = (int)blockIdx.x - a.plan_base, rg = RR == 8 ? local / a.parts : local;
  const int r0 = RR * rg, nr = min(RR, a.n_rows - r0);
  const int share = RR == 8 ? (a.n_tiles + a.parts - 1) / a.parts : a.n_tiles;
  const int t_first = RR == 8 ? (local - rg * a.parts) * share : 0, T = min(share, a.n_tiles - t_first);
  const int pitch = stage_pitch(a.len);
  float* const rows = s_x + 16;
  float* const plan = rows + RR * tab.pitch_max;
  float* const s_alpha = plan + RR * tab.plan_row_floats;
  int* const s_win = reinterpret_cast<int*>(s_alpha + RR * T);
  int* const s_mh = s_win + RR * T;
  if (tid == 0) {
    mbar_init(smem_addr(&s_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 4) s_x[tid] = -INFINITY;
  grid_wait();
  grid_launch_next();
  const bool bulk = (a.vec & 1) != 0;
  if (bulk && warp == 0) {
    const uint32_t bytes = (uint32_t)a.len * 4u;
    __syncwarp();
    if (lane == 0) mbar_expect(smem_addr(&s_bar), bytes * nr);
    __syncwarp();
    if (lane < nr) bulk_load(smem_addr(rows + lane * pitch), a.x + (size_t)(r0 + lane) * a.len, bytes, smem_addr(&s_bar));
  }
  const bool skip = error_latched(a.err);                 // an error is latched: write nothing
  if (!bulk) {
    stage_unaligned(rows, pitch, a.x + (size_t)r0 * a.len, a.len, a.len, nr, tid, (int)blockDim.x);
    async_loads_done();
  }
  __syncthreads();                                        // (the barrier's initialisation, the -inf, plain rows)
  const bool ok = !bulk || stage_wait(smem_addr(&s_bar), 0, tab.spin_limit, a.err);

  // the plan
  const int tpr = 1 << tab.plan_tpr_log2, rr = tid >> tab.plan_tpr_log2, ti = tid & (tpr - 1), q = ti & (kPlanQ - 1);
  float* const mine = plan + rr * tab.plan_row_floats;
  {
    const float* const src = rows + rr * pitch;
    const bool live = rr < nr;
    plan_stage(a, mine, ti, tpr, [&](int m0, float (&v)[8]) {
      if (live && m0 + 8 <= a.len) {
        const float4 p = *reinterpret_cast<const float4*>(src + m0), w = *reinterpret_cast<const float4*>(src + m0 + 4);
        v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w;
        v[4] = w.x; v[5] = w.y; v[6] = w.z; v[7] = w.w;
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = live && m0 + u < a.len ? src[m0 + u] : -INFINITY;
      }
    });
  }
  if (!__syncthreads_and(ok)) return;
  for (int t0 = 0; t0 < T; t0 += tpr / kPlanQ) {
    const int t = t0 + ti / kPlanQ;
    const PlanEntry e = plan_tile(a, mine, t_first + min(t, T - 1), q);
    if (t < T && q == 0) {
      s_alpha[t * RR + rr] = e.alpha;
      s_win[t * RR + rr] = e.lo | ((e.hi - e.lo) << 16);
      s_mh[t * RR + rr] = e.mh;
    }
  }
  __syncthreads();

  // the sums, a tile per warp
  unsigned long long* const terms = a.terms + 4 * (blockIdx.x & (kTermSlots - 1));
  const int lr = RR == 8 ? lane >> 2 : lane >> 4;
  Unit u;
  u.r0 = r0;
  u.row = r0 + lr;
  u.skip = skip;
  u.rv.staged = u.rv.vec = true;
  u.rv.row = rows + lr * pitch;
  u.rv.saddr = smem_addr(u.rv.row);
  u.rv.minf = smem_addr(s_x);
  auto open = [&](int tile) {
    const int i = tile * RR + lr;
    u.k0 = (t_first + tile) * a.tile_w;
    u.rv.alpha = s_alpha[i];
    u.rv.lo = s_win[i] & 0xffff;
    u.rv.wl = s_win[i] >> 16;
    u.rv.mh = s_mh[i];
  };
  if (RR == 2) {
#pragma unroll 1
    for (int tile = warp; tile < T; tile += (int)(blockDim.x >> 5)) {
      open(tile);
      exact_unit<MODE>(a, u, terms);
    }
  } else if (warp < T) {
    Tilt<FORM> tilt;
    tilt.load(a, a.tile_w);
    open(warp);
    product_unit<MODE, FORM>(a, u, tilt, terms);
  }
}

// the launch: RR rows per CTA; the table's plan fields are the small pass's (small_table, fot_band.cu)
template <int MODE, int FORM, int RR, int MAXP>
void launch_small(cudaStream_t s, const BandTable<MAXP>& t) {
  launch_dependent(small_pass_kernel<MODE, FORM, RR, MAXP>, dim3(t.plans), RR << t.plan_tpr_log2,
                   small_smem(RR, t.pitch_max, t.plan_row_floats, t.plan_items), s, t);
}

}  // namespace fot
