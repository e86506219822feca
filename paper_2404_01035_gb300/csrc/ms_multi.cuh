// Several steps of a small 2-D grid in one persistent launch.
//
// A small 2-D step is all latency: a launch, a tile's TMA, the dependent
// arithmetic of the few interface rows (which share a handful of CTAs when
// tiles are compact), and the host's time to enqueue it.  Here a cooperative
// grid advances n steps with a barrier between them (arrive and bounded spin
// on one counter).  The unit of work is a 32-cell row segment per warp, dealt
// round-robin over the CTAs, so that the rows of one interface, which cost
// many times a bulk row, sit on different SMs: what bounds an FP64 step is the
// FP64 pipe (2 FMA a clock and SM) of the SMs that hold the interface.  A warp
// reads its 3 x 34 cells of every field through L2 into shared memory and takes
// the bulk update when they hold one pure phase (tested on the values, so no
// segment codes are kept; a reader of codes recomputes them).
#pragma once

#include "ms_step.cuh"

namespace msgb {

template <int NP, int NM, class Real>
struct MultiShape {
  static constexpr int NF = NP + NM;
  static constexpr int WARPS = 4;
  static constexpr int THREADS = 32 * WARPS;
  static constexpr int BX = 34;
  static constexpr int BOX = NF * 3 * BX;
};

// Stencil accessor over a warp's staged rows; carries the step's temperature.
template <int NP, int NM, class Real>
struct MultiAcc {
  using Sh = MultiShape<NP, NM, Real>;
  const Real* s;   // this lane's cell in field 0, middle row
  const StepArgs<Real, NP, NM>* g;
  Real tz0;
  __device__ __forceinline__ Real phi(int a, int dx, int dy, int) const { return s[a * (3 * Sh::BX) + dy * Sh::BX + dx]; }
  __device__ __forceinline__ Real mu(int i, int dx, int dy, int) const { return phi(NP + i, dx, dy, 0); }
  __device__ __forceinline__ uint32_t mask() const { return stencil_mask<2, NP>(*this); }
  template <bool AT>
  __device__ __forceinline__ void mobility(int dx, int dy, int dz, Real* M) const {
    Real ph[NP];
#pragma unroll
    for (int a = 0; a < NP; ++a) ph[a] = phi(a, dx, dy, dz);
    cell_mobility<NP, NM, AT>(ph, g->DX, M);
  }
};
template <int NP, int NM, class Real>
__device__ __forceinline__ Real origin_temperature(const MultiAcc<NP, NM, Real>& A, const StepArgs<Real, NP, NM>&) {
  return A.tz0;
}

// One unit, by a warp: stages the 3 x 34 cells of every field around segment sg
// of row y in box and tells the pure phase + 1 that they all hold, or 0.
template <int NP, int NM, class Real>
__device__ __forceinline__ int stage_unit(const StepArgs<Real, NP, NM>& g, const Real* in, Real* box, int lane, int sg,
                                          int y) {
  using Sh = MultiShape<NP, NM, Real>;
  // columns 32 sg - 1 .. 32 sg + 32 (never past the ghost column nx)
  const Real* row = in + (long long)y * g.pitch + 32 * sg - 1 + g.xoff;
  const int c0 = min(lane, g.nx - 32 * sg + 1), c1 = min(lane + 32, g.nx - 32 * sg + 1);
#pragma unroll
  for (int f = 0; f < Sh::NF; ++f)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const Real* p = row + f * g.fstride + (long long)q * g.pitch;
      box[(f * 3 + q) * Sh::BX + lane] = __ldcg(p + c0);
      if (lane < 2) box[(f * 3 + q) * Sh::BX + 32 + lane] = __ldcg(p + c1);
    }
  __syncwarp();
  // one pure phase on this column's three rows (l + 1), 0 otherwise
  auto column = [&](int col) {
    int c = -1;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      uint32_t nz = 0, one = 0;
#pragma unroll
      for (int a = 0; a < NP; ++a) {
        const Real v = box[(a * 3 + q) * Sh::BX + col];
        nz |= (nonzero(v) ? 1u : 0u) << a;
        one |= (is_one(v) ? 1u : 0u) << a;
      }
      const int pc = (__popc(nz) == 1 && nz == one) ? __ffs(nz) : 0;
      c = (c == -1 || c == pc) ? pc : 0;
    }
    return c;
  };
  int mine = column(min(lane + 1, g.nx - 32 * sg + 1));
  if (lane == 0 || lane == 31) {
    const int side = column(lane == 0 ? 0 : min(33, g.nx - 32 * sg + 1));
    mine = mine == side ? mine : 0;
  }
  const int ref = __shfl_sync(0xffffffffu, mine, 0);
  return __all_sync(0xffffffffu, mine == ref) ? ref : 0;
}

// The staged unit's new cells (flag as stage_unit's).
template <int NP, int NM, class Real, class DP>
__device__ __forceinline__ void update_unit(const StepArgs<Real, NP, NM>& g, MultiAcc<NP, NM, Real>& acc, const DP& dp,
                                            const Real* box, Real* out, int lane, int sg, int y, int flag) {
  using Sh = MultiShape<NP, NM, Real>;
  const int x = 32 * sg + lane;
  if (x < g.nx) {
    acc.s = box + Sh::BX + lane + 1;
    Real pn[NP], mn[NM];
    if (flag != 0)
      bulk_cell<2, NP, NM, Real>(acc, g, flag - 1, pn, mn);
    else
      gp_cell<2, NP, NM, Real, Real, MultiAcc<NP, NM, Real>, kFeatNoAt>(acc, g, dp, y + g.zorg, 0ull, pn, mn);
    store_cell_to<2>(g, out, x, y, 0, pn, mn);
  }
}

__device__ __forceinline__ void multi_arrive(unsigned int* counter) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
}
// Waits until `target` arrivals are in; false after the time limit.
__device__ __forceinline__ bool multi_wait(unsigned int* counter, unsigned int target) {
  unsigned int v;
  unsigned long long t0 = 0;
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
      if (v >= target) return true;
    }
    const unsigned long long t = globaltimer();
    if (t0 == 0) t0 = t;
    if (t - t0 > kWaitLimitNs) return false;
  }
}

__device__ __forceinline__ bool multi_barrier(unsigned int* counter, unsigned int target) {
  multi_arrive(counter);
  return multi_wait(counter, target);
}

template <int NP, int NM, class Real>
__global__ void __launch_bounds__(MultiShape<NP, NM, Real>::THREADS)
    k_gp_multi(const __grid_constant__ StepArgs<Real, NP, NM> g, const __grid_constant__ MultiRun r) {
  using Sh = MultiShape<NP, NM, Real>;
  __shared__ Real s_box[Sh::WARPS][Sh::BOX];
  __shared__ int s_ok;
  __shared__ Real s_tz0;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  Real* const box = s_box[wid];
  const int units = g.segs * g.ny, total = gridDim.x * Sh::WARPS;
  DiffPrm<Real, StepArgs<Real, NP, NM>::P> dp;
  dp.mob = g.mob;
#pragma unroll
  for (int p = 0; p < StepArgs<Real, NP, NM>::P; ++p) dp.delta[p] = g.delta[p];
  bool ok = true;
  // T - T_ref at the origin of the last axis (rounded as temp_offset)
  auto origin = [&](double t) { return (Real)__dsub_rn(r.off, __dmul_rn(r.G, __dadd_rn(r.z0, __dmul_rn(r.V, t)))); };
  Real tz0 = origin(r.t);
  for (int k = 0; k < r.nsteps; ++k) {
    const Real* in = reinterpret_cast<const Real*>(r.slots ? r.slots + (size_t)k * r.slot_bytes : (char*)r.buf[k & 1]);
    Real* out = reinterpret_cast<Real*>(r.slots ? r.slots + (size_t)(k + 1) * r.slot_bytes : (char*)r.buf[(k + 1) & 1]);
    MultiAcc<NP, NM, Real> acc;
    acc.g = &g;
    acc.tz0 = tz0;
    for (int u = wid * gridDim.x + blockIdx.x; u < units; u += total) {
      const int y = u / g.segs, sg = u - y * g.segs;
      const int flag = stage_unit<NP, NM, Real>(g, in, box, lane, sg, y);
      update_unit(g, acc, dp, box, out, lane, sg, y, flag);
      __syncwarp();
    }
    if (k + 1 == r.nsteps) break;
    __syncthreads();
    if (threadIdx.x == 0) {
      multi_arrive(&r.counters[0]);
      // the time of step k + 1, rounded as launch_one_step's (the steps of a call may be
      // split over calls); by one thread while it waits: every FP64 instruction of a
      // warp holds the pipe for 16 cycles (by all warps: 5.4 us a step at 256^2, 4.5 so)
      s_tz0 = origin(__dadd_rn(r.t0, __dmul_rn((double)(r.step0 + k + 1), r.dt)));
      s_ok = multi_wait(&r.counters[0], (unsigned int)(k + 1) * gridDim.x) ? 1 : 0;
    }
    __syncthreads();
    ok = s_ok != 0;
    tz0 = s_tz0;
    if (!ok) {
      if (threadIdx.x == 0) atomicOr(g.status, kStatusTimeout);
      break;
    }
  }
  // the last CTA to leave clears the counters (the others are past every barrier)
  if (threadIdx.x == 0 && atomicAdd(&r.counters[1], 1u) == gridDim.x - 1) {
    r.counters[0] = 0u;
    r.counters[1] = 0u;
  }
}

}  // namespace msgb
