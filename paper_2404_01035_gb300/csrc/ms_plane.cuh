// Split 2-D FP32 step for grids beyond the multi-step kernel's sizes: a
// streaming kernel for the row segments whose 3 x 3 block of segments is one
// pure phase, which reads and writes mu alone (phi only where the output buffer
// does not hold it, as in the 3-D split step), and an interface kernel, a warp
// per remaining segment.  What bounds them is latency, of the loads and of the
// dependent arithmetic of a row.  Binary, 1537 x 1411 on a GB300: 6.8 + 9.1 us (18.6 a
// step with the gaps), 29.4 us in the fused kernel.  One kernel that keeps each CTA's list in shared memory
// takes 33: few CTAs hold all of an interface.  With three phases and interfaces
// over half of the grid the fused kernel is faster (1400^2 150 us, this form 220).
#pragma once

#include "ms_strip.cuh"

namespace msgb {

template <int NM>
struct PlaneShape {
  static constexpr int R = NM == 1 ? 8 : 4;   // rows per warp (registers: (R + 2) NM vectors)
  static constexpr int WARPS = 4;
  static constexpr int THREADS = 32 * WARPS;
  static constexpr int TX = 128;
};

template <int NP, int NM>
__global__ void __launch_bounds__(PlaneShape<NM>::THREADS)
    k_plane_stream(const __grid_constant__ StepArgs<float, NP, NM> g, const float* __restrict__ in) {
  using Sh = PlaneShape<NM>;
  using Strip = PlaneStrip<NP, NM, Sh::R, false>;
  __shared__ uint8_t s_code[Sh::WARPS][Strip::CODES];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned int strips = (unsigned int)(g.nx + Sh::TX - 1) / Sh::TX;
  const unsigned int w = blockIdx.x * Sh::WARPS + wid;
  const int sx = (int)(w % strips), y0 = (int)(w / strips) * Sh::R;
  if (y0 >= g.ny) return;
  Strip st;
  st.flags(g, sx, y0, lane, s_code[wid]);
  st.list(&g.iface[0], lane, [&](unsigned int at, int r) {
    if (at < g.iface_cap) g.iface[2 + at] = ((unsigned int)(y0 + r) << g.seg_bits) | (unsigned int)(4 * sx + (lane >> 3));
  });
  st.update(g, in, sx, y0, lane, s_code[wid]);
}

// Stencil accessor over the padded input (plain loads: the compiler keeps the
// 9-point neighbourhood in registers).
template <int NP, int NM>
struct PlaneAcc {
  const float* s;
  long long fs;
  int pitch;
  const StepArgs<float, NP, NM>* g;
  __device__ __forceinline__ float phi(int a, int dx, int dy, int) const { return __ldg(s + a * fs + dy * pitch + dx); }
  __device__ __forceinline__ float mu(int i, int dx, int dy, int) const { return phi(NP + i, dx, dy, 0); }
  __device__ __forceinline__ uint32_t mask() const { return stencil_mask<2, NP>(*this); }
  template <bool AT>
  __device__ __forceinline__ void mobility(int dx, int dy, int dz, float* M) const {
    float ph[NP];
#pragma unroll
    for (int a = 0; a < NP; ++a) ph[a] = phi(a, dx, dy, dz);
    cell_mobility<NP, NM, AT>(ph, g->DX, M);
  }
};

template <int NP, int NM, int FEAT>
__global__ void __launch_bounds__(128) k_plane_iface(const __grid_constant__ StepArgs<float, NP, NM> g,
                                                     const float* __restrict__ in) {
  const int lane = threadIdx.x & 31;
  unsigned int* const list = g.iface;
  const unsigned int count = min(*(volatile unsigned int*)&list[0], g.iface_cap);
  DiffPrm<float, StepArgs<float, NP, NM>::P> dp;
  dp.mob = g.mob;
#pragma unroll
  for (int p = 0; p < StepArgs<float, NP, NM>::P; ++p) dp.delta[p] = g.delta[p];
  for (unsigned int i = (blockIdx.x * 128u + threadIdx.x) >> 5; i < count; i += gridDim.x * 4u) {
    const unsigned int r = list[2 + i];
    const int sg = (int)(r & ((1u << g.seg_bits) - 1u)), y = (int)(r >> g.seg_bits);
    const int x = 32 * sg + lane;
    const bool active = x < g.nx;
    int code = 0;
    if (active) {
      PlaneAcc<NP, NM> A{in + (long long)(y + 1) * g.pitch + x + g.xoff, g.fstride, g.pitch, &g};
      float pn[NP], mn[NM];
      gp_cell<2, NP, NM, float, float, PlaneAcc<NP, NM>, FEAT>(A, g, dp, y + g.zorg, lab_cell<2>(g, x, y, 0), pn, mn);
      uint32_t nzm = 0, one = 0;
#pragma unroll
      for (int a = 0; a < NP; ++a) {
        nzm |= (pn[a] != 0.0f ? 1u : 0u) << a;
        one |= (pn[a] == 1.0f ? 1u : 0u) << a;
      }
      code = (__popc(nzm) == 1 && nzm == one) ? __ffs(nzm) : 0;
      store_cell<2>(g, x, y, 0, pn, mn);
    }
    const int ref = __shfl_sync(0xffffffffu, code, 0);
    const bool same = __all_sync(0xffffffffu, !active || code == ref);
    if (lane == 0) {
      const long long ci = (long long)y * g.segs + sg;
      int c = same ? ref : 0;
      if (c != 0 && (g.codes_in[ci] & kCodePhase) == c) c |= kCodeReuse;   // pure before and after
      g.codes_out[ci] = (uint8_t)c;
    }
  }
  // every CTA read the count before taking its ticket; the last one clears the list
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&list[1], 1u) == gridDim.x - 1) {
      list[0] = 0u;
      list[1] = 0u;
    }
  }
}

}  // namespace msgb
