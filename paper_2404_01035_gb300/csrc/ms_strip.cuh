// A strip of R rows x 128 cells of a 2-D FP32 grid, by one warp: which of its
// 32-cell segments are bulk (the 3 x 3 block of segments is one pure phase), the
// places of the others in a work list, and the bulk update, which reads and
// writes mu alone (phi only where the output buffer does not hold it, as in the
// 3-D split step).  What bounds it is memory: each lane holds 4 consecutive cells
// of R + 2 rows, all rows in flight at once, and updates R of them; x neighbours
// come by shuffle.
#pragma once

#include "ms_split.cuh"

namespace msgb {

// Loads of the input: through the read-only path, or (L2: several steps in one
// launch, the rows are other SMs' stores) past L1.
template <bool L2>
__device__ __forceinline__ float4 ld4(const float* p) {
  return L2 ? __ldcg(reinterpret_cast<const float4*>(p)) : __ldg(reinterpret_cast<const float4*>(p));
}
template <bool L2>
__device__ __forceinline__ float ld1(const float* p) {
  return L2 ? __ldcg(p) : __ldg(p);
}
template <bool L2>
__device__ __forceinline__ uint8_t ldc(const uint8_t* p) {
  return L2 ? __ldcg(p) : __ldg(p);
}

// One strip of R rows x 128 cells, rows y0 .., cells 128 sx .., by one warp:
// a lane's flags and the strip's bulk update.
// G: the launch arguments or a copy of the members used here.
template <int NP, int NM, int R, bool L2>
struct PlaneStrip {
  static constexpr int CS = 6;                       // segments of a strip with one on either side
  static constexpr int CODES = ((R + 2) * CS + 3) / 4 * 4;
  int rf[R + 2];              // pure phase + 1 of the row's three segments around this lane's, or 0
  uint32_t bulk, listed;      // rows of this lane's segment, by bit

  // code: CODES bytes of shared memory of this warp
  template <class G>
  __device__ __forceinline__ void flags(const G& g, int sx, int y0, int lane, uint8_t* code) {
    const int seg0 = 4 * sx, wc = lane >> 3, seg = seg0 + wc;
    for (int e = lane; e < (R + 2) * CS; e += 32) {
      const int r = e / CS, k = e - r * CS;
      code[e] = ldc<L2>(g.codes_in + (long long)bc_map(y0 - 1 + r, g.ny, g.bc[1]) * g.segs +
                        bc_map(seg0 - 1 + k, g.segs, g.bc[0]));
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R + 2; ++r) rf[r] = combine_codes(code + r * CS + wc);
    bulk = listed = 0u;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const bool inside = y0 + r < g.ny && seg < g.segs;
      const bool b = rf[r] != 0 && rf[r] == rf[r + 1] && rf[r + 1] == rf[r + 2];
      bulk |= (inside && b && 128 * sx + 4 * lane < g.nx ? 1u : 0u) << r;
      listed |= (inside && !b ? 1u : 0u) << r;
    }
  }

  // Places in a work list for the listed rows of each segment (by its first
  // lane), one atomic per warp: the first of this lane's; put(place, row bit).
  template <class Put>
  __device__ __forceinline__ void list(unsigned int* counter, int lane, Put put) const {
    const unsigned int mine = (lane & 7) == 0 ? __popc(listed) : 0u;
    unsigned int t = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int u = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += u;
    }
    const unsigned int total = __shfl_sync(0xffffffffu, t, 31);
    if (!total) return;
    unsigned int base = 0;
    if (lane == 31) base = atomicAdd(counter, total);
    base = __shfl_sync(0xffffffffu, base, 31) + t - mine;
    if ((lane & 7) == 0)
      for (uint32_t m = listed; m; m &= m - 1u, ++base) put(base, __ffs(m) - 1);
  }

  // The bulk rows: mu of rows y0 - 1 .. y0 + R in flight at once, x neighbours
  // by shuffle.
  template <class G>
  __device__ __forceinline__ void update(const G& g, const float* in, int sx, int y0, int lane,
                                         const uint8_t* code) const {
    if (!__any_sync(0xffffffffu, bulk != 0u)) return;
    const int wc = lane >> 3, seg = 4 * sx + wc, xs = 128 * sx + 4 * lane;
    const bool have = xs <= g.nx;   // (the lane past the row's end holds its ghost for its neighbour)
    const int keep = g.nx - xs;   // cells of this lane inside the row (4 and more: all)
    const bool first = xs == 0, last = keep >= 1 && keep <= 4, sider = lane == 0 || lane == 31;
    const float* row = in + (long long)NP * g.fstride + (long long)y0 * g.pitch + xs + g.xoff;
    float4 v[NM][R + 2];
    float e[NM][R + 2];   // the strip's neighbours in x (lanes 0 and 31)
#pragma unroll
    for (int r = 0; r < R + 2; ++r)
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        const float* p = row + i * g.fstride + (long long)r * g.pitch;
        const bool ok = have && y0 + r <= g.ny + 1;   // the grid's upper ghost row at most
        v[i][r] = ok ? ld4<L2>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
        e[i][r] = ok && sider && r >= 1 && r <= R ? ld1<L2>(p + (lane == 0 ? -1 : 4)) : 0.0f;
      }
    const int reuse = g.reuse_prev ? kCodeReuse : 0;
    const long long oxl = g.bc[0] == 3 ? g.nx : -1, oxr = g.bc[0] == 3 ? -xs - 1 : keep;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int y = y0 + r, l = rf[r + 1] - 1;
      float mn[NM][4], L[NM][4];
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        const float4 c = v[i][r + 1], n = v[i][r], s = v[i][r + 2];
        float xm = __shfl_up_sync(0xffffffffu, c.w, 1), xp = __shfl_down_sync(0xffffffffu, c.x, 1);
        if (lane == 0) xm = e[i][r + 1];
        if (lane == 31) xp = e[i][r + 1];
        L[i][0] = (xm + c.y) + (n.x + s.x) - 4.0f * c.x;
        L[i][1] = (c.x + c.z) + (n.y + s.y) - 4.0f * c.y;
        L[i][2] = (c.y + c.w) + (n.z + s.z) - 4.0f * c.z;
        L[i][3] = (c.z + xp) + (n.w + s.w) - 4.0f * c.w;
      }
      if (!((bulk >> r) & 1u)) continue;
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        const float4 c = v[i][r + 1];
        const float cv[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float d = cv[q] - g.eb[l][i];
#pragma unroll
          for (int j = 0; j < NM; ++j) d += g.Kb[l][i * NM + j] * L[j][q];
          mn[i][q] = d;
        }
      }
      const bool write_phi = (code[(r + 1) * CS + wc + 1] & reuse) == 0;
      float* const o0 = g.out + (long long)(y + 1) * g.pitch + xs + g.xoff;
      // the lane's cells and the x ghost images of the row's first and last
      auto cells = [&](float* q, const float* w) {
        if (keep >= 4) {
          stg4(q, w[0], w[1], w[2], w[3]);
        } else {   // the end of a ragged row
          q[0] = w[0];
          if (keep >= 2) q[1] = w[1];
          if (keep >= 3) q[2] = w[2];
        }
        if (first) q[oxl] = w[0];
        if (last) q[oxr] = keep == 4 ? w[3] : keep == 3 ? w[2] : keep == 2 ? w[1] : w[0];
      };
      auto put = [&](float* p) {
        if (write_phi) {
#pragma unroll
          for (int a = 0; a < NP; ++a) {
            const float f = a == l ? 1.0f : 0.0f;
            const float w[4] = {f, f, f, f};
            cells(p + a * g.fstride, w);
          }
        }
#pragma unroll
        for (int i = 0; i < NM; ++i) cells(p + (NP + i) * g.fstride, mn[i]);
      };
      put(o0);
      if (y == 0) put(o0 + (long long)(g.bc[1] == 3 ? g.ny : -1) * g.pitch);
      if (y == g.ny - 1) put(o0 + (long long)(g.bc[1] == 3 ? -g.ny : 1) * g.pitch);
      if ((lane & 7) == 0) g.codes_out[(long long)y * g.segs + seg] = (uint8_t)(rf[r + 1] | kCodeReuse);
    }
  }
};

}  // namespace msgb
