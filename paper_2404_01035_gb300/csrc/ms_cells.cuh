// Cell-list form of the 3-D step, for FP64.
//
// FP64 arithmetic is what bounds an FP64 step on this part (2 FMA a clock and
// SM: a warp instruction holds the pipe for 16 cycles, whatever its mask), so
// this form is built to issue as little of it as possible, and evenly over the
// SMs: single cells are listed, not whole rows; a face flux is evaluated once,
// by the cell below it, instead of by both of its cells; a cell's mobility
// once instead of by itself and its six neighbours; pairs with a phase absent
// from the cell's neighbourhood are skipped.  Three launches:
//   k_c_scan:   a warp per 32-cell row segment.  Cells whose 3 x 3 x 3 block is
//               one pure phase take the bulk update; the others are listed with
//               the mask of the phases in their block.
//   k_c_faces:  a thread per listed cell: J on its three upper faces, M(phi).
//   k_c_update: a thread per listed cell: divergence, centre term, potential,
//               projection and mu update from the stored fluxes and mobilities.
// A flux stored by no cell is zero: a face below a listed cell whose lower cell
// is not listed has its whole stencil inside that cell's pure block.
// eutectic 67x50x61 on a GB300: 894 us a step in the fused kernel, whose tiles
// put the interface planes on 63 CTAs, 145 us in this form (scan 15, faces 53,
// update 77).
#pragma once

#include "ms_step.cuh"

namespace msgb {

// Scratch of the cell-list step (one allocation, laid out by cells_layout).
template <class Real>
struct CellsScratch {
  unsigned int* list;      // [0] count, [1] exit ticket, [2..] listed cells (linear index)
  uint8_t* mask;           // phases in the block of listed cell k
  uint8_t* kind;           // per cell: pure phase + 1 where bulk, 0 where listed
  unsigned int* pos;       // per cell: its place in the list where listed; NULL: fluxes are stored by cell
  Real* J;                 // [3 NP][slots] upper-face fluxes of listed cells, [D NP + a], by cell or place
  Real* M;                 // [NM NM][slots] mobilities of listed cells
  long long slots;         // (see cell_slots)
  // where the fluxes of listed cell i, the k-th, are, or (place past the end) none are stored
  __device__ __forceinline__ unsigned int slot(unsigned int i, unsigned int k) const { return pos ? k : i; }
  __device__ __forceinline__ unsigned int slot_of(long long i) const { return pos ? pos[i] : (unsigned int)i; }
};

// (cells_scratch_bytes in ms_runtime.cu adds up the same parts)
template <class Real>
CellsScratch<Real> cells_layout(void* base, const HostModel& m) {
  CellsScratch<Real> c;
  const size_t cells = (size_t)m.nx * m.ny * m.nz, slots = cell_slots(cells);
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  char* p = static_cast<char*>(base);
  c.list = reinterpret_cast<unsigned int*>(p);
  p += up((cells + 2) * 4);
  c.mask = reinterpret_cast<uint8_t*>(p);
  p += up(cells);
  c.kind = reinterpret_cast<uint8_t*>(p);
  p += up(cells);
  c.pos = slots < cells ? reinterpret_cast<unsigned int*>(p) : nullptr;
  if (c.pos) p += up(cells * 4);
  c.J = reinterpret_cast<Real*>(p);
  p += up(3 * m.N * slots * sizeof(Real));
  c.M = reinterpret_cast<Real*>(p);
  c.slots = (long long)slots;
  return c;
}

// Stencil accessor over the padded input state.
template <int NP, int NM, class Real>
struct PadAcc {
  const Real* s;   // the cell in field 0
  long long fs, plane;
  int pitch;
  uint32_t m;
  const StepArgs<Real, NP, NM>* g;
  __device__ __forceinline__ Real phi(int a, int dx, int dy, int dz) const {
    return s[a * fs + dz * plane + (long long)dy * pitch + dx];
  }
  __device__ __forceinline__ Real mu(int i, int dx, int dy, int dz) const { return phi(NP + i, dx, dy, dz); }
  __device__ __forceinline__ uint32_t mask() const { return m; }
};

template <int NP, int NM, class Real>
__global__ void __launch_bounds__(256) k_c_scan(const __grid_constant__ StepArgs<Real, NP, NM> g,
                                                const Real* __restrict__ in,
                                                const __grid_constant__ CellsScratch<Real> c) {
  const int lane = threadIdx.x & 31;
  const unsigned int nseg = (unsigned int)g.segs * g.ny * g.nz, w0 = blockIdx.x * 8u + (threadIdx.x >> 5);
  const bool live = w0 < nseg;   // (warps past the end redo the last segment and list nothing)
  const unsigned int w = live ? w0 : nseg - 1;
  const int sg = (int)(w % g.segs), y = (int)((w / g.segs) % g.ny), z = (int)(w / ((unsigned int)g.segs * g.ny));
  const int x = 32 * sg + lane;
  const bool active = live && x < g.nx;
  const long long plane = (long long)g.nyp * g.pitch;
  const Real* s = in + (long long)(z + g.zoff) * plane + (long long)(y + 1) * g.pitch + g.xoff;
  // the 27 segment codes around: all one pure phase = the whole segment is bulk
  int code = 0;
  if (lane < 27) code = load_code(g, sg + lane % 3 - 1, y + (lane / 3) % 3 - 1, z + lane / 9 - 1) & kCodePhase;
  const int c0 = __shfl_sync(0xffffffffu, code, 0);
  int bulk;
  uint32_t present = 0;
  if (__all_sync(0xffffffffu, lane >= 27 || (code != 0 && code == c0))) {
    bulk = c0;
  } else {
    // common pure code of the 3 x 3 column at xx (0 if none), its phases OR-ed into nzm
    auto column = [&](int xx, uint32_t& nzm) {
      int col = -1;
#pragma unroll
      for (int r = 0; r < 9; ++r) {
        const Real* p = s + (long long)(r / 3 - 1) * plane + (long long)(r % 3 - 1) * g.pitch + xx;
        uint32_t nz = 0, one = 0;
#pragma unroll
        for (int a = 0; a < NP; ++a) {
          const Real v = p[a * g.fstride];
          nz |= (nonzero(v) ? 1u : 0u) << a;
          one |= (is_one(v) ? 1u : 0u) << a;
        }
        nzm |= nz;
        const int pc = (__popc(nz) == 1 && nz == one) ? __ffs(nz) : 0;
        col = (col == -1 || col == pc) ? pc : 0;
      }
      return col;
    };
    uint32_t mine = 0, side = 0;
    const int col = column(min(x, g.nx), mine);   // lanes past the row read its ghost column
    int edge = 0;
    if (lane == 0 || lane == 31) edge = column(lane == 0 ? 32 * sg - 1 : min(x + 1, g.nx), side);
    int left = __shfl_up_sync(0xffffffffu, col, 1), right = __shfl_down_sync(0xffffffffu, col, 1);
    uint32_t ml = __shfl_up_sync(0xffffffffu, mine, 1), mr = __shfl_down_sync(0xffffffffu, mine, 1);
    if (lane == 0) {
      left = edge;
      ml = side;
    }
    if (lane == 31) {
      right = edge;
      mr = side;
    }
    present = mine | ml | mr;
    bulk = (col != 0 && left == col && right == col) ? col : 0;
  }
  const unsigned int cell = ((unsigned int)z * g.ny + y) * g.nx + min(x, g.nx - 1);
  if (active) c.kind[cell] = (uint8_t)bulk;
  if (active && bulk != 0) {
    PadAcc<NP, NM, Real> A{s + x, g.fstride, plane, g.pitch, 0u, &g};
    Real pn[NP], mn[NM];
    bulk_cell<3, NP, NM, Real>(A, g, bulk - 1, pn, mn);
    store_cell<3>(g, x, y, z, pn, mn);
  }
  // code of the output segment: pure where every cell is bulk in one phase
  const int ref = __shfl_sync(0xffffffffu, bulk, 0);
  const bool same = __all_sync(0xffffffffu, !active || bulk == ref);
  if (live && lane == 0)
    g.codes_out[((long long)(z + g.zoff) * g.ny + y) * g.segs + sg] = same ? (uint8_t)ref : (uint8_t)0;
  const bool want = active && bulk == 0;
  const unsigned int k = block_append<256>(&c.list[0], want);
  if (want) {
    c.list[2 + k] = cell;
    c.mask[k] = (uint8_t)present;
    if (c.pos) c.pos[cell] = k;
  }
}

template <int NP, int NM, class Real>
__device__ __forceinline__ bool pair_aniso(const StepArgs<Real, NP, NM>& g, uint32_t mask) {
  bool r = false;
  int p = 0;
#pragma unroll
  for (int a = 0; a < NP; ++a)
#pragma unroll
    for (int b = a + 1; b < NP; ++b, ++p) r = r || ((((mask >> a) & (mask >> b)) & 1u) && g.aniso[p]);
  return r;
}

template <class Real, int NP, int NM>
__device__ __forceinline__ DiffPrm<Real, NP*(NP - 1) / 2> plain_prm(const StepArgs<Real, NP, NM>& g) {
  DiffPrm<Real, NP*(NP - 1) / 2> dp;
  dp.mob = g.mob;
#pragma unroll
  for (int p = 0; p < NP * (NP - 1) / 2; ++p) dp.delta[p] = g.delta[p];
  return dp;
}

template <int NP, int NM, class Real>
__global__ void __launch_bounds__(64) k_c_faces(const __grid_constant__ StepArgs<Real, NP, NM> g,
                                                const Real* __restrict__ in,
                                                const __grid_constant__ CellsScratch<Real> c) {
  const unsigned int count = *(volatile unsigned int*)&c.list[0];
  const long long plane = (long long)g.nyp * g.pitch;
  const auto dp = plain_prm<Real, NP, NM>(g);
  for (unsigned int k = blockIdx.x * 64u + threadIdx.x; k < count; k += gridDim.x * 64u) {
    const unsigned int i = c.list[2 + k], r = i / (unsigned int)g.nx, at = c.slot(i, k);
    if (at >= c.slots) break;   // (later cells have none either)
    const int x = (int)(i - r * g.nx), y = (int)(r % (unsigned int)g.ny), z = (int)(r / (unsigned int)g.ny);
    PadAcc<NP, NM, Real> A{in + (long long)(z + g.zoff) * plane + (long long)(y + 1) * g.pitch + x + g.xoff,
                           g.fstride, plane, g.pitch, c.mask[k], &g};
    const bool tan = pair_aniso<NP, NM, Real>(g, A.m);
    Real J[NP];
    face_flux<3, 0, NP, NM, Real, Real>(A, g, dp, A.m, 1, tan, J);
#pragma unroll
    for (int a = 0; a < NP; ++a) c.J[a * c.slots + at] = J[a];
    face_flux<3, 1, NP, NM, Real, Real>(A, g, dp, A.m, 1, tan, J);
#pragma unroll
    for (int a = 0; a < NP; ++a) c.J[(NP + a) * c.slots + at] = J[a];
    face_flux<3, 2, NP, NM, Real, Real>(A, g, dp, A.m, 1, tan, J);
#pragma unroll
    for (int a = 0; a < NP; ++a) c.J[(2 * NP + a) * c.slots + at] = J[a];
    if (!g.gg) {
      Real ph[NP], M[NM * NM];
#pragma unroll
      for (int a = 0; a < NP; ++a) ph[a] = A.phi(a, 0, 0, 0);
      cell_mobility<NP, NM>(ph, g.DX, M);
#pragma unroll
      for (int q = 0; q < NM * NM; ++q) c.M[q * c.slots + at] = M[q];
    }
  }
}

// One axis of a listed cell: adds (J_upper - J_lower) / dx to divJ and the mu
// flux through both faces to div.  `at`: where the cell's own fluxes are; `pos`, n,
// bc: its index along the axis, its extent and boundary code; `step`: linear cells to
// its neighbour.  What no cell stores (no cell below a boundary face, no place left)
// is evaluated here.  PLACES: there may be places for some cells only.
template <int D, bool PLACES, int NP, int NM, class Real, class DP>
__device__ __forceinline__ void axis_terms(const StepArgs<Real, NP, NM>& g, const CellsScratch<Real>& c,
                                           const PadAcc<NP, NM, Real>& A, const DP& dp, unsigned int i, unsigned int at, int pos, int n,
                                           int bc, long long step, bool tan, const Real* Mc, const Real* mc, Real* divJ,
                                           Real* div) {
  // linear index of the lower / upper neighbour where it is a cell of the grid
  const bool lo_in = pos > 0 || bc == 3, hi_in = pos < n - 1 || bc == 3;
  const long long lo = (long long)i + (pos > 0 ? -step : (long long)(n - 1) * step);
  const long long hi = (long long)i + (pos < n - 1 ? step : -(long long)(n - 1) * step);
  // flux of the lower (0) / upper (1) face: from its place, zero (listed = false:
  // the face lies in a pure block), or evaluated
  auto flux = [&](int side, bool listed, unsigned int place, bool eval, Real* J) {
    if (eval) {
      face_flux<3, D, NP, NM, Real, Real>(A, g, dp, A.m, side, tan, J);
    } else {
#pragma unroll
      for (int a = 0; a < NP; ++a) J[a] = listed ? c.J[(D * NP + a) * c.slots + place] : Real(0);
    }
  };
  const bool below = lo_in && c.kind[lo] == 0;
  const unsigned int pl = !below ? 0u : PLACES ? c.slot_of(lo) : (unsigned int)lo;
  Real Jl[NP], Ju[NP];
  flux(0, below, pl, !lo_in || (PLACES && pl >= c.slots), Jl);
  flux(1, true, at, PLACES && at >= c.slots, Ju);
#pragma unroll
  for (int a = 0; a < NP; ++a) divJ[a] += (Ju[a] - Jl[a]) * g.inv_dx;
  if (g.gg) return;
#pragma unroll
  for (int sd = 0; sd < 2; ++sd) {
    const bool inside = sd ? hi_in : lo_in;
    const long long nb = sd ? hi : lo;
    const int d = sd ? 1 : -1;
    Real Mn[NM * NM];
    const int kd = inside ? c.kind[nb] : 0;
    const unsigned int pn = !inside || kd != 0 ? 0u : PLACES ? c.slot_of(nb) : (unsigned int)nb;
    if (!inside || (PLACES && pn >= c.slots)) {
      Real ph[NP];
#pragma unroll
      for (int a = 0; a < NP; ++a) ph[a] = A.phi(a, D == 0 ? d : 0, D == 1 ? d : 0, D == 2 ? d : 0);
      cell_mobility<NP, NM>(ph, g.DX, Mn);
    } else {
#pragma unroll
      for (int q = 0; q < NM * NM; ++q) Mn[q] = kd == 0 ? c.M[q * c.slots + pn] : g.DX[kd - 1][q];
    }
#pragma unroll
    for (int r = 0; r < NM; ++r)
#pragma unroll
      for (int q = 0; q < NM; ++q) {
        const Real Mf = Real(0.5) * (Mc[r * NM + q] + Mn[r * NM + q]);
        div[r] += Mf * ((A.mu(q, D == 0 ? d : 0, D == 1 ? d : 0, D == 2 ? d : 0) - mc[q]) * g.inv_dx2);
      }
  }
}

template <int NP, int NM, class Real, bool PLACES>
__global__ void __launch_bounds__(64) k_c_update(const __grid_constant__ StepArgs<Real, NP, NM> g,
                                                 const Real* __restrict__ in,
                                                 const __grid_constant__ CellsScratch<Real> c) {
  const unsigned int count = *(volatile unsigned int*)&c.list[0];
  const long long plane = (long long)g.nyp * g.pitch;
  const auto dp = plain_prm<Real, NP, NM>(g);
  for (unsigned int k = blockIdx.x * 64u + threadIdx.x; k < count; k += gridDim.x * 64u) {
    const unsigned int i = c.list[2 + k], r = i / (unsigned int)g.nx, at = PLACES ? c.slot(i, k) : i;
    const int x = (int)(i - r * g.nx), y = (int)(r % (unsigned int)g.ny), z = (int)(r / (unsigned int)g.ny);
    PadAcc<NP, NM, Real> A{in + (long long)(z + g.zoff) * plane + (long long)(y + 1) * g.pitch + x + g.xoff,
                           g.fstride, plane, g.pitch, c.mask[k], &g};
    const bool tan = pair_aniso<NP, NM, Real>(g, A.m);
    Real ph[NP], mc[NM], Mc[NM * NM], divJ[NP], Gc[NP], div[NM];
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      ph[a] = A.phi(a, 0, 0, 0);
      divJ[a] = Real(0);
      Gc[a] = Real(0);
    }
#pragma unroll
    for (int q = 0; q < NM; ++q) {
      mc[q] = A.mu(q, 0, 0, 0);
      div[q] = Real(0);
    }
#pragma unroll
    for (int q = 0; q < NM * NM; ++q) Mc[q] = g.gg || (PLACES && at >= c.slots) ? Real(0) : c.M[q * c.slots + at];
    if (PLACES && !g.gg && at >= c.slots) cell_mobility<NP, NM>(ph, g.DX, Mc);
    axis_terms<0, PLACES>(g, c, A, dp, i, at, x, g.nx, g.bc[0], 1ll, tan, Mc, mc, divJ, div);
    axis_terms<1, PLACES>(g, c, A, dp, i, at, y, g.ny, g.bc[1], (long long)g.nx, tan, Mc, mc, divJ, div);
    axis_terms<2, PLACES>(g, c, A, dp, i, at, z, g.nz, g.bc[2], (long long)g.nx * g.ny, tan, Mc, mc, divJ, div);
    Real gcr[NP][3];
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      gcr[a][0] = A.phi(a, 1, 0, 0) - A.phi(a, -1, 0, 0);
      gcr[a][1] = A.phi(a, 0, 1, 0) - A.phi(a, 0, -1, 0);
      gcr[a][2] = A.phi(a, 0, 0, 1) - A.phi(a, 0, 0, -1);
    }
    centre_term<3, NP, NM, Real, Real, kFeatAll, false>(g, dp, ph, gcr, A.m, Gc);
    const Real sT = g.tz0 + g.tzg * (Real(z + g.zorg) + Real(0.5));
    Real pn[NP], mn[NM];
    phase_update<3, NP, NM, Real, Real>(g, dp, ph, mc, divJ, Gc, sT, lab_cell<3>(g, x, y, z), pn);
    if (g.gg) {   // grain growth: mu held
#pragma unroll
      for (int q = 0; q < NM; ++q) mn[q] = mc[q];
    } else {
      mu_update<NP, NM, Real>(g, ph, pn, mc, div, sT, false, mn);
    }
    store_cell<3>(g, x, y, z, pn, mn);
  }
  // every CTA read the count before taking its ticket; the last one clears the list
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&c.list[1], 1u) == gridDim.x - 1) {
      c.list[0] = 0u;
      c.list[1] = 0u;
    }
  }
}

}  // namespace msgb
