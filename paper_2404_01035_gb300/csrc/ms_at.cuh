// Anti-trapping current in the mu update (MICROSIM paper, arXiv 2404.01035,
// Sec. 2.1, Eq. jatr and the obstacle / well forms of j^{at,alpha} below it):
// j_at = sum_{alpha < liquid} A_alpha (c^alpha - c^liq) d phi_alpha/dt
// n_alpha (-n_alpha . n_liq), subtracted from M grad mu inside the divergence
// of Eq. (Mu_explicit_temperature).
//
// It needs d phi/dt at both cells of every face, so it runs after the step
// that wrote phi^{n+1} and mu* (the mu update without the current) into the
// output buffer: mu^{n+1} = mu* - chi(h(phi^{n+1}))^-1 dt div j_at (the update
// is linear in its right-hand side).  Two kernels: k_at_list lists the 32-cell
// row segments whose 3 x 3 (x 3) block of segments is not one pure phase in
// phi^n (elsewhere every phase gradient at every face of the segment's cells
// is zero, so no face has a normal and the current vanishes); k_at_work
// corrects mu on the listed segments (phi^n and mu^n from the input, phi^{n+1}
// from the output), one lane per cell.
#pragma once

#include "ms_step.cuh"

namespace msgb {

// 1 / sqrt(x): the hardware reciprocal square root in FP32 (rsqrtf, a few
// ulp: the current is a correction far inside the FP32 tolerance), exact in
// FP64.
__device__ __forceinline__ float inv_sqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double inv_sqrt(double x) { return 1.0 / sqrt(x); }

// Coefficient A of j^{at,alpha} at the face value p of phi_alpha (read as the
// 1-D equilibrium profile value there): obstacle pi eps p (1 - h(p)) /
// (4 sqrt(p (1 - p))) with the two-phase h(p) = p^2 (3 - 2p), 0 outside
// 0 < p < 1; well eps / (2 sqrt 2).
template <class Real>
__device__ __forceinline__ Real at_coefficient(int potential, Real eps, Real p) {
  if (potential != 1) return eps * Real(0.35355339059327376220);   // 1 / (2 sqrt 2)
  if (!(p > Real(0) && p < Real(1))) return Real(0);
  const Real h = p * p * (Real(3) - Real(2) * p);
  return Real(0.78539816339744830962) * eps * p * (Real(1) - h) * inv_sqrt(p * (Real(1) - p));   // pi / 4
}

// Reads relative to a cell: phi^n and mu^n from the input state, phi^{n+1} from
// the output (whose phi the correction does not write), offsets in [-1, 1].
template <int DIM, int NP, int NM, class Real>
struct AtBox {
  const Real* in;    // the cell in field 0 of the input
  const Real* out;   // and of the output
  long long fs, plane;
  int pitch;
  __device__ __forceinline__ long long off(int f, int dx, int dy, int dz) const {
    return f * fs + (DIM == 3 ? dz * plane : 0) + (long long)dy * pitch + dx;
  }
  __device__ __forceinline__ Real phi(int a, int dx, int dy, int dz) const { return __ldg(in + off(a, dx, dy, dz)); }
  __device__ __forceinline__ Real mu(int i, int dx, int dy, int dz) const { return __ldg(in + off(NP + i, dx, dy, dz)); }
  __device__ __forceinline__ Real phin(int a, int dx, int dy, int dz) const { return __ldg(out + off(a, dx, dy, dz)); }
};

template <class Real>
struct AtShape {
  static constexpr int THREADS = 128;
  static constexpr int WARPS = THREADS / 32;
  static constexpr int MIN_BLOCKS = sizeof(Real) == 4 ? 6 : 2;   // FP32: 24 warps per SM
};

// dt times the normal component along axis d of j_at_i (the rates are taken
// as phi^{n+1} - phi^n) at the face between the cell at
// offset (ox, oy, oz) from the lane's cell and its +d neighbour: face values
// as for the gradient-energy fluxes (means of the two cells; normal
// difference and 4-point averaged tangential differences of phi^n), T the
// mean of the two cells' temperatures; kl = index of the left cell along the
// last axis.
template <int DIM, int NP, int NM, class Real>
__device__ __forceinline__ void at_face(const StepArgs<Real, NP, NM>& g, const AtBox<DIM, NP, NM, Real>& A, int ox,
                                        int oy, int oz, int d, int kl, Real* J) {
  constexpr int L = NP - 1;   // the liquid
  const int rx = ox + (d == 0), ry = oy + (d == 1), rz = oz + (d == 2);
  Real pf[NP], rate[NP], nrm[NP][DIM];
  bool has_n[NP];
#pragma unroll
  for (int a = 0; a < NP; ++a) {
    const Real vl = A.phi(a, ox, oy, oz), vr = A.phi(a, rx, ry, rz);
    pf[a] = Real(0.5) * (vl + vr);
    rate[a] = Real(0.5) * ((A.phin(a, ox, oy, oz) - vl) + (A.phin(a, rx, ry, rz) - vr));   // dt d phi/dt
    Real gr[DIM], g2 = Real(0);
#pragma unroll
    for (int t = 0; t < DIM; ++t) {
      if (t == d) {
        gr[t] = (vr - vl) * g.inv_dx;
      } else {
        const int tx = t == 0, ty = t == 1, tz = t == 2;
        gr[t] = ((A.phi(a, ox + tx, oy + ty, oz + tz) + A.phi(a, rx + tx, ry + ty, rz + tz)) -
                 (A.phi(a, ox - tx, oy - ty, oz - tz) + A.phi(a, rx - tx, ry - ty, rz - tz))) *
                g.quarter_inv_dx;
      }
      g2 += gr[t] * gr[t];
    }
    has_n[a] = g2 >= Real(1e-12);
    const Real inv = has_n[a] ? inv_sqrt(g2) : Real(0);
#pragma unroll
    for (int t = 0; t < DIM; ++t) nrm[a][t] = gr[t] * inv;
  }
#pragma unroll
  for (int i = 0; i < NM; ++i) J[i] = Real(0);
  if (!has_n[L]) return;
  Real mf[NM];
#pragma unroll
  for (int i = 0; i < NM; ++i) mf[i] = Real(0.5) * (A.mu(i, ox, oy, oz) + A.mu(i, rx, ry, rz));
  // T - T_ref at the two cells (after the boundary mapping) and their mean
  const int n = DIM == 3 ? g.nz : g.ny, bc = g.bc[DIM - 1];
  const int kr = kl + (d == DIM - 1);
  const int kml = bc_map(kl, n, bc), kmr = bc_map(kr, n, bc);
  const Real sf = g.tz0 + g.tzg * (Real(0.5) * Real(kml + kmr) + Real(g.zorg) + Real(0.5));
  Real cl[NM];
#pragma unroll
  for (int i = 0; i < NM; ++i) {
    Real c = Real(0);
#pragma unroll
    for (int j = 0; j < NM; ++j) c += g.chi[L][i * NM + j] * (mf[j] - (g.B0[L][j] + g.B1[L][j] * sf));
    cl[i] = c;
  }
#pragma unroll
  for (int al = 0; al < L; ++al) {
    if (!has_n[al]) continue;
    Real proj = Real(0);   // -n_alpha . n_liq
#pragma unroll
    for (int t = 0; t < DIM; ++t) proj -= nrm[al][t] * nrm[L][t];
    const Real k = at_coefficient<Real>(g.potential, g.eps, pf[al]) * rate[al] * nrm[al][d] * proj;
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      Real c = Real(0);
#pragma unroll
      for (int j = 0; j < NM; ++j) c += g.chi[al][i * NM + j] * (mf[j] - (g.B0[al][j] + g.B1[al][j] * sf));
      J[i] += k * (c - cl[i]);
    }
  }
}

// dt times (j_at on the upper face along axis D minus on the lower one), FP32:
// at_face's arithmetic for both faces at once in paired registers, in its order:
// where a trace of a phase puts |grad phi|^2 near the cut-off of the normals, the
// last bit decides whether the current acts, so every launch takes the same sums.
// A face without a normal has a zero unit normal, so its current vanishes without a
// test.  lanes: the warp's lanes that call.
template <int DIM, int D, int NP, int NM>
__device__ __forceinline__ void at_axis(const StepArgs<float, NP, NM>& g, const AtBox<DIM, NP, NM, float>& A,
                                        int k, uint32_t lanes, float* dJ) {
  constexpr int L = NP - 1;   // the liquid
  constexpr int X = D == 0, Y = D == 1, Z = D == 2;
  F2 nL[DIM], cl[NM], mf[NM], J[NM], sf;
  // unit normal of phase a on both faces; false where no lane has one
  auto normal = [&](int a, F2 lr, F2* n) {
    F2 gr[DIM], g2 = f2s(0.0f);
#pragma unroll
    for (int t = 0; t < DIM; ++t) {
      if (t == D) {
        gr[t] = lr * f2s(g.inv_dx);
      } else {
        const int tx = t == 0, ty = t == 1, tz = t == 2;
        const float u = A.phi(a, tx, ty, tz), d = A.phi(a, -tx, -ty, -tz);
        gr[t] = ((f2(A.phi(a, tx - X, ty - Y, tz - Z), u) + f2(u, A.phi(a, tx + X, ty + Y, tz + Z))) -
                 (f2(A.phi(a, -tx - X, -ty - Y, -tz - Z), d) + f2(d, A.phi(a, X - tx, Y - ty, Z - tz)))) *
                f2s(g.quarter_inv_dx);
      }
      g2 = fma2(gr[t], gr[t], g2);
    }
    const float lo = f2lo(g2), hi = f2hi(g2);
    const F2 inv = f2(lo >= 1e-12f ? inv_sqrt(lo) : 0.0f, hi >= 1e-12f ? inv_sqrt(hi) : 0.0f);
#pragma unroll
    for (int t = 0; t < DIM; ++t) n[t] = gr[t] * inv;
    return lo >= 1e-12f || hi >= 1e-12f;
  };
#pragma unroll
  for (int i = 0; i < NM; ++i) J[i] = f2s(0.0f);
  const bool hasL = normal(L, f2(A.phi(L, 0, 0, 0), A.phi(L, X, Y, Z)) - f2(A.phi(L, -X, -Y, -Z), A.phi(L, 0, 0, 0)), nL);
  if (__any_sync(lanes, hasL)) {
    // T - T_ref: the mean of the two cells' temperatures (after the boundary mapping)
    const int n = DIM == 3 ? g.nz : g.ny, bc = g.bc[DIM - 1];
    const float zo = (float)g.zorg + 0.5f;
    const int kl = bc_map(k - (D == DIM - 1), n, bc), kh = bc_map(k + (D == DIM - 1), n, bc);
    sf = f2(g.tz0 + g.tzg * (0.5f * (float)(kl + k) + zo), g.tz0 + g.tzg * (0.5f * (float)(k + kh) + zo));
#pragma unroll
    for (int i = 0; i < NM; ++i)
      mf[i] = f2s(0.5f) * (f2(A.mu(i, -X, -Y, -Z), A.mu(i, 0, 0, 0)) + f2(A.mu(i, 0, 0, 0), A.mu(i, X, Y, Z)));
    auto conc = [&](int a, F2* c) {
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        c[i] = f2s(0.0f);
#pragma unroll
        for (int j = 0; j < NM; ++j)
          c[i] = fma2(f2s(g.chi[a][i * NM + j]), mf[j] - fma2(f2s(g.B1[a][j]), sf, f2s(g.B0[a][j])), c[i]);
      }
    };
    conc(L, cl);
#pragma unroll
    for (int a = 0; a < L; ++a) {
      const float vm = A.phi(a, -X, -Y, -Z), v0 = A.phi(a, 0, 0, 0), vp = A.phi(a, X, Y, Z);
      const F2 l = f2(vm, v0), r = f2(v0, vp);
      F2 na[DIM];
      if (!__any_sync(lanes, normal(a, r - l, na))) continue;
      const F2 pf = f2s(0.5f) * (l + r);
      const float d0 = A.phin(a, 0, 0, 0) - v0;
      const F2 rate = f2s(0.5f) * (f2(A.phin(a, -X, -Y, -Z) - vm, d0) + f2(d0, A.phin(a, X, Y, Z) - vp));
      F2 proj = f2s(0.0f);   // n_alpha . n_liq
#pragma unroll
      for (int t = 0; t < DIM; ++t) proj = fma2(na[t], nL[t], proj);
      const F2 co = f2(at_coefficient<float>(g.potential, g.eps, f2lo(pf)), at_coefficient<float>(g.potential, g.eps, f2hi(pf)));
      const F2 w = f2s(-1.0f) * co * rate * na[D] * proj;
      F2 ca[NM];
      conc(a, ca);
#pragma unroll
      for (int i = 0; i < NM; ++i) J[i] = fma2(w, ca[i] - cl[i], J[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < NM; ++i) dJ[i] = f2hi(J[i]) - f2lo(J[i]);
}

// One thread per row segment: append the segments whose block of segments is
// not one pure phase in phi^n to the work list ([0] count, [1] ticket).
template <int DIM, int NP, int NM, class Real>
__global__ void __launch_bounds__(256) k_at_list(const __grid_constant__ StepArgs<Real, NP, NM> g) {
  const long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int nzi = DIM == 3 ? g.nz : 1;
  const long long nseg = (long long)g.segs * g.ny * nzi;
  bool need = false;
  if (w < nseg) {
    const int s = (int)(w % g.segs);
    const int y = (int)((w / g.segs) % g.ny);
    const int z = (int)(w / ((long long)g.segs * g.ny));
    const int c0 = load_code_from(g.codes_in, g, s, y, z) & kCodePhase;
    bool pure = c0 != 0;
#pragma unroll
    for (int dz = (DIM == 3 ? -1 : 0); dz <= (DIM == 3 ? 1 : 0); ++dz)
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int ds = -1; ds <= 1; ++ds)
          pure = pure && (load_code_from(g.codes_in, g, s + ds, y + dy, z + dz) & kCodePhase) == c0;
    need = !pure;
  }
  const unsigned int i = block_append<256>(&g.at_list[0], need);
  if (need && i < g.at_cap) g.at_list[2 + i] = (unsigned int)w;
}

// Warps over the listed segments, a lane per cell, the stencil by plain loads
// (whole rows; L1 holds what the offsets share).  The last CTA to finish clears
// the list (ticket), so the launches replay from a graph.  FP32 evaluates the
// two faces of an axis together.  What bounds it: the latency of its loads, so 24
// warps per SM, also where the builds for that many spill a little (us a step of all
// kernels, 24 / 20 / 16 warps: three phases 133 / 135 / 142, two 67 / 69 / 71, eight
// 1616 / 1662 / 1681): eutectic 150x133x97 on a GB300 takes 42 us a step, 53 with 16
// warps, 63 with the block staged element by element in shared memory, every face
// on its own and the rows without a current corrected too.
template <int DIM, int NP, int NM, class Real>
__global__ void __launch_bounds__(AtShape<Real>::THREADS, AtShape<Real>::MIN_BLOCKS)
    k_at_work(const __grid_constant__ StepArgs<Real, NP, NM> g, const Real* __restrict__ in) {
  using Sh = AtShape<Real>;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned int count = min(*(volatile unsigned int*)&g.at_list[0], g.at_cap);
  const long long plane = (long long)g.nyp * g.pitch;
  for (unsigned int i = blockIdx.x * Sh::WARPS + wid; i < count; i += gridDim.x * Sh::WARPS) {
    const unsigned int r = g.at_list[2 + i];
    const int s = (int)(r % (unsigned int)g.segs);
    const unsigned int zy = r / (unsigned int)g.segs;
    const int y = (int)(zy % (unsigned int)g.ny), z = (int)(zy / (unsigned int)g.ny);
    const int x = 32 * s + lane;
    const uint32_t lanes = __ballot_sync(0xffffffffu, x < g.nx);
    if (x < g.nx) {
      const long long o = (long long)(DIM == 3 ? z + g.zoff : 0) * plane + (long long)(y + 1) * g.pitch + x + g.xoff;
      const AtBox<DIM, NP, NM, Real> A{in + o, g.out + o, g.fstride, plane, g.pitch};
      const int k = DIM == 3 ? z : y;   // index along the last axis
      Real div[NM];
#pragma unroll
      for (int q = 0; q < NM; ++q) div[q] = Real(0);
      if constexpr (sizeof(Real) == 4) {
        Real dJ[NM];
        at_axis<DIM, 0, NP, NM>(g, A, k, lanes, dJ);
#pragma unroll
        for (int q = 0; q < NM; ++q) div[q] += dJ[q] * g.inv_dx;
        at_axis<DIM, 1, NP, NM>(g, A, k, lanes, dJ);
#pragma unroll
        for (int q = 0; q < NM; ++q) div[q] += dJ[q] * g.inv_dx;
        if constexpr (DIM == 3) {
          at_axis<DIM, 2, NP, NM>(g, A, k, lanes, dJ);
#pragma unroll
          for (int q = 0; q < NM; ++q) div[q] += dJ[q] * g.inv_dx;
        }
      } else {
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
          Real Jp[NM], Jm[NM];
          at_face<DIM, NP, NM, Real>(g, A, 0, 0, 0, d, k, Jp);
          at_face<DIM, NP, NM, Real>(g, A, -(d == 0), -(d == 1), -(d == 2), d, k - (d == DIM - 1), Jm);
#pragma unroll
          for (int q = 0; q < NM; ++q) div[q] += (Jp[q] - Jm[q]) * g.inv_dx;
        }
      }
      bool moved = false;   // a row without a current keeps mu*
#pragma unroll
      for (int q = 0; q < NM; ++q) moved = moved || div[q] != Real(0);
      if (!__any_sync(lanes, moved)) continue;
      // mu^{n+1} = mu* + chi(h(phi^{n+1}))^-1 (-dt div j_at)
      Real pn[NP], h[NP];
#pragma unroll
      for (int a = 0; a < NP; ++a) pn[a] = A.phin(a, 0, 0, 0);
      interp_h<NP, true>(pn, h);
      Real chi[NM * NM], rhs[NM], dmu[NM], mn[NM];
#pragma unroll
      for (int q = 0; q < NM * NM; ++q) {
        chi[q] = h[0] * g.chi[0][q];
#pragma unroll
        for (int a = 1; a < NP; ++a) chi[q] += h[a] * g.chi[a][q];
      }
#pragma unroll
      for (int q = 0; q < NM; ++q) rhs[q] = -div[q];   // the rates above carry no 1/dt: dt div j_at
      solve_small<NM>(chi, rhs, dmu);
#pragma unroll
      for (int q = 0; q < NM; ++q) mn[q] = g.out[(long long)(NP + q) * g.fstride + o] + dmu[q];
      store_cell<DIM>(g, x, y, z, pn, mn, false);
    }
  }
  // every CTA read the count before taking its ticket; the last one clears the list
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&g.at_list[1], 1u) == gridDim.x - 1) {
      g.at_list[0] = 0u;
      g.at_list[1] = 0u;
    }
  }
}

}  // namespace msgb
