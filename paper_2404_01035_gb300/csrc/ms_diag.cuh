// Diagnostics of one state with FP64 reductions: solute mass sum_cells c_i
// with c = sum_a h_a c^a(mu, T) (the composition constraint under Eq.
// Mu_explicit_temperature), max |sum phi - 1|, min/max phi, the count of
// non-finite values, and the largest explicit mu-diffusion number
// dt sum_faces ||chi(phi)^-1 M_f||_inf / dx^2 (the device-side dt check).
// Per-cell values are evaluated in the state's precision and accumulated in
// FP64; the two-stage reduction runs in a fixed order (deterministic).
#pragma once

#include "ms_internal.h"
#include "ms_step.cuh"

namespace msgb {

constexpr int kDiagThreads = 256;

template <int NM, class R>
__device__ __forceinline__ void inv_small(const R* A, R* X) {
  if constexpr (NM == 1) {
    X[0] = R(1) / A[0];
  } else if constexpr (NM == 2) {
    R det = A[0] * A[3] - A[1] * A[2];
    X[0] = A[3] / det;
    X[1] = -A[1] / det;
    X[2] = -A[2] / det;
    X[3] = A[0] / det;
  } else {
    R c00 = A[4] * A[8] - A[5] * A[7], c01 = A[5] * A[6] - A[3] * A[8];
    R c02 = A[3] * A[7] - A[4] * A[6];
    R det = A[0] * c00 + A[1] * c01 + A[2] * c02;
    X[0] = c00 / det;
    X[3] = c01 / det;
    X[6] = c02 / det;
    X[1] = (A[2] * A[7] - A[1] * A[8]) / det;
    X[4] = (A[0] * A[8] - A[2] * A[6]) / det;
    X[7] = (A[1] * A[6] - A[0] * A[7]) / det;
    X[2] = (A[1] * A[5] - A[2] * A[4]) / det;
    X[5] = (A[2] * A[3] - A[0] * A[5]) / det;
    X[8] = (A[0] * A[4] - A[1] * A[3]) / det;
  }
}

// Per-thread running values of the diagnostics other than the solute sums:
// min / max phi, max |sum phi - 1|, max of the per-cell diffusion sum.  FP64
// states keep them in FP64.  FP32 states keep them in FP32 and convert once
// at the end (FP64 is a slow pipe): min and max are exact in either, the
// diffusion number dt num / dx^2 is monotone in num (its FP64 rounding
// commutes with the max), and |sum phi - 1| comes from an error-free FP32
// summation (TwoSum), so the result is the deviation rounded once to FP32.
template <class Real>
struct DiagRun {
  double lo = 1e300, hi = -1e300, dev = 0.0, num = 0.0;
  __device__ __forceinline__ void phase(Real v) {
    lo = fmin(lo, (double)v);
    hi = fmax(hi, (double)v);
  }
  template <int NP>
  __device__ __forceinline__ void sum_dev(const Real* ph) {
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < NP; ++a) s += (double)ph[a];
    dev = fmax(dev, fabs(s - 1.0));
  }
  __device__ __forceinline__ void diffusion(Real n, double dt, double inv_dx2) {
    num = fmax(num, dt * (double)n * inv_dx2);
  }
  __device__ __forceinline__ void finish(double dt, double inv_dx2, double* acc, int NM) {
    acc[NM] = dev;
    acc[NM + 1] = lo;
    acc[NM + 2] = hi;
    acc[NM + 4] = num;
  }
};

template <>
struct DiagRun<float> {
  float lo = INFINITY, hi = -INFINITY, dev = 0.0f, num = 0.0f;
  __device__ __forceinline__ void phase(float v) {
    lo = fminf(lo, v);
    hi = fmaxf(hi, v);
  }
  template <int NP>
  __device__ __forceinline__ void sum_dev(const float* ph) {
    float s = ph[0], e = 0.0f;
#pragma unroll
    for (int a = 1; a < NP; ++a) {   // TwoSum (Knuth): s + e is the exact sum
      const float t = __fadd_rn(s, ph[a]);
      const float bp = __fsub_rn(t, s);
      e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(ph[a], bp)));
      s = t;
    }
    dev = fmaxf(dev, fabsf(__fadd_rn(__fsub_rn(s, 1.0f), e)));
  }
  __device__ __forceinline__ void diffusion(float n, double, double) { num = fmaxf(num, n); }
  __device__ __forceinline__ void finish(double dt, double inv_dx2, double* acc, int NM) {
    acc[NM] = (double)dev;
    acc[NM + 1] = lo == INFINITY ? 1e300 : (double)lo;
    acc[NM + 2] = hi == -INFINITY ? -1e300 : (double)hi;
    acc[NM + 4] = dt * (double)num * inv_dx2;
  }
};

template <class Real, int NP, int NM>
struct DiagConsts {
  Real chi[NP][NM * NM];
  Real DX[NP][NM * NM];
  Real B0[NP][NM], B1[NP][NM];
};

struct DiagGeom {
  int nx, ny, nz, pitch, nyp, xoff, zoff, zorg, segs;
  int bc[3];
  long long fstride;
};

// Sum over the faces of a cell of ||chi^-1 M_f||_inf, from the cell's and its
// neighbours' mobilities (Mn(face) fills one).
template <int DIM, int NM, class Real, class Nb>
__device__ __forceinline__ Real diffusion_sum(const Real* chi, const Real* Mc, Nb neighbour) {
  Real chinv[NM * NM];
  inv_small<NM>(chi, chinv);
  Real num = Real(0);
#pragma unroll
  for (int d = 0; d < DIM; ++d)
#pragma unroll
    for (int sd = -1; sd <= 1; sd += 2) {
      Real Mn[NM * NM];
      neighbour(d, sd, Mn);
      Real rmax = Real(0);
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        Real r = Real(0);
#pragma unroll
        for (int j = 0; j < NM; ++j) {
          Real e = Real(0);
#pragma unroll
          for (int k = 0; k < NM; ++k) e += chinv[i * NM + k] * (Real(0.5) * (Mc[k * NM + j] + Mn[k * NM + j]));
          r += fabs(e);
        }
        rmax = fmax(rmax, r);
      }
      num += rmax;
    }
  return num;
}

// One warp per 32-cell row segment, grid-stride.  A segment whose code and whose
// neighbours' codes (x, y, z) name one pure phase needs no phi: h is 1 for that
// phase, the diffusion sum is that phase's constant.  codes: the state's segment
// codes, or NULL (every segment in full).  What bounds it is the FP64 conversions
// and sums: 256^3, 3 phases, FP32 on a GB300 take 321 us, 507 us when every
// stencil was read, with 64-bit cell indices.
template <int DIM, int NP, int NM, class Real>
__global__ void __launch_bounds__(kDiagThreads) k_diag(const Real* __restrict__ st, const uint8_t* __restrict__ codes,
                                                       const __grid_constant__ DiagGeom q, double tz0, double tzg,
                                                       double dt, double inv_dx2,
                                                       const __grid_constant__ DiagConsts<Real, NP, NM> c,
                                                       double* __restrict__ partials) {
  constexpr int NV = NM + 5;
  constexpr int WARPS = kDiagThreads / 32;
  __shared__ Real s_num[NP];   // diffusion sum inside each pure phase
  __shared__ double red[WARPS][NV];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  auto chi_of = [&](const Real* h, Real* chi) {
#pragma unroll
    for (int k = 0; k < NM * NM; ++k) {
      chi[k] = Real(0);
#pragma unroll
      for (int a = 0; a < NP; ++a) chi[k] += h[a] * c.chi[a][k];
    }
  };
  if (threadIdx.x < NP) {
    Real ph[NP], h[NP], chi[NM * NM], M[NM * NM];
#pragma unroll
    for (int a = 0; a < NP; ++a) ph[a] = a == (int)threadIdx.x ? Real(1) : Real(0);
    interp_h<NP>(ph, h);
    chi_of(h, chi);
    cell_mobility<NP, NM>(ph, c.DX, M);
    s_num[threadIdx.x] = diffusion_sum<DIM, NM, Real>(chi, M, [&](int, int, Real* Mn) {
#pragma unroll
      for (int k = 0; k < NM * NM; ++k) Mn[k] = M[k];
    });
  }
  __syncthreads();
  double acc[NV];
#pragma unroll
  for (int i = 0; i < NM; ++i) acc[i] = 0.0;
  acc[NM + 3] = 0.0;      // non-finite count
  DiagRun<Real> run;
  const long long plane = (long long)q.nyp * q.pitch;
  const unsigned int nseg = (unsigned int)q.segs * q.ny * q.nz;
  for (unsigned int w = blockIdx.x * WARPS + wid; w < nseg; w += gridDim.x * WARPS) {
    const unsigned int r = w / (unsigned int)q.segs;
    const int sg = (int)(w - r * q.segs), z = (int)(r / (unsigned int)q.ny), y = (int)(r - (unsigned int)z * q.ny);
    const int x = 32 * sg + lane;
    int l = 0;   // the pure phase + 1 of the segment and its neighbours, or 0
    if (codes) {
      int code = -1;
      if (lane < 1 + 2 * DIM) {
        const int d = (lane - 1) >> 1, o = lane == 0 ? 0 : (lane & 1 ? -1 : 1);
        const int zz = z + (lane && d == 2 ? o : 0);
        if (DIM == 3 && q.bc[2] == kBcHalo && (zz < 0 || zz >= q.nz))
          code = 0;
        else
          code = codes[((long long)(bc_map(zz, q.nz, q.bc[2]) + q.zoff) * q.ny +
                        bc_map(y + (lane && d == 1 ? o : 0), q.ny, q.bc[1])) * q.segs +
                       bc_map(sg + (lane && d == 0 ? o : 0), q.segs, q.bc[0])] & kCodePhase;
      }
      const int c0 = __shfl_sync(0xffffffffu, code, 0);
      l = __all_sync(0xffffffffu, code == -1 || code == c0) ? c0 : 0;
    }
    if (x >= q.nx) continue;
    const Real* p = st + (long long)(z + q.zoff) * plane + (long long)(y + 1) * q.pitch + x + q.xoff;
    Real ph[NP], mu[NM];
    bool finite = true;
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      ph[a] = l != 0 ? (a == l - 1 ? Real(1) : Real(0)) : p[a * q.fstride];
      finite = finite && isfinite(ph[a]);
      run.phase(ph[a]);
    }
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      mu[i] = p[(NP + i) * q.fstride];
      finite = finite && isfinite(mu[i]);
    }
    if (!finite) {
      acc[NM + 3] += 1.0;
      continue;
    }
    const Real s = (Real)(tz0 + tzg * ((DIM == 3 ? z : y) + q.zorg + 0.5));
    auto conc = [&](int a, int i) {
      Real ca = Real(0);
#pragma unroll
      for (int j = 0; j < NM; ++j) ca += c.chi[a][i * NM + j] * (mu[j] - (c.B0[a][j] + c.B1[a][j] * s));
      return ca;
    };
    if (l != 0) {
#pragma unroll
      for (int i = 0; i < NM; ++i) acc[i] += (double)conc(l - 1, i);
      run.diffusion(s_num[l - 1], dt, inv_dx2);
      continue;
    }
    run.template sum_dev<NP>(ph);
    Real h[NP];
    interp_h<NP>(ph, h);
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      Real ci = Real(0);
#pragma unroll
      for (int a = 0; a < NP; ++a) ci += h[a] * conc(a, i);
      acc[i] += (double)ci;
    }
    // explicit diffusion number of the mu update at this cell
    Real chi[NM * NM], Mc[NM * NM];
    chi_of(h, chi);
    cell_mobility<NP, NM>(ph, c.DX, Mc);
    run.diffusion(diffusion_sum<DIM, NM, Real>(chi, Mc,
                                               [&](int d, int sd, Real* Mn) {
                                                 const Real* n = p + (d == 0 ? sd : d == 1 ? sd * (long long)q.pitch : sd * plane);
                                                 Real pn[NP];
#pragma unroll
                                                 for (int a = 0; a < NP; ++a) pn[a] = n[a * q.fstride];
                                                 cell_mobility<NP, NM>(pn, c.DX, Mn);
                                               }),
                  dt, inv_dx2);
  }
  run.finish(dt, inv_dx2, acc, NM);
  // fixed shuffle tree per warp, then the warps in order
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    double t = acc[v];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double u = __shfl_down_sync(0xffffffffu, t, o);
      t = v < NM || v == NM + 3 ? t + u : v == NM + 1 ? fmin(t, u) : fmax(t, u);
    }
    if (lane == 0) red[wid][v] = t;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    const int v = threadIdx.x;
    double t = red[0][v];
    for (int k = 1; k < WARPS; ++k) {
      const double u = red[k][v];
      t = v < NM || v == NM + 3 ? t + u : v == NM + 1 ? fmin(t, u) : fmax(t, u);
    }
    partials[blockIdx.x * NV + v] = t;
  }
}

// One warp per value: lane l takes blocks l, l + 32, ... in order, then a fixed
// shuffle tree (7.3 us; one block-wide tree per value took 12.5 us).
template <int NM>
__global__ void __launch_bounds__(32 * (NM + 5)) k_diag_final(const double* __restrict__ partials, int nblocks,
                                                              double* __restrict__ out, int* status) {
  constexpr int NV = NM + 5;
  const int v = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool is_sum = v < NM || v == NM + 3, is_min = v == NM + 1;
  double r = is_sum ? 0.0 : (is_min ? 1e300 : -1e300);
  for (int b = lane; b < nblocks; b += 32) {
    const double o = partials[b * NV + v];
    r = is_sum ? r + o : (is_min ? fmin(r, o) : fmax(r, o));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double u = __shfl_down_sync(0xffffffffu, r, o);
    r = is_sum ? r + u : (is_min ? fmin(r, u) : fmax(r, u));
  }
  if (lane == 0) {
    out[v] = r;
    if (v == NM + 3 && r > 0.0) atomicOr(status, kStatusNonFinite);
  }
}

template <int DIM, int NP, int NM, class Real>
cudaError_t launch_diag(const void* state, const uint8_t* codes, const HostModel& m, double t, double* partials,
                        int nblocks, double* out, int* status, cudaStream_t st) {
  DiagConsts<Real, NP, NM> c;
  for (int a = 0; a < NP; ++a) {
    for (int k = 0; k < NM * NM; ++k) {
      c.chi[a][k] = (Real)m.chi[a][k];
      c.DX[a][k] = (Real)m.DX[a][k];
    }
    for (int i = 0; i < NM; ++i) {
      c.B0[a][i] = (Real)m.B0[a][i];
      c.B1[a][i] = (Real)m.B1[a][i];
    }
  }
  const double tz0 = m.T0 - m.T_ref - m.G * (m.z0 + m.V * t);
  DiagGeom q;
  q.nx = m.nx;
  q.ny = m.ny;
  q.nz = DIM == 3 ? m.nz : 1;
  q.pitch = m.pitch;
  q.nyp = m.nyp;
  q.xoff = m.xoff;
  q.zoff = m.zoff;
  q.zorg = m.zorg;
  q.segs = segments(m);
  for (int d = 0; d < 3; ++d) q.bc[d] = m.bc[d];
  q.fstride = m.fstride;
  // small grids: a warp per segment, no idle blocks to reduce over
  const long long nseg = (long long)q.segs * q.ny * q.nz, warps = kDiagThreads / 32;
  if (nseg > 0xFFFFFFF0ll) return cudaErrorInvalidValue;
  if ((nseg + warps - 1) / warps < nblocks) nblocks = (int)((nseg + warps - 1) / warps);
  k_diag<DIM, NP, NM, Real><<<nblocks, kDiagThreads, 0, st>>>(
      reinterpret_cast<const Real*>(state), codes, q, tz0, m.G * m.dx, m.dt, 1.0 / (m.dx * m.dx), c, partials);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_diag_final<NM><<<1, 32 * (NM + 5), 0, st>>>(partials, nblocks, out, status);
  return cudaGetLastError();
}

}  // namespace msgb
