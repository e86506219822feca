// Elasticity with a homogeneous stiffness (MICROSIM paper, arXiv 2404.01035,
// Sec. 2 "Elasticity implementation": the homogeneous case of its
// Fourier-space equilibrium).  The step needs w_b = -sigma : eps*^b of every
// phase b, sigma = C (eps - eps*), where the strain eps is in equilibrium with
// eps*(x) = sum_a eps*^a h_a(phi) (no homogeneous strain: zero at k = 0, and
// Nyquist wavenumbers taken as 0).
//
// The eigenstrains of the phases span few directions (one, when all grains
// share a dilatation): with a basis B^s of them, eps*^a = sum_s c_as B^s,
//   eps*(x)  = sum_s e_s(x) B^s,             e_s = sum_a c_as h_a
//   w_b      = -sum_s c_bs p_s(x),           p_s = B^s : sigma
//   p_s(k)   = sum_s' [ (P^s k) . G(k) (P^s' k) - B^s : C : B^s' ] e_s'(k),
// P^s = C : B^s, G = (C_ijkl k_j k_l)^-1, so the equilibrium takes rank
// transforms each way instead of one per strain component (6 in 3-D), and no
// pass over the cells after them.  Before a step:
//   1. k_el_eig:  e_s(x), the constant of its phase where a segment code says
//                 that the segment is pure
//   2. cuFFT R2C of the rank fields
//   3. k_el_spec: p_s(k) in place
//   4. cuFFT C2R: p_s(x), which the step reads where it needs them.
// What bounds it: memory passes.  7 grains with one dilatation, 128^3 FP32 on
// a GB300, without the step: 235 us with one transform per component and
// w_b stored per phase, 53 us here (k_el_eig 12.0, k_el_spec 11.2; 16 and 16
// with 64-bit index arithmetic and the stiffness contracted over all 81
// products per wavevector).
// cuFFT is opened at run time, so the library loads (and everything else runs)
// without it.
#include <cuda_runtime.h>
#include <cufft.h>
#include <dlfcn.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "ms_device.cuh"
#include "ms_rt.h"

namespace msgb {

// ------------------------------------------------------------------ cuFFT
namespace {

struct FftApi {
  decltype(&cufftCreate) create = nullptr;
  decltype(&cufftSetAutoAllocation) auto_allocation = nullptr;
  decltype(&cufftMakePlanMany) make_plan_many = nullptr;
  decltype(&cufftSetWorkArea) set_work_area = nullptr;
  decltype(&cufftSetStream) set_stream = nullptr;
  decltype(&cufftExecR2C) r2c = nullptr;
  decltype(&cufftExecC2R) c2r = nullptr;
  decltype(&cufftExecD2Z) d2z = nullptr;
  decltype(&cufftExecZ2D) z2d = nullptr;
  decltype(&cufftDestroy) destroy = nullptr;
  bool ok = false;
};

const FftApi& fft_api() {
  static FftApi api;
  static std::once_flag once;
  std::call_once(once, [] {
    const char* names[] = {"libcufft.so.12", "libcufft.so", "/usr/local/cuda/lib64/libcufft.so.12"};
    void* h = nullptr;
    for (const char* n : names)
      if ((h = dlopen(n, RTLD_NOW | RTLD_LOCAL)) != nullptr) break;
    if (!h) return;
    api.create = reinterpret_cast<decltype(api.create)>(dlsym(h, "cufftCreate"));
    api.auto_allocation = reinterpret_cast<decltype(api.auto_allocation)>(dlsym(h, "cufftSetAutoAllocation"));
    api.make_plan_many = reinterpret_cast<decltype(api.make_plan_many)>(dlsym(h, "cufftMakePlanMany"));
    api.set_work_area = reinterpret_cast<decltype(api.set_work_area)>(dlsym(h, "cufftSetWorkArea"));
    api.set_stream = reinterpret_cast<decltype(api.set_stream)>(dlsym(h, "cufftSetStream"));
    api.r2c = reinterpret_cast<decltype(api.r2c)>(dlsym(h, "cufftExecR2C"));
    api.c2r = reinterpret_cast<decltype(api.c2r)>(dlsym(h, "cufftExecC2R"));
    api.d2z = reinterpret_cast<decltype(api.d2z)>(dlsym(h, "cufftExecD2Z"));
    api.z2d = reinterpret_cast<decltype(api.z2d)>(dlsym(h, "cufftExecZ2D"));
    api.destroy = reinterpret_cast<decltype(api.destroy)>(dlsym(h, "cufftDestroy"));
    api.ok = api.create && api.auto_allocation && api.make_plan_many && api.set_work_area && api.set_stream && api.r2c &&
             api.c2r && api.d2z && api.z2d && api.destroy;
  });
  return api;
}

template <class Real>
struct ElConst {
  Real c[kNMax][kElRank];          // e_s = sum_a c_as h_a
  Real Pl[kElRank][3][3];          // B_ij C_ijkl
  Real Pr[kElRank][3][3];          // C_ijkl B_kl
  Real Q[kElRank][kElRank];        // B^s : C : B^s'
  Real D[3][3][6];                 // A_ik = C_ijkl k_j k_l over the products k_j k_l, j <= l
  Real kstep[3];                   // 2 pi / (n dx) per axis
  int rank, nx, ny, nz, nxh, pitch, nyp, xoff, zoff, segs;
  long long fstride, cells, ncplx;
};

// One warp per 32-cell row segment.
template <int DIM, int NP, class Real>
__global__ void __launch_bounds__(256) k_el_eig(const __grid_constant__ ElConst<Real> q, const Real* __restrict__ st,
                                                const uint8_t* __restrict__ codes, Real* __restrict__ E) {
  // (32-bit indices: elastic_grid_fits bounds the cells by 2^31)
  const unsigned w = blockIdx.x * 8u + (threadIdx.x >> 5), row = w / (unsigned)q.segs;
  const int lane = threadIdx.x & 31;
  const int sg = (int)(w - row * q.segs), z = (int)(row / (unsigned)q.ny), y = (int)(row - (unsigned)z * q.ny);
  if (z >= q.nz) return;
  const int x = 32 * sg + lane;
  if (x >= q.nx) return;
  const long long idx = ((long long)z * q.ny + y) * q.nx + x;
  const int code = codes[((long long)(z + q.zoff) * q.ny + y) * q.segs + sg] & kCodePhase;
  if (code != 0) {   // the segment is pure: h is 1 for that phase, 0 for the others
    for (int s = 0; s < q.rank; ++s) E[s * q.cells + idx] = q.c[code - 1][s];
    return;
  }
  const long long o = (long long)(DIM == 3 ? z + q.zoff : 0) * q.nyp * q.pitch + (long long)(y + 1) * q.pitch + x + q.xoff;
  Real ph[NP], h[NP];
#pragma unroll
  for (int a = 0; a < NP; ++a) ph[a] = st[a * q.fstride + o];
  interp_h<NP>(ph, h);
  for (int s = 0; s < q.rank; ++s) {
    Real e = Real(0);
#pragma unroll
    for (int a = 0; a < NP; ++a) e += h[a] * q.c[a][s];
    E[s * q.cells + idx] = e;
  }
}

template <class Real>
struct Cplx {
  Real re, im;
};

// Wavenumber of FFT index i of an extent n (the Nyquist index of an even n -> 0).
template <class Real>
__device__ __forceinline__ Real wavenumber(int i, int n, Real step) {
  if (2 * i == n) return Real(0);
  return step * Real(2 * i < n ? i : i - n);
}

// One thread per wavevector, all fields of it in place.
template <int DIM, int RANK, class Real>
__global__ void __launch_bounds__(256) k_el_spec(const __grid_constant__ ElConst<Real> q, Cplx<Real>* __restrict__ S) {
  const unsigned idx = blockIdx.x * 256u + threadIdx.x, row = idx / (unsigned)q.nxh;
  if (idx >= (unsigned long long)q.ncplx) return;
  const int mx = (int)(idx - row * q.nxh), mz = (int)(row / (unsigned)q.ny), my = (int)(row - (unsigned)mz * q.ny);
  Real k[3] = {wavenumber<Real>(mx, q.nx, q.kstep[0]), wavenumber<Real>(my, q.ny, q.kstep[1]),
               DIM == 3 ? wavenumber<Real>(mz, q.nz, q.kstep[2]) : Real(0)};
  Real k2 = Real(0);
#pragma unroll
  for (int d = 0; d < DIM; ++d) k2 += k[d] * k[d];
  Cplx<Real> e[RANK];
#pragma unroll
  for (int s = 0; s < RANK; ++s) e[s] = S[s * q.ncplx + idx];
  // v^s = Pr^s k and y^s = G v^s, G = A^-1 (adjugate over the determinant), A_ik = C_ijkl k_j k_l
  Real yv[RANK][DIM];
  if (k2 != Real(0)) {
    Real A[DIM][DIM], kk[DIM * (DIM + 1) / 2];
    int n = 0;
#pragma unroll
    for (int j = 0; j < DIM; ++j)
#pragma unroll
      for (int l = j; l < DIM; ++l) kk[n++] = k[j] * k[l];
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
      for (int j = 0; j < DIM; ++j) {
        Real a = Real(0);
#pragma unroll
        for (int p = 0; p < DIM * (DIM + 1) / 2; ++p) a += q.D[i][j][p] * kk[p];
        A[i][j] = a;
      }
    Real adj[DIM][DIM], det;
    if constexpr (DIM == 2) {
      det = A[0][0] * A[1][1] - A[0][1] * A[1][0];
      adj[0][0] = A[1][1];
      adj[0][1] = -A[0][1];
      adj[1][0] = -A[1][0];
      adj[1][1] = A[0][0];
    } else {
      adj[0][0] = A[1][1] * A[2][2] - A[1][2] * A[2][1];
      adj[1][0] = A[1][2] * A[2][0] - A[1][0] * A[2][2];
      adj[2][0] = A[1][0] * A[2][1] - A[1][1] * A[2][0];
      det = A[0][0] * adj[0][0] + A[0][1] * adj[1][0] + A[0][2] * adj[2][0];
      adj[0][1] = A[0][2] * A[2][1] - A[0][1] * A[2][2];
      adj[1][1] = A[0][0] * A[2][2] - A[0][2] * A[2][0];
      adj[2][1] = A[0][1] * A[2][0] - A[0][0] * A[2][1];
      adj[0][2] = A[0][1] * A[1][2] - A[0][2] * A[1][1];
      adj[1][2] = A[0][2] * A[1][0] - A[0][0] * A[1][2];
      adj[2][2] = A[0][0] * A[1][1] - A[0][1] * A[1][0];
    }
#pragma unroll
    for (int s = 0; s < RANK; ++s) {
      Real v[DIM];
#pragma unroll
      for (int i = 0; i < DIM; ++i) {
        v[i] = Real(0);
#pragma unroll
        for (int j = 0; j < DIM; ++j) v[i] += q.Pr[s][i][j] * k[j];
      }
#pragma unroll
      for (int i = 0; i < DIM; ++i) {
        Real t = Real(0);
#pragma unroll
        for (int j = 0; j < DIM; ++j) t += adj[i][j] * v[j];
        yv[s][i] = t / det;
      }
    }
  } else {
#pragma unroll
    for (int s = 0; s < RANK; ++s)
#pragma unroll
      for (int i = 0; i < DIM; ++i) yv[s][i] = Real(0);
  }
  const Real scale = Real(1) / Real(q.cells);   // the inverse transform is unnormalised
#pragma unroll
  for (int s = 0; s < RANK; ++s) {
    Real v[DIM];
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      v[i] = Real(0);
#pragma unroll
      for (int j = 0; j < DIM; ++j) v[i] += q.Pl[s][i][j] * k[j];
    }
    Real re = Real(0), im = Real(0);
#pragma unroll
    for (int t = 0; t < RANK; ++t) {
      Real K = -q.Q[s][t];
#pragma unroll
      for (int i = 0; i < DIM; ++i) K += v[i] * yv[t][i];
      re += K * e[t].re;
      im += K * e[t].im;
    }
    S[s * q.ncplx + idx] = Cplx<Real>{re * scale, im * scale};
  }
}

template <class Real>
ElConst<Real> make_const(const HostModel& m) {
  ElConst<Real> q{};
  const ElasticBasis eb = elastic_basis(m);
  q.rank = eb.rank;
  for (int a = 0; a < m.N; ++a)
    for (int s = 0; s < eb.rank; ++s) q.c[a][s] = (Real)eb.c[a][s];
  const int dim = m.dim;
  for (int i = 0; i < dim; ++i)
    for (int k = 0; k < dim; ++k) {
      int n = 0;
      for (int j = 0; j < dim; ++j)
        for (int l = j; l < dim; ++l)
          q.D[i][k][n++] = (Real)(j == l ? m.elC[i][j][k][j] : m.elC[i][j][k][l] + m.elC[i][l][k][j]);
    }
  for (int s = 0; s < eb.rank; ++s) {
    for (int k = 0; k < dim; ++k)
      for (int l = 0; l < dim; ++l) {
        double pl = 0.0, pr = 0.0;
        for (int i = 0; i < dim; ++i)
          for (int j = 0; j < dim; ++j) {
            pl += eb.B[s][i][j] * m.elC[i][j][k][l];
            pr += m.elC[k][l][i][j] * eb.B[s][i][j];
          }
        q.Pl[s][k][l] = (Real)pl;
        q.Pr[s][k][l] = (Real)pr;
      }
    for (int t = 0; t < eb.rank; ++t) {
      double v = 0.0;
      for (int i = 0; i < dim; ++i)
        for (int j = 0; j < dim; ++j)
          for (int k = 0; k < dim; ++k)
            for (int l = 0; l < dim; ++l) v += eb.B[s][i][j] * m.elC[i][j][k][l] * eb.B[t][k][l];
      q.Q[s][t] = (Real)v;
    }
  }
  const double two_pi = 6.28318530717958647692;
  q.kstep[0] = (Real)(two_pi / (m.nx * m.dx));
  q.kstep[1] = (Real)(two_pi / (m.ny * m.dx));
  q.kstep[2] = (Real)(two_pi / ((m.dim == 3 ? m.nz : 1) * m.dx));
  q.nx = m.nx;
  q.ny = m.ny;
  q.nz = m.dim == 3 ? m.nz : 1;
  q.nxh = m.nx / 2 + 1;
  q.pitch = m.pitch;
  q.nyp = m.nyp;
  q.xoff = m.xoff;
  q.zoff = m.zoff;
  q.segs = segments(m);
  q.fstride = m.fstride;
  q.cells = (long long)m.nx * m.ny * q.nz;
  q.ncplx = (long long)q.nxh * m.ny * q.nz;
  return q;
}

template <int DIM, class Real>
cudaError_t launch_eig(int np, const ElConst<Real>& q, const void* st, const uint8_t* codes, ElasticState& s,
                       cudaStream_t str) {
  const unsigned blocks = (unsigned)(((long long)q.segs * q.ny * q.nz * 32 + 255) / 256);
  const Real* p = static_cast<const Real*>(st);
  Real* E = static_cast<Real*>(s.E);
  switch (np) {
    case 2: k_el_eig<DIM, 2, Real><<<blocks, 256, 0, str>>>(q, p, codes, E); break;
    case 3: k_el_eig<DIM, 3, Real><<<blocks, 256, 0, str>>>(q, p, codes, E); break;
    case 8: k_el_eig<DIM, 8, Real><<<blocks, 256, 0, str>>>(q, p, codes, E); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <int DIM, class Real>
cudaError_t launch_spec(const ElConst<Real>& q, ElasticState& s, cudaStream_t str) {
  const unsigned blocks = (unsigned)((q.ncplx + 255) / 256);
  Cplx<Real>* S = static_cast<Cplx<Real>*>(s.spec);
  switch (q.rank) {
    case 1: k_el_spec<DIM, 1, Real><<<blocks, 256, 0, str>>>(q, S); break;
    case 2: k_el_spec<DIM, 2, Real><<<blocks, 256, 0, str>>>(q, S); break;
    case 3: k_el_spec<DIM, 3, Real><<<blocks, 256, 0, str>>>(q, S); break;
    case 4: k_el_spec<DIM, 4, Real><<<blocks, 256, 0, str>>>(q, S); break;
    case 5: k_el_spec<DIM, 5, Real><<<blocks, 256, 0, str>>>(q, S); break;
    case 6: k_el_spec<DIM, 6, Real><<<blocks, 256, 0, str>>>(q, S); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <class Real>
cudaError_t solve(const HostModel& m, const void* st, const uint8_t* codes, ElasticState& s, cudaStream_t str) {
  const FftApi& f = fft_api();
  const ElConst<Real> q = make_const<Real>(m);
  if (q.rank == 0) return cudaSuccess;   // no eigenstrain: no stress
  cudaError_t e = m.dim == 3 ? launch_eig<3, Real>(m.N, q, st, codes, s, str) : launch_eig<2, Real>(m.N, q, st, codes, s, str);
  if (e != cudaSuccess) return e;
  const bool dbl = sizeof(Real) == 8;
  cufftResult r = dbl ? f.d2z(s.plan_r2c, static_cast<cufftDoubleReal*>(s.E), static_cast<cufftDoubleComplex*>(s.spec))
                      : f.r2c(s.plan_r2c, static_cast<cufftReal*>(s.E), static_cast<cufftComplex*>(s.spec));
  if (r != CUFFT_SUCCESS) return cudaErrorUnknown;
  e = m.dim == 3 ? launch_spec<3, Real>(q, s, str) : launch_spec<2, Real>(q, s, str);
  if (e != cudaSuccess) return e;
  r = dbl ? f.z2d(s.plan_c2r, static_cast<cufftDoubleComplex*>(s.spec), static_cast<cufftDoubleReal*>(s.E))
          : f.c2r(s.plan_c2r, static_cast<cufftComplex*>(s.spec), static_cast<cufftReal*>(s.E));
  return r == CUFFT_SUCCESS ? cudaSuccess : cudaErrorUnknown;
}

}  // namespace

bool elastic_available() { return fft_api().ok; }

ElasticBasis elastic_basis(const HostModel& m) {
  // Gram-Schmidt with the largest remainder next; a remainder below 1e-12 of
  // the largest eigenstrain is rounding
  ElasticBasis b;
  double rem[kNMax][3][3] = {}, top = 0.0;
  auto norm2 = [&](const double (*t)[3]) {
    double s = 0.0;
    for (int i = 0; i < m.dim; ++i)
      for (int j = 0; j < m.dim; ++j) s += t[i][j] * t[i][j];
    return s;
  };
  for (int a = 0; a < m.N; ++a) {
    for (int i = 0; i < m.dim; ++i)
      for (int j = 0; j < m.dim; ++j) rem[a][i][j] = m.eig[a][std::max(i, j)][std::min(i, j)];   // symmetric
    top = std::max(top, norm2(rem[a]));
  }
  for (int a = 0; a < m.N; ++a)
    if (!std::isfinite(norm2(rem[a]))) {   // no comparison below holds: passed on, the state becomes non-finite
      b.rank = 1;
      b.B[0][0][0] = 1.0;
      for (int p = 0; p < m.N; ++p) b.c[p][0] = norm2(rem[a]);
      return b;
    }
  while (b.rank < kElRank) {
    int pick = 0;
    for (int a = 1; a < m.N; ++a)
      if (norm2(rem[a]) > norm2(rem[pick])) pick = a;
    const double n2 = norm2(rem[pick]);
    if (!(n2 > 1e-24 * top)) break;
    double (*B)[3] = b.B[b.rank];
    for (int i = 0; i < m.dim; ++i)
      for (int j = 0; j < m.dim; ++j) B[i][j] = rem[pick][i][j] / std::sqrt(n2);
    for (int a = 0; a < m.N; ++a) {
      double c = 0.0;
      for (int i = 0; i < m.dim; ++i)
        for (int j = 0; j < m.dim; ++j) c += rem[a][i][j] * B[i][j];
      b.c[a][b.rank] = c;
      for (int i = 0; i < m.dim; ++i)
        for (int j = 0; j < m.dim; ++j) rem[a][i][j] -= c * B[i][j];
    }
    ++b.rank;
  }
  return b;
}

namespace {
void release_state(ms_ctx* c, ElasticState& s) {
  const FftApi& f = fft_api();
  if (f.ok) {
    if (s.has_r2c) f.destroy(s.plan_r2c);
    if (s.has_c2r) f.destroy(s.plan_c2r);
  }
  dev_free(c->hook, s.E);
  dev_free(c->hook, s.spec);
  dev_free(c->hook, s.work);
  s = ElasticState{};
}
// The context's buffers and plans of another rank, once the stream is done with them.
void drop_state(ms_ctx* c) {
  if (c->el.E) cudaStreamSynchronize(c->stream);
  release_state(c, c->el);
}
}  // namespace

bool elastic_grid_fits(const HostModel& m) {
  // the batched plans take the per-transform distance (cells) as an int
  const long long cells = (long long)m.nx * m.ny * (m.dim == 3 ? m.nz : 1);
  return cells <= 0x7FFFFFFFll;
}

ms_status elastic_setup(ms_ctx* c) {
  const HostModel& m = c->m;
  // the step kernels read the elastic fields only while elasticity is on
  // (ms_update_params may turn it on or off, or change the eigenstrains' rank)
  const int rank_now = m.el ? elastic_basis(m).rank : 0;
  c->lg.elw = m.el && c->el.ready && c->el.rank == rank_now ? c->el.E : nullptr;
  if (!m.el || (c->el.ready && c->el.rank == rank_now)) return MS_OK;
  const FftApi& f = fft_api();
  if (!f.ok) return fail(c, MS_ERR_UNSUPPORTED, "elasticity needs cuFFT (libcufft.so.12), which could not be opened");
  if (m.N != 2 && m.N != 3 && m.N != 8) return fail(c, MS_ERR_UNSUPPORTED, "elasticity: phases must be 2, 3 or 8");
  if (!elastic_grid_fits(m)) return fail(c, MS_ERR_UNSUPPORTED, "grid too large for the FFT plans of the elasticity");
  // everything is built in a local state and handed to the context only when
  // every buffer and both plans exist; a failure part-way frees what was made
  ElasticState s;
  s.rank = rank_now;
  if (rank_now == 0) {   // no eigenstrain in the plane of the grid: nothing to transform
    s.ready = true;
    drop_state(c);
    c->el = s;
    return MS_OK;
  }
  const int nz = m.dim == 3 ? m.nz : 1;
  const long long cells = (long long)m.nx * m.ny * nz;
  const long long ncplx = (long long)(m.nx / 2 + 1) * m.ny * nz;
  const size_t real = m.dtype == MS_F64 ? 8 : 4;
  s.E = alloc_with_room(c, s.rank * cells * real);
  s.spec = alloc_with_room(c, s.rank * ncplx * 2 * real);
  if (!s.E || !s.spec) {
    release_state(c, s);
    return fail(c, MS_ERR_OOM, "elasticity buffers");
  }
  int n3[3] = {nz, m.ny, m.nx};
  int* n = m.dim == 3 ? n3 : n3 + 1;
  const int rank = m.dim;
  const int idist = (int)cells, odist = (int)ncplx;
  int inr[3] = {nz, m.ny, m.nx}, onr[3] = {nz, m.ny, m.nx / 2 + 1};
  int* inb = m.dim == 3 ? inr : inr + 1;
  int* onb = m.dim == 3 ? onr : onr + 1;
  const bool dbl = m.dtype == MS_F64;
  // the plans' work area (one: they run one after the other) comes from the
  // context's allocator like the rest, and can have a split step's scratch for room
  cufftHandle p1 = 0, p2 = 0;
  size_t w1 = 0, w2 = 0;
  bool ok = f.create(&p1) == CUFFT_SUCCESS;
  s.plan_r2c = p1;
  s.has_r2c = ok;
  ok = ok && f.auto_allocation(p1, 0) == CUFFT_SUCCESS &&
       f.make_plan_many(p1, rank, n, inb, 1, idist, onb, 1, odist, dbl ? CUFFT_D2Z : CUFFT_R2C, s.rank, &w1) ==
           CUFFT_SUCCESS &&
       f.create(&p2) == CUFFT_SUCCESS;
  s.plan_c2r = p2;
  s.has_c2r = ok;
  ok = ok && f.auto_allocation(p2, 0) == CUFFT_SUCCESS &&
       f.make_plan_many(p2, rank, n, onb, 1, odist, inb, 1, idist, dbl ? CUFFT_Z2D : CUFFT_C2R, s.rank, &w2) ==
           CUFFT_SUCCESS;
  if (!ok) {
    release_state(c, s);
    return fail(c, MS_ERR_CUDA, "cuFFT plan creation failed");
  }
  const size_t work = std::max(w1, w2);
  if (work > 0 && !(s.work = alloc_with_room(c, work))) {
    release_state(c, s);
    return fail(c, MS_ERR_OOM, "cuFFT work area");
  }
  if (work > 0 && (f.set_work_area(p1, s.work) != CUFFT_SUCCESS || f.set_work_area(p2, s.work) != CUFFT_SUCCESS)) {
    release_state(c, s);
    return fail(c, MS_ERR_CUDA, "cuFFT work area");
  }
  if (f.set_stream(p1, c->stream) != CUFFT_SUCCESS || f.set_stream(p2, c->stream) != CUFFT_SUCCESS) {
    release_state(c, s);
    return fail(c, MS_ERR_CUDA, "cuFFT stream");
  }
  s.ready = true;
  drop_state(c);
  c->el = s;
  c->lg.elw = s.E;
  return MS_OK;
}

ms_status elastic_solve(ms_ctx* c, const void* state, const uint8_t* codes) {
  cudaError_t e = c->m.dtype == MS_F64 ? solve<double>(c->m, state, codes, c->el, c->stream)
                                       : solve<float>(c->m, state, codes, c->el, c->stream);
  if (e != cudaSuccess) return cuda_fail(c, e, "elastic equilibrium");
  return MS_OK;
}

void elastic_free(ms_ctx* c) { release_state(c, c->el); }

}  // namespace msgb
