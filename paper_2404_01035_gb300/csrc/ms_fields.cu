// Device-resident fields in and out of a context: dense [f][z][y][x] arrays
// against the padded state, one pass over memory each way.
//
// Loading writes the interior, every ghost image and the segment codes from
// one read of the fields.  What bounds it is DRAM: 512^3 with 9 FP32 fields (9.7
// GB moved) on a GB300 loads in 1.59 ms and unloads in 1.42 ms (6.8 TB/s); one
// strided copy per field (2.4 TB/s), a ghost pass per axis and a code pass took
// 5.3 ms, the copies back 4.0 ms.  A warp takes one row piece of every field, 16 bytes per
// lane where rows allow it (extent a multiple of the vector, aligned pointers),
// else one element per lane.
#include <cuda_runtime.h>
#include <stdint.h>

#include "ms_pointer.h"
#include "ms_rt.h"

namespace msgb {
namespace {

struct FieldGeom {
  int nx, ny, nz, n_phi, n_mu, pitch, nyp, xoff, zoff, segs, pieces, three_d;
  int bc[3];
  long long fstride, cells;
};

template <class Real, int VEC>
struct alignas(sizeof(Real) * VEC) Vec {
  Real v[VEC];
};

constexpr int kBatch = 4;   // fields in flight per lane

template <class Real, int VEC>
__global__ void __launch_bounds__(256) k_load_fields(const __grid_constant__ FieldGeom q, const Real* __restrict__ phi,
                                                     const Real* __restrict__ mu, Real* __restrict__ out,
                                                     uint8_t* __restrict__ codes) {
  using V = Vec<Real, VEC>;
  const unsigned int w = blockIdx.x * 8u + (threadIdx.x >> 5);   // (warps: threads would pass 2^32 with the grid)
  const int lane = threadIdx.x & 31;
  if (w >= (unsigned int)q.pieces * q.ny * q.nz) return;
  const unsigned int r = w / (unsigned int)q.pieces;
  const int z = (int)(r / (unsigned int)q.ny), y = (int)(r - (unsigned int)z * q.ny);
  const int x = ((int)(w - r * q.pieces) * 32 + lane) * VEC;
  const bool have = x < q.nx;
  const long long plane = (long long)q.nyp * q.pitch;
  const long long d0 = ((long long)z * q.ny + y) * q.nx + x;
  const long long p0 = (long long)(z + q.zoff) * plane + (long long)(y + 1) * q.pitch + x + q.xoff;
  // ghost images of the row's ends, and of the whole row on y / z boundaries
  const long long xl = x == 0 ? (q.bc[0] == 3 ? q.nx : -1) : 0;                                  // image of the first cell
  const long long xr = x + VEC == q.nx ? VEC - 1 + (q.bc[0] == 3 ? -q.nx : 1) : 0;               // of the last
  const bool have_xr = x + VEC == q.nx;
  long long oy[3] = {0, 0, 0}, oz[3] = {0, 0, 0};
  bool hy[3] = {true, y == 0, y == q.ny - 1}, hz[3] = {true, false, false};
  if (hy[1]) oy[1] = (long long)(q.bc[1] == 3 ? q.ny : -1) * q.pitch;
  if (hy[2]) oy[2] = (long long)(q.bc[1] == 3 ? -q.ny : 1) * q.pitch;
  if (q.three_d && q.bc[2] != kBcHalo) {   // internal cuts get their ghosts from the exchange
    hz[1] = z == 0;
    hz[2] = z == q.nz - 1;
    if (hz[1]) oz[1] = (long long)(q.bc[2] == 3 ? q.nz : -1) * plane;
    if (hz[2]) oz[2] = (long long)(q.bc[2] == 3 ? -q.nz : 1) * plane;
  }
  const bool edge = hy[1] || hy[2] || hz[1] || hz[2];
  uint32_t nz_[VEC], one[VEC];
#pragma unroll
  for (int k = 0; k < VEC; ++k) nz_[k] = one[k] = 0;
  const int nf = q.n_phi + q.n_mu;
  auto put = [&](Real* p, const V& v) {
    *reinterpret_cast<V*>(p) = v;
    if (x == 0) p[xl] = v.v[0];
    if (have_xr) p[xr] = v.v[VEC - 1];
  };
  for (int f0 = 0; f0 < nf; f0 += kBatch) {
    V b[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int f = f0 + u;
      if (have && f < nf) {
        const Real* s = f < q.n_phi ? phi + f * q.cells : mu + (f - q.n_phi) * q.cells;
        b[u] = *reinterpret_cast<const V*>(s + d0);
      }
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int f = f0 + u;
      if (!have || f >= nf) continue;
      Real* p = out + f * q.fstride + p0;
      put(p, b[u]);
      if (f < q.n_phi) {
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
          nz_[k] |= (b[u].v[k] != Real(0) ? 1u : 0u) << f;
          one[k] |= (b[u].v[k] == Real(1) ? 1u : 0u) << f;
        }
      }
      if (edge) {
#pragma unroll
        for (int iz = 0; iz < 3; ++iz)
#pragma unroll
          for (int iy = 0; iy < 3; ++iy)
            if ((iy | iz) != 0 && hy[iy] && hz[iz]) put(p + oy[iy] + oz[iz], b[u]);
      }
    }
  }
  if (!codes) return;
  // a segment's code: the pure phase + 1 that all its cells hold, else 0
  int code = -1;
  if (have) {
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
      const int c = (__popc(nz_[k]) == 1 && nz_[k] == one[k]) ? __ffs(nz_[k]) : 0;
      code = (code == -1 || code == c) ? c : 0;
    }
  }
  constexpr int LPS = 32 / VEC;   // lanes per segment
  const int first = lane / LPS * LPS;
  const int ref = __shfl_sync(0xffffffffu, code, first);
  const uint32_t same = __ballot_sync(0xffffffffu, !have || code == ref);
  const uint32_t mask = (LPS == 32 ? 0xffffffffu : ((1u << (LPS & 31)) - 1u)) << first;
  if (lane == first && have)
    codes[((long long)(z + q.zoff) * q.ny + y) * q.segs + (x >> 5)] = (same & mask) == mask ? (uint8_t)ref : (uint8_t)0;
}

template <class Real, int VEC>
__global__ void __launch_bounds__(256) k_unload_fields(const __grid_constant__ FieldGeom q, const Real* __restrict__ in,
                                                       Real* __restrict__ phi, Real* __restrict__ mu) {
  using V = Vec<Real, VEC>;
  const unsigned int w = blockIdx.x * 8u + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= (unsigned int)q.pieces * q.ny * q.nz) return;
  const unsigned int r = w / (unsigned int)q.pieces;
  const int z = (int)(r / (unsigned int)q.ny), y = (int)(r - (unsigned int)z * q.ny);
  const int x = ((int)(w - r * q.pieces) * 32 + lane) * VEC;
  if (x >= q.nx) return;
  const long long d0 = ((long long)z * q.ny + y) * q.nx + x;
  const long long p0 =
      (long long)(z + q.zoff) * q.nyp * q.pitch + (long long)(y + 1) * q.pitch + x + q.xoff;
  const int nf = q.n_phi + q.n_mu;
  for (int f0 = 0; f0 < nf; f0 += kBatch) {
    V b[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
      if (f0 + u < nf && (f0 + u >= q.n_phi || phi)) b[u] = *reinterpret_cast<const V*>(in + (f0 + u) * q.fstride + p0);
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int f = f0 + u;
      if (f >= nf) continue;
      Real* d = f < q.n_phi ? phi : mu;
      if (d) *reinterpret_cast<V*>(d + (f < q.n_phi ? f : f - q.n_phi) * q.cells + d0) = b[u];
    }
  }
}

FieldGeom geom(const HostModel& m, int vec) {
  FieldGeom q = {};
  q.nx = m.nx;
  q.ny = m.ny;
  q.nz = m.nz;
  q.n_phi = m.N;
  q.n_mu = m.NM;
  q.pitch = m.pitch;
  q.nyp = m.nyp;
  q.xoff = m.xoff;
  q.zoff = m.zoff;
  q.segs = segments(m);
  q.pieces = (m.nx + 32 * vec - 1) / (32 * vec);
  q.three_d = m.dim == 3;
  for (int d = 0; d < 3; ++d) q.bc[d] = m.bc[d];
  q.fstride = m.fstride;
  q.cells = (long long)m.nx * m.ny * m.nz;
  return q;
}

bool aligned(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

template <class Real>
cudaError_t load(const HostModel& m, void* padded, const void* phi, const void* mu, uint8_t* codes, cudaStream_t st) {
  constexpr int VEC = 16 / (int)sizeof(Real);
  const bool vec = m.nx % VEC == 0 && aligned(phi) && aligned(mu) && aligned(padded);
  const FieldGeom q = geom(m, vec ? VEC : 1);
  const unsigned blocks = (unsigned)(((long long)q.pieces * q.ny * q.nz + 7) / 8);
  const Real *a = static_cast<const Real*>(phi), *b = static_cast<const Real*>(mu);
  if (vec)
    k_load_fields<Real, VEC><<<blocks, 256, 0, st>>>(q, a, b, static_cast<Real*>(padded), codes);
  else
    k_load_fields<Real, 1><<<blocks, 256, 0, st>>>(q, a, b, static_cast<Real*>(padded), codes);
  return cudaGetLastError();
}

template <class Real>
cudaError_t unload(const HostModel& m, const void* padded, void* phi, void* mu, cudaStream_t st) {
  constexpr int VEC = 16 / (int)sizeof(Real);
  const bool vec = m.nx % VEC == 0 && aligned(phi) && aligned(mu) && aligned(padded);
  FieldGeom q = geom(m, vec ? VEC : 1);
  const Real* in = static_cast<const Real*>(padded);
  if (!mu) q.n_mu = 0;
  const unsigned blocks = (unsigned)(((long long)q.pieces * q.ny * q.nz + 7) / 8);
  if (vec)
    k_unload_fields<Real, VEC><<<blocks, 256, 0, st>>>(q, in, static_cast<Real*>(phi), static_cast<Real*>(mu));
  else
    k_unload_fields<Real, 1><<<blocks, 256, 0, st>>>(q, in, static_cast<Real*>(phi), static_cast<Real*>(mu));
  return cudaGetLastError();
}

static_assert((int)cudaMemoryTypeDevice == kMemDevice && (int)cudaMemoryTypeManaged == kMemManaged, "ms_pointer.h");

}  // namespace

// Row pieces are counted with 32 bits.
bool field_kernels_fit(const HostModel& m) {
  return (long long)((m.nx + 31) / 32) * m.ny * m.nz < 0x7FFFFFF0ll;
}

bool field_kernel_reaches(const void* p) {
  if (!p) return true;
  cudaPointerAttributes a;
  int here = 0;
  if (cudaGetDevice(&here) != cudaSuccess || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return kernel_reaches((int)a.type, a.device, here);
}

cudaError_t load_fields(const HostModel& m, void* padded, const void* phi, const void* mu, uint8_t* codes,
                        cudaStream_t st) {
  return m.dtype == 1 ? load<double>(m, padded, phi, mu, codes, st) : load<float>(m, padded, phi, mu, codes, st);
}

cudaError_t unload_fields(const HostModel& m, const void* padded, void* phi, void* mu, cudaStream_t st) {
  return m.dtype == 1 ? unload<double>(m, padded, phi, mu, st) : unload<float>(m, padded, phi, mu, st);
}

}  // namespace msgb
