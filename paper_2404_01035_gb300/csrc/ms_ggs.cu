// Sparse grain growth: many grains (up to 64), each cell storing only the
// grains non-zero there (MICROSIM paper, arXiv 2404.01035, Sec. 4
// "Grain-growth": the phi equation of Sec. 2.1 without the chemical driving
// force; isotropic boundary energies, multi-obstacle potential with the
// triple term Gamma_abc).
//
// Reading (locally active phases): the Lagrange multiplier acts on the grains
// present at the cell or at one of its face neighbours -- the projection onto
// the simplex runs over them alone and every other grain stays 0 -- so a grain
// can only appear next to where it already is, and a cell holds few grains.
// With isotropic pairs (g = 2 gamma q) the update of a cell reads only its
// 7-point stencil (face fluxes need the normal differences alone).
//
// State per buffer: for every cell the number of stored grains, up to kSlots
// (grain index, value) pairs sorted by grain index (slot-major arrays), and a
// code byte (grain + 1 when the cell is that grain alone with value 1, else 0).
// One step = two launches:
//   k_ggs_classify: a cell whose 7 codes name one grain keeps it (written only
//     when the destination buffer, which holds the state one step back, does
//     not already hold it); the others are appended to a work list (one atomic
//     per 1024 cells).
//   k_ggs_update: grid-stride over the list (a build for unions of up to 4
//     grains, which defers larger ones to a second list and build); the grains
//     of the 7 stencil cells (a 64-bit union mask), their values, the face
//     fluxes, centre term, potential derivative and rate over that union in
//     increasing grain order (the order of the dense sums, whose other terms
//     are exact zeros), the projection over the union, and the non-zero results
//     stored.
// A cell that would need more than kSlots grains (or a stencil union above
// kUnion) sets the sticky status MS_ERR_BOUNDS instead of losing a grain.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/microsim_gb.h"
#include "ms_device.cuh"
#include "ms_rt.h"
#include "ms_trace.h"

namespace msgb {
ms_status build_model(ms_ctx* c, const ms_grid* g, int N, int K, const ms_params* p, HostModel& m);
}

using namespace msgb;

namespace {

constexpr int kSlots = 8;        // grains stored per cell
constexpr int kUnion = 8;        // grains in a 7-point stencil at most
constexpr int kUnionSmall = 4;   // the union size of the first update build
constexpr int kMaxGrains = 64;   // union masks are 64-bit
constexpr int kStatusOverflow = 8;

template <class Real>
struct GgsArgs {
  int nx, ny, nz, dim, N;
  int bc[3];
  long long cells;
  Real dt, eps, inv_eps, mob, inv_dx, half_inv_dx, g3;
  int has_g3;
  const Real* gam2;   // [N][N] 2 gamma_ab
  const Real* cw;     // [N][N] 16 gamma_ab / pi^2
  Real gam2_0, cw_0;  // their value when one gamma holds for every pair
  // input / output state
  const uint8_t* cnt_in;
  const uint8_t* code_in;
  const uint8_t* idx_in;   // [kSlots][cells]
  const Real* val_in;      // [kSlots][cells]
  uint8_t* cnt_out;
  uint8_t* code_out;
  uint8_t* idx_out;
  Real* val_out;
  unsigned int* list;      // [0] count, [1..] cell indices
  unsigned int* list2;     // the cells whose stencil holds more than kUnionSmall grains
  unsigned int list_cap;
  int* status;             // [0] sticky status, [1] cells listed by the last step, [2] exit ticket
};

__device__ __forceinline__ int wrap_axis(int i, int n, int bc) {
  if (i >= 0 && i < n) return i;
  if (bc == 3) return i < 0 ? i + n : i - n;
  return i < 0 ? 0 : n - 1;   // no-flux: mirror ghost = adjacent interior cell
}

// Linear index of the cell at (x, y, z) + unit step s along axis d (boundary
// mapped; grids hold fewer than 2^32 cells, and 32-bit index arithmetic is
// suffices).
template <class Real>
__device__ __forceinline__ unsigned int nb_index(const GgsArgs<Real>& g, int x, int y, int z, int d, int s) {
  if (d == 0) x = wrap_axis(x + s, g.nx, g.bc[0]);
  if (d == 1) y = wrap_axis(y + s, g.ny, g.bc[1]);
  if (d == 2) z = wrap_axis(z + s, g.nz, g.bc[2]);
  return ((unsigned int)z * (unsigned int)g.ny + (unsigned int)y) * (unsigned int)g.nx + (unsigned int)x;
}
template <class Real>
__device__ __forceinline__ void cell_of(const GgsArgs<Real>& g, unsigned int i, int& x, int& y, int& z) {
  const unsigned int r = i / (unsigned int)g.nx;
  x = (int)(i - r * (unsigned int)g.nx);
  z = (int)(r / (unsigned int)g.ny);
  y = (int)(r - (unsigned int)z * (unsigned int)g.ny);
}

// Each block takes 1024 consecutive cells and its places in the list with one
// atomic (one per warp serialised on the counter: 37 us at 128^3 on a GB300).
constexpr int kClassifyRounds = 4;
template <class Real>
__global__ void __launch_bounds__(256) k_ggs_classify(const __grid_constant__ GgsArgs<Real> g) {
  __shared__ unsigned int s_place[8 * kClassifyRounds + 1];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long long first = blockIdx.x * (256ll * kClassifyRounds) + threadIdx.x;
  unsigned int need[kClassifyRounds];
#pragma unroll
  for (int rnd = 0; rnd < kClassifyRounds; ++rnd) {
    const long long li = first + 256 * rnd;
    const unsigned int i = (unsigned int)li;
    bool listed = false;
    if (li < g.cells) {
      int x, y, z;
      cell_of(g, i, x, y, z);
      const uint8_t c0 = g.code_in[i];
      bool bulk = c0 != 0;
      if (bulk) {
        // (every neighbour's code at once: the loads are in flight together)
        uint8_t nb[6];
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
          for (int s = 0; s < 2; ++s) nb[2 * d + s] = d < g.dim ? g.code_in[nb_index(g, x, y, z, d, s ? 1 : -1)] : c0;
#pragma unroll
        for (int k = 0; k < 6; ++k) bulk = bulk && nb[k] == c0;
      }
      if (bulk) {
        // the destination holds the state one step back: rewrite only when it differs
        if (g.code_out[i] != c0 || g.cnt_out[i] != 1) {
          g.cnt_out[i] = 1;
          g.idx_out[i] = (uint8_t)(c0 - 1);
          g.val_out[i] = Real(1);
          g.code_out[i] = c0;
        }
      } else {
        listed = true;
      }
    }
    need[rnd] = __ballot_sync(0xffffffffu, listed);
    if (lane == 0) s_place[rnd * 8 + wid] = __popc(need[rnd]);
  }
  __syncthreads();
  if (wid == 0) {   // exclusive sums of the 32 warp counts, in cell order
    const unsigned int c = s_place[lane];
    unsigned int t = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int u = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += u;
    }
    s_place[lane] = t - c;
    if (lane == 31) s_place[32] = t ? atomicAdd(&g.list[0], t) : 0u;
  }
  __syncthreads();
#pragma unroll
  for (int rnd = 0; rnd < kClassifyRounds; ++rnd)
    if ((need[rnd] >> lane) & 1u) {
      const unsigned int k = s_place[32] + s_place[rnd * 8 + wid] + __popc(need[rnd] & ((1u << lane) - 1u));
      if (k < g.list_cap) g.list[1 + k] = (unsigned int)(first + 256 * rnd);
    }
}
static_assert(8 * kClassifyRounds == 32, "one warp sums the counts");

// The same for rows of a multiple of 4 cells, 4 consecutive cells of a row per
// thread: the codes of a cell's six neighbours are compared four at a time (at
// 128^3 on a GB300: 7.8 us against 17 for a cell per thread and round).
template <class Real>
__global__ void __launch_bounds__(256) k_ggs_classify4(const __grid_constant__ GgsArgs<Real> g) {
  __shared__ unsigned int s_place[9];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long long first = blockIdx.x * 1024ll + 4 * threadIdx.x;
  unsigned int listed = 0u;   // by bit
  if (first < g.cells) {
    const unsigned int i = (unsigned int)first;
    int x, y, z;
    cell_of(g, i, x, y, z);
    auto word = [&](const uint8_t* p, unsigned int at) { return *reinterpret_cast<const unsigned int*>(p + at); };
    const unsigned int c = word(g.code_in, i);
    const unsigned int left = g.code_in[nb_index(g, x, y, z, 0, -1)], right = g.code_in[nb_index(g, x + 3, y, z, 0, 1)];
    const unsigned int ym = word(g.code_in, nb_index(g, x, y, z, 1, -1)), yp = word(g.code_in, nb_index(g, x, y, z, 1, 1));
    unsigned int zm = c, zp = c;
    if (g.dim == 3) {
      zm = word(g.code_in, nb_index(g, x, y, z, 2, -1));
      zp = word(g.code_in, nb_index(g, x, y, z, 2, 1));
    }
    const unsigned int co = word(g.code_out, i), no = word(g.cnt_out, i);
    const unsigned int bulk = __vcmpeq4(c, (c << 8) | left) & __vcmpeq4(c, (c >> 8) | (right << 24)) & __vcmpeq4(c, ym) &
                              __vcmpeq4(c, yp) & __vcmpeq4(c, zm) & __vcmpeq4(c, zp) & ~__vcmpeq4(c, 0u);
    // the destination holds the state one step back: rewrite only what differs
    const unsigned int stale = bulk & ~(__vcmpeq4(c, co) & __vcmpeq4(no, 0x01010101u));
    if (stale) {
      for (int k = 0; k < 4; ++k) {
        if (!((stale >> (8 * k)) & 1u)) continue;
        const uint8_t ck = (uint8_t)(c >> (8 * k));
        g.cnt_out[i + k] = 1;
        g.idx_out[i + k] = (uint8_t)(ck - 1);
        g.val_out[i + k] = Real(1);
        g.code_out[i + k] = ck;
      }
    }
    const unsigned int l = ~bulk & 0x01010101u;
    listed = (l | (l >> 7) | (l >> 14) | (l >> 21)) & 15u;
  }
  const unsigned int mine = __popc(listed);
  unsigned int t = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int u = __shfl_up_sync(0xffffffffu, t, o);
    if (lane >= o) t += u;
  }
  if (lane == 31) s_place[wid] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int sum = 0u;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      const unsigned int n = s_place[w];
      s_place[w] = sum;
      sum += n;
    }
    s_place[8] = sum ? atomicAdd(&g.list[0], sum) : 0u;
  }
  __syncthreads();
  unsigned int at = s_place[8] + s_place[wid] + t - mine;
  for (unsigned int m = listed; m; m &= m - 1u, ++at)
    if (at < g.list_cap) g.list[1 + at] = (unsigned int)first + __ffs(m) - 1;
}

// Simplex projection (Held-Wolfe-Crowder 1974; Duchi et al. 2008) of the
// first n <= kUnion values: the threshold theta (phi = max(v - theta, 0)).
template <class Real, int K>
__device__ __forceinline__ Real simplex_theta(const Real* v, int n) {
  Real u[K];
#pragma unroll
  for (int a = 0; a < K; ++a) u[a] = a < n ? v[a] : Real(-INFINITY);
  // descending, by Batcher's odd-even merge network (5 and 19 exchanges)
  auto order = [&](int i, int j) {
    if (u[j] > u[i]) {
      const Real t = u[j];
      u[j] = u[i];
      u[i] = t;
    }
  };
  static_assert(K == 2 || K == 4 || K == 8, "networks of 2, 4 and 8");
  if constexpr (K == 2) order(0, 1);
#pragma unroll
  for (int h = 0; h + 4 <= K; h += 4) {
    order(h, h + 1), order(h + 2, h + 3);
    order(h, h + 2), order(h + 1, h + 3);
    order(h + 1, h + 2);
  }
  if constexpr (K == 8) {
    order(0, 4), order(1, 5), order(2, 6), order(3, 7);
    order(2, 4), order(3, 5);
    order(1, 2), order(3, 4), order(5, 6);
  }
  Real csum = Real(0), theta = Real(0);
#pragma unroll
  for (int j = 0; j < K; ++j) {
    if (j >= n) break;
    csum += u[j];
    const Real t = (csum - Real(1)) * Real(1.0 / (j + 1));
    if (u[j] - t > Real(0)) theta = t;
  }
  return theta;
}

// Threads per block of the update kernel: its shared memory holds 7 x KU
// values per thread.
template <class Real, int KU>
struct UpdShape {
  static constexpr int THREADS = sizeof(Real) * KU > 16 ? 64 : 128;
  static constexpr int MIN_BLOCKS = 8;   // registers for 16 / 32 warps per SM
};

// Projection of the values v of the union's grains over the union, and the cell's
// new slots.
template <class Real, int K>
__device__ __forceinline__ void store_union(const GgsArgs<Real>& g, unsigned int i, const Real* v, const int* uid, int nu) {
  // projection over the locally active grains (the union)
  const Real theta = simplex_theta<Real, K>(v, nu);
  int n_out = 0;
  uint8_t code = 0;
#pragma unroll
  for (int a = 0; a < K; ++a) {
    if (a >= nu) break;
    const Real dd = v[a] - theta;
    const Real pn = dd > Real(0) ? dd : Real(0);
    if (pn > Real(0)) {
      if (n_out < kSlots) {
        g.idx_out[(size_t)n_out * g.cells + i] = (uint8_t)uid[a];
        g.val_out[(size_t)n_out * g.cells + i] = pn;
        if (pn == Real(1)) code = (uint8_t)(uid[a] + 1);
      }
      ++n_out;
    }
  }
  if (n_out > kSlots) {
    atomicOr(g.status, kStatusOverflow);
    n_out = kSlots;
  }
  g.cnt_out[i] = (uint8_t)n_out;
  g.code_out[i] = n_out == 1 ? code : 0;
}

// One gamma: the update of cell i, whose stencil (cells ci, their first PRE slots
// in pidx / pval, cntc stored) holds the nu <= K grains uid.
template <class Real, int K, int PRE>
__device__ __forceinline__ void update_uniform(const GgsArgs<Real>& g, unsigned int i, const unsigned int* ci,
                                               const int* cntc, const int (*pidx)[PRE], const Real (*pval)[PRE],
                                               const int* uid, int nu, int most) {
  Real v[K];
  // a stencil cell's values of the union's grains
  auto gather = [&](int c, Real* out) {
#pragma unroll
    for (int u = 0; u < K; ++u) {
      Real r = Real(0);
#pragma unroll
      for (int k = 0; k < PRE; ++k) r = pidx[c][k] == uid[u] ? pval[c][k] : r;
      out[u] = u < nu ? r : Real(0);
    }
    for (int k = PRE; k < most; ++k) {
      if (k >= cntc[c]) continue;
      const int a = g.idx_in[(size_t)k * g.cells + ci[c]];
      const Real r = g.val_in[(size_t)k * g.cells + ci[c]];
#pragma unroll
      for (int u = 0; u < K; ++u) out[u] = u < nu && a == uid[u] ? r : out[u];
    }
  };
  Real ph[K], dg[K];
  Real e1 = Real(0), e2 = Real(0), C2 = Real(0);
  gather(0, ph);
#pragma unroll
  for (int a = 0; a < K; ++a) {
    dg[a] = Real(0);
    e2 += ph[a] * e1;
    e1 += ph[a];
    C2 += ph[a] * ph[a];
  }
  const Real kf = g.gam2_0 * g.inv_dx * g.inv_dx;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (d >= g.dim) continue;
    Real w[K], u[K];   // differences to the two neighbours (see k_ggs_update)
    gather(1 + 2 * d, w);
    gather(2 + 2 * d, u);
    Real S = Real(0), Xw = Real(0), Xu = Real(0), Y = Real(0);
#pragma unroll
    for (int a = 0; a < K; ++a) {
      w[a] -= ph[a];
      u[a] -= ph[a];
      S += w[a] * w[a] + u[a] * u[a];
      Xw += w[a] * ph[a];
      Xu += u[a] * ph[a];
      Y += w[a] * u[a];
    }
    const Real V = Real(0.25) * (Xu - Xw), Tt = Real(0.25) * S - Real(0.5) * Y;
    const Real kw = kf * ((C2 + Real(0.5) * Xw) - V), ku = kf * ((C2 + Real(0.5) * Xu) + V);
    const Real kc = -kf * (((Xu + Xw) + Real(0.5) * S) + Tt);
#pragma unroll
    for (int a = 0; a < K; ++a) dg[a] += (w[a] * kw + u[a] * ku) + ph[a] * kc;
  }
#pragma unroll
  for (int a = 0; a < K; ++a) {
    // S4 potential derivative (obstacle, with the triple term), S5 rate and explicit Euler
    const Real others = e1 - ph[a];
    Real W = g.cw_0 * others;
    if (g.has_g3) W += g.g3 * (e2 - ph[a] * others);
    const Real r = g.mob * (g.eps * dg[a] - W * g.inv_eps) * g.inv_eps;
    v[a] = ph[a] + g.dt * r;
  }
  store_union<Real, K>(g, i, v, uid, nu);
}

// Two builds: KU = kUnionSmall takes the cells of the first list whose
// stencil holds at most that many grains (nearly all) and moves the others to
// the second list, which the KU = kUnion build then updates (each build's
// registers fit its own union size).
//
// UNI: one gamma for every pair (the rule; a table of gammas takes the other
// build).  The sums over pairs then factorise: with a cell's values c and the
// differences u = n_+ - c, w = n_- - c to its neighbours along an axis, X = sum u c,
// S = sum u^2 (of u, of w), Y = sum u w, C2 = sum c^2, V = (X_u - X_w) / 4 and T =
// (S_u + S_w - 2 Y) / 4,
//   dx^2 (div J - Gc)_a = 2 gamma [ u_a (C2 + X_u / 2 + V) + w_a (C2 + X_w / 2 - V)
//                                   - c_a (X_u + X_w + (S_u + S_w) / 2 + T) ]
// (differences, or terms of order 1 cancel: see k_gp_rows), summed over the axes: O(grains) instead of O(grains^2), and straight-line
// (absent grains of the union hold zeros); warps whose stencils hold two grains at
// most, as most of a boundary does, take a build of the update for two.  What
// bounds it is integer and FP32 instruction issue (gathering the values of the
// seven cells by grain is two thirds of it).  The first kPre slots of the seven
// cells are loaded at once, before their counts are known (a stale slot is then
// ignored), and matched to the union in registers.  8 grains in 128^3, FP32, GB300,
// KU = 4 / KU = 8 a step: 144 / 23 us by pairs, 61 / 17 us with the sums face by face
// and the values scattered to shared memory, 53 / 12 us here (55 with 24 warps per
// SM instead of 32).
template <class Real, int KU, bool UNI>
__global__ void __launch_bounds__(UpdShape<Real, KU>::THREADS, UpdShape<Real, KU>::MIN_BLOCKS)
    k_ggs_update(const __grid_constant__ GgsArgs<Real> g) {
  constexpr int T = UpdShape<Real, KU>::THREADS;
  constexpr bool kFirst = KU < kUnion;
  unsigned int* list = kFirst ? g.list : g.list2;
  constexpr int kPre = kFirst ? 2 : 3;
  __shared__ Real s_val[UNI ? 1 : 7 * KU][T];   // by pairs: [cell][slot][thread], a warp never shares a bank
  const int tid = threadIdx.x;
  auto sv = [&](int c, int u) -> Real& { return s_val[c * KU + u][tid]; };
  const unsigned int count = min(*(volatile const unsigned int*)&list[0], g.list_cap);
  const int nst = 2 * g.dim + 1;   // stencil cells: 0 the centre, 1 + 2d the -d and 2 + 2d the +d neighbour
  const unsigned int stride = gridDim.x * T;
  for (unsigned int w0 = blockIdx.x * T; w0 < count; w0 += stride) {
    const unsigned int w = w0 + tid;
    const bool live = w < count;
    const unsigned int i = live ? list[1 + w] : 0u;
    unsigned int ci[7];
    int cntc[7];
    int x, y, z;
    cell_of(g, i, x, y, z);
    ci[0] = i;
    auto neighbours = [&](int d, int pos, int n, int bc, unsigned int step) {
      const unsigned int wrap = (unsigned int)(n - 1) * step;
      ci[1 + 2 * d] = pos > 0 ? i - step : bc == 3 ? i + wrap : i;
      ci[2 + 2 * d] = pos < n - 1 ? i + step : bc == 3 ? i - wrap : i;
    };
    neighbours(0, x, g.nx, g.bc[0], 1u);
    neighbours(1, y, g.ny, g.bc[1], (unsigned int)g.nx);
    ci[5] = ci[6] = i;
    if (g.dim == 3) neighbours(2, z, g.nz, g.bc[2], (unsigned int)g.nx * (unsigned int)g.ny);
    int most = 0;
    int pidx[7][kPre];
    Real pval[7][kPre];
#pragma unroll
    for (int c = 0; c < 7; ++c) {
      cntc[c] = live && c < nst ? (int)g.cnt_in[ci[c]] : 0;
#pragma unroll
      for (int k = 0; k < kPre; ++k) {
        pidx[c][k] = g.idx_in[(size_t)k * g.cells + ci[c]];
        if constexpr (UNI) pval[c][k] = g.val_in[(size_t)k * g.cells + ci[c]];
      }
    }
#pragma unroll
    for (int c = 0; c < 7; ++c) {
      most = max(most, cntc[c]);
#pragma unroll
      for (int k = 0; k < kPre; ++k)
        if (k >= cntc[c]) pidx[c][k] = kMaxGrains;   // no grain
    }
    most = __reduce_max_sync(0xffffffffu, most);   // slots in use anywhere in the warp
    // union of the grains present on the stencil
    uint32_t lo = 0u, hi = 0u;
    // bit a (bits past 31 and 63 shift out: lshift clamps)
    auto lshift = [](int a) {
      uint32_t r;
      asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(a));
      return r;
    };
#pragma unroll
    for (int c = 0; c < 7; ++c)
#pragma unroll
      for (int k = 0; k < kPre; ++k) lo |= lshift(pidx[c][k]);
    if (g.N > 32) {
#pragma unroll
      for (int c = 0; c < 7; ++c)
#pragma unroll
        for (int k = 0; k < kPre; ++k) hi |= lshift(pidx[c][k] - 32);
    }
    for (int k = kPre; k < most; ++k) {
#pragma unroll
      for (int c = 0; c < 7; ++c)
        if (k < cntc[c]) {
          const int a = g.idx_in[(size_t)k * g.cells + ci[c]];
          lo |= lshift(a);
          hi |= lshift(a - 32);
        }
    }
    const unsigned long long mask = ((unsigned long long)hi << 32) | lo;
    const int nu = __popcll(mask);
    if (live && nu > KU) {
      if constexpr (kFirst) {
        const unsigned int k2 = atomicAdd(&g.list2[0], 1u);
        if (k2 < g.list_cap) g.list2[1 + k2] = i;
      } else {
        atomicOr(g.status, kStatusOverflow);
      }
    }
    const bool two = __all_sync(0xffffffffu, !live || nu <= 2);   // anywhere in the warp
    if (!live || nu > KU) continue;
    int uid[KU];
    {
      unsigned long long m = mask;
#pragma unroll
      for (int u = 0; u < KU; ++u) {
        uid[u] = m ? __ffsll((long long)m) - 1 : 0;   // (the entries past nu are not used)
        m &= m - 1ull;
      }
    }
    // S1-S3: divergence of the face fluxes (isotropic: the normal component
    // of g = 2 gamma q needs the normal differences only) and the centre term
    if constexpr (UNI) {
      if constexpr (kFirst) {   // two grains: most cells of a boundary
        if (two)
          update_uniform<Real, 2, kPre>(g, i, ci, cntc, pidx, pval, uid, nu, 0);
        else
          update_uniform<Real, KU, kPre>(g, i, ci, cntc, pidx, pval, uid, nu, most);
      } else {
        update_uniform<Real, KU, kPre>(g, i, ci, cntc, pidx, pval, uid, nu, most);
      }
    } else {
      Real v[KU];
#pragma unroll
      for (int c = 0; c < 7; ++c)
#pragma unroll
        for (int u = 0; u < KU; ++u) sv(c, u) = Real(0);
      for (int k = 0; k < most; ++k) {
#pragma unroll
        for (int c = 0; c < 7; ++c)
          if (k < cntc[c]) {
            const int a = g.idx_in[(size_t)k * g.cells + ci[c]];
            sv(c, __popcll(mask & ((1ull << a) - 1ull))) = g.val_in[(size_t)k * g.cells + ci[c]];
          }
      }
      Real divJ[KU], Gc[KU];
#pragma unroll
      for (int u = 0; u < KU; ++u) {
        divJ[u] = Real(0);
        Gc[u] = Real(0);
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        if (d >= g.dim) break;
        Real Jm[KU], Jp[KU];
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          // side 0: the face with the -d neighbour (left = it, right = the
          // cell); side 1: with the +d neighbour (left = the cell)
          const int cl = side ? 0 : 1 + 2 * d, cr = side ? 2 + 2 * d : 0;
          Real* J = side ? Jp : Jm;
          Real pf[KU], gr[KU];
#pragma unroll
          for (int a = 0; a < KU; ++a) {
            J[a] = Real(0);
            if (a >= nu) continue;
            const Real vl = sv(cl, a), vr = sv(cr, a);
            pf[a] = Real(0.5) * (vl + vr);
            gr[a] = (vr - vl) * g.inv_dx;
          }
#pragma unroll
          for (int a = 0; a < KU; ++a) {
            if (a >= nu) break;
#pragma unroll
            for (int b = a + 1; b < KU; ++b) {
              if (b >= nu) break;
              const Real q = pf[a] * gr[b] - pf[b] * gr[a];
              const Real gq = g.gam2[uid[a] * g.N + uid[b]] * q;
              J[a] -= pf[b] * gq;
              J[b] += pf[a] * gq;
            }
          }
        }
#pragma unroll
        for (int a = 0; a < KU; ++a)
          if (a < nu) divJ[a] += (Jp[a] - Jm[a]) * g.inv_dx;
      }
      // centre term, central differences
      Real gc[KU][3];
#pragma unroll
      for (int a = 0; a < KU; ++a)
#pragma unroll
        for (int d = 0; d < 3; ++d)
          gc[a][d] = d < g.dim ? (sv(2 + 2 * d, a) - sv(1 + 2 * d, a)) * g.half_inv_dx : Real(0);
#pragma unroll
      for (int a = 0; a < KU; ++a) {
        if (a >= nu) break;
#pragma unroll
        for (int b = a + 1; b < KU; ++b) {
          if (b >= nu) break;
          const Real gm = g.gam2[uid[a] * g.N + uid[b]];
          Real gq[3];
#pragma unroll
          for (int d = 0; d < 3; ++d) gq[d] = gm * (sv(0, a) * gc[b][d] - sv(0, b) * gc[a][d]);
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            if (d >= g.dim) break;
            Gc[a] += gq[d] * gc[b][d];
            Gc[b] -= gq[d] * gc[a][d];
          }
        }
      }
      // S4 potential derivative (obstacle, with the triple term), S5 rate and
      // explicit Euler (no chemical driving force in grain growth)
#pragma unroll
      for (int a = 0; a < KU; ++a) {
        v[a] = Real(0);
        if (a >= nu) continue;
        Real W = Real(0);
#pragma unroll
        for (int b = 0; b < KU; ++b)
          if (b < nu && b != a) W += g.cw[uid[a] * g.N + uid[b]] * sv(0, b);
        if (g.has_g3) {
#pragma unroll
          for (int b = 0; b < KU; ++b)
#pragma unroll
            for (int e = b + 1; e < KU; ++e)
              if (e < nu && b != a && e != a) W += g.g3 * sv(0, b) * sv(0, e);
        }
        const Real r = g.mob * (g.eps * (divJ[a] - Gc[a]) - W * g.inv_eps) * g.inv_eps;
        v[a] = sv(0, a) + g.dt * r;
      }
      store_union<Real, KU>(g, i, v, uid, nu);
    }
  }
  if constexpr (!kFirst) {
    // the last CTA of the step's last kernel keeps the listed count and
    // clears both lists for the next step
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      if (atomicAdd(&g.status[2], 1) == (int)gridDim.x - 1) {
        g.status[1] = (int)*(volatile unsigned int*)&g.list[0];
        g.list[0] = 0u;
        g.list2[0] = 0u;
        g.status[2] = 0;
      }
    }
  }
}

// dense [N][cells] -> slots (sorted by grain), codes; overflow -> status
template <class Real>
__global__ void k_ggs_pack(const Real* __restrict__ dense, int N, long long cells, uint8_t* cnt, uint8_t* code,
                           uint8_t* idx, Real* val, int* status) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= cells) return;
  int n = 0;
  uint8_t c = 0;
  for (int a = 0; a < N; ++a) {
    const Real v = dense[a * cells + i];
    if (v > Real(0)) {
      if (n < kSlots) {
        idx[n * cells + i] = (uint8_t)a;
        val[n * cells + i] = v;
        if (v == Real(1)) c = (uint8_t)(a + 1);
      }
      ++n;
    } else if (!(v == Real(0))) {
      atomicOr(status, kStatusOverflow);   // negative or non-finite input
    }
  }
  if (n > kSlots) {
    atomicOr(status, kStatusOverflow);
    n = kSlots;
  }
  cnt[i] = (uint8_t)n;
  code[i] = n == 1 ? c : 0;
}

template <class Real>
__global__ void k_ggs_unpack(Real* __restrict__ dense, long long cells, const uint8_t* cnt, const uint8_t* idx,
                             const Real* val) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= cells) return;
  const int n = cnt[i];
  for (int k = 0; k < n; ++k) dense[idx[k * cells + i] * cells + i] = val[k * cells + i];
}

}  // namespace

struct ms_ggs {
  HostModel m;
  int N = 0;
  long long cells = 0;
  size_t s = 4;
  void* buf[2] = {nullptr, nullptr};   // cnt | code | idx | val per buffer
  void* tables = nullptr;              // gam2 [N][N], cw [N][N]
  unsigned int* list = nullptr;
  unsigned int* list2 = nullptr;
  int* status = nullptr;
  int cur = 0;
  int64_t step = 0;
  int sms = 0;
  bool uniform = false;                // one gamma for every pair
  double gamma0 = 0.0;                 // gamma of the first pair
  double g3 = 0.0;
  int has_g3 = 0;
  cudaStream_t stream = nullptr;
  AllocHook hook;
  std::string err;
};

namespace {

ms_status gfail(ms_ggs* s, ms_status st, const std::string& m) {
  if (s) s->err = m;
  return fail(nullptr, st, m);
}

size_t buf_bytes(const ms_ggs* s) {
  const size_t c = (size_t)s->cells;
  const size_t head = (2 * c + (size_t)kSlots * c + 255) / 256 * 256;
  return head + (size_t)kSlots * c * s->s;
}
uint8_t* cnt_of(const ms_ggs* s, int b) { return static_cast<uint8_t*>(s->buf[b]); }
uint8_t* code_of(const ms_ggs* s, int b) { return cnt_of(s, b) + s->cells; }
uint8_t* idx_of(const ms_ggs* s, int b) { return cnt_of(s, b) + 2 * s->cells; }
void* val_of(const ms_ggs* s, int b) {
  const size_t c = (size_t)s->cells;
  return cnt_of(s, b) + (2 * c + (size_t)kSlots * c + 255) / 256 * 256;
}

template <class Real>
GgsArgs<Real> make_args(const ms_ggs* s, int src) {
  GgsArgs<Real> g;
  std::memset(&g, 0, sizeof(g));
  const HostModel& m = s->m;
  g.nx = m.nx;
  g.ny = m.ny;
  g.nz = m.dim == 3 ? m.nz : 1;
  g.dim = m.dim;
  g.N = s->N;
  for (int d = 0; d < 3; ++d) g.bc[d] = m.bc[d];
  g.cells = s->cells;
  g.dt = (Real)m.dt;
  g.eps = (Real)m.eps;
  g.inv_eps = (Real)(1.0 / m.eps);
  g.mob = (Real)(1.0 / m.tau);
  g.inv_dx = (Real)(1.0 / m.dx);
  g.half_inv_dx = (Real)(0.5 / m.dx);
  g.g3 = (Real)s->g3;
  g.has_g3 = s->has_g3;
  g.gam2 = static_cast<const Real*>(s->tables);
  g.cw = static_cast<const Real*>(s->tables) + s->N * s->N;
  g.gam2_0 = (Real)(2.0 * s->gamma0);
  g.cw_0 = (Real)((16.0 / (3.14159265358979323846 * 3.14159265358979323846)) * s->gamma0);
  g.cnt_in = cnt_of(s, src);
  g.code_in = code_of(s, src);
  g.idx_in = idx_of(s, src);
  g.val_in = static_cast<const Real*>(val_of(s, src));
  g.cnt_out = cnt_of(s, 1 - src);
  g.code_out = code_of(s, 1 - src);
  g.idx_out = idx_of(s, 1 - src);
  g.val_out = static_cast<Real*>(val_of(s, 1 - src));
  g.list = s->list;
  g.list2 = s->list2;
  g.list_cap = (unsigned int)s->cells;
  g.status = s->status;
  return g;
}

template <class Real>
cudaError_t step_once(ms_ggs* s) {
  const GgsArgs<Real> g = make_args<Real>(s, s->cur);
  const unsigned int blocks = (unsigned int)((s->cells + 1023) / 1024);
  if (g.nx % 4 == 0)   // (rows, and the code array behind the counts, start on words then)
    k_ggs_classify4<Real><<<blocks, 256, 0, s->stream>>>(g);
  else
    k_ggs_classify<Real><<<blocks, 256, 0, s->stream>>>(g);
  const auto small = s->uniform ? k_ggs_update<Real, kUnionSmall, true> : k_ggs_update<Real, kUnionSmall, false>;
  const auto large = s->uniform ? k_ggs_update<Real, kUnion, true> : k_ggs_update<Real, kUnion, false>;
  using Ss = UpdShape<Real, kUnionSmall>;
  using Sl = UpdShape<Real, kUnion>;
  small<<<s->sms * Ss::MIN_BLOCKS, Ss::THREADS, 0, s->stream>>>(g);
  large<<<s->sms * Sl::MIN_BLOCKS, Sl::THREADS, 0, s->stream>>>(g);
  return cudaGetLastError();
}

}  // namespace

extern "C" {

ms_status ms_ggs_create(const ms_grid* grid, int n_grains, const ms_params* p, void* stream,
                        const ms_allocator* alloc, ms_ggs** out) {
  if (!out || !grid || !p) return gfail(nullptr, MS_ERR_ARG, "grid, params and out are required");
  *out = nullptr;
  if (n_grains < 2 || n_grains > kMaxGrains)
    return gfail(nullptr, MS_ERR_ARG, "sparse grain growth takes 2 to 64 grains");
  if (p->potential != MS_POT_OBSTACLE)
    return gfail(nullptr, MS_ERR_UNSUPPORTED, "sparse grain growth needs the obstacle potential");
  if (p->noise_amp != 0.0 || p->anti_trapping || p->elastic_C)
    return gfail(nullptr, MS_ERR_UNSUPPORTED, "sparse grain growth takes no noise, anti-trapping or elasticity");
  const int N = n_grains;
  for (int a = 0; a < N; ++a)
    for (int b = 0; b < N; ++b)
      if (a != b && p->delta && p->delta[a * N + b] != 0.0)
        return gfail(nullptr, MS_ERR_UNSUPPORTED, "sparse grain growth is isotropic (delta = 0 for every pair)");
  double g3 = 0.0;
  int has_g3 = 0;
  if (p->gamma3) {
    // a uniform triple term over distinct triples (the only form stored)
    bool first = true;
    for (int a = 0; a < N; ++a)
      for (int b = 0; b < N; ++b)
        for (int c = 0; c < N; ++c) {
          const double v = p->gamma3[(a * N + b) * N + c];
          if (a == b || b == c || a == c) {
            if (v != 0.0) return gfail(nullptr, MS_ERR_ARG, "gamma3 must vanish unless the three phases differ");
            continue;
          }
          if (first) {
            g3 = v;
            first = false;
          } else if (v != g3) {
            return gfail(nullptr, MS_ERR_UNSUPPORTED, "sparse grain growth takes a uniform gamma3");
          }
        }
    has_g3 = g3 != 0.0;
  }
  if (grid->dim == 3 && grid->bc[2] == MS_BC_HALO)
    return gfail(nullptr, MS_ERR_UNSUPPORTED, "sparse grain growth runs on the whole domain");
  ensure_registered();
  ms_ggs* s = new ms_ggs();
  // the model checks of a context (grid, boundaries, dt bound, gamma): one
  // solute field stands in for the held mu, with the values build_model needs
  ms_params q = *p;
  std::vector<double> D(N, 0.0), A(N, 1.0), ceq(N, 0.5), sl(N, 0.0);
  q.D = D.data();
  q.A = A.data();
  q.ceq = ceq.data();
  q.slopes = sl.data();
  q.f0 = nullptr;
  q.gamma3 = nullptr;
  q.grain_growth = 1;
  q.rot = nullptr;
  q.delta = nullptr;
  std::vector<double> zero(N * N, 0.0);
  q.delta = zero.data();
  if (N > kNMax) {
    // build_model checks at most kNMax phases: check the shape here
    if (grid->dim != 2 && grid->dim != 3) {
      delete s;
      return gfail(nullptr, MS_ERR_ARG, "dim must be 2 or 3");
    }
    if (grid->nx < 1 || grid->ny < 1 || (grid->dim == 3 && grid->nz < 1) || !(grid->dx > 0.0)) {
      delete s;
      return gfail(nullptr, MS_ERR_ARG, "bad grid");
    }
    for (int d = 0; d < grid->dim; ++d)
      if (grid->bc[d] != MS_BC_PERIODIC && grid->bc[d] != MS_BC_NOFLUX) {
        delete s;
        return gfail(nullptr, MS_ERR_ARG, "boundaries must be periodic or no-flux");
      }
    if (!(p->eps > 0.0) || !(p->tau > 0.0) || !(p->dt > 0.0) || !p->gamma) {
      delete s;
      return gfail(nullptr, MS_ERR_ARG, "eps, tau, dt and gamma are required");
    }
    s->m.dim = grid->dim;
    s->m.nx = grid->nx;
    s->m.ny = grid->ny;
    s->m.nz = grid->dim == 3 ? grid->nz : 1;
    s->m.dx = grid->dx;
    for (int d = 0; d < 3; ++d) s->m.bc[d] = d < grid->dim ? grid->bc[d] : 3;
    s->m.dtype = p->dtype;
    s->m.eps = p->eps;
    s->m.tau = p->tau;
    s->m.dt = p->dt;
  } else {
    ms_status st = build_model(nullptr, grid, N, 2, &q, s->m);
    if (st != MS_OK) {
      std::string msg = ms_last_error(nullptr);
      delete s;
      return gfail(nullptr, st, msg);
    }
  }
  // explicit stability of the phase equation (isotropic): dt <= (dx^2 / 2d) tau / gamma_max
  double gmax = 0.0;
  for (int a = 0; a < N; ++a)
    for (int b = 0; b < N; ++b)
      if (a != b) {
        const double v = p->gamma[a * N + b];
        if (!(v >= 0.0) || v != p->gamma[b * N + a]) {
          delete s;
          return gfail(nullptr, MS_ERR_ARG, "gamma must be symmetric and non-negative");
        }
        gmax = std::max(gmax, v);
      }
  const double bound = grid->dx * grid->dx / (2.0 * grid->dim) * p->tau / (gmax > 0 ? gmax : 1.0);
  if (p->dt > bound) {
    delete s;
    return gfail(nullptr, MS_ERR_DT_UNSTABLE, "dt above the explicit stability bound");
  }
  s->N = N;
  s->gamma0 = p->gamma[1];
  s->uniform = true;
  for (int a = 0; a < N; ++a)
    for (int b = 0; b < N; ++b)
      if (a != b && p->gamma[a * N + b] != s->gamma0) s->uniform = false;
  s->g3 = g3;
  s->has_g3 = has_g3;
  s->cells = (long long)grid->nx * grid->ny * (grid->dim == 3 ? grid->nz : 1);
  if (s->cells >= 0xFFFFFFFFll) {
    delete s;
    return gfail(nullptr, MS_ERR_BOUNDS, "grid too large for the work list");
  }
  s->s = p->dtype == MS_F64 ? 8 : 4;
  s->stream = static_cast<cudaStream_t>(stream);
  if (alloc) s->hook = AllocHook{alloc->alloc, alloc->release, alloc->user};
  for (int b = 0; b < 2; ++b) s->buf[b] = dev_alloc(s->hook, buf_bytes(s));
  s->tables = dev_alloc(s->hook, 2 * (size_t)N * N * s->s);
  s->list = static_cast<unsigned int*>(dev_alloc(s->hook, 2 * (size_t)(s->cells + 1) * sizeof(unsigned int) + 256));
  if (!s->buf[0] || !s->buf[1] || !s->tables || !s->list) {
    ms_ggs_destroy(s);
    return gfail(nullptr, MS_ERR_OOM, "sparse grain-growth allocation failed");
  }
  s->list2 = s->list + (s->cells + 1);
  s->status = reinterpret_cast<int*>(s->list2 + (s->cells + 1));
  const double PI = 3.14159265358979323846;
  std::vector<double> tab(2 * (size_t)N * N);
  for (int a = 0; a < N; ++a)
    for (int b = 0; b < N; ++b) {
      tab[a * N + b] = 2.0 * p->gamma[a * N + b];
      tab[N * N + a * N + b] = (16.0 / (PI * PI)) * p->gamma[a * N + b];   // as the obstacle term forms it
    }
  cudaError_t e = cudaSuccess;
  if (s->s == 8) {
    e = cudaMemcpyAsync(s->tables, tab.data(), tab.size() * 8, cudaMemcpyHostToDevice, s->stream);
  } else {
    std::vector<float> tf(tab.begin(), tab.end());
    e = cudaMemcpyAsync(s->tables, tf.data(), tf.size() * 4, cudaMemcpyHostToDevice, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  }
  for (int b = 0; b < 2 && e == cudaSuccess; ++b) e = cudaMemsetAsync(s->buf[b], 0, buf_bytes(s), s->stream);
  // the lists' counts and the status words (cleared by the steps themselves afterwards)
  if (e == cudaSuccess) e = cudaMemsetAsync(s->list, 0, sizeof(unsigned int), s->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(s->list2, 0, sizeof(unsigned int), s->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(s->status, 0, 4 * sizeof(int), s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  s->sms = sms;
  if (e != cudaSuccess) {
    std::string m = std::string("sparse grain growth set-up: ") + cudaGetErrorString(e);
    ms_ggs_destroy(s);
    return gfail(nullptr, MS_ERR_CUDA, m);
  }
  *out = s;
  return MS_OK;
}

void ms_ggs_destroy(ms_ggs* s) {
  if (!s) return;
  cudaStreamSynchronize(s->stream);
  for (int b = 0; b < 2; ++b) dev_free(s->hook, s->buf[b]);
  dev_free(s->hook, s->tables);
  dev_free(s->hook, s->list);
  delete s;
}

const char* ms_ggs_last_error(const ms_ggs* s) { return s ? s->err.c_str() : ms_last_error(nullptr); }

ms_status ms_ggs_set_fields(ms_ggs* s, const void* phi, int on_device) {
  if (!s || !phi) return gfail(s, MS_ERR_ARG, "ctx and phi are required");
  const size_t bytes = (size_t)s->N * s->cells * s->s;
  void* dense = const_cast<void*>(phi);
  void* tmp = nullptr;
  cudaError_t e = cudaSuccess;
  if (!on_device) {
    tmp = dev_alloc(s->hook, bytes);
    if (!tmp) return gfail(s, MS_ERR_OOM, "staging allocation failed");
    e = cudaMemcpyAsync(tmp, phi, bytes, cudaMemcpyHostToDevice, s->stream);
    dense = tmp;
  }
  const unsigned int blocks = (unsigned int)((s->cells + 255) / 256);
  if (e == cudaSuccess) {
    if (s->s == 8)
      k_ggs_pack<double><<<blocks, 256, 0, s->stream>>>(static_cast<const double*>(dense), s->N, s->cells,
                                                         cnt_of(s, s->cur), code_of(s, s->cur), idx_of(s, s->cur),
                                                         static_cast<double*>(val_of(s, s->cur)), s->status);
    else
      k_ggs_pack<float><<<blocks, 256, 0, s->stream>>>(static_cast<const float*>(dense), s->N, s->cells,
                                                        cnt_of(s, s->cur), code_of(s, s->cur), idx_of(s, s->cur),
                                                        static_cast<float*>(val_of(s, s->cur)), s->status);
    e = cudaGetLastError();
  }
  // the other buffer holds nothing of this state
  if (e == cudaSuccess) e = cudaMemsetAsync(s->buf[1 - s->cur], 0, 2 * (size_t)s->cells, s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  dev_free(s->hook, tmp);
  if (e != cudaSuccess) return gfail(s, MS_ERR_CUDA, std::string("sparse set fields: ") + cudaGetErrorString(e));
  s->step = 0;
  return ms_ggs_sync(s);
}

ms_status ms_ggs_get_fields(ms_ggs* s, void* phi, int on_device) {
  if (!s || !phi) return gfail(s, MS_ERR_ARG, "ctx and phi are required");
  const size_t bytes = (size_t)s->N * s->cells * s->s;
  void* dense = phi;
  void* tmp = nullptr;
  if (!on_device) {
    tmp = dev_alloc(s->hook, bytes);
    if (!tmp) return gfail(s, MS_ERR_OOM, "staging allocation failed");
    dense = tmp;
  }
  cudaError_t e = cudaMemsetAsync(dense, 0, bytes, s->stream);
  const unsigned int blocks = (unsigned int)((s->cells + 255) / 256);
  if (e == cudaSuccess) {
    if (s->s == 8)
      k_ggs_unpack<double><<<blocks, 256, 0, s->stream>>>(static_cast<double*>(dense), s->cells, cnt_of(s, s->cur),
                                                           idx_of(s, s->cur), static_cast<double*>(val_of(s, s->cur)));
    else
      k_ggs_unpack<float><<<blocks, 256, 0, s->stream>>>(static_cast<float*>(dense), s->cells, cnt_of(s, s->cur),
                                                          idx_of(s, s->cur), static_cast<float*>(val_of(s, s->cur)));
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && !on_device) e = cudaMemcpyAsync(phi, dense, bytes, cudaMemcpyDeviceToHost, s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  dev_free(s->hook, tmp);
  if (e != cudaSuccess) return gfail(s, MS_ERR_CUDA, std::string("sparse get fields: ") + cudaGetErrorString(e));
  return MS_OK;
}

ms_status ms_ggs_step(ms_ggs* s, int64_t n) {
  TraceRange trace("ms_ggs_step");
  if (!s || n < 0) return gfail(s, MS_ERR_ARG, "bad argument");
  for (int64_t k = 0; k < n; ++k) {
    cudaError_t e = s->s == 8 ? step_once<double>(s) : step_once<float>(s);
    if (e != cudaSuccess) return gfail(s, MS_ERR_CUDA, std::string("sparse step: ") + cudaGetErrorString(e));
    s->cur = 1 - s->cur;
    s->step += 1;
  }
  return MS_OK;
}

ms_status ms_ggs_sync(ms_ggs* s) {
  if (!s) return gfail(nullptr, MS_ERR_ARG, "ctx is NULL");
  int st = 0;
  cudaError_t e = cudaMemcpyAsync(&st, s->status, sizeof(int), cudaMemcpyDeviceToHost, s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  if (e != cudaSuccess) return gfail(s, MS_ERR_CUDA, std::string("sparse sync: ") + cudaGetErrorString(e));
  if (st & kStatusOverflow)
    return gfail(s, MS_ERR_BOUNDS, "a cell needed more than 8 grains (or its stencil more than 8), or the input "
                                   "held a negative or non-finite value");
  return MS_OK;
}

ms_status ms_ggs_stats(ms_ggs* s, int64_t* listed_cells, int64_t* step) {
  if (!s) return gfail(nullptr, MS_ERR_ARG, "ctx is NULL");
  unsigned int cnt = 0;
  cudaError_t e = cudaMemcpyAsync(&cnt, s->status + 1, sizeof(unsigned int), cudaMemcpyDeviceToHost, s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  if (e != cudaSuccess) return gfail(s, MS_ERR_CUDA, std::string("sparse stats: ") + cudaGetErrorString(e));
  if (listed_cells) *listed_cells = s->step > 0 ? (int64_t)cnt : 0;
  if (step) *step = s->step;
  return MS_OK;
}

}  // extern "C"
