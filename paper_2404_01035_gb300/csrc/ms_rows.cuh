// Interface rows of the split 3-D FP32 step for models with many phases and one
// boundary energy: gamma_ab = gamma for every pair (what the infile's single
// GAMMA value gives).
//
// With one gamma the isotropic part of the sums over pairs (MICROSIM paper,
// arXiv 2404.01035, Sec. 2.1) factorises.  With q_ab = phi_a grad phi_b -
// phi_b grad phi_a and g_ab = 2 gamma q_ab,
//   J_a  = -sum_b phi_b g_ab  = 2 gamma (grad phi_a S2 - phi_a S1),
//          S1 = sum_b phi_b grad phi_b, S2 = sum_b phi_b^2,
//   Gc_a = sum_b g_ab . grad phi_b = 2 gamma (phi_a T - grad phi_a . S1),
//          T = sum_b |grad phi_b|^2,
// and likewise the obstacle and well derivatives and the driving force, so a
// cell costs O(N) instead of O(N^2).  Written out in the cell's value c and the
// differences u = n_+ - c, w = n_- - c to its neighbours along an axis, the two
// faces of the axis and its part of the centre term need the sums over the phases
// X = sum u c, S = sum u^2 (of u, of w), Y = sum u w and C2 = sum c^2:
//   dx^2 (div J - Gc)_a = 2 gamma [ u_a (C2 + X_u / 2 + V) + w_a (C2 + X_w / 2 - V)
//                                   - c_a (X_u + X_w + (S_u + S_w) / 2 + T) ],
//   V = (X_u - X_w) / 4, T = (S_u + S_w - 2 Y) / 4.
// (In the neighbours' values themselves terms of order 1 cancel: ten times the
// rounding error, 8.8e-8 rms for profiles of three phases against 8.5e-9 here and
// 9.0e-9 by pairs.)
// An anisotropic pair adds the difference of its g to 2 gamma q.
//
// Without the triple term gamma_abc the multi-obstacle potential puts every
// phase on every boundary, so a listed row of an 8-phase grid usually holds all
// 8 phases and the pair form pays for all 28 pairs (and spills: 255 registers).
// What bounds it: instruction issue, the latency of its loads, and with
// anisotropic pairs the instruction cache (so one code path for rotated and
// unrotated pairs, and builds of their own for grain growth).  Measured on a
// GB300, interface rows of one step, by pairs / with the sums taken face by
// face / here: 8 grains filling 192^3 (isotropic) 5846 / 340 / 222 us; 7 rotated
// grains in 128^3 with an eigenstrain - / 141 / 111 us; in 512^3 (few interface
// rows) 698 / 186 / 144 us.  Models with unequal gamma, the triple term or the
// anti-trapping current keep the pair form (k_gp_iface).
#pragma once

#include "ms_split.cuh"

namespace msgb {

template <int NP, int NM, bool ANISO, bool GG>
struct RowsShape {
  static constexpr int WARPS = 4;
  static constexpr int THREADS = 32 * WARPS;
  // (isotropic rows with the driving force: 54 us a step of 7 grains in 128^3 with 24 warps
  // per SM, which spill, 50 with 16)
  static constexpr int MIN_BLOCKS = GG && !ANISO ? 8 : 4;   // 32 / 16 warps per SM
};

// Threshold of the simplex projection (phi = max(v - theta, 0)): sorted values,
// running sums (project's rule).  Eight values go through Batcher's odd-even
// merge network (19 exchanges of two instructions; insertion takes 28 of three).
template <int NP>
__device__ __forceinline__ float simplex_shift(const float* v) {
  float u[NP];
#pragma unroll
  for (int a = 0; a < NP; ++a) u[a] = v[a];
  auto order = [&](int i, int j) {   // u[i] >= u[j]
    const float hi = fmaxf(u[i], u[j]), lo = fminf(u[i], u[j]);
    u[i] = hi;
    u[j] = lo;
  };
  if constexpr (NP == 8) {
    order(0, 1), order(2, 3), order(4, 5), order(6, 7);
    order(0, 2), order(1, 3), order(4, 6), order(5, 7);
    order(1, 2), order(5, 6);
    order(0, 4), order(1, 5), order(2, 6), order(3, 7);
    order(2, 4), order(3, 5);
    order(1, 2), order(3, 4), order(5, 6);
  } else {
#pragma unroll
    for (int i = 1; i < NP; ++i)
#pragma unroll
      for (int j = i; j > 0; --j) order(j - 1, j);
  }
  float csum = u[0], theta = u[0] - 1.0f;
#pragma unroll
  for (int j = 1; j < NP; ++j) {
    csum += u[j];
    const float t = (csum - 1.0f) * float(1.0 / (j + 1));
    theta = u[j] - t > 0.0f ? t : theta;
  }
  return theta;
}

// g = dA/dq of an anisotropic pair minus its isotropic part 2 gamma q, for the
// two faces of an axis (or, in both halves, one cell) in paired FP32: the
// factored form of aniso_grad_factored applied to R q, g := 0 where |q|^2 <
// 1e-12 (pair_grad's rule; the isotropic part is then taken off as well).
// ONLY >= 0: that component alone.
template <int ONLY>
__device__ __forceinline__ void aniso_excess(const F2* q, float gam2, float del, const float* R, F2* out) {
  // (unrotated pairs too: R is the identity then, and one code path keeps the
  // kernel nearer the instruction cache's size)
  F2 r[3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
    r[i] = fma2(f2s(R[i * 3 + 2]), q[2], fma2(f2s(R[i * 3 + 1]), q[1], f2s(R[i * 3]) * q[0]));
  F2 r2[3], Q = q[0] * q[0];
  Q = fma2(q[2], q[2], fma2(q[1], q[1], Q));
#pragma unroll
  for (int i = 0; i < 3; ++i) r2[i] = r[i] * r[i];
  const F2 s4 = fma2(r2[2], r2[2], fma2(r2[1], r2[1], r2[0] * r2[0]));
  const float Ql = f2lo(Q), Qh = f2hi(Q);
  const bool tl = Ql < 1e-12f, th = Qh < 1e-12f;
  const F2 invQ = f2(recip(tl ? 1.0f : Ql), recip(th ? 1.0f : Qh));
  const F2 rr = s4 * invQ * invQ;
  const F2 ac = fma2(f2s(4.0f * del), rr, f2s(1.0f - 3.0f * del));
  const F2 ga = f2s(gam2) * ac;
  F2 g[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) g[i] = ga * r[i] * fma2(f2s(16.0f * del), r2[i] * invQ - rr, ac);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    if (ONLY >= 0 && j != ONLY) continue;
    F2 v = fma2(f2s(R[6 + j]), g[2], fma2(f2s(R[3 + j]), g[1], f2s(R[j]) * g[0]));
    v = f2(tl ? 0.0f : f2lo(v), th ? 0.0f : f2hi(v));
    out[j] = fma2(f2s(-gam2), q[j], v);
  }
}

// The 19-point neighbourhood of one phase at a cell (the 3 x 3 x 3 block
// without its corners), and whether any of it is non-zero.
struct Edge19 {
  float c, m[3], p[3];     // centre, the -d and +d neighbours
  float e[3][4];           // edges of the axis pair (t, u) = (d+1, d+2): -t-u, +t-u, -t+u, +t+u
};
__device__ __forceinline__ bool load19(const float* s, const long long* o, Edge19& v) {
  v.c = s[0];
  bool any = v.c != 0.0f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    v.m[d] = s[-o[d]];
    v.p[d] = s[o[d]];
    any = any || v.m[d] != 0.0f || v.p[d] != 0.0f;
    const long long t = o[(d + 1) % 3], u = o[(d + 2) % 3];
    v.e[d][0] = s[-t - u];
    v.e[d][1] = s[t - u];
    v.e[d][2] = s[u - t];
    v.e[d][3] = s[t + u];
    any = any || v.e[d][0] != 0.0f || v.e[d][1] != 0.0f || v.e[d][2] != 0.0f || v.e[d][3] != 0.0f;
  }
  return any;
}
// phi(m_D + t) - phi(m_D - t) at the -D neighbour (low half) and the +D one.
template <int D, int T>
__device__ __forceinline__ F2 edge_diff(const Edge19& v) {
  if constexpr (T == (D + 1) % 3) {        // axis of the edge list is the third one, (t', u') = (D, T)
    constexpr int A = (D + 2) % 3;
    return f2(v.e[A][2] - v.e[A][0], v.e[A][3] - v.e[A][1]);
  } else {                                 // (t', u') = (T, D)
    constexpr int A = (D + 1) % 3;
    return f2(v.e[A][1] - v.e[A][0], v.e[A][3] - v.e[A][2]);
  }
}

// Excess flux of the pair through the two faces along D: adds its divergence
// to (da, db).
template <int D>
__device__ __forceinline__ void pair_faces(const Edge19& va, const Edge19& vb, float gam2, float del, const float* R,
                                           float inv_dx, float qdx, float& da, float& db) {
  constexpr int T = (D + 1) % 3, U = (D + 2) % 3;
  auto grads = [&](const Edge19& v, F2& pf, F2* gr) {
    const F2 l = f2(v.m[D], v.c), r = f2(v.c, v.p[D]);
    pf = f2s(0.5f) * (l + r);
    gr[D] = (r - l) * f2s(inv_dx);
    gr[T] = (edge_diff<D, T>(v) + f2s(v.p[T] - v.m[T])) * f2s(qdx);
    gr[U] = (edge_diff<D, U>(v) + f2s(v.p[U] - v.m[U])) * f2s(qdx);
  };
  F2 pa, pb, ga[3], gb[3], q[3], x[3];
  grads(va, pa, ga);
  grads(vb, pb, gb);
#pragma unroll
  for (int i = 0; i < 3; ++i) q[i] = pa * gb[i] - pb * ga[i];
  aniso_excess<D>(q, gam2, del, R, x);
  const F2 ja = pb * x[D], jb = pa * x[D];   // J_a = -ja, J_b = jb
  da -= (f2hi(ja) - f2lo(ja)) * inv_dx;
  db += (f2hi(jb) - f2lo(jb)) * inv_dx;
}

// One warp per listed 32-cell row segment, grid-stride; stencil values by
// plain loads (a warp's loads are whole rows, and neighbouring list entries
// share them through L1 and L2), which leaves shared memory and the registers
// of a staging ring to more warps.
template <int NP, int NM, bool ANISO, bool GG>
__global__ void __launch_bounds__(RowsShape<NP, NM, ANISO, GG>::THREADS, RowsShape<NP, NM, ANISO, GG>::MIN_BLOCKS)
    k_gp_rows(const __grid_constant__ StepArgs<float, NP, NM> g, const float* __restrict__ in) {
  using Sh = RowsShape<NP, NM, ANISO, GG>;
  __shared__ unsigned int s_count;
  __shared__ float s_dg[ANISO ? Sh::WARPS : 1][ANISO ? NP : 1][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned int* const list = g.iface;
  if (threadIdx.x == 0) s_count = min(*(volatile unsigned int*)&list[0], g.iface_cap);
  __syncthreads();
  const unsigned int count = s_count;
  const unsigned int seg_mask = (1u << g.seg_bits) - 1u, y_mask = (1u << g.y_bits) - 1u;
  const long long plane = (long long)g.nyp * g.pitch, fs = g.fstride;
  const long long o[3] = {1, g.pitch, plane};
  const float gam2 = g.gam2[0];
  for (unsigned int i = blockIdx.x * Sh::WARPS + wid; i < count; i += gridDim.x * Sh::WARPS) {
    const unsigned int r = list[2 + i];
    const int sg = (int)(r & seg_mask), y = (int)((r >> g.seg_bits) & y_mask), z = (int)(r >> (g.seg_bits + g.y_bits));
    const int x = 32 * sg + lane;
    const bool active = x < g.nx;
    // lanes past the end of a ragged row repeat its last cell (in bounds)
    const float* s = in + (long long)(z + g.zoff) * plane + (long long)(y + 1) * g.pitch + min(x, g.nx - 1) + g.xoff;
    float ph[NP], dg[NP];
    float e1 = 0.0f, p2s = 0.0f;
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      ph[a] = s[a * fs];
      dg[a] = 0.0f;
      e1 += ph[a];
      p2s += ph[a] * ph[a];
    }
    float mc[NM];
    F2 dv[NM];
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      mc[k] = s[(NP + k) * fs];
      dv[k] = f2s(0.0f);
    }
    float Mc[NM * NM];
    if constexpr (!GG) cell_mobility<NP, NM>(ph, g.DX, Mc);
    // isotropic part, axis by axis (see the file comment)
    const float kf = gam2 * g.inv_dx * g.inv_dx;
#pragma unroll
    for (int D = 0; D < 3; ++D) {
      F2 nb[NP], S = f2s(0.0f), X = f2s(0.0f);   // (low halves: w, high halves: u)
      float Y = 0.0f;
#pragma unroll
      for (int a = 0; a < NP; ++a) {
        nb[a] = f2(s[a * fs - o[D]], s[a * fs + o[D]]);
        const F2 d = nb[a] - f2s(ph[a]);
        S = fma2(d, d, S);
        X = fma2(d, f2s(ph[a]), X);
        Y += f2lo(d) * f2hi(d);
      }
      const float Xw = f2lo(X), Xu = f2hi(X), S2 = f2lo(S) + f2hi(S);
      const float V = 0.25f * (Xu - Xw), T = 0.25f * S2 - 0.5f * Y;
      const F2 wd = f2(kf * ((p2s + 0.5f * Xw) - V), kf * ((p2s + 0.5f * Xu) + V));
      const float wc = -kf * (((Xu + Xw) + 0.5f * S2) + T);
#pragma unroll
      for (int a = 0; a < NP; ++a) {
        const F2 d = (nb[a] - f2s(ph[a])) * wd;
        dg[a] += (f2lo(d) + f2hi(d)) + ph[a] * wc;
      }
      if constexpr (!GG) {
        // mu fluxes through the two faces (mobility_pair's form)
        F2 e1n = nb[0], e2n = f2s(0.0f), run = nb[0], Mn[NM * NM];
#pragma unroll
        for (int a = 1; a < NP; ++a) {
          e1n = e1n + nb[a];
          e2n = fma2(nb[a], run, e2n);
          run = run + nb[a];
        }
#pragma unroll
        for (int a = 0; a < NP; ++a) {
          const F2 rest = e2n - nb[a] * (e1n - nb[a]);
          const F2 q2 = nb[a] * nb[a];
          const F2 h = f2s(3.0f) * q2 - f2s(2.0f) * q2 * nb[a] + f2s(2.0f) * nb[a] * rest;
#pragma unroll
          for (int k = 0; k < NM * NM; ++k) Mn[k] = a == 0 ? h * f2s(g.DX[0][k]) : fma2(h, f2s(g.DX[a][k]), Mn[k]);
        }
#pragma unroll
        for (int k = 0; k < NM; ++k)
#pragma unroll
          for (int j = 0; j < NM; ++j) {
            const F2 Mf = f2s(0.5f) * (f2s(Mc[k * NM + j]) + Mn[k * NM + j]);
            const F2 dm = f2(s[(NP + j) * fs - o[D]], s[(NP + j) * fs + o[D]]) - f2s(mc[j]);
            dv[k] = fma2(Mf, dm * f2s(g.inv_dx2), dv[k]);
          }
      }
    }
    if constexpr (ANISO) {
      // anisotropic pairs: a run-time loop (indices of phases are data, so the
      // sums live in shared memory, one column per lane)
#pragma unroll
      for (int a = 0; a < NP; ++a) s_dg[wid][a][lane] = dg[a];
      __syncwarp();
      int last = -1;
      bool hb = false;
      Edge19 vb;
      for (int k = 0; k < g.n_apairs; ++k) {
        const int a = g.apair[k][0], b = g.apair[k][1], p = g.apair[k][2];
        // a phase absent from every lane's neighbourhood: q = 0 on every face
        // (the list is sorted by b: the grains share the liquid's values)
        if (b != last) {
          hb = __any_sync(0xffffffffu, load19(s + b * fs, o, vb));
          last = b;
        }
        if (!hb) continue;
        Edge19 va;
        const bool ha = load19(s + a * fs, o, va);
        if (!__any_sync(0xffffffffu, ha)) continue;
        float da = 0.0f, db = 0.0f;
        const float del = g.delta[p];
        pair_faces<0>(va, vb, gam2, del, g.rot[p], g.inv_dx, g.quarter_inv_dx, da, db);
        pair_faces<1>(va, vb, gam2, del, g.rot[p], g.inv_dx, g.quarter_inv_dx, da, db);
        pair_faces<2>(va, vb, gam2, del, g.rot[p], g.inv_dx, g.quarter_inv_dx, da, db);
        float Ga = 0.0f, Gb = 0.0f;
        {
          float ca[3], cb[3];
          F2 q[3], xs[3];
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            ca[d] = (va.p[d] - va.m[d]) * g.half_inv_dx;
            cb[d] = (vb.p[d] - vb.m[d]) * g.half_inv_dx;
            q[d] = f2s(va.c * cb[d] - vb.c * ca[d]);
          }
          aniso_excess<-1>(q, gam2, del, g.rot[p], xs);
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            Ga += f2lo(xs[d]) * cb[d];
            Gb -= f2lo(xs[d]) * ca[d];
          }
        }
        s_dg[wid][a][lane] += da - Ga;
        s_dg[wid][b][lane] += db - Gb;
      }
      __syncwarp();
#pragma unroll
      for (int a = 0; a < NP; ++a) dg[a] = s_dg[wid][a][lane];
    }
    // potential derivative, driving force, rate, projection (phase_update's
    // terms with the sums over the other phases taken as total minus own)
    const float sT = g.tz0 + g.tzg * (float(z + g.zorg) + 0.5f);
    float pn[NP], mn[NM];
    {
      const float cw = g.cw[0][1];
      float psi[NP], A1 = 0.0f, A2 = 0.0f;
      if constexpr (!GG) {
#pragma unroll
        for (int a = 0; a < NP; ++a) psi[a] = grand_potential<NP, NM, float>(g, a, mc, sT);
        if (g.elw) {
          const unsigned long long cells = (unsigned long long)g.nx * g.ny * g.nz;
          const unsigned long long cell = ((unsigned long long)z * g.ny + y) * g.nx + min(x, g.nx - 1);
          add_elastic<NP, NM, float, float>(g, cell, cells, psi);
        }
#pragma unroll
        for (int a = 0; a < NP; ++a) {
          A1 += psi[a] * ph[a];
          A2 += psi[a] * (ph[a] * ph[a]);
        }
      }
      float e2 = 0.0f, run = ph[0];
      if constexpr (!GG) {
#pragma unroll
        for (int a = 1; a < NP; ++a) {
          e2 += ph[a] * run;
          run += ph[a];
        }
      }
      float v[NP];
#pragma unroll
      for (int a = 0; a < NP; ++a) {
        const float q2 = ph[a] * ph[a], others = e1 - ph[a];
        const float W = g.potential == 1 ? cw * others : cw * (ph[a] * (p2s - q2));
        float P = 0.0f;
        if constexpr (!GG) {
          const float rest = e2 - ph[a] * others;
          P = psi[a] * (6.0f * ph[a] - 6.0f * q2 + 2.0f * rest);
          P += 2.0f * (others * (A1 - psi[a] * ph[a]) - (A2 - psi[a] * q2));
        }
        const float rate = g.mob * ((g.eps * dg[a] - W * g.inv_eps - P) * g.inv_eps);
        v[a] = ph[a] + g.dt * rate;
        if (g.noise_amp != 0.0f && ph[a] > 0.0f && ph[a] < 1.0f)
          v[a] += g.dt * g.noise_amp *
                  noise_variate<float>(g.noise_seed, g.step, lab_cell<3>(g, min(x, g.nx - 1), y, z) * NP + a);
      }
      if (g.potential == 1) {
        const float theta = simplex_shift<NP>(v);
#pragma unroll
        for (int a = 0; a < NP; ++a) {
          const float d = v[a] - theta;
          pn[a] = d > 0.0f ? d : 0.0f;
        }
      } else {
        project<NP>(g.potential, v, pn);
      }
    }
    if constexpr (GG) {   // grain growth: mu held
#pragma unroll
      for (int k = 0; k < NM; ++k) mn[k] = mc[k];
    } else {
      float div[NM];
#pragma unroll
      for (int k = 0; k < NM; ++k) div[k] = f2lo(dv[k]) + f2hi(dv[k]);
      mu_update<NP, NM, float>(g, ph, pn, mc, div, sT, false, mn);
    }
    uint32_t nzm = 0, one = 0;
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      nzm |= (pn[a] != 0.0f ? 1u : 0u) << a;
      one |= (pn[a] == 1.0f ? 1u : 0u) << a;
    }
    const int code = (__popc(nzm) == 1 && nzm == one) ? __ffs(nzm) : 0;
    if (active) store_cell<3>(g, x, y, z, pn, mn);
    const int ref = __shfl_sync(0xffffffffu, code, 0);
    const bool same = __all_sync(0xffffffffu, !active || code == ref);
    if (lane == 0) {
      const long long ci = ((long long)(z + g.zoff) * g.ny + y) * g.segs + sg;
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
