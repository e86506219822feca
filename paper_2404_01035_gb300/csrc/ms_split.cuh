// Split 3-D step (FP32): a streaming kernel that updates every 32-cell row
// segment whose stencil lies in one pure phase, and lists the others for the
// interface kernel, which applies the full cell update (Sec. 2.1) to them.
//
// Bulk rows (MICROSIM paper, arXiv 2404.01035, Sec. 2.1 with a single
// phase present): every q_ab vanishes and the projection keeps the vertex,
// so phi^{n+1} = phi^n, and the mu update of Eq. (Mu_explicit_temperature)
// reduces to the constant-coefficient form mu + Kb_l Lap(mu) - eb_l with
// M = D^l chi^l, chi = chi^l and dh = 0.  The streaming kernel therefore
// reads only mu (phi is the pure phase the segment codes name) and writes phi
// only where the output buffer does not already hold it.
#pragma once

#include "ms_step.cuh"

namespace msgb {

// ---------------------------------------------------------------- streaming
// A CTA takes a tile of 128 x TY cells through `zchunk` planes, a warp per row
// and 4 consecutive cells per lane; a producer warp streams the mu planes of
// the tile through a TMA ring.  While the first planes are on their way the CTA
// reads the segment codes of its block (its planes, rows and segments with one
// of each on either side) and derives a flag per segment: the pure phase + 1
// when the 3 x 3 x 3 segments around it hold that phase alone, else 0, in which
// case the segment goes on the interface list.  Then each warp with bulk
// segments marches in z: the plane below and the plane itself stay in
// registers, the plane above and the two rows beside come from the ring, the x
// neighbours by shuffle.
//
// What bounds it: DRAM (mu in and out) and instruction issue.  Measured on a
// GB300, with flags, list places and ghost images in the march / here: 66 / 66 us
// at 256^3 with 3 phases and 2 solutes, 374 / 330 us at 512^3 and 64 / 21 us at
// 192^3 (all interface) with 8 phases and 1 solute.  The same march on plain
// loads one plane ahead in registers, without the ring: 75, 331 and 17 us.
template <int NP, int NM, int TY>
struct StreamShape {
  static constexpr int VEC = 4;                   // cells per lane (float4)
  static constexpr int TX = 32 * VEC;             // cells per warp row
  static constexpr int WCS = TX / 32;             // 32-cell segments per warp row
  static constexpr int H = 4;                     // 16-byte halo of the TMA box
  static constexpr int SX = TX + 2 * H;
  static constexpr int SY = TY + 2;
  static constexpr int NT = 32 * TY;              // consumer threads
  static constexpr int NTHREADS = NT + 32;
  static constexpr int FSTRIDE = SY * SX;         // elements per field in a stage
  static constexpr int STAGE_BYTES = NM * FSTRIDE * 4;
  static constexpr int STAGE_STRIDE = (STAGE_BYTES + 127) / 128 * 128;
  static constexpr int NST_RAW = (44 * 1024) / STAGE_STRIDE;   // 4 CTAs per SM
  static constexpr int NST = NST_RAW < 4 ? 4 : (NST_RAW > 12 ? 12 : NST_RAW);
  static constexpr int CSEG = WCS + 2;
  static constexpr int MAXE = kMaxZChunk + 2;     // ring entries at most
  static constexpr int NCOEF = NM * NM + NM;      // Kb_l and eb_l of one phase
  static constexpr int OFF_CODE = NST * STAGE_STRIDE;
  static constexpr int OFF_ROW = OFF_CODE + (MAXE * SY * CSEG + 15) / 16 * 16;
  static constexpr int OFF_FLAG = OFF_ROW + (MAXE * SY * WCS + 15) / 16 * 16;
  static constexpr int OFF_COEF = OFF_FLAG + (kMaxZChunk * TY * WCS + 15) / 16 * 16;
  static constexpr int OFF_BAR = OFF_COEF + (NP * NCOEF * 4 + 15) / 16 * 16;
  static constexpr int OFF_ABORT = OFF_BAR + 2 * NST * 8;
  static constexpr int SMEM_BYTES = OFF_ABORT + 16 + 128;
  static constexpr int MIN_BLOCKS = 4;
};

// Four cells' worth of one field.
__device__ __forceinline__ void stg4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }

//
// RAGGED: rows that are no multiple of 4 cells, whose last lane stores cell by
// cell (the others keep the shorter code: 66 against 69 us at 256^3).  Listing
// every segment cut by a row's end instead cost the interface kernel 11 of 54 us
// at 150x133x97.
template <int NP, int NM, int TY, bool RAGGED>
__global__ void __launch_bounds__(StreamShape<NP, NM, TY>::NTHREADS, StreamShape<NP, NM, TY>::MIN_BLOCKS)
    k_gp_stream(const __grid_constant__ CUtensorMap tm, const __grid_constant__ StepArgs<float, NP, NM> g) {
  using Sh = StreamShape<NP, NM, TY>;
  constexpr int NST = Sh::NST;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  uint8_t* const s_code = smem + Sh::OFF_CODE;
  uint8_t* const s_row = smem + Sh::OFF_ROW;
  uint8_t* const s_flag = smem + Sh::OFF_FLAG;
  float* const s_coef = reinterpret_cast<float*>(smem + Sh::OFF_COEF);
  uint64_t* const full = reinterpret_cast<uint64_t*>(smem + Sh::OFF_BAR);
  uint64_t* const empty = full + NST;
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(smem + Sh::OFF_ABORT);
  auto stage = [&](int i) { return reinterpret_cast<float*>(smem + i * Sh::STAGE_STRIDE); };
  const int tid = threadIdx.x, lane = tid & 31, ty = tid >> 5;
  const int tiles_x = (g.nx + Sh::TX - 1) / Sh::TX;
  const int x0 = (blockIdx.x % tiles_x) * Sh::TX;
  const int y0 = (blockIdx.x / tiles_x) * TY;
  const int zb = blockIdx.y * g.zchunk;
  const int nk = min(g.nz, zb + g.zchunk) - zb;   // planes of this CTA
  const int nplanes = nk + 2;                     // ring entries j <-> plane zb - 1 + j
  if (nk > kMaxZChunk) {   // the host clamps z-chunks; never touch smem beyond its size
    if (tid == 0) atomicOr(g.status, kStatusLaunch);
    return;
  }
  // the first ring entries
  const int npre = nplanes < NST ? nplanes : NST;
  auto load = [&](int j) {   // by one thread
    const int i = j % NST;
    mbar_expect_tx(&full[i], Sh::STAGE_BYTES);
    tma_load_4d(stage(i), &tm, &full[i], x0 + g.xoff - Sh::H, y0, zb - 1 + j + g.zoff, 0);
  };
  if (tid == Sh::NT) {
    for (int i = 0; i < NST; ++i) mbar_init(&full[i], 1);
    *abort_flag = 0;
    mbar_fence_init();
    prefetch_tensormap(&tm);
    for (int j = 0; j < npre; ++j) load(j);
  }
  const int seg0 = x0 >> 5;
  // codes: thread (row, segment), boundary-mapped once, for planes zb - 1 + j
  {
    constexpr int PAIRS = Sh::SY * Sh::CSEG;
    constexpr int GROUPS = Sh::NTHREADS / PAIRS;
    static_assert(GROUPS >= 1, "the code preload needs one thread per (row, segment)");
    if (tid < GROUPS * PAIRS) {
      const int pr = tid % PAIRS, j0 = tid / PAIRS;
      const int k = pr % Sh::CSEG, ay = pr / Sh::CSEG;
      const long long rowoff =
          (long long)bc_map(y0 - 1 + ay, g.ny, g.bc[1]) * g.segs + bc_map(seg0 - 1 + k, g.segs, g.bc[0]);
      const long long pstride = (long long)g.ny * g.segs;
#pragma unroll 4
      for (int j = j0; j < nk + 2; j += GROUPS) {
        const int z = zb - 1 + j;
        int zz;   // as load_code: ghost code planes at internal cuts
        if (z >= 0 && z < g.nz)
          zz = z + g.zoff;
        else if (g.bc[2] == kBcHalo)
          zz = z < 0 ? 0 : g.nz + 1;
        else
          zz = bc_map(z, g.nz, g.bc[2]) + g.zoff;
        s_code[j * PAIRS + pr] = __ldg(g.codes_in + zz * pstride + rowoff);
      }
    }
    // bulk coefficients of every phase (indexed by the flag)
    for (int e = tid; e < NP * Sh::NCOEF; e += Sh::NTHREADS) {
      const int a = e / Sh::NCOEF, r = e % Sh::NCOEF;
      s_coef[e] = r < NM * NM ? g.Kb[a][r] : g.eb[a][r - NM * NM];
    }
  }
  __syncthreads();
  // rows: three adjacent segments of one pure phase
  for (int e = tid; e < (nk + 2) * Sh::SY * Sh::WCS; e += Sh::NTHREADS) {
    const int wc = e % Sh::WCS, ja = e / Sh::WCS;
    s_row[e] = (uint8_t)combine_codes(s_code + ja * Sh::CSEG + wc);
  }
  __syncthreads();
  const int reuse = g.reuse_prev ? kCodeReuse : 0;
  for (int e0 = 0; e0 < nk * TY * Sh::WCS; e0 += Sh::NTHREADS) {
    const int e = e0 + tid, wc = e % Sh::WCS, row = e / Sh::WCS % TY, k = e / (Sh::WCS * TY);
    const int y = y0 + row, seg = seg0 + wc;
    const bool inside = e < nk * TY * Sh::WCS && y < g.ny && seg < g.segs;
    int f = 0;
    if (inside) {
      const uint8_t* r = s_row + (k * Sh::SY + row) * Sh::WCS + wc;
      f = r[0];
#pragma unroll
      for (int q = 1; q < 9; ++q) f = r[((q / 3) * Sh::SY + q % 3) * Sh::WCS] == f ? f : 0;
    }
    if (e < nk * TY * Sh::WCS) {
      // bit kCodeReuse of the flag: the output buffer holds phi already (the
      // state before the input held the phase there too)
      const int reused = f != 0 ? s_code[((k + 1) * Sh::SY + row + 1) * Sh::CSEG + wc + 1] & reuse : 0;
      s_flag[e] = (uint8_t)(f | reused);
    }
    const long long ci = ((long long)(zb + k + g.zoff) * g.ny + y) * g.segs + seg;
    if (f != 0) g.codes_out[ci] = (uint8_t)(f | kCodeReuse);   // input and output pure phase l
    const bool want = inside && f == 0;
    const unsigned int i = block_append<Sh::NTHREADS>(&g.iface[0], want);
    if (want && i < g.iface_cap)
      g.iface[2 + i] = ((unsigned int)(zb + k) << (g.seg_bits + g.y_bits)) | ((unsigned int)y << g.seg_bits) |
                       (unsigned int)seg;
  }
  __syncthreads();
  // a row without bulk segments has nothing to stream; the others share the ring
  uint32_t any = 0u;
  if (tid < Sh::NT) {
    for (int k = lane; k < nk; k += 32) any |= *reinterpret_cast<const uint32_t*>(s_flag + (k * TY + ty) * Sh::WCS);
    any = __reduce_or_sync(0xffffffffu, any);
  }
  const int streaming = __syncthreads_count(lane == 0 && any != 0u);   // warps
  if (tid == 0) {
    for (int i = 0; i < NST; ++i) mbar_init(&empty[i], streaming > 0 ? streaming : 1);   // (a count is at least 1)
    mbar_fence_init();
  }
  __syncthreads();   // the last CTA-wide barrier: roles split below

  if (tid >= Sh::NT) {
    // ---------------- producer
    if (lane != 0) return;
    int issued = npre;
    bool ok = true;
    for (int j = npre; j < nplanes && streaming > 0; ++j) {
      ok = mbar_wait_bounded(&empty[j % NST], ((j / NST) - 1) & 1) && *abort_flag == 0;
      if (!ok) break;
      load(j);
      issued = j + 1;
    }
    if (!ok) {
      atomicOr(g.status, kStatusTimeout);
      *abort_flag = 1;
    }
    // nobody may be left to wait for the copies in flight (no streaming warp, or
    // an abort): see them land before this warp leaves
    if (!ok || streaming == 0)
      for (int i = 0; i < NST; ++i) {
        if (issued <= i) continue;
        const int j = i + ((issued - 1 - i) / NST) * NST;
        mbar_wait_bounded(&full[i], (j / NST) & 1);
      }
    return;
  }
  if (any == 0u) return;

  // -------------------- consumer warps: 4 cells per lane, one plane at a time
  const int xs = x0 + 4 * lane, y = y0 + ty;
  const int keep = g.nx - xs;                // cells of this lane inside the row (4 and more: all)
  const bool last = RAGGED ? keep >= 1 && keep <= 4 : keep == 4;
  const long long plane = (long long)g.nyp * g.pitch, fs = g.fstride;
  const int pitch = g.pitch;
  float* o = g.out + (long long)(zb + g.zoff) * plane + (long long)(y + 1) * pitch + xs + g.xoff;
  const bool first = xs == 0;
  const long long oxl = g.bc[0] == 3 ? g.nx : -1, oxr = g.bc[0] == 3 ? -xs - 1 : RAGGED ? keep : 4;   // images of their cells
  const bool yend = y == 0 || y == g.ny - 1;
  const bool zcut = g.bc[2] == kBcHalo;                 // internal cuts get their ghost planes from the exchange
  const int sidx = (ty + 1) * Sh::SX + Sh::H + 4 * lane;   // this lane's cells in a stage
  // a lane's cells of a row, and the x ghost images of the row's first and last
  auto put = [&](float* r, float a, float b, float e, float f) {
    if (!RAGGED || keep >= 4) {
      stg4(r, a, b, e, f);
    } else {   // the end of a ragged row
      r[0] = a;
      if (keep >= 2) r[1] = b;
      if (keep >= 3) r[2] = e;
    }
    if (first) r[oxl] = a;
    if (last) r[oxr] = !RAGGED || keep == 4 ? f : keep == 3 ? e : keep == 2 ? b : a;
  };
  float4 d[NM], c[NM];
  bool ok = mbar_wait_bounded(&full[0], 0) && mbar_wait_bounded(&full[1], 0);
  if (__all_sync(0xffffffffu, ok)) {
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      d[i] = lds4(stage(0) + i * Sh::FSTRIDE + sidx);
      c[i] = lds4(stage(1) + i * Sh::FSTRIDE + sidx);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[0]);
  }
  int s1 = 1, s2 = 2 % NST;
  uint32_t par2 = (2 / NST) & 1;
  int lk = 0;              // phase + 1 whose coefficients are loaded
  float kb[NM * NM], eb[NM];
#pragma unroll
  for (int q = 0; q < NM * NM; ++q) kb[q] = 0.0f;
#pragma unroll
  for (int q = 0; q < NM; ++q) eb[q] = 0.0f;
  for (int k = 0; k < nk; ++k, o += plane) {
    ok = ok && mbar_wait_bounded(&full[s2], par2) && *abort_flag == 0;
    if (!__all_sync(0xffffffffu, ok)) {   // the warp leaves together (shuffles below)
      if (lane == 0) {
        atomicOr(g.status, kStatusTimeout);
        *abort_flag = 1;
      }
      return;
    }
    const int z = zb + k;
    float4 u[NM], n[NM], s[NM];
    float xm[NM], xp[NM];
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      const float* const q = stage(s1) + i * Sh::FSTRIDE + sidx;
      u[i] = lds4(stage(s2) + i * Sh::FSTRIDE + sidx);
      n[i] = lds4(q - Sh::SX);
      s[i] = lds4(q + Sh::SX);
      xm[i] = __shfl_up_sync(0xffffffffu, c[i].w, 1);
      xp[i] = __shfl_down_sync(0xffffffffu, c[i].x, 1);
      if (lane == 0) xm[i] = q[-1];
      if (lane == 31) xp[i] = q[4];
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s1]);   // entry k + 1 is read: the rest of it is in registers
    const int fl = s_flag[(k * TY + ty) * Sh::WCS + (lane >> 3)];
    float L[NM][4];
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      L[i][0] = (xm[i] + c[i].y) + (n[i].x + s[i].x) + (d[i].x + u[i].x) - 6.0f * c[i].x;
      L[i][1] = (c[i].x + c[i].z) + (n[i].y + s[i].y) + (d[i].y + u[i].y) - 6.0f * c[i].y;
      L[i][2] = (c[i].y + c[i].w) + (n[i].z + s[i].z) + (d[i].z + u[i].z) - 6.0f * c[i].z;
      L[i][3] = (c[i].z + xp[i]) + (n[i].w + s[i].w) + (d[i].w + u[i].w) - 6.0f * c[i].w;
    }
    if (fl != 0 && keep > 0) {
      const int l1 = fl & kCodePhase;
      if (l1 != lk) {
        lk = l1;
        const float* cf = s_coef + (l1 - 1) * Sh::NCOEF;
#pragma unroll
        for (int q = 0; q < NM * NM; ++q) kb[q] = cf[q];
#pragma unroll
        for (int q = 0; q < NM; ++q) eb[q] = cf[NM * NM + q];
      }
      float mn[NM][4];
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        const float cv[4] = {c[i].x, c[i].y, c[i].z, c[i].w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float t = cv[q] - eb[i];
#pragma unroll
          for (int j = 0; j < NM; ++j) t += kb[i * NM + j] * L[j][q];
          mn[i][q] = t;
        }
      }
      const bool write_phi = (fl & kCodeReuse) == 0;
#pragma unroll
      for (int i = 0; i < NM; ++i) put(o + (NP + i) * fs, mn[i][0], mn[i][1], mn[i][2], mn[i][3]);
      if (write_phi) {
#pragma unroll 1
        for (int a = 0; a < NP; ++a) {
          const float v = a == l1 - 1 ? 1.0f : 0.0f;
          put(o + a * fs, v, v, v, v);
        }
      }
      if (yend || (!zcut && (z == 0 || z == g.nz - 1))) {
        // ghost images of the whole row (with those) on y and z boundaries: a
        // loop over (iz, iy), not unrolled
#pragma unroll 1
        for (int v = 1; v < 9; ++v) {
          const int iz = v / 3, iy = v % 3;
          long long off = 0;
          if (iy == 1) {
            if (y != 0) continue;
            off += (long long)(g.bc[1] == 3 ? g.ny : -1) * pitch;
          } else if (iy == 2) {
            if (y != g.ny - 1) continue;
            off += (long long)(g.bc[1] == 3 ? -g.ny : 1) * pitch;
          }
          if (iz == 1) {
            if (zcut || z != 0) continue;
            off += (g.bc[2] == 3 ? g.nz : -1) * plane;
          } else if (iz == 2) {
            if (zcut || z != g.nz - 1) continue;
            off += (g.bc[2] == 3 ? -g.nz : 1) * plane;
          }
          float* const q = o + off;
#pragma unroll
          for (int i = 0; i < NM; ++i) put(q + (NP + i) * fs, mn[i][0], mn[i][1], mn[i][2], mn[i][3]);
          if (write_phi) {
#pragma unroll 1
            for (int a = 0; a < NP; ++a) {
              const float f = a == l1 - 1 ? 1.0f : 0.0f;
              put(q + a * fs, f, f, f, f);
            }
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      d[i] = c[i];
      c[i] = u[i];
    }
    s1 = s2;
    if (++s2 == NST) {
      s2 = 0;
      par2 ^= 1u;
    }
  }
}

// Phases the compact update of the interface kernel handles (more phases
// than this around a row take the full update).
constexpr int kSparseK = 4;

// Interface kernel of the split 3-D step (shape of its shared memory).  Each
// warp owns two buffers of one TMA box: 32 + 2H cells x 3 rows x 3 planes x
// all fields around one listed 32-cell row, so the next row is in flight
// while the current one is updated.
template <int NP, int NM, class Real>
struct IfaceShape {
  static constexpr int NF = NP + NM;
  static constexpr int H = Halo<Real>::H;
  static constexpr int BX = 32 + 2 * H;                 // box extent along x
  static constexpr int BOX_ELEMS = NF * 9 * BX;
  static constexpr int BOX_BYTES = BOX_ELEMS * (int)sizeof(Real);
  static constexpr int BOX_STRIDE = (BOX_BYTES + 127) / 128 * 128;
  static constexpr int WARPS = 4;                       // warps per CTA
  static constexpr int THREADS = 32 * WARPS;
  static constexpr int OFF_BAR = WARPS * 2 * BOX_STRIDE;
  static constexpr int SMEM_BYTES = OFF_BAR + WARPS * 2 * 8 + 128;   // + alignment slack
  static constexpr int MIN_BLOCKS = NP <= 4 ? 3 : 2;
};

// Stencil accessor over one interface box ([field][plane][row][x]).
template <int DIM, int NP, int NM, class Real>
struct BoxAcc {
  using Sh = IfaceShape<NP, NM, Real>;
  const Real* s;
  const StepArgs<Real, NP, NM>* g;
  int sidx;         // centre of this lane's cell: plane 1, row 1, x = H + lane
  uint32_t wmask;   // phases present anywhere in the warp's box (a superset of
                    // each cell's stencil: absent phases then contribute exact
                    // zeros, so the update is the same as with the cell's own)

  __device__ __forceinline__ Real ld(int f, int dx, int dy, int dz) const {
    return s[f * (9 * Sh::BX) + sidx + dz * (3 * Sh::BX) + dy * Sh::BX + dx];
  }
  __device__ __forceinline__ Real phi(int a, int dx, int dy, int dz) const { return ld(a, dx, dy, dz); }
  __device__ __forceinline__ Real mu(int i, int dx, int dy, int dz) const { return ld(NP + i, dx, dy, dz); }
  __device__ __forceinline__ uint32_t mask() const { return wmask; }
  template <bool AT>
  __device__ __forceinline__ void mobility(int dx, int dy, int dz, Real* M) const {
    Real ph[NP];
#pragma unroll
    for (int a = 0; a < NP; ++a) ph[a] = phi(a, dx, dy, dz);
    cell_mobility<NP, NM, AT>(ph, g->DX, M);
  }
};

// Phases present anywhere in an interface box, OR-ed over the warp (every
// lane its own column of the 3 x 3 rows, lanes 0 and 31 also the halo column
// on their side).  Called by all lanes of the warp.
template <int NP, int NM, class Real>
__device__ __forceinline__ uint32_t box_phase_mask(const Real* box, int lane) {
  using Sh = IfaceShape<NP, NM, Real>;
  uint32_t m = 0;
  if constexpr (sizeof(Real) == 4) {
    // phase fractions are never negative: the OR of the bit patterns is
    // non-zero exactly when some value is (a -0.0 could only mark a phase
    // present, which costs work, never correctness)
    const unsigned int* bx = reinterpret_cast<const unsigned int*>(box);
    const int xh = lane == 0 ? Sh::H - 1 : Sh::H + 32;
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      unsigned int any = 0u;
#pragma unroll
      for (int r = 0; r < 9; ++r) any |= bx[a * (9 * Sh::BX) + r * Sh::BX + Sh::H + lane];
      if (lane == 0 || lane == 31) {
#pragma unroll
        for (int r = 0; r < 9; ++r) any |= bx[a * (9 * Sh::BX) + r * Sh::BX + xh];
      }
      m |= (any != 0u ? 1u : 0u) << a;
    }
  } else {
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      bool any = false;
#pragma unroll
      for (int r = 0; r < 9; ++r) any = any || box[a * (9 * Sh::BX) + r * Sh::BX + Sh::H + lane] != Real(0);
      if (lane == 0 || lane == 31) {
        const int xh = lane == 0 ? Sh::H - 1 : Sh::H + 32;
#pragma unroll
        for (int r = 0; r < 9; ++r) any = any || box[a * (9 * Sh::BX) + r * Sh::BX + xh] != Real(0);
      }
      m |= (any ? 1u : 0u) << a;
    }
  }
  return __reduce_or_sync(0xffffffffu, m);
}

// Scan of an interface box by the warp: lane = column H + lane of the 3 x 3
// rows; lanes 0..17 also take one cell of the halo column on either side
// (lanes 0..8 the left one, 9..17 the right one, row lane % 9).  Returns the
// phases present anywhere in the box (OR over the warp: a superset of every
// cell's stencil) and sets `bulk` to l + 1 when every cell of the 3 x 3 x 3
// block around the lane's cell is exactly pure phase l (phi_l = 1, all others
// 0), else 0.  Called by all lanes of the warp.
template <int NP, int NM, class Real>
__device__ __forceinline__ uint32_t box_scan(const Real* box, int lane, int& bulk) {
  using Sh = IfaceShape<NP, NM, Real>;
  uint32_t m = 0;
  // pure code of one box cell (l + 1 or 0); ORs its nonzero phases into nzm
  auto code_of = [&](int r, int x, uint32_t& nzm) {
    uint32_t nz = 0, one = 0;
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      const Real v = box[a * (9 * Sh::BX) + r * Sh::BX + x];
      nz |= (v != Real(0) ? 1u : 0u) << a;
      one |= (v == Real(1) ? 1u : 0u) << a;
    }
    nzm |= nz;
    return (__popc(nz) == 1 && nz == one) ? __ffs(nz) : 0;
  };
  int col = code_of(0, Sh::H + lane, m);   // common code of the lane's 9 cells, or 0
#pragma unroll
  for (int r = 1; r < 9; ++r) {
    const int c = code_of(r, Sh::H + lane, m);
    col = c == col ? col : 0;
  }
  uint32_t hm = 0;
  const int hc = code_of(lane % 9, lane < 9 ? Sh::H - 1 : Sh::H + 32, hm);
  if (lane < 18) m |= hm;
  const uint32_t wmask = __reduce_or_sync(0xffffffffu, m);
  const int lc = __shfl_sync(0xffffffffu, hc, 0), rc = __shfl_sync(0xffffffffu, hc, 9);
  const uint32_t lb = __ballot_sync(0xffffffffu, lane < 9 && hc == lc);
  const uint32_t rb = __ballot_sync(0xffffffffu, lane >= 9 && lane < 18 && hc == rc);
  int left = __shfl_up_sync(0xffffffffu, col, 1), right = __shfl_down_sync(0xffffffffu, col, 1);
  if (lane == 0) left = lb == 0x1FFu ? lc : 0;
  if (lane == 31) right = rb == (0x1FFu << 9) ? rc : 0;
  bulk = (col != 0 && left == col && right == col) ? col : 0;
  return wmask;
}

// Bulk update of one cell of an interface box whose 3 x 3 x 3 block is pure
// phase l (c = the cell in field 0, cf = Kb_l then eb_l): phi unchanged and
// mu + Kb_l Lap(mu) - eb_l, the form of the streaming kernel.
template <int NP, int NM, class Real>
__device__ __forceinline__ void box_bulk_mu(const Real* c, const Real* cf, Real* mn) {
  using Sh = IfaceShape<NP, NM, Real>;
  Real L[NM], mc[NM];
#pragma unroll
  for (int i = 0; i < NM; ++i) {
    const Real* f = c + (NP + i) * (9 * Sh::BX);
    const Real v = f[0];
    Real sum = (f[-1] + f[1]) + (f[-Sh::BX] + f[Sh::BX]);
    sum += f[-3 * Sh::BX] + f[3 * Sh::BX];
    L[i] = sum - Real(6) * v;
    mc[i] = v;
  }
#pragma unroll
  for (int i = 0; i < NM; ++i) {
    Real dd = mc[i] - cf[NM * NM + i];
#pragma unroll
    for (int j = 0; j < NM; ++j) dd += cf[i * NM + j] * L[j];
    mn[i] = dd;
  }
}

// Interface kernel of the split 3-D step: the full cell update of every warp
// row the streaming kernel listed (32 cells of one row of one plane per
// warp), from a TMA box of the input state; writes phi, mu, their ghost
// images and the row's segment code.  With more than kSparseK phases the
// work is shared by two launches: MODE 0 takes the rows whose box holds at
// most kSparseK phases (the compact update) and moves the others to a second
// list, which MODE 1 updates with the full one (each kernel's registers then
// fit its own path); with one gamma for every pair k_gp_rows takes all rows
// instead.  The last CTA to finish clears its list (ticket in
// list[1]), so the launches can be replayed from a CUDA graph.
template <int DIM, int NP, int NM, class Real, int MODE, int FEAT = kFeatAll>
__global__ void __launch_bounds__(IfaceShape<NP, NM, Real>::THREADS, IfaceShape<NP, NM, Real>::MIN_BLOCKS)
    k_gp_iface(const __grid_constant__ CUtensorMap tmi, const __grid_constant__ StepArgs<Real, NP, NM> g) {
  static_assert(DIM == 3, "the interface list is built by the 3-D streaming kernel");
  constexpr bool kSparse = NP > kSparseK && MODE == 0;   // compact update, defer the rest
  unsigned int* const list = MODE == 0 ? g.iface : g.iface2;
  using Sh = IfaceShape<NP, NM, Real>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  __shared__ unsigned int s_count;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + Sh::OFF_BAR) + 2 * wid;
  Real* buf0 = reinterpret_cast<Real*>(smem + (2 * wid) * Sh::BOX_STRIDE);
  if (threadIdx.x == 0) s_count = min(*(volatile unsigned int*)&list[0], g.iface_cap);
  if (MODE == 0 && g.at_list && blockIdx.x == 0 && threadIdx.x == 0)   // see the copy below
    g.at_list[0] = min(*(volatile unsigned int*)&list[0], g.at_cap);
  if (lane == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
    prefetch_tensormap(&tmi);
  }
  __syncthreads();
  const unsigned int count = s_count;
  const unsigned int stride = gridDim.x * Sh::WARPS;
  DiffPrm<Real, StepArgs<Real, NP, NM>::P> dp;
  dp.mob = g.mob;
#pragma unroll
  for (int p = 0; p < StepArgs<Real, NP, NM>::P; ++p) dp.delta[p] = g.delta[p];

  // list entry r -> (segment, y, z) (bit fields)
  const unsigned int seg_mask = (1u << g.seg_bits) - 1u, y_mask = (1u << g.y_bits) - 1u;
  const int zshift = g.seg_bits + g.y_bits;
  // row -> box origin (x, y - 1, z - 1 in padded coordinates)
  auto issue = [&](unsigned int i, int b) {
    const unsigned int r = list[2 + i];
    const int sg = (int)(r & seg_mask);
    const int y = (int)((r >> g.seg_bits) & y_mask), z = (int)(r >> zshift);
    fence_proxy_async_shared();
    mbar_expect_tx(&bar[b], Sh::BOX_BYTES);
    tma_load_4d(reinterpret_cast<unsigned char*>(buf0) + b * Sh::BOX_STRIDE, &tmi, &bar[b],
                32 * sg + g.xoff - Sh::H, y, z + g.zoff - 1, 0);
  };
  // bit b of `pending` / `phase`: buffer b has a copy in flight / the
  // parity its barrier completes next (bits, not arrays: a runtime index
  // would put them in local memory)
  uint32_t pending = 0u, phase = 0u;
  bool aborted = false;
  unsigned int i = blockIdx.x * Sh::WARPS + wid;
  if (i < count && lane == 0) issue(i, 0);
  if (i < count) pending = 1u;
  int b = 0;
  while (i < count) {
    const unsigned int nxt = i + stride;
    if (nxt < count) {
      if (lane == 0) issue(nxt, b ^ 1);
      pending |= 1u << (b ^ 1);
    }
    const bool ok = mbar_wait_bounded(&bar[b], (phase >> b) & 1u);
    if (!__all_sync(0xffffffffu, ok)) {
      aborted = true;
      break;
    }
    pending &= ~(1u << b);
    phase ^= 1u << b;
    const unsigned int r = list[2 + i];
    const int sg = (int)(r & seg_mask);
    const int y = (int)((r >> g.seg_bits) & y_mask), z = (int)(r >> zshift);
    // with the anti-trapping current on, its correction works on the same
    // segments (those whose block of segments is not one pure phase in phi^n):
    // the list is copied, by linear segment index, at the same positions
    if (MODE == 0 && g.at_list && lane == 0 && i < g.at_cap)
      g.at_list[2 + i] = (unsigned int)(((long long)z * g.ny + y) * g.segs + sg);
    const int x = 32 * sg + lane;
    const bool active = x < g.nx;
    const Real* box = reinterpret_cast<const Real*>(reinterpret_cast<unsigned char*>(buf0) + b * Sh::BOX_STRIDE);
    uint32_t wmask;
    if constexpr (kSparse) {
      // many phases: rows whose cells all have a pure 3 x 3 x 3 block (listed
      // only because a segment next to them is not pure) take the bulk update
      int bk = 0;
      wmask = box_scan<NP, NM, Real>(box, lane, bk);
      if (__all_sync(0xffffffffu, !active || bk != 0)) {
        if (active) {
          Real pn[NP], mn[NM], cf[NM * NM + NM];
#pragma unroll
          for (int a = 0; a < NP; ++a) pn[a] = a == bk - 1 ? Real(1) : Real(0);
#pragma unroll
          for (int k = 0; k < NM * NM; ++k) cf[k] = g.Kb[bk - 1][k];
#pragma unroll
          for (int k = 0; k < NM; ++k) cf[NM * NM + k] = g.eb[bk - 1][k];
          box_bulk_mu<NP, NM, Real>(box + 4 * Sh::BX + Sh::H + lane, cf, mn);
          store_cell<DIM>(g, x, y, z, pn, mn);
        }
        const int ref = __shfl_sync(0xffffffffu, bk, 0);
        const bool same = __all_sync(0xffffffffu, !active || bk == ref);
        if (lane == 0) {
          const long long ci = ((long long)(z + g.zoff) * g.ny + y) * g.segs + sg;
          int c = same ? ref : 0;
          if (c != 0 && (g.codes_in[ci] & kCodePhase) == c) c |= kCodeReuse;   // pure before and after
          g.codes_out[ci] = (uint8_t)c;
        }
        __syncwarp();
        b ^= 1;
        i = nxt;
        continue;
      }
    } else {
      wmask = box_phase_mask<NP, NM, Real>(box, lane);
    }
    if constexpr (kSparse) {
      if (__popc(wmask) > kSparseK) {   // for the MODE 1 launch
        if (lane == 0) {
          const unsigned int k = atomicAdd(&g.iface2[0], 1u);
          if (k < g.iface_cap) g.iface2[2 + k] = r;
        }
        __syncwarp();
        b ^= 1;
        i = nxt;
        continue;
      }
    }
    int code = 0;
    if (active) {
      BoxAcc<DIM, NP, NM, Real> acc;
      acc.s = box;
      acc.g = &g;
      acc.sidx = 3 * Sh::BX + Sh::BX + Sh::H + lane;
      acc.wmask = wmask;
      Real pn[NP], mn[NM];
      if constexpr (kSparse)   // many phases, at most kSparseK of them around this row
        gp_cell_sparse<DIM, NP, NM, kSparseK, Real, BoxAcc<DIM, NP, NM, Real>, FEAT>(acc, g, z + g.zorg,
                                                                                   lab_cell<DIM>(g, x, y, z), pn, mn);
      else
        gp_cell<DIM, NP, NM, Real, Real, BoxAcc<DIM, NP, NM, Real>, FEAT>(acc, g, dp, z + g.zorg,
                                                                         lab_cell<DIM>(g, x, y, z), pn, mn);
      uint32_t nzm = 0, one = 0;
#pragma unroll
      for (int a = 0; a < NP; ++a) {
        nzm |= (pn[a] != Real(0) ? 1u : 0u) << a;
        one |= (pn[a] == Real(1) ? 1u : 0u) << a;
      }
      code = (__popc(nzm) == 1 && nzm == one) ? __ffs(nzm) : 0;
      store_cell<DIM>(g, x, y, z, pn, mn);
    }
    const int ref = __shfl_sync(0xffffffffu, code, 0);
    const bool same = __all_sync(0xffffffffu, !active || code == ref);
    if (lane == 0) {
      const long long ci = ((long long)(z + g.zoff) * g.ny + y) * g.segs + sg;
      int c = same ? ref : 0;
      if (c != 0 && (g.codes_in[ci] & kCodePhase) == c) c |= kCodeReuse;   // pure before and after
      g.codes_out[ci] = (uint8_t)c;
    }
    __syncwarp();   // every lane is done with buffer b before it is refilled
    b ^= 1;
    i = nxt;
  }
  if (aborted) {
    // a copy did not complete in time: record it and wait (bounded) for the
    // copies still in flight before the CTA exits
    if (lane == 0) {
      atomicOr(g.status, kStatusTimeout);
      for (int k = 0; k < 2; ++k)
        if ((pending >> k) & 1u) mbar_wait_bounded(&bar[k], (phase >> k) & 1u);
    }
  }
  // every CTA read the count before taking its ticket
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
