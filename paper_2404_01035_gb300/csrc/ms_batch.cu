// Batched form: hundreds of independent 2-D simulations of different sizes
// and parameters advanced by ONE persistent, cooperative kernel launch
// (captured once into a CUDA graph and replayed).
//
// A step has two phases with a grid-wide barrier (atomic counter, bounded spin
// on %globaltimer) after each.  In the first, a warp per strip of 128 x R cells
// (work list of precomputed descriptors, a contiguous range per CTA) updates
// the segments whose 3 x 3 block of segment codes is one pure phase, which
// touches mu alone (PlaneStrip, as in the split 2-D step), and lists the others.
// In the second, a warp per listed 32-cell segment of any simulation stages its
// 3 x 34 cells and takes the full cell update.  The list spreads the interface
// rows, which cost many times a bulk row, over all warps.  Reads go past L1:
// the rows are other SMs' stores of the previous phase.
//
// What bounds it: the two barriers and the latency of each phase.  32 simulations
// of 64^2 .. 512^2 (3.2 M cells) on a GB300: 20.4 us a step; 60 us with every tile
// staged through a TMA ring, a cell per thread, and phi tested cell by cell.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/microsim_gb.h"
#include "ms_launch.cuh"
#include "ms_rt.h"
#include "ms_strip.cuh"
#include "ms_trace.h"

namespace msgb {

ms_status build_model(ms_ctx* c, const ms_grid* g, int N, int K, const ms_params* p, HostModel& m);

// Per-simulation constants for one buffer parity (out points at the
// destination of a step that reads the other buffer).
template <class Real, int NP, int NM>
struct alignas(64) BatchSim {
  StepArgs<Real, NP, NM> g[2];   // [parity of the source buffer]
  const Real* in[2];             // the source buffer
};

// One work item: simulation, strip (128 cells wide) and first row.
struct alignas(16) BatchItem {
  int sim, sx, y0, pad;
};

// A listed row segment: simulation, (y << seg_bits) | segment.
struct alignas(8) BatchRow {
  unsigned int sim, row;
};

// What a strip reads of a simulation's arguments, copied to shared memory (the
// arguments themselves lie in global memory, where every store might alias them).
template <int NP, int NM>
struct StripArgs {
  long long fstride;
  const uint8_t* codes_in;
  uint8_t* codes_out;
  float* out;
  const float* in;
  int nx, ny, pitch, xoff, segs, reuse_prev, seg_bits;
  int bc[3];
  float Kb[NP][NM * NM], eb[NP][NM];
};

template <int R>
struct BatchShape {
  static constexpr int WARPS = 4;
  static constexpr int THREADS = 32 * WARPS;
  static constexpr int MIN_BLOCKS = R <= 8 ? 5 : 4;
};

// counters: [0] barrier arrivals, [1 + (step & 1)] rows listed by the step;
// all zero at the launch.
template <int NP, int NM, int R>
__global__ void __launch_bounds__(BatchShape<R>::THREADS, BatchShape<R>::MIN_BLOCKS)
    k_batch(const BatchSim<float, NP, NM>* __restrict__ sims, const BatchItem* __restrict__ items, int nitems,
            BatchRow* rows, int nsteps, int parity0, unsigned int* counters, int* status) {
  using Bs = BatchShape<R>;
  using Strip = PlaneStrip<NP, NM, R, true>;
  using Ms = MultiShape<NP, NM, float>;
  __shared__ StripArgs<NP, NM> s_args[Bs::WARPS];
  __shared__ uint8_t s_code[Bs::WARPS][Strip::CODES];
  __shared__ float s_box[Bs::WARPS][Ms::BOX];
  __shared__ int s_ok;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  StripArgs<NP, NM>& a = s_args[wid];
  float* const box = s_box[wid];
  const int per = (nitems + (int)gridDim.x - 1) / (int)gridDim.x;
  const int ibeg = min(nitems, (int)blockIdx.x * per), iend = min(nitems, ibeg + per);
  auto barrier = [&](unsigned int round) {
    __syncthreads();
    if (threadIdx.x == 0) {
      s_ok = multi_barrier(&counters[0], round * gridDim.x) ? 1 : 0;
      if (!s_ok) atomicOr(status, kStatusTimeout);
    }
    __syncthreads();
    return s_ok != 0;
  };
  for (int step = 0; step < nsteps; ++step) {
    const int par = (parity0 + step) & 1;
    unsigned int* const listed = &counters[1 + (step & 1)];
    // ---- bulk
    int cur = -1;
    for (int k = ibeg + wid; k < iend; k += Bs::WARPS) {
      const BatchItem it = items[k];
      if (it.sim != cur) {
        cur = it.sim;
        __syncwarp();
        if (lane == 0) {
          const StepArgs<float, NP, NM>& g = sims[cur].g[par];
          a.fstride = g.fstride;
          a.codes_in = g.codes_in;
          a.codes_out = g.codes_out;
          a.out = g.out;
          a.in = sims[cur].in[par];
          a.nx = g.nx;
          a.ny = g.ny;
          a.pitch = g.pitch;
          a.xoff = g.xoff;
          a.segs = g.segs;
          a.reuse_prev = g.reuse_prev;
          a.seg_bits = g.seg_bits;
#pragma unroll
          for (int d = 0; d < 3; ++d) a.bc[d] = g.bc[d];
#pragma unroll
          for (int p = 0; p < NP; ++p) {
#pragma unroll
            for (int q = 0; q < NM * NM; ++q) a.Kb[p][q] = g.Kb[p][q];
#pragma unroll
            for (int q = 0; q < NM; ++q) a.eb[p][q] = g.eb[p][q];
          }
        }
        __syncwarp();
      }
      Strip st;
      st.flags(a, it.sx, it.y0, lane, s_code[wid]);
      st.list(listed, lane, [&](unsigned int at, int r) {
        __stcg(reinterpret_cast<uint2*>(rows) + at,
               make_uint2((unsigned int)it.sim,
                          ((unsigned int)(it.y0 + r) << a.seg_bits) | (unsigned int)(4 * it.sx + (lane >> 3))));
      });
      st.update(a, a.in, it.sx, it.y0, lane, s_code[wid]);
      __syncwarp();
    }
    if (!barrier(2u * step + 1u)) break;
    // ---- interface rows
    if (blockIdx.x == 0 && threadIdx.x == 0) counters[1 + ((step + 1) & 1)] = 0u;   // last read a phase ago
    const unsigned int count = __ldcg(listed);
    for (unsigned int k = wid * gridDim.x + blockIdx.x; k < count; k += gridDim.x * Bs::WARPS) {
      const uint2 e = __ldcg(reinterpret_cast<const uint2*>(rows) + k);
      const StepArgs<float, NP, NM>& g = sims[e.x].g[par];
      const float* in = sims[e.x].in[par];
      const int nx = g.nx, sg = (int)(e.y & ((1u << g.seg_bits) - 1u)), y = (int)(e.y >> g.seg_bits);
      const int x = 32 * sg + lane;
      const bool active = x < nx;
      // columns 32 sg - 1 .. 32 sg + 32 (never past the ghost column nx)
      const float* row = in + (long long)y * g.pitch + 32 * sg - 1 + g.xoff;
      const int c0 = min(lane, nx - 32 * sg + 1), c1 = min(lane + 32, nx - 32 * sg + 1);
#pragma unroll
      for (int f = 0; f < Ms::NF; ++f)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const float* p = row + f * g.fstride + (long long)q * g.pitch;
          box[(f * 3 + q) * Ms::BX + lane] = __ldcg(p + c0);
          if (lane < 2) box[(f * 3 + q) * Ms::BX + 32 + lane] = __ldcg(p + c1);
        }
      __syncwarp();
      int code = 0;
      if (active) {
        MultiAcc<NP, NM, float> acc;
        acc.s = box + Ms::BX + lane + 1;
        acc.g = &g;
        acc.tz0 = g.tz0;
        DiffPrm<float, StepArgs<float, NP, NM>::P> dp;
        dp.mob = g.mob;
#pragma unroll
        for (int p = 0; p < StepArgs<float, NP, NM>::P; ++p) dp.delta[p] = g.delta[p];
        float pn[NP], mn[NM];
        gp_cell<2, NP, NM, float, float, MultiAcc<NP, NM, float>, kFeatNoAt>(acc, g, dp, y + g.zorg, 0ull, pn, mn);
        uint32_t nzm = 0, one = 0;
#pragma unroll
        for (int q = 0; q < NP; ++q) {
          nzm |= (pn[q] != 0.0f ? 1u : 0u) << q;
          one |= (pn[q] == 1.0f ? 1u : 0u) << q;
        }
        code = (__popc(nzm) == 1 && nzm == one) ? __ffs(nzm) : 0;
        store_cell<2>(g, x, y, 0, pn, mn);
      }
      const int ref = __shfl_sync(0xffffffffu, code, 0);
      const bool same = __all_sync(0xffffffffu, !active || code == ref);
      if (lane == 0) {
        const long long ci = (long long)y * g.segs + sg;
        int c = same ? ref : 0;
        if (c != 0 && (__ldcg(g.codes_in + ci) & kCodePhase) == c) c |= kCodeReuse;   // pure before and after
        g.codes_out[ci] = (uint8_t)c;
      }
      __syncwarp();
    }
    if (step + 1 < nsteps && !barrier(2u * step + 2u)) break;
  }
}

// The same steps for batches whose strips would be few: a warp per 32-cell
// segment of any simulation (item: simulation, segment, row), as k_gp_multi, with
// one barrier a step and no codes.
template <int NP, int NM>
__global__ void __launch_bounds__(MultiShape<NP, NM, float>::THREADS)
    k_batch_units(const BatchSim<float, NP, NM>* __restrict__ sims, const BatchItem* __restrict__ items, int nitems,
                  int nsteps, int parity0, unsigned int* counters, int* status) {
  using Sh = MultiShape<NP, NM, float>;
  __shared__ float s_box[Sh::WARPS][Sh::BOX];
  __shared__ int s_ok;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float* const box = s_box[wid];
  for (int step = 0; step < nsteps; ++step) {
    const int par = (parity0 + step) & 1;
    for (int k = wid * gridDim.x + blockIdx.x; k < nitems; k += gridDim.x * Sh::WARPS) {
      const BatchItem it = items[k];
      const StepArgs<float, NP, NM>& g = sims[it.sim].g[par];
      MultiAcc<NP, NM, float> acc;
      acc.g = &g;
      acc.tz0 = g.tz0;
      DiffPrm<float, StepArgs<float, NP, NM>::P> dp;
      dp.mob = g.mob;
#pragma unroll
      for (int p = 0; p < StepArgs<float, NP, NM>::P; ++p) dp.delta[p] = g.delta[p];
      const int flag = stage_unit<NP, NM, float>(g, sims[it.sim].in[par], box, lane, it.sx, it.y0);
      update_unit(g, acc, dp, box, g.out, lane, it.sx, it.y0, flag);
      __syncwarp();
    }
    if (step + 1 == nsteps) break;
    __syncthreads();
    if (threadIdx.x == 0) {
      s_ok = multi_barrier(&counters[0], (unsigned int)(step + 1) * gridDim.x) ? 1 : 0;
      if (!s_ok) atomicOr(status, kStatusTimeout);
    }
    __syncthreads();
    if (!s_ok) break;
  }
}

}  // namespace msgb

using namespace msgb;

struct ms_batch {
  bool units = false;                   // steps by k_batch_units
  bool units_fit = false;               // few enough cells for it
  bool codes_ok = true;                 // the segment codes describe the states (k_batch_units keeps none)
  int nsims = 0, N = 0, NM = 0, dtype = 0;
  std::vector<HostModel> models;
  std::vector<size_t> off;              // byte offset of each simulation's two state buffers
  std::vector<size_t> sbytes;           // state bytes per simulation (one buffer)
  std::vector<size_t> coff;             // byte offset of its two segment-code arrays
  size_t total = 0;                     // bytes of states and codes
  void* state = nullptr;                // all state buffers, then all codes
  void* stage = nullptr;                // dense fields of the largest simulation, on their way to or from the host
                                        // (NULL: strided copies)
  void* sims = nullptr;                 // BatchSim array (device)
  BatchItem* items = nullptr;
  int nitems = 0;
  BatchRow* rows = nullptr;             // interface rows of a step (room for every row segment)
  unsigned int* barrier = nullptr;      // counters of the kernel (see k_batch)
  int* status = nullptr;
  int parity = 0;                       // buffer holding the current state
  int64_t steps_done = 0;
  cudaStream_t stream = nullptr;
  AllocHook hook;
  int grid = 0;
  int ty = 0;                           // rows of a strip (kBTYs)
  cudaGraphExec_t graph = nullptr;
  int64_t graph_n = -1;
  std::string err;
};

namespace {

// Strips are 128 cells wide; their height is chosen at run time among the
// compiled ones (ms_batch_set_tile / ms_batch_tune).
constexpr int kBTY = 8;
constexpr int kBTYs[] = {4, 8, 16};
constexpr int kNBTY = 3;

// Cells of all simulations up to which a batch steps by units: below, the strips'
// two phases and barriers dominate (us a step on a GB300, units / strips: 8 x 64^2
// 4.7 / 14.0, 30 x 77^2 10.8 / 15.9, 8 x 200^2 11.5 / 13.9, 2 x 512^2 14.6 / 13.1,
// 4 x 400^2 17.8 / 13.5, 64 x 128^2 31.0 / 20.8).
constexpr long long kBatchUnitCells = 400000;

void* batch_kernel_for(bool units, int ty) {
  return units      ? reinterpret_cast<void*>(k_batch_units<2, 1>)
         : ty == 4  ? reinterpret_cast<void*>(k_batch<2, 1, 4>)
         : ty == 16 ? reinterpret_cast<void*>(k_batch<2, 1, 16>)
                    : reinterpret_cast<void*>(k_batch<2, 1, 8>);
}

uint8_t* codes_of(const ms_batch* b, int sim, int par) {
  return static_cast<uint8_t*>(b->state) + b->coff[sim] + par * code_bytes(b->models[sim]);
}

ms_status bfail(ms_batch* b, ms_status s, const std::string& m) {
  if (b) b->err = m;
  return fail(nullptr, s, m);
}

void batch_free(ms_batch* b) {
  if (!b) return;
  if (b->stream) cudaStreamSynchronize(b->stream);
  if (b->graph) cudaGraphExecDestroy(b->graph);
  dev_free(b->hook, b->state);
  dev_free(b->hook, b->stage);
  dev_free(b->hook, b->sims);
  dev_free(b->hook, b->items);
  dev_free(b->hook, b->rows);
  dev_free(b->hook, b->barrier);
  delete b;
}

cudaError_t launch_batch(ms_batch* b, int64_t n) {
  cudaError_t e = cudaMemsetAsync(b->barrier, 0, 4 * sizeof(unsigned int), b->stream);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(b->grid);
  cfg.blockDim = dim3(BatchShape<kBTY>::THREADS);
  cfg.stream = b->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const BatchSim<float, 2, 1>* sims = (const BatchSim<float, 2, 1>*)b->sims;
  const BatchItem* items = b->items;
  if (b->units)
    return cudaLaunchKernelEx(&cfg, k_batch_units<2, 1>, sims, items, b->nitems, (int)n, b->parity, b->barrier, b->status);
  auto kern = b->ty == 4 ? k_batch<2, 1, 4> : b->ty == 16 ? k_batch<2, 1, 16> : k_batch<2, 1, 8>;
  return cudaLaunchKernelEx(&cfg, kern, sims, items, b->nitems, b->rows, (int)n, b->parity, b->barrier, b->status);
}

// Work list and persistent grid for strips of ty rows (one of kBTYs), or for
// units: items are (simulation, strip or segment) pairs in simulation order.  Drops
// the captured graph.
cudaError_t batch_set_tiles(ms_batch* b, int ty, bool units) {
  std::vector<BatchItem> items;
  for (int i = 0; i < b->nsims; ++i) {
    const HostModel& m = b->models[i];
    for (int y0 = 0; y0 < m.ny; y0 += units ? 1 : ty)
      for (int sx = 0; (units ? 32 : 128) * sx < m.nx; ++sx) items.push_back(BatchItem{i, sx, y0, 0});
  }
  cudaError_t e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return e;
  BatchItem* dev_items = static_cast<BatchItem*>(dev_alloc(b->hook, sizeof(BatchItem) * items.size()));
  if (!dev_items) return cudaErrorMemoryAllocation;   // (the batch keeps the list it has)
  dev_free(b->hook, b->items);
  b->items = dev_items;
  b->nitems = (int)items.size();
  if (b->graph) {   // (it reads the old list)
    cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
  }
  b->graph_n = -1;
  e = cudaMemcpyAsync(b->items, items.data(), sizeof(BatchItem) * items.size(), cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  b->ty = ty;
  b->units = units;
  int per_sm = 0, dev = 0, sms = 0;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel_for(units, ty), BatchShape<kBTY>::THREADS, 0);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  b->grid = std::max(1, per_sm) * sms;
  if (b->units) b->grid = std::min(b->grid, std::max(sms, (b->nitems + BatchShape<kBTY>::WARPS - 1) / BatchShape<kBTY>::WARPS));
  return cudaSuccess;
}

// Codes of the current states, none of which lets a step keep phi.
cudaError_t batch_refresh_codes(ms_batch* b) {
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < b->nsims && e == cudaSuccess; ++i) {
    const size_t half = (b->sbytes[i] + 255) / 256 * 256;
    e = step_variants(2, 2, 1, 0).front()->codes(static_cast<char*>(b->state) + b->off[i] + b->parity * half, b->models[i],
                                                 codes_of(b, i, b->parity), b->stream);
  }
  b->codes_ok = e == cudaSuccess;
  return e;
}

}  // namespace

extern "C" {

ms_status ms_batch_create(int nsims, const ms_grid* grids, int n_phases, int n_components,
                          const ms_params* params, void* stream, const ms_allocator* alloc, ms_batch** out) {
  if (!out || nsims < 1 || !grids || !params) return bfail(nullptr, MS_ERR_ARG, "bad batch arguments");
  *out = nullptr;
  ensure_registered();
  ms_batch* b = new ms_batch();
  b->nsims = nsims;
  b->stream = static_cast<cudaStream_t>(stream);
  if (alloc) b->hook = AllocHook{alloc->alloc, alloc->release, alloc->user};
  b->models.resize(nsims);
  for (int i = 0; i < nsims; ++i) {
    ms_status s = build_model(nullptr, &grids[i], n_phases, n_components, &params[i], b->models[i]);
    if (s != MS_OK) {
      std::string m = "simulation " + std::to_string(i) + ": " + ms_last_error(nullptr);
      batch_free(b);
      return bfail(nullptr, s, m);
    }
    HostModel& m = b->models[i];
    if (m.dim != 2 || m.N != 2 || m.NM != 1 || m.dtype != MS_F32) {
      batch_free(b);
      return bfail(nullptr, MS_ERR_UNSUPPORTED, "the batched kernel is compiled for 2-D, N=2, K=2, FP32");
    }
    if (m.noise_amp != 0.0) {
      batch_free(b);
      return bfail(nullptr, MS_ERR_UNSUPPORTED, "batched simulations do not support phi noise (noise_amp != 0)");
    }
    if (m.at || m.gg || m.el) {
      batch_free(b);
      return bfail(nullptr, MS_ERR_UNSUPPORTED,
                   "batched simulations do not support the anti-trapping current, grain growth or elasticity");
    }
    if (m.G * m.V != 0.0) {
      batch_free(b);
      return bfail(nullptr, MS_ERR_UNSUPPORTED, "batched simulations must be isothermal in time (G V = 0)");
    }
    set_layout(m);
  }
  b->N = 2;
  b->NM = 1;
  b->dtype = MS_F32;
  // one allocation for all states (2 buffers each) and segment codes
  size_t tot = 0, nrows = 0;
  for (int i = 0; i < nsims; ++i) {
    const HostModel& m = b->models[i];
    if (!list_entry_fits(m)) {
      batch_free(b);
      return bfail(nullptr, MS_ERR_UNSUPPORTED, "grid too large for the batched work list");
    }
    const size_t sb = (size_t)m.fstride * (m.N + m.NM) * 4;
    b->sbytes.push_back(sb);
    b->off.push_back(tot);
    tot += 2 * ((sb + 255) / 256 * 256);
    nrows += (size_t)segments(m) * m.ny;
  }
  b->units_fit = ms_batch_cells(b) <= kBatchUnitCells;
  for (int i = 0; i < nsims; ++i) {
    b->coff.push_back(tot);
    tot += (2 * code_bytes(b->models[i]) + 15) / 16 * 16;
  }
  b->total = tot;
  b->state = dev_alloc(b->hook, tot);
  size_t dense = 0;
  for (auto& m : b->models) dense = std::max(dense, sizeof(float) * (m.N + m.NM) * (size_t)m.nx * m.ny);
  b->stage = dev_alloc(b->hook, dense);
  b->sims = dev_alloc(b->hook, sizeof(BatchSim<float, 2, 1>) * nsims);
  b->rows = static_cast<BatchRow*>(dev_alloc(b->hook, sizeof(BatchRow) * nrows));
  b->barrier = static_cast<unsigned int*>(dev_alloc(b->hook, 256));
  if (!b->state || !b->sims || !b->rows || !b->barrier) {
    batch_free(b);
    return bfail(nullptr, MS_ERR_OOM, "batch allocation failed");
  }
  b->status = reinterpret_cast<int*>(reinterpret_cast<char*>(b->barrier) + 128);
  cudaError_t e = cudaMemsetAsync(b->state, 0, tot, b->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(b->barrier, 0, 256, b->stream);
  // per-simulation constants
  std::vector<BatchSim<float, 2, 1>> hs(nsims);
  const StepKernel* k = step_variants(2, 2, 1, 0).front();
  for (int i = 0; i < nsims && e == cudaSuccess; ++i) {
    const HostModel& m = b->models[i];
    const size_t half = (b->sbytes[i] + 255) / 256 * 256;
    char* base = static_cast<char*>(b->state) + b->off[i];
    for (int par = 0; par < 2; ++par) {
      StepArgs<float, 2, 1>& g = hs[i].g[par];
      k->fill(&g, m, 1, b->status);
      g.out = reinterpret_cast<float*>(base + (1 - par) * half);
      g.tz0 = (float)temp_offset(m, m.t0);
      g.codes_in = codes_of(b, i, par);
      g.codes_out = codes_of(b, i, 1 - par);
      g.reuse_prev = 1;
      hs[i].in[par] = reinterpret_cast<const float*>(base + par * half);
    }
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->sims, hs.data(), sizeof(hs[0]) * nsims, cudaMemcpyHostToDevice, b->stream);
  // work list and persistent grid (every CTA resident at once)
  if (e == cudaSuccess) e = batch_set_tiles(b, kBTY, b->units_fit);
  if (e != cudaSuccess) {
    std::string m = std::string("batch set-up: ") + cudaGetErrorString(e);
    batch_free(b);
    return bfail(nullptr, e == cudaErrorMemoryAllocation ? MS_ERR_OOM : MS_ERR_CUDA, m);
  }
  *out = b;
  return MS_OK;
}

void ms_batch_destroy(ms_batch* b) { batch_free(b); }

const char* ms_batch_last_error(const ms_batch* b) { return b ? b->err.c_str() : ms_last_error(nullptr); }

ms_status ms_batch_set_fields(ms_batch* b, int sim, const void* phi, const void* mu, int on_device) {
  if (!b || sim < 0 || sim >= b->nsims || !phi || !mu) return bfail(b, MS_ERR_ARG, "bad argument");
  const HostModel& m = b->models[sim];
  const size_t half = (b->sbytes[sim] + 255) / 256 * 256;
  char* buf = static_cast<char*>(b->state) + b->off[sim] + b->parity * half;
  cudaError_t e = cudaSuccess;
  if (on_device ? field_kernel_reaches(phi) && field_kernel_reaches(mu) : b->stage != nullptr) {
    // (host fields: dense copies; strided ones run at a tenth of their rate)
    const void *p = phi, *q = mu;
    if (!on_device) {
      char* s = static_cast<char*>(b->stage);
      const size_t np = sizeof(float) * m.N * m.nx * m.ny, nm = sizeof(float) * m.NM * m.nx * m.ny;
      e = cudaMemcpyAsync(s, phi, np, cudaMemcpyHostToDevice, b->stream);
      if (e == cudaSuccess) e = cudaMemcpyAsync(s + np, mu, nm, cudaMemcpyHostToDevice, b->stream);
      p = s;
      q = s + np;
    }
    if (e == cudaSuccess) e = load_fields(m, buf, p, q, codes_of(b, sim, b->parity), b->stream);
  } else {
    e = copy_fields(m, buf, 0, m.N, phi, nullptr, on_device, b->stream);
    if (e == cudaSuccess) e = copy_fields(m, buf, m.N, m.NM, mu, nullptr, on_device, b->stream);
    if (e == cudaSuccess) e = fill_ghosts(m, buf, m.N + m.NM, b->stream);
    if (e == cudaSuccess) e = step_variants(2, 2, 1, 0).front()->codes(buf, m, codes_of(b, sim, b->parity), b->stream);
  }
  if (e == cudaSuccess && !on_device) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return bfail(b, MS_ERR_CUDA, std::string("batch set fields: ") + cudaGetErrorString(e));
  return MS_OK;
}

ms_status ms_batch_get_fields(ms_batch* b, int sim, void* phi, void* mu, int on_device) {
  if (!b || sim < 0 || sim >= b->nsims) return bfail(b, MS_ERR_ARG, "bad argument");
  const HostModel& m = b->models[sim];
  const size_t half = (b->sbytes[sim] + 255) / 256 * 256;
  char* buf = static_cast<char*>(b->state) + b->off[sim] + b->parity * half;
  cudaError_t e = cudaSuccess;
  if (on_device && field_kernel_reaches(phi) && field_kernel_reaches(mu)) {
    e = unload_fields(m, buf, phi, mu, b->stream);
  } else if (!on_device && b->stage) {   // as the way in
    char* s = static_cast<char*>(b->stage);
    const size_t np = sizeof(float) * m.N * m.nx * m.ny, nm = sizeof(float) * m.NM * m.nx * m.ny;
    e = unload_fields(m, buf, phi ? s : nullptr, mu ? s + np : nullptr, b->stream);
    if (e == cudaSuccess && phi) e = cudaMemcpyAsync(phi, s, np, cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess && mu) e = cudaMemcpyAsync(mu, s + np, nm, cudaMemcpyDeviceToHost, b->stream);
  } else {
    if (phi) e = copy_fields(m, buf, 0, m.N, nullptr, phi, on_device, b->stream);
    if (e == cudaSuccess && mu) e = copy_fields(m, buf, m.N, m.NM, nullptr, mu, on_device, b->stream);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return bfail(b, MS_ERR_CUDA, std::string("batch get fields: ") + cudaGetErrorString(e));
  return MS_OK;
}

ms_status ms_batch_step(ms_batch* b, int64_t n) {
  TraceRange trace("ms_batch_step");
  if (!b || n < 0) return bfail(b, MS_ERR_ARG, "bad argument");
  if (n == 0) return MS_OK;
  // the grid barrier counts (2 steps x CTAs) in 32 bits: at most 2^20 steps per launch
  if (n > ((int64_t)1 << 20)) return bfail(b, MS_ERR_BOUNDS, "at most 1048576 steps per ms_batch_step call");
  // the launch (barrier reset + cooperative kernel) is captured once per
  // (n, parity) and replayed
  cudaError_t e = b->units || b->codes_ok ? cudaSuccess : batch_refresh_codes(b);
  if (e != cudaSuccess) return bfail(b, MS_ERR_CUDA, std::string("batch codes: ") + cudaGetErrorString(e));
  if (!b->graph || b->graph_n != n * 2 + b->parity) {
    if (b->graph) {
      cudaGraphExecDestroy(b->graph);
      b->graph = nullptr;
    }
    cudaStream_t cap;
    e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
    if (e == cudaSuccess) {
      cudaStream_t keep = b->stream;
      b->stream = cap;
      cudaGraph_t graph;
      e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
      if (e == cudaSuccess) {
        cudaError_t le = launch_batch(b, n);
        e = cudaStreamEndCapture(cap, &graph);
        if (le != cudaSuccess) e = le;
      }
      b->stream = keep;
      if (e == cudaSuccess) {
        e = cudaGraphInstantiate(&b->graph, graph, 0);
        cudaGraphDestroy(graph);
      }
      cudaStreamDestroy(cap);
    }
    if (e != cudaSuccess) return bfail(b, MS_ERR_CUDA, std::string("batch graph: ") + cudaGetErrorString(e));
    b->graph_n = n * 2 + b->parity;
  }
  e = cudaGraphLaunch(b->graph, b->stream);
  if (e != cudaSuccess) return bfail(b, MS_ERR_CUDA, std::string("batch launch: ") + cudaGetErrorString(e));
  b->parity = (int)((b->parity + n) & 1);
  b->steps_done += n;
  b->codes_ok = !b->units;
  return MS_OK;
}

ms_status ms_batch_sync(ms_batch* b) {
  if (!b) return bfail(nullptr, MS_ERR_ARG, "batch is NULL");
  int st = 0;
  cudaError_t e = cudaMemcpyAsync(&st, b->status, sizeof(int), cudaMemcpyDeviceToHost, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return bfail(b, MS_ERR_CUDA, std::string("batch sync: ") + cudaGetErrorString(e));
  if (st & kStatusTimeout) return bfail(b, MS_ERR_TIMEOUT, "a bounded device wait timed out");
  return MS_OK;
}

ms_status ms_batch_set_tile(ms_batch* b, int ty) {
  if (!b) return bfail(nullptr, MS_ERR_ARG, "batch is NULL");
  bool ok = false;
  for (int k = 0; k < kNBTY; ++k) ok = ok || kBTYs[k] == ty;
  if (!ok) return bfail(b, MS_ERR_ARG, "tile height must be one of 4, 8, 16");
  if (ty == b->ty && !b->units) return MS_OK;
  cudaError_t e = batch_set_tiles(b, ty, false);   // strips, also where units were the default
  if (e != cudaSuccess) return bfail(b, MS_ERR_CUDA, std::string("batch tiles: ") + cudaGetErrorString(e));
  return MS_OK;
}

int ms_batch_tile(const ms_batch* b) { return b ? b->ty : 0; }

ms_status ms_batch_tune(ms_batch* b, int steps_per_trial, double* best_ms_per_step) {
  TraceRange trace("ms_batch_tune");
  if (!b || steps_per_trial < 1) return bfail(b, MS_ERR_ARG, "bad argument");
  const size_t tot = b->total;
  void* save = dev_alloc(b->hook, tot);
  if (!save) return bfail(b, MS_ERR_OOM, "batch tuner: state copy allocation failed");
  const int parity0 = b->parity;
  const int64_t done0 = b->steps_done;
  const bool codes0 = b->codes_ok;
  cudaError_t e = cudaMemcpyAsync(save, b->state, tot, cudaMemcpyDeviceToDevice, b->stream);
  cudaEvent_t t0 = nullptr, t1 = nullptr;
  if (e == cudaSuccess) e = cudaEventCreate(&t0);
  if (e == cudaSuccess) e = cudaEventCreate(&t1);
  int best = b->ty;
  bool best_units = b->units;
  float best_ms = 0.0f;
  for (int k = 0; k < kNBTY + (b->units_fit ? 1 : 0) && e == cudaSuccess; ++k) {   // the heights, then the units
    const bool units = k == kNBTY;
    e = batch_set_tiles(b, units ? kBTY : kBTYs[k], units);
    if (e != cudaSuccess) break;
    // a warm-up launch captures the graph for this step count
    if (ms_batch_step(b, steps_per_trial) != MS_OK) {
      e = cudaErrorUnknown;
      break;
    }
    e = cudaEventRecord(t0, b->stream);
    if (e == cudaSuccess && ms_batch_step(b, steps_per_trial) != MS_OK) e = cudaErrorUnknown;
    if (e == cudaSuccess) e = cudaEventRecord(t1, b->stream);
    if (e == cudaSuccess) e = cudaEventSynchronize(t1);
    float ms = 0.0f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, t0, t1);
    if (e == cudaSuccess && (k == 0 || ms < best_ms)) {
      best_ms = ms;
      best = b->ty;
      best_units = units;
    }
    // back to the saved state
    if (e == cudaSuccess) e = cudaMemcpyAsync(b->state, save, tot, cudaMemcpyDeviceToDevice, b->stream);
    b->parity = parity0;
    b->steps_done = done0;
    b->codes_ok = codes0;   // (the copy holds the codes as well)
  }
  if (t0) cudaEventDestroy(t0);
  if (t1) cudaEventDestroy(t1);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  dev_free(b->hook, save);
  if (e == cudaSuccess) e = batch_set_tiles(b, best, best_units);
  if (e != cudaSuccess) return bfail(b, MS_ERR_CUDA, std::string("batch tuner: ") + cudaGetErrorString(e));
  if (best_ms_per_step) *best_ms_per_step = best_ms / steps_per_trial;
  return ms_batch_sync(b);
}

int64_t ms_batch_cells(const ms_batch* b) {
  if (!b) return 0;
  int64_t c = 0;
  for (auto& m : b->models) c += (int64_t)m.nx * m.ny * m.nz;
  return c;
}

}  // extern "C"
