// Host-side internals shared by the runtime and the kernel instantiation units.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

namespace msgb {

constexpr int kNMax = 8;
constexpr int kKMax = 3;
constexpr int kElRank = 6;   // independent eigenstrains at most (symmetric tensors)

// Boundary code of an internal cut whose ghost plane is filled by a halo
// exchange (same value as MS_BC_HALO in the public header).
constexpr int kBcHalo = 16;

// Status bits OR-ed into the device status word.
constexpr int kStatusNonFinite = 1;
constexpr int kStatusTimeout = 2;
constexpr int kStatusLaunch = 4;   // launch geometry beyond a compiled limit (no work done)
// Planes marched by one CTA of the 3-D step at most (bounds the shared-memory
// copy of the segment codes a CTA reads).
constexpr int kMaxZChunk = 64;
// Segment-code byte: pure phase + 1 in the low bits (phases <= kNMax), and a
// bit saying that the state one step earlier held the same pure phase there.
constexpr int kCodePhase = 0x7F;
constexpr int kCodeReuse = 0x80;

// Model constants derived in FP64 from the paper's inputs (Sec. 3).
struct HostModel {
  int dim = 2, N = 2, NM = 1, dtype = 0;
  int nx = 1, ny = 1, nz = 1, bc[3] = {3, 3, 3};
  int zorg = 0;   // lab index of the first cell along the last axis (slabs, moving frame)
  // padded layout (elements)
  int pitch = 0, nyp = 0, nzp = 0, xoff = 0, zoff = 0;
  long long fstride = 0;
  double dx = 1, dt = 0, eps = 1, tau = 1;
  int potential = 1;
  double gamma[kNMax][kNMax] = {};
  double delta[kNMax][kNMax] = {};
  double rot[kNMax][kNMax][9] = {};
  bool rotated[kNMax][kNMax] = {};
  double g3[kNMax][kNMax][kNMax] = {};
  bool has_g3 = false;
  double chi[kNMax][kKMax * kKMax] = {};   // (Hessian)^-1
  double D[kNMax][kKMax * kKMax] = {};
  double DX[kNMax][kKMax * kKMax] = {};    // D chi
  double B0[kNMax][kKMax] = {}, B1[kNMax][kKMax] = {};
  double C0[kNMax] = {}, C1[kNMax] = {}, C2[kNMax] = {};
  double T0 = 0, G = 0, z0 = 0, V = 0, T_ref = 0, t0 = 0;
  double noise_amp = 0;                    // phi noise (0 = off)
  unsigned long long noise_seed = 0;
  int at = 0;                              // anti-trapping current in the mu update
  int gg = 0;                              // grain growth: no chemical driving force, mu held
  int el = 0;                              // elasticity (homogeneous stiffness)
  double elC[3][3][3][3] = {};             // stiffness tensor
  double eig[kNMax][3][3] = {};            // eigenstrain of each phase
};

// Basis of the phases' eigenstrains (in-plane components in 2-D): tensors
// B[s], orthonormal, and E^a = sum_s c[a][s] B[s].  rank = number of tensors.
struct ElasticBasis {
  int rank = 0;
  double B[kElRank][3][3] = {};
  double c[kNMax][kElRank] = {};
};
ElasticBasis elastic_basis(const HostModel& m);

// Launch geometry of one step.
struct LaunchGeom {
  int tiles = 0;       // gridDim.x
  int zchunks = 1;     // gridDim.y
  int zchunk = 1;
  unsigned int* iface = nullptr;   // work lists of split kernels (see StepArgs)
  unsigned int* iface2 = nullptr;
  unsigned int iface_cap = 0;
  int iface_blocks = 0;            // SMs: the interface grid is this x resident CTAs per SM
  void* cells = nullptr;           // scratch of the cell-list step (ms_cells.cuh)
  int sms = 0;                     // multiprocessors of the device
  unsigned int* at_list = nullptr; // anti-trapping work list (see StepArgs)
  const void* elw = nullptr;       // fields of the elastic phase potentials (see StepArgs)
  unsigned int at_cap = 0;
  int reuse_prev = 1;              // output buffer = state one step before the input (see StepArgs)
  long long step = 0;              // step index of the input state (phi-noise counter)
};

// Where the states of a run live: state k at slots + k slot_bytes, or, without
// slots, alternating between two buffers (state 0 in buf[0]).
struct MultiRun {
  void* buf[2];
  char* slots;
  size_t slot_bytes;
  int nsteps;
  double t;                    // time of state 0
  double t0, dt;               // and of state k > 0: t0 + (step0 + k) dt
  long long step0;
  double off, G, z0, V;        // T - T_ref = off - G (z0 + V t) at the origin of the last axis
  unsigned int* counters;      // [0] barrier arrivals, [1] exit tickets; zero between launches
};

// One compiled forward-step instantiation.
struct StepKernel {
  int dim, np, nm, dtype, tx, ty;
  int split;   // 1: the bulk and the rest by kernels of their own (FP32: streaming kernel and interface rows;
               // FP64: cell list, ms_cells.cuh), 0: one fused kernel
  int smem_bytes;
  size_t args_bytes;
  // Fill the launch-argument blob from the model (all constants).
  void (*fill)(void* blob, const HostModel& m, int zchunk, int* status);
  // Launch one step: tm = tensor map of the input state (tile box), tmi =
  // its interface-box map (split variants; may be NULL otherwise), in = the
  // input state itself, t = time
  // of the input state, out = destination buffer, codes_in / codes_out =
  // segment codes of the input / output state.
  cudaError_t (*launch)(const CUtensorMap* tm, const CUtensorMap* tmi, const void* in, void* blob, const HostModel& m,
                        double t, void* out, const uint8_t* codes_in, uint8_t* codes_out, const LaunchGeom& lg,
                        cudaStream_t st);
  // Several steps in one persistent launch (2-D; NULL otherwise); segment
  // codes are neither read nor written.
  cudaError_t (*multi)(const void* blob, const MultiRun& run, int sms, cudaStream_t st);
  // Recompute the segment codes of a state loaded from outside.
  cudaError_t (*codes)(const void* state, const HostModel& m, uint8_t* codes, cudaStream_t st);
  // Anti-trapping correction of the mu just written by launch (same
  // arguments; in = the input state).
  cudaError_t (*at)(const void* in, void* blob, const HostModel& m, double t, void* out, const uint8_t* codes_in,
                    uint8_t* codes_out, const LaunchGeom& lg, cudaStream_t st);
};

// Cells up to which a 2-D grid is stepped by the persistent multi-step kernel
// (FP32, FP64): us a step on a GB300, one launch a step / multi-step: FP32
// binary 128^2 6.2 / 3.7, 256^2 6.2 / 4.5, 384^2 6.2 / 7.7, ternary 200^2
// 10.3 / 9.0, 400^2 18.3 / 20.3; FP64 binary 128^2 24.6 / 11.6, 512^2 50 / 20,
// 900^2 77 / 51, ternary 512^2 344 / 307.  (The FP64 line stands below the crossover.)
constexpr long long kMultiMaxCells[2] = {80000, 300000};
// Cells from which a binary 2-D FP32 context starts with the split step: its two
// launches cost 13 us however small the grid (us a step on a GB300, fused / split,
// a dendrite: 290^2 6.2 / 13.4, 700^2 10.9 / 16.3, 1000^2 16.4 / 16.4, 1537x1411
// 29.4 / 18.6, 2048^2 52.7 / 28.2).
constexpr long long kPlaneMinCells = 1200000;
// Steps of one multi-step launch at most (the barrier counts steps x CTAs in 32 bits).
constexpr int kMultiMaxSteps = 1 << 16;

// Number of 32-cell segments per row.
inline int segments(const HostModel& m) { return (m.nx + 31) / 32; }
// Bits that hold the values 0 .. n - 1.
inline int bits_for(int n) {
  int b = 0;
  while ((1ll << b) < n) ++b;
  return b;
}
// An interface-list entry (z, y, segment) packs into 31 bits (every shift
// of its fields stays below 32).
inline bool list_entry_fits(const HostModel& m) {
  return bits_for(segments(m)) + bits_for(m.ny) + bits_for(m.nz) <= 31;
}
// Bytes of one segment-code array (3-D arrays carry a ghost plane per side).
inline size_t code_bytes(const HostModel& m) { return (size_t)segments(m) * m.ny * m.nzp; }

// One compiled FP64 diagnostics instantiation.
struct DiagKernel {
  int dim, np, nm, dtype;
  // codes: the state's segment codes, or NULL where they do not describe it
  cudaError_t (*launch)(const void* state, const uint8_t* codes, const HostModel& m, double t, double* partials,
                        int nblocks, double* out, int* status, cudaStream_t st);
};

size_t cells_scratch_bytes(const HostModel& m);   // of the cell-list step
// Listed cells whose fluxes and mobilities the cell-list step stores (8 (3 N +
// (K-1)^2) bytes each): all there can be on grids of up to 2^22 cells, an eighth of
// the cells beyond, where the rest, if that many are ever listed, evaluate the faces
// of a neighbour without a place themselves.  By cell instead, the scratch of a
// 3-D FP64 context was more than its state (110 bytes a cell beside 80 for N = 3, 206
// beside 144 for N = 8), now 22 and 34.
constexpr size_t kCellSlots = size_t(1) << 22;
inline size_t cell_slots(size_t cells) { return cells <= kCellSlots ? cells : cells / 8 > kCellSlots ? cells / 8 : kCellSlots; }
// The cell-list step indexes cells with 32 bits.
inline bool cells_fit(const HostModel& m) { return (long long)m.nx * m.ny * m.nz < 0xFFFFFFF0ll; }

std::vector<StepKernel>& step_registry();
std::vector<DiagKernel>& diag_registry();
void ensure_registered();

}  // namespace msgb
