// Arguments of one pass over a lattice, shared by the step kernels.
#pragma once

#include <cuda.h>

#include "node.cuh"

namespace lbm {

enum : uint32_t { kStatusNonFinite = 1u, kStatusTimeout = 2u };

enum StepMode : int {
  kModeStep = 0,      // write post-collision populations to fout
  kModeMoments = 1,   // write rho and u = (j + F/2) / rho (FP64) instead
};

// Which run-time switches of the update are fixed at compile time:
// kFlRuntime reads psi_kind, project and the rounding mode from the
// arguments; kFlExpPlain is the exponential pseudo-potential without the
// projection step, with stochastic rounding for 16-bit storage, kFlExpNearest the
// same with rounding to nearest (16-bit D2Q9 tiles: 1024x512 7.66 -> 6.30 us per
// step, 128x64 1.89 -> 1.52); the other settings run the kFlRuntime kernel.  All
// give the same bits.
enum StepFlags : int { kFlRuntime = 0, kFlExpPlain = 1, kFlExpNearest = 2 };
template <int FL> constexpr int kPsiOf = FL == kFlRuntime ? -1 : 0;  // psi kind, -1: P.psi_kind

// Wall-flag words per lattice row: one per 32 columns, padded to 16 bytes.
__host__ __device__ constexpr int flag_words_per_row(int nx) { return ((nx + 31) / 32 + 3) / 4 * 4; }

template <typename T, typename S> struct StepCore {
  Physics<T> phys;
  WallFields<T> wall;
  int32_t nx, ny;
  int32_t pitch;       // elements per padded row
  int32_t tile_rows;   // L
  int64_t plane;       // elements per population plane
  S* fout;             // kModeStep: destination buffer (same layout as the source)
  uint32_t* status;    // error bits (kStatus*)
  uint64_t wait_ns;    // bound of every stage wait
  uint32_t extra_tx;   // test hook: bytes each stage expects beyond its copies (0 normally)
  // Step counter of the stochastic rounding: two words indexed by the source
  // buffer; a step reads rng[rng_idx] and one CTA writes rng[rng_idx ^ 1] =
  // rng[rng_idx] + 1 for the next step (kModeStep only).
  uint32_t* rng;
  int32_t rng_idx;
  int32_t stochastic;  // 16-bit storage: 1 = stochastic rounding, 0 = nearest-even
};
template <typename T, typename S> struct StepArgs : StepCore<T, S> {
  double* out_rho;     // kModeMoments: [ny][nx]
  double* out_ux;
  double* out_uy;
  int32_t momentum;    // kModeMoments: 1 -> out_ux/out_uy get j + F/2 instead of u
};

template <int FL, typename Args> __device__ __forceinline__ bool rounds_stochastically(const Args& a) {
  return FL == kFlRuntime ? a.stochastic != 0 : FL == kFlExpPlain;
}

// Counter of the step about to run (0 unless it is needed).
template <typename S, int MODE, int FL, typename Args>
__device__ __forceinline__ uint32_t step_key(const Args& a) {
  if constexpr (MODE == kModeStep && Codec<S>::kShifted) {
    if (rounds_stochastically<FL>(a)) return a.rng[a.rng_idx];
  }
  return 0u;
}

// Advances the counter past the launch's steps; called by one thread of one CTA.
template <int MODE, typename Args>
__device__ __forceinline__ void advance_key(const Args& a, uint32_t steps = 1u) {
  if constexpr (MODE == kModeStep) a.rng[a.rng_idx ^ 1] = a.rng[a.rng_idx] + steps;
}

// TMA maps of one population buffer, one per distinct box depth of the
// lattice's plane groups (D2Q9 uses one, D2Q21 three).
constexpr int kMaxMaps = 3;
template <int Q> constexpr int kMapsOf = Q == 9 ? 1 : kMaxMaps;
struct PopMaps {
  CUtensorMap m[kMaxMaps];
};

}  // namespace lbm
