// Launch-side view of the kernels: per-(lattice, storage) shapes and the
// host launchers that the engine dispatches to.  Each storage type's kernels
// are compiled in their own translation unit (step_<type>.cu).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "step_kernel.cuh"
#include "tile_kernel.cuh"

namespace lbm {

// CTA width, TMA pipeline depth and the CTAs per SM the register budget is
// sized for, per (lattice, storage).  Shared memory per CTA is
// NS * (Q box slots + flag slot) + the psi ring.
// (Measured on GB300, 8192x4096: D2Q9 NS 4 / MINB 8 for FP32 and MINB 10 for
// 16-bit storage beat NS 5 / MINB 6 and MINB 8 or 12 (16-bit at MINB 12: 76
// registers, 0.243 ms against 0.233); D2Q21 needs NS >= R + 2 = 5, and NS 5
// with 3 CTAs per SM (FP32) or 5 (16-bit) beat NS 6 with 2 or 3 by 21% and
// 5%.  16-bit D2Q21 runs CTAs of 64 threads (node pairs), its plane groups
// arriving as boxes of depth 1, 3 and 7: NS 6 (43 KB, 5 CTAs per SM: two rows
// in flight besides the four the collision re-reads) beat NS 5 (6 CTAs) by 1.1%
// and NS 7 (4 CTAs) by 8%.)
template <int Q, typename S> struct StepConfig {
  static constexpr int W = 128;
  static constexpr int NS = (Q == 9) ? (sizeof(S) == 8 ? 4 : (sizeof(S) == 4 ? 4 : 5))
                                     : (sizeof(S) == 2 ? 6 : 5);
  static constexpr int MINB = (Q == 9) ? (sizeof(S) == 8 ? 2 : (sizeof(S) == 4 ? 8 : 10))
                                       : (sizeof(S) == 8 ? 1 : (sizeof(S) == 4 ? 3 : 6));
  // The persistent batch kernel carries its tile loop on top of the march:
  // 16-bit D2Q9 targets 8 CTAs per SM there, so that it does not spill.
  static constexpr int BATCH_MINB = (Q == 9 && sizeof(S) == 2) ? 8 : MINB;
  // One CTA per tile, the compile-time-flag kernel (kFlExpPlain): D2Q9 FP32
  // and 16-bit batches run 12 CTAs per SM (76-80 registers, no spills; the
  // 256-lattice sweep 6% faster than at 10 for FP16S, 1.4% than at 8 for
  // FP32): short tiles of many small lattices need more CTAs in flight than
  // the single lattice's long strips.  The run-time-flag kernel keeps MINB (it
  // would spill at 12).
  static constexpr int BATCH_MINB_PLAIN = (Q == 9 && sizeof(S) != 8) ? 12 : MINB;
  template <int FL> static constexpr int batch_minb_tile() {
    return FL == kFlExpPlain ? BATCH_MINB_PLAIN : MINB;
  }
};

template <int Q, typename S>
using ConfigShape = StepShape<Q, S, StepConfig<Q, S>::W, StepConfig<Q, S>::NS>;

// Launches the fused step as a row march.  (device, here and below: the lattice's.)
template <int Q, typename S>
cudaError_t launch_step(const PopMaps& src, const CUtensorMap& flags,
                        const StepArgs<typename Codec<S>::T, S>& a, dim3 grid, int device,
                        cudaStream_t stream);

// Shapes of the tile kernel per (lattice, storage): tile width and height,
// threads, time steps per launch, whether tiles without edges or walls run a
// copy of the update without that code, CTAs per SM the registers are sized for,
// and the microseconds of a launch, us0 + us per round of resident CTAs (FP64: per
// tile of the SM with the most tiles), fitted to GB300 times on 128x64 to 4096x2048 lattices (within about 15%).  The shape with
// the least time per step by this estimate runs (choose_tiles); on the lattices
// of the fit that is the fastest one or within 6% of it.  (At these register
// budgets the 64-wide D2Q9 and 16-bit D2Q21 shapes and the 32x28 one spill: 4-16
// bytes with the common settings fixed at compile time, 32-72 with all of them
// at run time.)
struct TileCfg {
  int tw, th, nt, steps;
  bool in;
  int minb;
  double us0, us;
};
constexpr int kMaxTileShapes = 7;
struct TileList {
  TileCfg t[kMaxTileShapes];
  int n;
  int moments;  // the shape that also reads out the moments
};
template <int Q, typename S> constexpr TileList tile_list() {
  if constexpr (sizeof(S) == 8 && Q == 9)
    return {{{16, 4, 64, 1, false, 4, 5.6, 2.8},
             {32, 8, 256, 1, false, 3, 3.8, 9.85},
             {32, 16, 256, 1, true, 2, 4.7, 19.1}}, 3, 2};
  else if constexpr (sizeof(S) == 8)
    return {{{16, 4, 64, 1, false, 4, 10.0, 5.95},
             {32, 8, 256, 1, false, 3, 5.3, 19.6},
             {32, 16, 256, 1, true, 2, 2.0, 39.0}}, 3, 2};
  else if constexpr (Q == 21 && sizeof(S) == 4)
    return {{{16, 4, 64, 1, false, 4, 3.9, 3.3},
             {32, 8, 256, 1, false, 3, 3.2, 4.1},
             {64, 8, 256, 1, true, 2, 6.0, 4.7}}, 3, 1};
  else if constexpr (Q == 21)
    return {{{32, 4, 64, 1, false, 8, 3.6, 3.85},
             {64, 8, 128, 1, true, 4, 6.0, 5.6}}, 2, 1};
  else if constexpr (sizeof(S) == 4)
    return {{{32, 4, 64, 1, false, 8, 2.4, 2.6},
             {64, 8, 128, 1, true, 7, 2.3, 6.6},
             {32, 4, 160, 2, false, 4, 2.0, 3.35},
             {32, 8, 224, 2, false, 3, 2.6, 3.9},
             {32, 28, 288, 2, true, 3, 6.3, 7.3},
             {64, 12, 288, 2, true, 3, 5.0, 6.6},
             {64, 22, 448, 2, true, 2, 7.0, 7.4}}, 7, 0};
  else
    return {{{32, 4, 64, 1, false, 8, 2.2, 2.9},
             {64, 8, 128, 1, true, 7, 3.0, 3.85},
             {32, 4, 160, 2, false, 4, 1.7, 3.2},
             {32, 8, 224, 2, false, 3, 2.5, 3.3},
             {32, 28, 288, 2, true, 3, 4.4, 6.6},
             {64, 12, 288, 2, true, 3, 4.5, 5.85},
             {64, 22, 448, 2, true, 2, 5.5, 6.6}}, 7, 0};
}
template <int Q, typename S, int K> struct TileConfig {
  static constexpr TileCfg kCfg = tile_list<Q, S>().t[K];
  using Sh = TileShape<Q, S, kCfg.tw, kCfg.th, kCfg.nt, kCfg.steps, kCfg.in>;
};

// Launches tile shape `shape`: its steps (kModeStep), or the read-out pass
// (kModeMoments; the list's `moments` shape only).
template <int Q, typename S>
cudaError_t launch_tile(int shape, const PopMaps& src, const uint32_t* flags, int flag_pitch,
                        const StepArgs<typename Codec<S>::T, S>& a, int device, cudaStream_t stream,
                        int mode);

// What the host needs of a tile shape: its TMA boxes, and the tiles that one
// round of resident CTAs takes (0 if the kernel cannot run).
struct TileInfo {
  int bw, bh, nmap, depth[kMaxMaps], slots, sms;
};
template <int Q, typename S> TileInfo tile_info(int shape, int device);

// CTAs of the step kernel that fit on one SM (occupancy query).
template <int Q, typename S> int step_ctas_per_sm(int device);

// One time step of up to BatchArgs::kChunk members of a batch: nctas CTAs, one per
// tile of the chunk, or (persistent) each marching every nctas-th tile; and
// the batch kernel's residency per SM.  `plain`: every member has the
// exponential psi, no projection and (16-bit storage) stochastic rounding, so
// the kernel with those settings fixed runs.
template <int Q, typename S>
cudaError_t launch_batch(const BatchArgs<Q, typename Codec<S>::T, S>& args, int nctas,
                         bool persistent, bool plain, int device, cudaStream_t stream);
template <int Q, typename S> int batch_ctas_per_sm(int device);

// The same on tiles of shape `shape`, one CTA per tile.
template <int Q, typename S>
cudaError_t launch_batch_tiles(int shape, const BatchArgs<Q, typename Codec<S>::T, S>& args,
                               int ntiles, bool plain, cudaStream_t stream);
// Sets the shared-memory attribute of its kernels (outside any stream capture).
template <int Q, typename S> cudaError_t prepare_batch_tiles(int shape, int device);

// Auxiliary kernels (aux.cu).
template <int Q, typename S>
cudaError_t launch_encode(const double* f, S* buf, int nx, int ny, int64_t pitch, int64_t plane,
                          double rho_s, cudaStream_t st);
template <int Q, typename S>
cudaError_t launch_equilibrium(const double* rho, const double* ux, const double* uy,
                               const double* dfi, S* buf, int nx, int ny, int64_t pitch,
                               int64_t plane, double rho_s, cudaStream_t st);
template <int Q, typename S>
cudaError_t launch_decode(const S* buf, double* f, int nx, int ny, int64_t pitch, int64_t plane,
                          double rho_s, cudaStream_t st);
template <int Q, typename T>
cudaError_t launch_wall_prepare(const double* phi, const double* psr, const double* psa,
                                const double* uw, double G_R, double G_A, double eps, int nx,
                                int ny, T* phie, T* sx, T* sy, T* uwx, T* uwy, uint32_t* flags,
                                int nchunk_pad, cudaStream_t st);

// Compensated (Neumaier) FP64 sums of up to three [N] arrays (NULL sums to
// 0) into out[3]: nparts blocks each reduce a grid-stride share into
// partials[6 * nparts], then one thread merges them in block order
// (deterministic).  lbm_totals and lbm_reduce3_noalloc both use kReduceParts
// blocks.
constexpr int kReduceParts = 1024;
cudaError_t launch_reduce3(const double* a, const double* b, const double* c, int64_t n,
                           double* partials, int nparts, double* out, cudaStream_t st);
cudaError_t launch_colsum(const double* f, int q, int64_t n, double* out_n, cudaStream_t st);

cudaError_t launch_filter_pass(int q, const double* g, double* out, const uint8_t* solid, int nx,
                               int ny, cudaStream_t st);

}  // namespace lbm
