// Definitions of the step launchers; included by one translation unit per
// storage type, which instantiates them for D2Q9 and D2Q21.
#pragma once

#include <algorithm>
#include <atomic>
#include <mutex>

#include "launch.cuh"

namespace lbm {

// A value computed once per device: kernel attributes and residency belong to the
// device that was current when they were set or asked for, and a process may
// hold lattices on several.  The caller names its lattice's device, which is
// current for any launch that can succeed: asking the runtime each time cost
// 0.1 us of a launch's 2.2 on the host.
template <typename T> class PerDevice {
 public:
  template <typename F> T get(int device, F&& compute) {
    if (device < 0 || device >= kDevices) return compute();
    if (!ready_[device].load(std::memory_order_acquire)) {
      int current = -1;
      if (cudaGetDevice(&current) != cudaSuccess || current != device) return compute();
      std::lock_guard<std::mutex> lock(mu_);
      if (!ready_[device].load(std::memory_order_relaxed)) {
        value_[device] = compute();
        ready_[device].store(true, std::memory_order_release);
      }
    }
    return value_[device];
  }

 private:
  static constexpr int kDevices = 64;
  std::mutex mu_;
  std::atomic<bool> ready_[kDevices] = {};
  T value_[kDevices] = {};
};

// The common settings (exponential psi, no projection, stochastic rounding of
// 16-bit storage) run kernels with them fixed at compile time.
template <typename T, typename S> static bool plain_flags(const StepArgs<T, S>& a) {
  return a.phys.psi_kind == 0 && !a.phys.project && (a.stochastic || !Codec<S>::kShifted);
}

template <int Q, typename S, int FL>
static cudaError_t prepare_kernel(int device) {
  using Cfg = StepConfig<Q, S>;
  using Sh = ConfigShape<Q, S>;
  static PerDevice<cudaError_t> once;
  return once.get(device, [] {
    return cudaFuncSetAttribute(step_kernel<Q, S, Cfg::W, Cfg::NS, Cfg::MINB, FL>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, Sh::SMEM);
  });
}

// The fused step as a programmatic dependent launch: the step may begin
// launching while the previous kernel in the stream drains (the kernel waits
// before touching global memory).
template <int Q, typename S, int FL>
static cudaError_t launch_step_pdl(const PopMaps& src, const CUtensorMap& flags,
                                   const StepArgs<typename Codec<S>::T, S>& a, dim3 grid,
                                   int device, cudaStream_t stream) {
  using Cfg = StepConfig<Q, S>;
  using Sh = ConfigShape<Q, S>;
  cudaError_t e;
  if ((e = prepare_kernel<Q, S, FL>(device)) != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(Sh::NT);
  cfg.dynamicSmemBytes = Sh::SMEM;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, step_kernel<Q, S, Cfg::W, Cfg::NS, Cfg::MINB, FL>,
                            src, flags, a);
}

template <int Q, typename S>
cudaError_t launch_step(const PopMaps& src, const CUtensorMap& flags,
                        const StepArgs<typename Codec<S>::T, S>& a, dim3 grid, int device,
                        cudaStream_t stream) {
  return plain_flags(a) ? launch_step_pdl<Q, S, kFlExpPlain>(src, flags, a, grid, device, stream)
                        : launch_step_pdl<Q, S, kFlRuntime>(src, flags, a, grid, device, stream);
}

template <int Q, typename S, int K, int MODE, int FL>
static cudaError_t prepare_tile(int device) {
  using Cfg = TileConfig<Q, S, K>;
  static PerDevice<cudaError_t> once;
  return once.get(device, [] {
    return cudaFuncSetAttribute(tile_kernel<typename Cfg::Sh, MODE, FL, Cfg::kCfg.minb>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::Sh::SMEM);
  });
}

static int sm_count(int device) {
  static PerDevice<int> sms;
  return sms.get(device, [=] {
    int n = 0;
    return cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device) == cudaSuccess ? n : 0;
  });
}

// CTAs of the K-th shape that the GPU holds at once (0 if the kernel cannot run).
template <int Q, typename S, int K> static int tile_slots(int device) {
  using Cfg = TileConfig<Q, S, K>;
  using Sh = typename Cfg::Sh;
  static PerDevice<int> slots;
  return slots.get(device, [=] {
    int n = 0;
    if (prepare_tile<Q, S, K, kModeStep, kFlExpPlain>(device) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &n, tile_kernel<Sh, kModeStep, kFlExpPlain, Cfg::kCfg.minb>, Sh::NT, Sh::SMEM) != cudaSuccess)
      return 0;
    return n * sm_count(device);
  });
}

template <int Q, typename S, int K, int MODE, int FL>
static cudaError_t launch_tile_k(const PopMaps& src, const uint32_t* flags, int flag_pitch,
                                 const StepArgs<typename Codec<S>::T, S>& a, int device,
                                 cudaStream_t stream) {
  using Cfg = TileConfig<Q, S, K>;
  using Sh = typename Cfg::Sh;
  cudaError_t e = prepare_tile<Q, S, K, MODE, FL>(device);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  const int nty = (a.ny + Sh::TH - 1) / Sh::TH;
  cfg.gridDim = dim3((a.nx + Sh::TW - 1) / Sh::TW);
  const int slots = Sh::IN ? tile_slots<Q, S, K>(device) : 0;
  const int ahead = (int64_t)cfg.gridDim.x * nty > slots ? slots / 2 : 0;
  cfg.blockDim = dim3(Sh::NT);
  cfg.dynamicSmemBytes = Sh::SMEM;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  for (int ty0 = 0; ty0 < nty && e == cudaSuccess; ty0 += 65535) {
    cfg.gridDim.y = std::min(nty - ty0, 65535);
    e = cudaLaunchKernelEx(&cfg, tile_kernel<Sh, MODE, FL, Cfg::kCfg.minb>, src, flags, flag_pitch, ahead, ty0, a);
  }
  return e;
}

// Calls fn<K>() for the K-th shape of the list.
template <int Q, typename S, int K = 0, typename F> auto with_shape(int shape, F&& fn) {
  if constexpr (K + 1 < tile_list<Q, S>().n)
    if (shape != K) return with_shape<Q, S, K + 1>(shape, fn);
  return fn.template operator()<K>();
}

template <int Q, typename S>
cudaError_t launch_tile(int shape, const PopMaps& src, const uint32_t* flags, int flag_pitch,
                        const StepArgs<typename Codec<S>::T, S>& a, int device, cudaStream_t stream,
                        int mode) {
  if (mode == kModeMoments)
    return launch_tile_k<Q, S, tile_list<Q, S>().moments, kModeMoments, kFlRuntime>(
        src, flags, flag_pitch, a, device, stream);
  return with_shape<Q, S>(shape, [&]<int K>() {
    if constexpr (Q == 9 && sizeof(S) == 2)
      if (a.phys.psi_kind == 0 && !a.phys.project && !a.stochastic)
        return launch_tile_k<Q, S, K, kModeStep, kFlExpNearest>(src, flags, flag_pitch, a, device, stream);
    return plain_flags(a) ? launch_tile_k<Q, S, K, kModeStep, kFlExpPlain>(src, flags, flag_pitch, a, device, stream)
                          : launch_tile_k<Q, S, K, kModeStep, kFlRuntime>(src, flags, flag_pitch, a, device, stream);
  });
}

template <int Q, typename S> TileInfo tile_info(int shape, int device) {
  return with_shape<Q, S>(shape, [&]<int K>() {
    using Cfg = TileConfig<Q, S, K>;
    using Sh = typename Cfg::Sh;
    TileInfo t{Sh::BW, Sh::BH, Sh::NMAP, {}, 0, 0};
    for (int k = 0; k < Sh::NMAP; ++k) t.depth[k] = Sh::kTab.depth[k];
    t.slots = tile_slots<Q, S, K>(device);
    t.sms = sm_count(device);
    return t;
  });
}

template <int Q, typename S> int step_ctas_per_sm(int device) {
  using Cfg = StepConfig<Q, S>;
  using Sh = ConfigShape<Q, S>;
  if (prepare_kernel<Q, S, kFlRuntime>(device) != cudaSuccess) return 0;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &n, step_kernel<Q, S, Cfg::W, Cfg::NS, Cfg::MINB, kFlRuntime>, Sh::NT,
          Sh::SMEM) != cudaSuccess)
    return 0;
  return n;
}

template <int Q, typename S, int FL>
static cudaError_t prepare_batch_kernel(int device) {
  using Cfg = StepConfig<Q, S>;
  using Sh = ConfigShape<Q, S>;
  static PerDevice<cudaError_t> once;
  return once.get(device, [] {
    cudaError_t e = cudaFuncSetAttribute(
        batch_step_kernel<Q, S, Cfg::W, Cfg::NS, Cfg::template batch_minb_tile<FL>(), false, FL>,
        cudaFuncAttributeMaxDynamicSharedMemorySize, Sh::SMEM);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(batch_step_kernel<Q, S, Cfg::W, Cfg::NS, Cfg::BATCH_MINB, true, FL>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, Sh::SMEM);
  });
}

template <int Q, typename S, int FL>
static cudaError_t launch_batch_fl(const BatchArgs<Q, typename Codec<S>::T, S>& args, int nctas,
                                   bool persistent, int device, cudaStream_t stream) {
  using Cfg = StepConfig<Q, S>;
  using Sh = ConfigShape<Q, S>;
  cudaError_t e = prepare_batch_kernel<Q, S, FL>(device);
  if (e != cudaSuccess) return e;
  // A programmatic dependent launch, as for the single-lattice step.
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nctas);
  cfg.blockDim = dim3(Sh::NT);
  cfg.dynamicSmemBytes = Sh::SMEM;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (persistent)
    return cudaLaunchKernelEx(&cfg, batch_step_kernel<Q, S, Cfg::W, Cfg::NS, Cfg::BATCH_MINB, true, FL>,
                              args);
  return cudaLaunchKernelEx(&cfg, batch_step_kernel<Q, S, Cfg::W, Cfg::NS, Cfg::template batch_minb_tile<FL>(), false, FL>,
                            args);
}

template <int Q, typename S>
cudaError_t launch_batch(const BatchArgs<Q, typename Codec<S>::T, S>& args, int nctas,
                         bool persistent, bool plain, int device, cudaStream_t stream) {
  return plain ? launch_batch_fl<Q, S, kFlExpPlain>(args, nctas, persistent, device, stream)
               : launch_batch_fl<Q, S, kFlRuntime>(args, nctas, persistent, device, stream);
}

// Residency per SM of the persistent batch kernel; also sets the shared-memory
// attribute of every batch kernel variant (outside any stream capture).
template <int Q, typename S> int batch_ctas_per_sm(int device) {
  using Cfg = StepConfig<Q, S>;
  using Sh = ConfigShape<Q, S>;
  if (prepare_batch_kernel<Q, S, kFlRuntime>(device) != cudaSuccess) return 0;
  if (prepare_batch_kernel<Q, S, kFlExpPlain>(device) != cudaSuccess) return 0;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &n, batch_step_kernel<Q, S, Cfg::W, Cfg::NS, Cfg::BATCH_MINB, true, kFlRuntime>, Sh::NT,
          Sh::SMEM) != cudaSuccess)
    return 0;
  return n;
}

template <int Q, typename S, int K, int FL> static cudaError_t prepare_batch_tile_k(int device) {
  using Cfg = TileConfig<Q, S, K>;
  static PerDevice<cudaError_t> once;
  return once.get(device, [] {
    return cudaFuncSetAttribute(batch_tile_kernel<typename Cfg::Sh, FL, Cfg::kCfg.minb>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::Sh::SMEM);
  });
}

template <int Q, typename S> cudaError_t prepare_batch_tiles(int shape, int device) {
  return with_shape<Q, S>(shape, [&]<int K>() {
    if constexpr (TileConfig<Q, S, K>::kCfg.steps != 1) return cudaErrorInvalidValue;
    else {
    const cudaError_t e = prepare_batch_tile_k<Q, S, K, kFlExpPlain>(device);
    return e != cudaSuccess ? e : prepare_batch_tile_k<Q, S, K, kFlRuntime>(device);
    }
  });
}

template <int Q, typename S>
cudaError_t launch_batch_tiles(int shape, const BatchArgs<Q, typename Codec<S>::T, S>& args,
                               int ntiles, bool plain, cudaStream_t stream) {
  return with_shape<Q, S>(shape, [&]<int K>() {
    using Cfg = TileConfig<Q, S, K>;
    using Sh = typename Cfg::Sh;
    if constexpr (Sh::TS != 1) {
      return cudaErrorInvalidValue;
    } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ntiles);
    cfg.blockDim = dim3(Sh::NT);
    cfg.dynamicSmemBytes = Sh::SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return plain ? cudaLaunchKernelEx(&cfg, batch_tile_kernel<Sh, kFlExpPlain, Cfg::kCfg.minb>, args)
                 : cudaLaunchKernelEx(&cfg, batch_tile_kernel<Sh, kFlRuntime, Cfg::kCfg.minb>, args);
    }
  });
}

}  // namespace lbm

#define LBM_INSTANTIATE_STEP(Q, S)                                                         \
  template cudaError_t lbm::launch_step<Q, S>(const PopMaps&, const CUtensorMap&,      \
                                              const lbm::StepArgs<lbm::Codec<S>::T, S>&,   \
                                              dim3, int, cudaStream_t);                    \
  template cudaError_t lbm::launch_tile<Q, S>(int, const PopMaps&, const uint32_t*, int, const lbm::StepArgs<lbm::Codec<S>::T, S>&, int, cudaStream_t, int); \
  template lbm::TileInfo lbm::tile_info<Q, S>(int, int); \
  template int lbm::step_ctas_per_sm<Q, S>(int);                                         \
  template cudaError_t lbm::launch_batch<Q, S>(                                          \
      const lbm::BatchArgs<Q, lbm::Codec<S>::T, S>&, int, bool, bool, int, cudaStream_t);     \
  template cudaError_t lbm::launch_batch_tiles<Q, S>(                                    \
      int, const lbm::BatchArgs<Q, lbm::Codec<S>::T, S>&, int, bool, cudaStream_t);           \
  template cudaError_t lbm::prepare_batch_tiles<Q, S>(int, int);                         \
  template int lbm::batch_ctas_per_sm<Q, S>(int);
