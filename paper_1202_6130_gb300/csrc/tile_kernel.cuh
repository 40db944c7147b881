// The fused time step on two-dimensional tiles: a CTA updates TW x TH nodes at
// once, for TS time steps, instead of marching row by row (step_kernel.cuh).
//
// What bounds a march on small and middle lattices is its serial chain: about
// 0.9 us per row (stage wait, psi, barrier, collision), with too few strips and
// segments to fill the chip.  A tile does all its rows at once: one load of
// everything it reads, psi of the tile and its halo, one barrier, the
// collision.  GB300, us per step, march -> tiles: D2Q9 128x64 FP32 6.4 -> 3.0 and
// FP64 40.6 -> 9.9, 400x200 FP32 7.9 -> 4.3, 1024x512 FP16S 9.2 -> 6.7, D2Q21
// 650x150 FP32 10.8 -> 6.4.  Tiles also need a quarter fewer instructions per
// node (no ring or stage bookkeeping per row: 5.8 warp instructions against 8.2
// on 2048x1024 FP16S) and, for D2Q21, no second read of the row from its stage
// with four stages pinned: D2Q21 4096x2048 FP32 314 -> 256 and FP16S 175 -> 155;
// FP64 2048x1024 726 -> 637.  Tiles that touch no edge and no wall run a second
// copy of the update without that code (IN): 63.3 against 65.4 us on 4096x2048
// FP16S; on small lattices, where every tile has an edge, it only costs.
//
// Two steps per launch (TS = 2, D2Q9 node pairs): the tile's populations stay in
// shared memory between the steps, so a pair of steps costs one launch, one load
// latency and one trip through HBM; the price is the first step on 2 more nodes
// on every side (larger tiles for the lattices that can afford them).  GB300, us
// per step, best one-step kernel -> two steps when they came -> with the shapes of
// launch.cuh, wall fields ahead of the wait and boxes fetched ahead into L2:
// 128x64 FP32 3.0 -> 2.1 -> 1.7, 400x200 FP32 4.3 -> 2.9 -> 2.4, 1024x512 FP32 8.3 ->
// 7.6 -> 7.3, 4096x2048 FP32 96 -> 80 -> 76, 8192x4096 FP32 368 -> 304 -> 290.  The DRAM
// traffic of the large ones halves; what bounds them then is latency between
// barriers, at 28 warps per SM and 52% of issue slots.  16-bit storage is bound by
// instruction issue on large lattices and stays at one step there.
//
// Tried and dropped: persistent CTAs that prefetch the next tile's boxes under
// the last collision (loop-invariant values took the registers: 184-628 bytes
// of spills, 1.3x slower with two steps; no gain with one step, which did not
// spill).
#pragma once

#include "node_update.cuh"
#include "step_kernel.cuh"
#include "tma.cuh"

namespace lbm {

// Shape and shared-memory layout of a tile CTA.
//
// The populations that the tile's TS steps read arrive as one TMA box per plane
// group (the planes with one c_y): BW columns (the tile and GX ghost columns on
// either side, so that the box starts on 16 bytes) by BH rows.  Row b of a
// group's box is the source row of node row y0 - BR + b, so a node pulls every
// population from the same box row.  Step s updates the tile and margin(s)
// nodes around it, which is what the later steps still read; nodes around the
// tile are other tiles' nodes (or their periodic images), recomputed with the
// same arithmetic.  Post-collision values go back into the boxes, to the place
// the next step pulls them from.
template <int Q_, typename S_, int TW_, int TH_, int NT_, int TS_, bool IN_> struct TileShape {
  using S = S_;
  using L = Lattice<Q_>;
  using P = Planes<Q_>;
  using T = typename Codec<S>::T;
  static constexpr int Q = Q_, R = L::R, TW = TW_, TH = TH_, NT = NT_, TS = TS_;
  static constexpr bool IN = IN_;  // a second copy of the update without edge and wall code
  static constexpr int GX = ghost_x<S, R>(), GY = ghost_y<R>();
  static constexpr int V = (sizeof(T) == 4 && (Q == 9 || sizeof(S) == 2)) ? 2 : 1;  // as StepShape
  static constexpr int margin(int s) { return 2 * R * (TS - 1 - s); }
  static constexpr int BR = R + margin(0);
  static constexpr int BW = TW + 2 * GX, BH = TH + 2 * BR;
  static constexpr int NBOX = 2 * R + 1;
  // Work items (node pairs, or nodes) of step s: prow(s) per row, over the
  // tile and its margin; slots(s) of them per thread.
  static constexpr int prow(int s) { return (TW + 2 * margin(s)) / V; }
  static constexpr int items(int s) { return prow(s) * (TH + 2 * margin(s)); }
  static constexpr int slots(int s) { return (items(s) + NT - 1) / NT; }
  // psi: RO columns and BR rows around the tile (RO even for pairs).
  static constexpr int RP = V == 2 ? (R + 1) / 2 * 2 : R;
  static constexpr int RO = margin(0) + RP;
  static constexpr int PW = TW + 2 * RO;
  // The psi columns beside the updated nodes are formed as whole items where
  // the boxes hold what their outer nodes pull, else node by node.
  static constexpr bool kHaloItems = RO + R <= GX;
  static constexpr uint32_t TX = Q * BW * BH * (uint32_t)sizeof(S);
  struct Tables {
    int pop[Q];  // element offset of population i of node column -GX, row -BR
    int box_cy[NBOX], box_plane[NBOX], box_depth[NBOX], box_off[NBOX], box_map[NBOX];
    int depth[kMaxMaps];
    int nmap, bytes;
  };
  static constexpr Tables make() {
    Tables t{};
    int off = 0;
    for (int j = 0; j < NBOX; ++j) {
      const int cy = j - R;
      int first = Q, n = 0;
      for (int i = 0; i < Q; ++i) {
        if (L::cy(i) != cy) continue;
        ++n;
        if (P::kTable.plane[i] < first) first = P::kTable.plane[i];
      }
      t.box_cy[j] = cy;
      t.box_plane[j] = first;
      t.box_depth[j] = n;
      t.box_off[j] = off;
      int k = 0;
      while (k < t.nmap && t.depth[k] != n) ++k;
      if (k == t.nmap) t.depth[t.nmap++] = n;
      t.box_map[j] = k;
      off += (n * BW * BH * (int)sizeof(S) + 127) / 128 * 128;
    }
    t.bytes = off;
    for (int i = 0; i < Q; ++i) {
      const int j = L::cy(i) + R;
      t.pop[i] = t.box_off[j] / (int)sizeof(S) + (P::kTable.plane[i] - t.box_plane[j]) * BW * BH;
    }
    return t;
  }
  static constexpr Tables kTab = make();
  static constexpr int NMAP = kTab.nmap;
  static constexpr int SMEM = 128 /*alignment slack*/ + kTab.bytes + PW * BH * (int)sizeof(T) + 16;
  static_assert(TW % 16 == 0 && NT % 32 == 0, "tile shape");
  static_assert(BW <= 256 && BH <= 256 && NMAP == kMapsOf<Q>, "tensor-map boxes");
  static_assert(margin(0) + 2 * R <= GX && margin(0) + 2 * R <= GY, "ghost frame");
  static_assert(TS == 1 || (TS % 2 == 0 && V == 2 && R == 1), "several steps: D2Q9 node pairs");
  static_assert(kHaloItems || R == 1, "halo columns node by node: R = 1");
};

// Advances the tile with origin (x0, y0) by TS time steps (kModeStep), or writes
// its moments (kModeMoments, TS = 1).  (xn, yn): a later CTA's tile to fetch into
// L2 meanwhile (xn < 0: none).
template <typename Sh, int MODE, int FL, typename Args>
__device__ __forceinline__ void tile_update(const CUtensorMap* src, const uint32_t* __restrict__ flags,
                                            int flag_pitch, const Args& a, int x0, int y0,
                                            int xn, int yn, unsigned char* smem_raw) {
  using S = typename Sh::S;
  using T = typename Sh::T;
  using C = Codec<S>;
  using L = typename Sh::L;
  constexpr int Q = Sh::Q, R = Sh::R, GX = Sh::GX, GY = Sh::GY, V = Sh::V, NT = Sh::NT;
  constexpr int PW = Sh::PW, BW = Sh::BW, BR = Sh::BR, TS = Sh::TS;
  unsigned char* const base = smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u);
  S* const st = reinterpret_cast<S*>(base);
  constexpr int kPopBytes = Sh::kTab.bytes;
  T* const psi = reinterpret_cast<T*>(base + kPopBytes);
  uint64_t* const bar = reinterpret_cast<uint64_t*>(psi + PW * Sh::BH);
  int* const s_abort = reinterpret_cast<int*>(bar + 1);
  const int tid = threadIdx.x;

  if (tid == 0) {
    mbar_init(bar, 1);
    *s_abort = 0;
    fence_barrier_init();
    static_for<0, Sh::NMAP>([&](auto kc) { prefetch_tensormap(&src[decltype(kc)::value]); });
  }
  auto wrap_x = [&](int x) { return x < 0 ? x + a.nx : (x >= a.nx ? x - a.nx : x); };
  auto wrap_y = [&](int y) { return y < 0 ? y + a.ny : (y >= a.ny ? y - a.ny : y); };
  // Column and row of the thread's k-th item of step s, whether it is updated
  // (its nodes exist, or are images of nodes), and its wall flag.
  auto item = [&](auto sc, int k, int& col, int& row) -> bool {
    constexpr int s = decltype(sc)::value;
    constexpr int M = Sh::margin(s), PROW = Sh::prow(s), NI = Sh::items(s);
    if constexpr (NT % PROW == 0) {  // every slot in the thread's first column
      row = tid / PROW + k * (NT / PROW) - M;
      col = V * (tid % PROW) - M;
    } else {
      const int p = tid + k * NT, q = p / PROW;
      row = q - M;
      col = V * (p - q * PROW) - M;
    }
    return (NI % NT == 0 || tid + k * NT < NI) && x0 + col < a.nx + M && y0 + row < a.ny + M;
  };
  auto flag_of = [&](auto sc, bool on, int col, int row) -> uint32_t {
    constexpr int M = Sh::margin(decltype(sc)::value);
    if (!a.wall.active || !on) return 0u;
    const int xw = M ? wrap_x(x0 + col) : x0 + col, yw = M ? wrap_y(y0 + row) : y0 + row;
    return flags[(int64_t)yw * flag_pitch + (xw >> 5)];
  };
  // Shapes for small lattices (one item per thread and step, every tile at an
  // edge or a wall) fetch the flags and wall fields of all steps ahead of the
  // wait for the previous launch: set_wall ran to its end before this launch was
  // enqueued, so they are static, and their latency leaves the step's chain
  // (0.25 of 2.1 us per step on 128x64).
  constexpr bool kEarlyWall = !Sh::IN && MODE == kModeStep;
  using Wall = std::conditional_t<V == 2, PairWall, NodeWall<T>>;
  uint32_t early_flag[kEarlyWall ? TS : 1];
  Wall early_wall[kEarlyWall ? TS : 1];
  if constexpr (kEarlyWall) {
    static_for<0, TS>([&](auto sc) {
      constexpr int s = decltype(sc)::value;
      static_assert(Sh::slots(s) == 1, "one item per thread and step");
      int c, r;
      const bool on = item(sc, 0, c, r);
      early_flag[s] = flag_of(sc, on, c, r);
      early_wall[s] = Wall{};
      if (early_flag[s]) {
        const int x = x0 + c, y = y0 + r;
        if constexpr (V == 2)
          early_wall[s] = load_wall(a, PairAt{wrap_x(x), wrap_y(y), true, TS > 1 || x + 1 < a.nx});
        else
          early_wall[s] = load_wall<T>(a, x, y);
      }
    });
  }
  griddep_wait();  // a programmatic dependent of the previous launch
  if (tid == 0) {
    mbar_arrive_expect_tx(bar, Sh::TX + a.extra_tx);
    static_for<0, Sh::NBOX>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      constexpr int cy = Sh::kTab.box_cy[j], off = Sh::kTab.box_off[j], map = Sh::kTab.box_map[j];
      constexpr int plane = Sh::kTab.box_plane[j];
      tma_load_3d(base + off, &src[map], bar, x0, y0 - BR - cy + GY, plane);
    });
    if (xn >= 0)  // the lines of a tile some waves ahead, into L2
      static_for<0, Sh::NBOX>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        constexpr int cy = Sh::kTab.box_cy[j], map = Sh::kTab.box_map[j], plane = Sh::kTab.box_plane[j];
        tma_prefetch_3d(&src[map], xn, yn - BR - cy + GY, plane);
      });
  }
  const uint32_t key = step_key<S, MODE, FL>(a);
  const bool simple_images = a.nx >= 2 * GX && a.ny >= 2 * GY && (V == 1 || (a.nx & 1) == 0);
  __syncthreads();  // the barrier is initialised

  // Address of population i as the node at (c, r) of the tile pulls it.
  auto pop = [&](auto ic, int c, int r) -> S* {
    constexpr int off = Sh::kTab.pop[decltype(ic)::value] + GX - L::cx(decltype(ic)::value);
    return st + (off + (r + BR) * BW + c);
  };
  auto psi_at = [&](int c, int r) -> T* { return psi + (r + BR) * PW + Sh::RO + c; };
  // psi of one node from its populations.
  auto node_psi = [&](int c, int r) {
    T H;
    static_for<0, Q>([&](auto ic) {
      const T v = C::load(*pop(ic, c, r));
      H = (decltype(ic)::value == 0) ? v : H + v;
    });
    if constexpr (V == 2)
      *psi_at(c, r) = pseudo_potential<Q, T, kPsiOf<FL>, C::kShifted>(
          a.phys, PairRho<S>::of(a.phys, H));
    else
      *psi_at(c, r) = pseudo_potential<Q, T, kPsiOf<FL>>(a.phys, H);
  };
  // Loads the item at (c, r) (a node pair or a node) into f, its sum into H,
  // and forms its psi.
  using F = std::conditional_t<V == 2, F2, T>;
  auto item_psi = [&](int c, int r, F (&f)[Q], F& H) {
    static_for<0, Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      const S* p = pop(ic, c, r);
      if constexpr (V == 1) {
        f[i] = C::load(*p);
      } else if constexpr ((L::cx(i) & 1) == 0) {
        f[i] = Pair<S>::load(*reinterpret_cast<const typename Pair<S>::Raw*>(p));
      } else {
        f[i] = Pair<S>::load1(p[0], p[1]);
      }
      H = (i == 0) ? f[i] : H + f[i];
    });
    if constexpr (V == 2)
      *reinterpret_cast<float2*>(psi_at(c, r)) =
          pair_psi<Q, S, FL>(a.phys, PairRho<S>::of(a.phys, H));
    else
      *psi_at(c, r) = pseudo_potential<Q, T, kPsiOf<FL>>(a.phys, H);
  };
  const bool strip_edge = x0 < GX || x0 + Sh::TW > a.nx - GX;
  // Tiles inside the lattice: no edge, no images.
  const bool interior = Sh::IN && x0 >= GX && x0 + Sh::TW <= a.nx - GX && y0 >= GY &&
                        y0 + Sh::TH <= a.ny - GY &&
                        (uint64_t)a.pitch * Sh::TH * sizeof(S) < (1ull << 32);  // 32-bit store offsets
  bool aborted = false, inside = false;
  static_for<0, TS>([&](auto sc) {
    constexpr int s = decltype(sc)::value;
    constexpr int M = Sh::margin(s), SL = Sh::slots(s), PROW = Sh::prow(s), NI = Sh::items(s);
    F f[SL][Q], H[SL];
    int col[SL], row[SL];
    uint32_t flag[SL];
    bool on[SL];
#pragma unroll
    for (int k = 0; k < SL; ++k) {
      on[k] = item(sc, k, col[k], row[k]);
      // A tile found inside by the first step's (larger) region stays so.
      flag[k] = kEarlyWall ? early_flag[kEarlyWall ? s : 0]
                           : (s > 0 && inside ? 0u : flag_of(sc, on[k], col[k], row[k]));
    }
    if constexpr (s == 0) {
      if (!mbar_wait_bounded(bar, 0, a.wait_ns)) *s_abort = 1;
    } else {
      __syncthreads();  // the previous step's populations are in place, its psi read
    }
#pragma unroll
    for (int k = 0; k < SL; ++k)
      if (NI % NT == 0 || tid + k * NT < NI) item_psi(col[k], row[k], f[k], H[k]);
    // psi of the rows above and below the updated nodes, then of the columns
    // on either side.
    constexpr int HP = Sh::kHaloItems ? PROW + 2 * Sh::RP / V : PROW;
    constexpr int HC = Sh::kHaloItems ? 2 * Sh::RP / V * (Sh::TH + 2 * M) : 0;
    for (int h = tid; h < 2 * R * HP + HC; h += NT) {
      int c, r;
      if (HC == 0 || h < 2 * R * HP) {
        const int q = h / HP;
        c = V * (h - q * HP) - M - (Sh::kHaloItems ? Sh::RP : 0);
        r = q < R ? q - R - M : Sh::TH + M + q - R;
      } else {
        constexpr int HR = Sh::TH + 2 * M;
        const int q = (h - 2 * R * HP) / HR;
        c = q < Sh::RP / V ? V * q - Sh::RP - M : Sh::TW + M + V * (q - Sh::RP / V);
        r = h - 2 * R * HP - q * HR - M;
      }
      F fh[Q], Hh;
      item_psi(c, r, fh, Hh);
    }
    if constexpr (!Sh::kHaloItems) {
      constexpr int NR = Sh::TH + 2 * M + 2;
      for (int h = NT - 1 - tid; h < 2 * NR; h += NT)
        node_psi(h < NR ? -M - 1 : Sh::TW + M, (h < NR ? h : h - NR) - M - 1);
    }
    if constexpr (Sh::IN && s == 0) {
      uint32_t any = 0;
#pragma unroll
      for (int k = 0; k < SL; ++k) any |= flag[k];
      inside = !__syncthreads_or((int)any) && interior;
    } else {
      __syncthreads();
    }
    // psi is complete; every population has been read.
    aborted = *s_abort != 0;
    if (aborted) return;
    auto collide = [&](auto ec) {
      constexpr bool E = decltype(ec)::value;
#pragma unroll
      for (int k = 0; k < SL; ++k) {
        if (E ? !on[k] : !(NI % NT == 0 || tid + k * NT < NI)) continue;
        const int x = x0 + col[k], y = y0 + row[k];
        auto psi_row = [&](int cy) -> const T* { return psi_at(col[k], row[k] + cy); };
        auto wall = [&]() -> Wall {
          if constexpr (kEarlyWall) return early_wall[s];
          else if constexpr (V == 2)
            return load_wall(a, PairAt{M ? wrap_x(x) : x, M ? wrap_y(y) : y, true, TS > 1 || x + 1 < a.nx});
          else return load_wall<T>(a, x, y);
        };
        if constexpr (V == 1) {
          node_update<Q, S, MODE, FL, E>(a, f[k], flag[k], x, y, strip_edge, simple_images, psi_row,
                                         wall);
        } else if constexpr (s == TS - 1 && (E || MODE != kModeStep)) {
          pair_update<Q, S, MODE, FL, true>(a, f[k], H[k], flag[k], x, y, strip_edge, simple_images,
                                            key + (uint32_t)s, psi_row, wall);
        } else {
          // Whole pairs: inside the lattice, or (two steps: even nx) images of
          // pairs of whole nodes.
          const PairAt at{E ? wrap_x(x) : x, E ? wrap_y(y) : y, true, true};
          const PairState<Q, S, E> n(a, f[k], H[k], flag[k], psi_row, wall);
          typename Pair<S>::Raw raw[Q];
          pair_collide<Q, S, FL>(a, n, f[k], H[k], at, key + (uint32_t)s, raw);
          if constexpr (s == TS - 1) {
            S* org = a.fout + (int64_t)(y0 + GY) * a.pitch + x0 + GX;
            pair_store_inside<Q, S>(a, raw, org, (uint32_t)row[k] * (uint32_t)a.pitch + (uint32_t)col[k]);
          } else {
            static_for<0, Q>([&](auto ic) {
              constexpr int i = decltype(ic)::value;
              constexpr int off = Sh::kTab.pop[i] + GX;
              *reinterpret_cast<typename Pair<S>::Raw*>(
                  st + (off + (row[k] + L::cy(i) + BR) * BW + col[k])) = raw[i];
            });
          }
        }
      }
    };
    if constexpr (Sh::IN) {
      if (inside) {
        collide(std::false_type{});
        return;
      }
    }
    collide(std::true_type{});
  });
  // Only now may the next launch's CTAs come: those that come while this one's
  // still compute pile up on the SMs that are free at that moment, and several
  // steps ahead, since each lets the next one in (GB300, us per step with the
  // trigger at the start / here: 128x64 FP64 17 / 7.8, 400x200 FP64 43 / 30, 128x64
  // FP32 1.85 / 1.69, D2Q21 FP32 4.4 / 3.3, 650x150 6.3 / 5.9).
  griddep_launch_dependents();
  if (aborted && tid == 0) {
    // The boxes never arrived in full.  Record it, retire the bytes that the
    // barrier was told to expect beyond its copies (the test hook), and wait
    // (bounded) for the copies still in flight.
    atomicOr(a.status, kStatusTimeout);
    if (a.extra_tx) mbar_complete_tx(bar, a.extra_tx);
    mbar_wait_bounded(bar, 0, a.wait_ns);
  }
}

// TS time steps of one lattice, one CTA per tile; ty0: the launch's first row of
// tiles (a grid holds 65,535 of them, taller lattices take several launches).
// ahead > 0: each CTA also brings the boxes of the tile `ahead` places on into L2,
// half a round of resident CTAs early, so that its loads find them there instead
// of waiting for HBM (8192x4096 FP32 301 -> 286 us per step, 4096x2048 FP16S 62.6 ->
// 61.0; a whole round or more ahead gains nothing for FP32).
template <typename Sh, int MODE, int FL, int MINB>
__global__ void __launch_bounds__(Sh::NT, MINB)
    tile_kernel(const __grid_constant__ PopMaps src, const uint32_t* __restrict__ flags,
                int flag_pitch, int ahead, int ty0, const StepArgs<typename Sh::T, typename Sh::S> a) {
  extern __shared__ unsigned char smem_raw[];
  const int ty = blockIdx.y + ty0;
  int xn = -1, yn = 0;
  if (ahead > 0) {
    const int next = ty * gridDim.x + blockIdx.x + ahead, tn = next / gridDim.x;
    if (tn * Sh::TH < a.ny) {
      xn = (next - tn * gridDim.x) * Sh::TW;
      yn = tn * Sh::TH;
    }
  }
  tile_update<Sh, MODE, FL>(src.m, flags, flag_pitch, a, blockIdx.x * Sh::TW, ty * Sh::TH, xn, yn,
                            smem_raw);
  if constexpr (MODE == kModeStep)
    if (blockIdx.x == 0 && ty == 0 && threadIdx.x == 0) advance_key<MODE>(a, Sh::TS);
}

// One step of up to kChunk lattices of a batch on tiles: CTA b updates tile b of
// the chunk, numbered member by member and, within a member, row by row
// (nstrip tiles per row).  Arguments as for batch_step_kernel.
template <typename Sh, int FL, int MINB>
__global__ void __launch_bounds__(Sh::NT, MINB)
    batch_tile_kernel(const __grid_constant__ BatchArgs<Sh::Q, typename Sh::T, typename Sh::S> P) {
  extern __shared__ unsigned char smem_raw[];
  const int m = batch_member(P, (int)blockIdx.x);
  const int local = (int)blockIdx.x - P.tile0[m], ty = local / P.nstrip[m];
  const auto& a = P.a[m];
  tile_update<Sh, kModeStep, FL>(P.map[m], P.flag_words[m], flag_words_per_row(a.nx), a,
                                 (local - ty * P.nstrip[m]) * Sh::TW, ty * Sh::TH, -1, 0, smem_raw);
  if (threadIdx.x == 0 && local == 0) advance_key<kModeStep>(a, Sh::TS);
}

}  // namespace lbm
