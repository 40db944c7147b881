// The update of one node, and of a pair of horizontally adjacent nodes in packed
// FP32: moments, force, EDM-BGK collision, rounding and the store with its
// periodic images.  Shared by the row march (step_kernel.cuh) and the tile
// kernel (tile_kernel.cuh), so that both give the same bits.
#pragma once

#include "f2.cuh"
#include "lattice.cuh"
#include "node.cuh"
#include "step_args.cuh"

namespace lbm {

// rho from the sum H of a node's stored values: H itself, or for 16-bit
// storage H / sigma + rho_s (the shifts w_i rho_s sum to rho_s).
template <typename S> struct PairRho {
  using C = Codec<S>;
  static constexpr float kInvScale = 1.0f / float(C::kScale);
  __device__ __forceinline__ static float of(const Physics<float>& P, float H) {
    if constexpr (C::kShifted) return fmaf(H, kInvScale, P.rho_s);
    else return H;
  }
  __device__ __forceinline__ static F2 of(const Physics<float>& P, F2 H) {
    if constexpr (C::kShifted) return fma2(H, F2::splat(kInvScale), F2::splat(P.rho_s));
    else return H;
  }
};

// psi of both nodes of a pair.
template <int Q, typename S, int FL>
__device__ __forceinline__ float2 pair_psi(const Physics<float>& P, F2 rho) {
  constexpr int kPsiKind = kPsiOf<FL>;
  constexpr bool kFastExp = Codec<S>::kShifted;
  if constexpr (kPsiKind == 0 && kFastExp) {
    // psi_exp_fast of both nodes, the product and the fused multiply-add packed
    const F2 e2 = rho * F2::splat(P.exp2_scale);
    return fma2(F2(ex2_approx(e2.x()), ex2_approx(e2.y())), F2::splat(-P.rho0), F2::splat(P.rho0)).v;
  } else {
    return make_float2(pseudo_potential<Q, float, kPsiKind, kFastExp>(P, rho.x()),
                       pseudo_potential<Q, float, kPsiKind, kFastExp>(P, rho.y()));
  }
}

// rho and u = (j + F / 2) / rho (or j + F / 2) of node n, FP64.
template <typename T, typename Args>
__device__ __forceinline__ void write_moments(const Args& a, int64_t n, T rho, T jx, T jy, T Fx,
                                              T Fy) {
  a.out_rho[n] = (double)rho;
  if (a.momentum) {
    a.out_ux[n] = (double)jx + 0.5 * (double)Fx;
    a.out_uy[n] = (double)jy + 0.5 * (double)Fy;
  } else if constexpr (sizeof(T) == 4) {
    const float r2 = __fadd_rn(rho, rho), rc2 = __frcp_rn(r2);
    a.out_ux[n] = half_force_velocity(jx, Fx, rho, r2, rc2);
    a.out_uy[n] = half_force_velocity(jy, Fy, rho, r2, rc2);
  } else {
    const T y = T(1) / rho;
    a.out_ux[n] = div_rho<T>(jx + 0.5 * Fx, rho, y);
    a.out_uy[n] = div_rho<T>(jy + 0.5 * Fy, rho, y);
  }
}

// The rows of psi around a node: operator()(c_y) is the shared-memory row c_y above
// it, at its column.  (A march passes the pointers themselves: computing them
// on demand cost the batch march 4 registers and 7% of its time.)
template <typename T, int R> struct PsiRows {
  const T* row[2 * R + 1];
  __device__ __forceinline__ const T* operator()(int cy) const { return row[R + cy]; }
};

// Where a pair sits in the lattice (its first node; for an image of a pair, the
// pair itself), and which of its nodes exist.
struct PairAt {
  int x, y;
  bool ok0, ok1;
};

// The wall fields of a pair (phi_S^eps, S, U_wall; zero where a node does not
// exist), and of a node.
struct PairWall {
  F2 phe, Sx, Sy, ux, uy;
};
template <typename Args> __device__ __forceinline__ PairWall load_wall(const Args& a, const PairAt& at) {
  float v[5][2] = {};
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    if (e == 0 ? at.ok0 : at.ok1) {
      const int64_t n = (int64_t)at.y * a.nx + at.x + e;
      v[0][e] = a.wall.phie[n];
      v[1][e] = a.wall.sx[n];
      v[2][e] = a.wall.sy[n];
      if (a.wall.uwx) {
        v[3][e] = a.wall.uwx[n];
        v[4][e] = a.wall.uwy[n];
      }
    }
  }
  return {F2(v[0][0], v[0][1]), F2(v[1][0], v[1][1]), F2(v[2][0], v[2][1]), F2(v[3][0], v[3][1]),
          F2(v[4][0], v[4][1])};
}
template <typename T> struct NodeWall {
  T phe, Sx, Sy, ux, uy;
};
template <typename T, typename Args>
__device__ __forceinline__ NodeWall<T> load_wall(const Args& a, int x, int y) {
  const int64_t n = (int64_t)y * a.nx + x;
  NodeWall<T> w{a.wall.phie[n], a.wall.sx[n], a.wall.sy[n], T(0), T(0)};
  if (a.wall.uwx) {
    w.ux = a.wall.uwx[n];
    w.uy = a.wall.uwy[n];
  }
  return w;
}

// A pair's moments, velocity and total force.  f_: its stored values (f, or
// h = sigma (f - w rho_s) for 16-bit storage); Hm: their sum in table order.
// psi_row(c_y): the shared-memory row of psi at c_y rows above, at the pair's
// first column.  flag: non-zero where wall terms act; wall(): the wall fields,
// called there only.
template <int Q, typename S, bool EDGE = true> struct PairState {
  using L = Lattice<Q>;
  using C = Codec<S>;
  using T = float;
  static constexpr T kInvScale = PairRho<S>::kInvScale;
  F2 rho, inv_rho, ux, uy, Jx, Jy, jx, jy, Fx, Fy;

  template <typename Args, typename Row, typename Wall>
  __device__ __forceinline__ PairState(const Args& a, const F2 (&f_)[Q], const F2 Hm, uint32_t flag,
                                       Row&& psi_row, Wall&& wall) {
    // J = sum f_i c_i (D2Q9: the diagonal differences f5 - f7 and f8 - f6 shared
    // by its two components; otherwise in table order), j = J / sigma (the
    // shifts carry no momentum).
    rho = PairRho<S>::of(a.phys, Hm);
    if constexpr (Q == 9) {
      const F2 d57 = f_[5] - f_[7], d86 = f_[8] - f_[6];
      Jx = ((f_[1] - f_[3]) + d57) + d86;
      Jy = ((f_[2] - f_[4]) + d57) - d86;
    } else {
      Jx = F2::splat(0.f);
      Jy = F2::splat(0.f);
      static_for<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        if constexpr (L::cx(i) != 0) Jx = fma2(f_[i], F2::splat(T(L::cx(i))), Jx);
        if constexpr (L::cy(i) != 0) Jy = fma2(f_[i], F2::splat(T(L::cy(i))), Jy);
      });
    }
    jx = Jx;
    jy = Jy;
    if constexpr (C::kShifted && C::kScale != 1.0f) {
      jx = Jx * F2::splat(kInvScale);
      jy = Jy * F2::splat(kInvScale);
    }
    inv_rho = F2(rcp_node<S, float>(rho.x()), rcp_node<S, float>(rho.y()));
    ux = jx * inv_rho;
    uy = jy * inv_rho;

    // Neighbour psi, sum_i w_i psi(x + c_i) c_i.
    F2 sfx = F2::splat(0.f), sfy = F2::splat(0.f), psi_c;
    if constexpr (Q != 9) {
      // The psi pair at column offset c_x is one aligned pair (c_x even) or the
      // halves of two.
      auto ring_at = [&](int cy, int o) -> float2 {
        return *reinterpret_cast<const float2*>(psi_row(cy) + o);
      };
      psi_c = F2(ring_at(0, 0));
      static_for<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        constexpr int cx = L::cx(i), cy = L::cy(i);
        if constexpr (i == L::REST) return;
        F2 nb;
        if constexpr ((cx & 1) == 0) {
          nb = F2(ring_at(cy, cx));
        } else {
          nb = F2(ring_at(cy, cx - 1).y, ring_at(cy, cx + 1).x);
        }
        if constexpr (cx != 0) sfx = fma2(nb, F2::splat(T(L::w(i) * cx)), sfx);
        if constexpr (cy != 0) sfy = fma2(nb, F2::splat(T(L::w(i) * cy)), sfy);
      });
    } else {
      // D2Q9: three aligned pairs per ring row cover the pair's columns
      // and one more on either side.
      static_for<0, 3>([&](auto rc) {
        constexpr int cy = decltype(rc)::value - 1;
        const T* row = psi_row(cy);
        const float2 A = *reinterpret_cast<const float2*>(row - 2);
        const float2 B = *reinterpret_cast<const float2*>(row);
        const float2 Cc = *reinterpret_cast<const float2*>(row + 2);
        const F2 pm(A.y, B.x), p0(B), pp(B.y, Cc.x);   // psi at c_x = -1, 0, +1
        if constexpr (cy == 0) {
          psi_c = p0;
          sfx = fma2(pp - pm, F2::splat(T(L::w(1))), sfx);  // (1,0) and (-1,0)
        } else {
          // (0,cy): weight w_axis; (+-1, cy): weight w_diag
          constexpr T sg = cy > 0 ? T(1) : T(-1);
          sfy = fma2(p0, F2::splat(sg * T(L::w(2))), sfy);
          sfy = fma2(pp + pm, F2::splat(sg * T(L::w(5))), sfy);
          sfx = fma2(pp - pm, F2::splat(T(L::w(5))), sfx);
        }
      });
    }

    // Force: F_FF, then the wall terms on flagged chunks, then body force.
    const F2 mg = F2::splat(-a.phys.G) * psi_c;
    if (EDGE && flag != 0u) {
      const F2 ffx = mg * sfx, ffy = mg * sfy;
      const PairWall w = wall();
      const F2 rp = rho * w.phe;
      const F2 dfx = rp * (w.ux - ux - ffx * inv_rho);
      const F2 dfy = rp * (w.uy - uy - ffy * inv_rho);
      Fx = ((ffx + rho * w.Sx) + dfx) + F2::splat(a.phys.bfx);
      Fy = ((ffy + rho * w.Sy) + dfy) + F2::splat(a.phys.bfy);
    } else {
      Fx = fma2(mg, sfx, F2::splat(a.phys.bfx));
      Fy = fma2(mg, sfy, F2::splat(a.phys.bfy));
    }
  }
};

// The collision of a pair and its rounding to storage.  f_ is overwritten.
template <int Q, typename S, int FL, typename Args, typename St>
__device__ __forceinline__ void pair_collide(const Args& a, const St& n, F2 (&f_)[Q],
                                             const F2 Hm, const PairAt& at, uint32_t key,
                                             typename Pair<S>::Raw (&raw)[Q]) {
  using L = Lattice<Q>;
  using E = EqConst<Q>;
  using C = Codec<S>;
  using PR = Pair<S>;
  using T = float;
  const F2 rho = n.rho, inv_rho = n.inv_rho, ux = n.ux, uy = n.uy;
  if (!(fabsf(rho.x()) <= 3.0e38f) || (at.ok1 && !(fabsf(rho.y()) <= 3.0e38f)))
    atomicOr(a.status, kStatusNonFinite);
  const F2 usx = fma2(n.Fx, inv_rho, ux);
  const F2 usy = fma2(n.Fy, inv_rho, uy);
  // EDM-BGK in pair form (see node_collide), packed over the two nodes
  // and written as fused multiply-adds: with ca = c.(u* - g u) / theta
  // and sb = omega - B + ((c.u*)^2 - g (c.u)^2) / (2 theta^2),
  // f_post(+-c) = g f(+-c) + w rho (sb +- ca).
  const F2 gg = F2::splat(a.phys.one_m_omega), ngg = F2::splat(-a.phys.one_m_omega);
  const F2 ax3 = fma2(ngg, ux, usx) * F2::splat(T(E::inv_theta));
  const F2 ay3 = fma2(ngg, uy, usy) * F2::splat(T(E::inv_theta));
  const F2 us2 = fma2(usy, usy, usx * usx), u2 = fma2(uy, uy, ux * ux);
  const F2 wB = fma2(fma2(ngg, u2, us2), F2::splat(-T(E::inv_2theta)),
                     F2::splat(a.phys.omega));
  if (FL == kFlRuntime && a.phys.project) {
    // rare path: per node.  The projection is linear and maps the
    // shift w_i rho_s to itself, so it acts on h with (H, J) as it
    // acts on f with (rho, j).
    T fa[Q], fb[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      fa[i] = f_[i].x();
      fb[i] = f_[i].y();
    }
    project<Q, T>(fa, Hm.x(), n.Jx.x(), n.Jy.x());
    project<Q, T>(fb, Hm.y(), n.Jx.y(), n.Jy.y());
#pragma unroll
    for (int i = 0; i < Q; ++i) f_[i] = F2(fa[i], fb[i]);
  }
  if constexpr (C::kShifted) {
    // The same update on h = sigma (f - w rho_s):
    //   h_post(+-c) = g h(+-c) + sigma w [rho (sb +- ca) - omega rho_s].
    const F2 nwr = F2::splat(a.phys.neg_omega_rho_s);
    static_for<0, Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      constexpr int j = opposite<Q>(i);
      if constexpr (i != L::REST && i < j) {
        const F2 cs = cdot2<L::cx(i), L::cy(i)>(usx, usy);
        const F2 cu = cdot2<L::cx(i), L::cy(i)>(ux, uy);
        const F2 ca = cdot2<L::cx(i), L::cy(i)>(ax3, ay3);
        const F2 t = fma2(ngg, cu * cu, cs * cs);
        const F2 sb = fma2(t, F2::splat(T(E::inv_2theta2)), wB);
        const F2 z = fma2(rho, sb, nwr);
        const F2 sw = F2::splat(T(C::kScale * L::w(i)));
        const F2 hi = fma2(gg, f_[i], sw * fma2(rho, ca, z));
        const F2 hj = fma2(gg, f_[j], sw * fma2(rho, -ca, z));
        f_[i] = hi;
        f_[j] = hj;
      }
    });
  } else {
    static_for<0, Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      constexpr int j = opposite<Q>(i);
      // The rest population comes from the mass closure below.
      if constexpr (i != L::REST && i < j) {
        const F2 cs = cdot2<L::cx(i), L::cy(i)>(usx, usy);
        const F2 cu = cdot2<L::cx(i), L::cy(i)>(ux, uy);
        const F2 ca = cdot2<L::cx(i), L::cy(i)>(ax3, ay3);
        const F2 wr = F2::splat(T(L::w(i))) * rho;
        const F2 t = fma2(ngg, cu * cu, cs * cs);
        const F2 sb = fma2(t, F2::splat(T(E::inv_2theta2)), wB);
        const F2 fi = fma2(gg, f_[i], wr * (sb + ca));
        const F2 fj = fma2(gg, f_[j], wr * (sb - ca));
        f_[i] = fi;
        f_[j] = fj;
      }
    });
  }
  {  // mass closure of the rest population: the stored values sum to
     // H (rho, or sigma (rho - rho_s) for 16-bit storage) after the
     // collision as before it
    constexpr int i0 = L::REST == 0 ? 1 : 0;
    F2 moving = f_[i0];
#pragma unroll
    for (int i = i0 + 1; i < Q; ++i)
      if (i != L::REST) moving += f_[i];
    f_[L::REST] = Hm - moving;
  }
  // Round both nodes once (stochastic rounding: bits from the node pair and
  // the step).
  if constexpr (C::kShifted) {
    if (rounds_stochastically<FL>(a)) {
      const uint32_t h = sr_hash((uint32_t)at.x, (uint32_t)at.y, key);
      static_for<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        raw[i] = PR::store_sr(f_[i], h * sr_multiplier(i));
      });
    } else {
#pragma unroll
      for (int i = 0; i < Q; ++i) raw[i] = PR::store_rn(f_[i]);
    }
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i) raw[i] = PR::store_rn(f_[i]);
  }
}

// The primary store of a pair at (xp, yo) plus its periodic images.
// LANES: on lattices of odd width whose nodes have at most one image column and
// row, the images go out node by node without the general loop.
// strip_edge: the pair may lie within GX of a side; simple_images: every pair
// has at most one image column and one image row, and they are pairs again.
template <int Q, typename S, bool LANES, typename Args>
__device__ __forceinline__ void pair_store(const Args& a, const typename Pair<S>::Raw (&raw)[Q],
                                           int xp, int yo, bool strip_edge, bool simple_images) {
  using PR = Pair<S>;
  constexpr int GX = ghost_x<S, Lattice<Q>::R>(), GY = ghost_y<Lattice<Q>::R>();
  const bool pair_ok = xp + 1 < a.nx;  // both nodes exist
  S* out = a.fout + (int64_t)(yo + GY) * a.pitch + xp + GX;
  if (pair_ok) {
    static_for<0, Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      *reinterpret_cast<typename PR::Raw*>(out + Planes<Q>::template plane<i> * a.plane) =
          raw[i];
    });
  } else {
    static_for<0, Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      out[Planes<Q>::template plane<i> * a.plane] = PR::lane(raw[i], 0);
    });
  }
  const bool xedge = strip_edge && (xp < GX || xp + 1 >= a.nx - GX);
  const bool yedge = yo < GY || yo >= a.ny - GY;
  if ((xedge || yedge) && pair_ok && simple_images) {
    // Both nodes of the pair have the same images: at most one
    // column shift (+-nx) and one row shift (+-ny), stored as pairs.
    const int sx = !xedge ? 0 : (xp < GX ? a.nx : -a.nx);
    const int64_t sy = !yedge ? 0 : (int64_t)(yo < GY ? a.ny : -a.ny) * a.pitch;
    auto put = [&](int64_t d) {
      static_for<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        *reinterpret_cast<typename PR::Raw*>(out + d + Planes<Q>::template plane<i> * a.plane) =
            raw[i];
      });
    };
    if (sx != 0) put(sx);
    if (sy != 0) {
      put(sy);
      if (sx != 0) put(sy + sx);
    }
  } else if (LANES && (xedge || yedge) && a.nx >= 2 * GX && a.ny >= 2 * GY) {
    const int64_t sy = !yedge ? 0 : (int64_t)(yo < GY ? a.ny : -a.ny) * a.pitch;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (xp + e >= a.nx) break;
      const int sx = xp + e < GX ? a.nx : (xp + e >= a.nx - GX ? -a.nx : 0);
      auto put = [&](int64_t d) {
        static_for<0, Q>([&](auto ic) {
          constexpr int i = decltype(ic)::value;
          out[d + e + Planes<Q>::template plane<i> * a.plane] = PR::lane(raw[i], e);
        });
      };
      if (sx != 0) put(sx);
      if (sy != 0) {
        put(sy);
        if (sx != 0) put(sy + sx);
      }
    }
  } else if (xedge || yedge) {
#pragma unroll 1
    for (int e = 0; e < 2; ++e) {
      const int xn = xp + e;
      if (xn >= a.nx) break;
      int xs = xn;
      while (xs - a.nx >= -GX) xs -= a.nx;
      int ya = yo;
      while (ya - a.ny >= -GY) ya -= a.ny;
      for (int ym = ya; ym < a.ny + GY; ym += a.ny) {
        for (int xm = xs; xm < a.nx + GX; xm += a.nx) {
          if (xm == xn && ym == yo) continue;
          S* o2 = a.fout + (int64_t)(ym + GY) * a.pitch + xm + GX;
          static_for<0, Q>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            o2[Planes<Q>::template plane<i> * a.plane] = PR::lane(raw[i], e);
          });
        }
      }
    }
  }
}

// The store of a pair without images, off elements after org: with the CTA's
// origin and the pair's offset in it kept apart, a plane's address is a base that
// the CTA shares plus one 32-bit offset.
template <int Q, typename S, typename Args>
__device__ __forceinline__ void pair_store_inside(const Args& a, const typename Pair<S>::Raw (&raw)[Q],
                                                  S* org, uint32_t off) {
  static_for<0, Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    char* base = reinterpret_cast<char*>(org + Planes<Q>::template plane<i> * a.plane);
    *reinterpret_cast<typename Pair<S>::Raw*>(base + off * (uint32_t)sizeof(S)) = raw[i];
  });
}

// Updates the node pair (xp, yo), (xp + 1, yo) and stores the result
// (kModeStep) or the moments (kModeMoments).
template <int Q, typename S, int MODE, int FL, bool LANES, typename Args, typename Row, typename Wall>
__device__ __forceinline__ void pair_update(const Args& a, F2 (&f_)[Q], const F2 Hm, uint32_t flag,
                                            int xp, int yo, bool strip_edge, bool simple_images,
                                            uint32_t key, Row&& psi_row, Wall&& wall) {
  const PairAt at{xp, yo, xp < a.nx, xp + 1 < a.nx};
  const PairState<Q, S> n(a, f_, Hm, flag, psi_row, wall);
  if (!at.ok0) return;
  if constexpr (MODE == kModeStep) {
    typename Pair<S>::Raw raw[Q];
    pair_collide<Q, S, FL>(a, n, f_, Hm, at, key, raw);
    pair_store<Q, S, LANES>(a, raw, xp, yo, strip_edge, simple_images);
  } else {
    if (!(fabsf(n.rho.x()) <= 3.0e38f) || (at.ok1 && !(fabsf(n.rho.y()) <= 3.0e38f)))
      atomicOr(a.status, kStatusNonFinite);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (e == 1 && !at.ok1) break;
      const int64_t i = (int64_t)yo * a.nx + xp + e;
      const float r = e == 0 ? n.rho.x() : n.rho.y();
      write_moments(a, i, r, e == 0 ? n.jx.x() : n.jx.y(), e == 0 ? n.jy.x() : n.jy.y(),
                    e == 0 ? n.Fx.x() : n.Fx.y(), e == 0 ? n.Fy.x() : n.Fy.y());
    }
  }
}

// Updates the node (x, yo) from its populations f and stores the result
// (kModeStep) or the moments (kModeMoments).  Arguments as for pair_update.
template <int Q, typename S, int MODE, int FL, bool EDGE = true, typename T, typename Args,
          typename Row, typename Wall>
__device__ __forceinline__ void node_update(const Args& a, T (&f)[Q], uint32_t flag, int x, int yo,
                                            bool strip_edge, bool simple_images, Row&& psi_row,
                                            Wall&& wall) {
  using L = Lattice<Q>;
  using C = Codec<S>;
  constexpr int R = L::R;
  constexpr int GX = ghost_x<S, R>(), GY = ghost_y<R>();
  T rho, jx, jy;
  node_moments<Q, T>(f, rho, jx, jy);
  const T inv_rho = rcp_node<S, T>(rho);
  const T ux = div_rho<T>(jx, rho, inv_rho);
  const T uy = div_rho<T>(jy, rho, inv_rho);

  // sum_i w_i psi(x + c_i) c_i (rest state contributes 0).
  // prow[R + c_y]: psi of node row yo + c_y, at this node's column.
  const T* prow[2 * R + 1];
  static_for<0, 2 * R + 1>([&](auto rc) {
    constexpr int cy = decltype(rc)::value - R;
    prow[R + cy] = psi_row(cy);
  });
  const T psi_c = prow[R][0];
  T sfx = 0, sfy = 0;
  if constexpr (sizeof(T) == 8) {
    // Opposite neighbours differenced first, one product per pair and
    // component (as many operations on the FP64 pipe as there are pairs).
    static_for<0, Q>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      constexpr int cx = L::cx(i), cy = L::cy(i);
      if constexpr (i < opposite<Q>(i)) {
        const T nb = prow[R + cy][cx] - prow[R - cy][-cx];
        if constexpr (cx != 0) sfx = fma(L::w(i) * cx, nb, sfx);
        if constexpr (cy != 0) sfy = fma(L::w(i) * cy, nb, sfy);
      }
    });
  } else static_for<0, Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    if constexpr (L::cx(i) != 0 || L::cy(i) != 0) {
      const T nb = prow[R + L::cy(i)][L::cx(i)];
      const T wn = T(L::w(i)) * nb;
      if constexpr (L::cx(i) != 0) sfx += cmul<L::cx(i)>(wn);
      if constexpr (L::cy(i) != 0) sfy += cmul<L::cy(i)>(wn);
    }
  });

  // Wall terms only on flagged (row, 32-column chunk) pairs.
  const bool has_wall = EDGE && flag != 0u && x < a.nx;
  NodeWall<T> w{};
  if (has_wall) w = wall();
  T Fx, Fy;
  node_force<T>(a.phys, rho, ux, uy, psi_c, sfx, sfy, has_wall, w.phe, w.Sx, w.Sy, w.ux, w.uy,
                inv_rho, Fx, Fy);

  if (!EDGE || x < a.nx) {
    if (!(fabs(rho) <= T(3.0e38))) atomicOr(a.status, kStatusNonFinite);
    if constexpr (MODE == kModeStep) {
      const T usx = ux + div_rho<T>(Fx, rho, inv_rho);
      const T usy = uy + div_rho<T>(Fy, rho, inv_rho);
      if (FL == kFlRuntime && a.phys.project) project<Q, T>(f, rho, jx, jy);
      node_collide<Q, T>(a.phys, f, rho, ux, uy, usx, usy);
      // The primary store plus periodic images inside the ghost frame.
      S e[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) e[i] = C::store_rn(f[i]);
      S* out = a.fout + (int64_t)(yo + GY) * a.pitch + x + GX;
      static_for<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        out[Planes<Q>::template plane<i> * a.plane] = e[i];
      });
      // Periodic images exist only for nodes within GX of a side or GY of
      // the top or bottom; the strip test is per CTA, the row test per row.
      if constexpr (!EDGE) return;
      const bool xedge = strip_edge && (x < GX || x >= a.nx - GX);
      const bool yedge = yo < GY || yo >= a.ny - GY;
      if ((xedge || yedge) && simple_images) {
        // at most one image column (+-nx) and one image row (+-ny)
        const int sx = !xedge ? 0 : (x < GX ? a.nx : -a.nx);
        const int64_t sy = !yedge ? 0 : (int64_t)(yo < GY ? a.ny : -a.ny) * a.pitch;
        auto put = [&](int64_t d) {
          static_for<0, Q>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            out[d + Planes<Q>::template plane<i> * a.plane] = e[i];
          });
        };
        if (sx != 0) put(sx);
        if (sy != 0) {
          put(sy);
          if (sx != 0) put(sy + sx);
        }
      } else if (xedge || yedge) {
        int xa = x;
        while (xa - a.nx >= -GX) xa -= a.nx;
        int ya = yo;
        while (ya - a.ny >= -GY) ya -= a.ny;
        for (int ym = ya; ym < a.ny + GY; ym += a.ny) {
          for (int xm = xa; xm < a.nx + GX; xm += a.nx) {
            if (xm == x && ym == yo) continue;
            S* o2 = a.fout + (int64_t)(ym + GY) * a.pitch + xm + GX;
            static_for<0, Q>([&](auto ic) {
              constexpr int i = decltype(ic)::value;
              o2[Planes<Q>::template plane<i> * a.plane] = e[i];
            });
          }
        }
      }
    } else {
      const int64_t n = (int64_t)yo * a.nx + x;
      write_moments(a, n, rho, jx, jy, Fx, Fy);
    }
  }
}

}  // namespace lbm
