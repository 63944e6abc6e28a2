// lbpf_plane.cuh -- the 2D step of large planes: one warp per tile, two x-adjacent nodes per lane.
//
// A warp covers 60 interior columns (lanes 1 to 30; lanes 0 and 31 recompute the neighbours' edge
// nodes) and marches along the paper's y (the kernels' z) over a chunk of rows.  phi of three rows
// sits in registers, neighbours along x come from the next lanes by shuffle, and the moments of
// the next step are gathered from the lane's own collisions and its neighbours' by shuffle, so
// there is no shared memory and no barrier, and the distributions are read once.  Rows of even
// length; bit for bit the results of the other forms.
#pragma once

#include "lbpf_nodepair.cuh"

namespace lbpf {

static_assert(2 * TILE_X == 60, "lanes 1 to 30 of a warp, two nodes each");

// The stored numbers that a pair of values becomes.
template <typename S>
__device__ __forceinline__ F2 as_stored(F2 v) {
  using C = Codec<S>;
  return F2{C::raw(C::pack(v.x)), C::raw(C::pack(v.y))};
}

// Neighbours of a pair along x in a row held by the warp: .x left of the first node, .y right of the
// second, mirror ghosts at the walls.
__device__ __forceinline__ F2 beside(F2 v, bool wl, bool wr) {
  const float l = __shfl_up_sync(0xffffffffu, v.y, 1), r = __shfl_down_sync(0xffffffffu, v.x, 1);
  return F2{wl ? v.x : l, wr ? v.y : r};
}

// Adds a pair's arriving populations to the moments of rows z-1 (a0), z (a1) and z+1 (a2), the
// links in index order; g: the pair's own post-collision populations (all lanes take part; only
// those with `add` add).  The wall choices are selects on every lane.  A form with a separate path
// without them, a branch around part of this loop of full-mask shuffles, gave wrong moments in FP32
// and was dropped; its cause was not found.
template <int Q>
__device__ __forceinline__ void gather_row(const PairAt<false>& at, int z, bool add, const F2 (&g)[Q], F2& a0, F2& a1,
                                           F2& a2) {
  using L = Lat<Q>;
  const bool wl = at.a.x == 0, wr = at.b.x == at.b.nx - 1;
  const bool below = z == 0, above = z == at.a.nz - 1;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int ex = L::ex(i), ez = L::ez(i);
    const F2 o = g[L::opp(i)];  // what comes back from a wall
    F2 v = g[i];
    if (ex > 0) v = F2{__shfl_up_sync(0xffffffffu, g[i].y, 1), g[i].x};
    if (ex < 0) v = F2{g[i].y, __shfl_down_sync(0xffffffffu, g[i].x, 1)};
    if (!add) continue;
    // the link arrives at row z + ez from inside along x, or comes back at row z from beyond a wall
    const bool outx = ex > 0 && wl, outy = ex < 0 && wr;
    const bool outz = (ez > 0 && below) || (ez < 0 && above);
    if (ez == 0) {
      a1.x = radd(a1.x, outx ? o.x : v.x);
      a1.y = radd(a1.y, outy ? o.y : v.y);
    } else {
      F2& a = ez < 0 ? a0 : a2;
      a.x = radd(a.x, outx ? 0.0f : v.x);
      a.y = radd(a.y, outy ? 0.0f : v.y);
      a1.x = radd(a1.x, outx || outz ? o.x : 0.0f);
      a1.y = radd(a1.y, outy || outz ? o.y : 0.0f);
    }
  }
}

// Resident one-warp blocks per SM that set the register budget (80): 8000^2 FP16 1773 us per step
// (20 blocks, 96 registers: 1967), FP32 2143 (2137; 28 blocks 2136).
#ifndef LBPF_PLANE_BLOCKS
#define LBPF_PLANE_BLOCKS 24
#endif

// phi collision and phi^{n+1}
template <int QP, typename S>
__global__ void __launch_bounds__(32, LBPF_PLANE_BLOCKS)
    k_phi_plane(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items, int s6) {
  using C = Codec<S>;
  using L = Lat<QP>;
  const WorkItem it = items[blockIdx.x];
  const SimDev& sd = sims[it.sim];
  const int tx = threadIdx.x;
  const PairAt<false> at(sd, it.x0 - 2 + 2 * tx, 0);
  const int nx = at.a.nx, nz = at.a.nz;
  const unsigned NS = at.a.NS;
  const bool in = at.a.x >= 0 && at.a.x < nx, mine = in && tx >= 1 && tx <= 30;
  const bool wl = at.a.x == 0, wr = at.b.x == nx - 1;
  const Consts<float> P = sd.c32;
  const int par = s6 & 1;
  const S* __restrict__ gin = (const S*)sd.pop[par][0];
  S* __restrict__ gout = (S*)sd.pop[par ^ 1][0];
  const float* __restrict__ phin = (const float*)sd.phi[s6 % 3];
  const float* __restrict__ phim = (const float*)sd.phi[(s6 + 2) % 3];
  float* __restrict__ phinew = (float*)sd.phi[(s6 + 1) % 3];
  const float* __restrict__ Un = (const float*)sd.U[par];
  const float* __restrict__ thn = (const float*)sd.th[s6 % 3];
  const bool has_th = sd.q_theta != 0;
  const int zlo = max(it.z0 - 1, 0), zhi = min(it.z1, nz - 1);
  unsigned site = (unsigned)zlo * (unsigned)nx + (unsigned)(in ? at.a.x : 0);
  F2 cm = ld2<true>(phin + (zlo > 0 ? site - nx : site)), c = ld2<true>(phin + site);
  F2 a0 = both(0.0f), a1 = a0, a2 = a0;
  for (int z = zlo; z <= zhi; ++z, site += nx) {
    const F2 cp = z < nz - 1 ? ld2<true>(phin + (site + nx)) : c;
    const F2 n = beside(c, wl, wr);
    F2 g[QP];
#pragma unroll
    for (int i = 0; i < QP; ++i) g[i] = both(0.0f);
    if (in) {
      const F2 dx = rsub(F2{c.y, n.y}, F2{n.x, c.x}), dz = rsub(cp, cm);
      const F2 U = ld2<true>(Un + site), th = has_th ? ld2<true>(thn + site) : both(P.theta0);
      pull2<QP, S, false, C::shifted, true, true>(at, z, site, gin, phim, P.scale[0], g);
      const bool fa = !has_gradient(P, dx.x, 0.0f, dz.x), fb = !has_gradient(P, dx.y, 0.0f, dz.y);
      PhiCoef<float> ca, cb;
      if (fa && fb) {  // bulk: no non-local term
        phi_coef<QP, S, true>(P, c.x, U.x, th.x, dx.x, 0.0f, dz.x, false, 0.0f, ca);
        phi_coef<QP, S, true>(P, c.y, U.y, th.y, dx.y, 0.0f, dz.y, false, 0.0f, cb);
#pragma unroll
        for (int i = 0; i < QP; ++i) g[i] = rfma(g[i], F2{ca.omw, cb.omw}, F2{ca.K[L::cls(i)], cb.K[L::cls(i)]});
      } else {
        F2 gn[QP];
#pragma unroll
        for (int i = 0; i < QP; ++i) gn[i] = ld2<true>(gin + ((unsigned)i * NS + site));  // factor 0 at walls
        F2 ref = both(0.0f);
        if (C::shifted) ref = ld2<true>(phim + site);
        phi_coef<QP, S, false>(P, c.x, U.x, th.x, dx.x, 0.0f, dz.x, !at.a.inner(z), ref.x, ca);
        phi_coef<QP, S, false>(P, c.y, U.y, th.y, dx.y, 0.0f, dz.y, !at.b.inner(z), ref.y, cb);
        const F2 omw{ca.omw, cb.omw}, noma2{-ca.oma2, -cb.oma2}, inv_a2{ca.inv_a2, cb.inv_a2};
#pragma unroll
        for (int i = 0; i < QP; ++i) {
          const int k = L::cls(i);
          const F2 eq = eq_of<L>(i, F2{ca.K[k], cb.K[k]}, F2{ca.nx[k], cb.nx[k]}, F2{ca.ny[k], cb.ny[k]},
                                 F2{ca.nz[k], cb.nz[k]});
          g[i] = rmul(rfma(noma2, gn[i], rfma(g[i], omw, eq)), inv_a2);
        }
      }
      if (mine && z >= it.z0 && z < it.z1) {
#pragma unroll
        for (int i = 0; i < QP; ++i) st2(gout + ((unsigned)i * NS + site), g[i]);
      }
      if (C::shifted) {  // what was stored, with its shift
#pragma unroll
        for (int i = 0; i < QP; ++i)
          g[i] = shifted<false>(rmul(P.scale[0], (float)L::w(i)), c, as_stored<S>(g[i]));
      }
    }
    gather_row<QP>(at, z, mine, g, a0, a1, a2);
    if (mine) {
      const F2 sc = both(P.inv_scale[0]);
      if (z - 1 >= it.z0 && z - 1 < it.z1) st2(phinew + (site - nx), C::shifted ? rmul(a0, sc) : a0);
      if (z == nz - 1 && z >= it.z0 && z < it.z1) st2(phinew + site, C::shifted ? rmul(a1, sc) : a1);
    }
    a0 = a1;
    a1 = a2;
    a2 = both(0.0f);
    cm = c;
    c = cp;
  }
}

// U and theta collisions with phi^{n+1}, U^{n+1} and theta^{n+1}
template <int QU, int QT, typename S>
__global__ void __launch_bounds__(32, LBPF_PLANE_BLOCKS)
    k_uth_plane(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items, int s6) {
  using C = Codec<S>;
  constexpr int QTL = QT > 0 ? QT : 5;
  using LU = Lat<QU>;
  using LT = Lat<QTL>;
  const WorkItem it = items[blockIdx.x];
  const SimDev& sd = sims[it.sim];
  const int tx = threadIdx.x;
  const PairAt<false> at(sd, it.x0 - 2 + 2 * tx, 0);
  const int nx = at.a.nx, nz = at.a.nz;
  const unsigned NS = at.a.NS;
  const bool in = at.a.x >= 0 && at.a.x < nx, mine = in && tx >= 1 && tx <= 30;
  const bool wl = at.a.x == 0, wr = at.b.x == nx - 1;
  const Consts<float> P = sd.c32;
  const int par = s6 & 1;
  const S* __restrict__ hin = (const S*)sd.pop[par][1];
  S* __restrict__ hout = (S*)sd.pop[par ^ 1][1];
  const S* __restrict__ fin = (const S*)sd.pop[par][2];
  S* __restrict__ fout = (S*)sd.pop[par ^ 1][2];
  const float* __restrict__ phin = (const float*)sd.phi[s6 % 3];
  const float* __restrict__ phi1 = (const float*)sd.phi[(s6 + 1) % 3];
  const float* __restrict__ Un = (const float*)sd.U[par];
  float* __restrict__ Unew = (float*)sd.U[par ^ 1];
  const float* __restrict__ thn = (const float*)sd.th[s6 % 3];
  const float* __restrict__ thm = (const float*)sd.th[(s6 + 2) % 3];
  float* __restrict__ thnew = (float*)sd.th[(s6 + 1) % 3];
  const bool at_on = sd.antitrapping != 0;
  const int zlo = max(it.z0 - 1, 0), zhi = min(it.z1, nz - 1);
  unsigned site = (unsigned)zlo * (unsigned)nx + (unsigned)(in ? at.a.x : 0);
  F2 cm = ld2<true>(phi1 + (zlo > 0 ? site - nx : site)), c = ld2<true>(phi1 + site);
  F2 u0 = both(0.0f), u1 = u0, u2 = u0, t0 = u0, t1 = u0, t2 = u0;
  for (int z = zlo; z <= zhi; ++z, site += nx) {
    const F2 cp = z < nz - 1 ? ld2<true>(phi1 + (site + nx)) : c;
    const F2 n = beside(c, wl, wr);
    F2 h[QU], f[QTL];
#pragma unroll
    for (int i = 0; i < QU; ++i) h[i] = both(0.0f);
#pragma unroll
    for (int i = 0; i < QTL; ++i) f[i] = both(0.0f);
    if (in) {
      const F2 U = ld2<true>(Un + site), pn = ld2<true>(phin + site), th = QT > 0 ? ld2<true>(thn + site) : both(0.0f);
      pull2<QU, S, false, false, true, true>(at, z, site, hin, nullptr, 0.0f, h);
      if (QT > 0) pull2<QTL, S, false, C::shifted, true, true>(at, z, site, fin, thm, P.scale[2], f);
      UthCoef<float> ca, cb;
      uth_coef<QU, QT, S>(P, at_on, U.x, th.x, pn.x, c.x, c.y, n.x, c.x, c.x, cp.x, cm.x, ca);
      uth_coef<QU, QT, S>(P, at_on, U.y, th.y, pn.y, c.y, n.y, c.x, c.y, c.y, cp.y, cm.y, cb);
      const bool store = mine && z >= it.z0 && z < it.z1;
      const F2 A = both(ca.A);
#pragma unroll
      for (int i = 0; i < QU; ++i) {
        const int k = LU::cls(i);
        h[i] = rfma(h[i], A, eq_of<LU>(i, F2{ca.K[k], cb.K[k]}, F2{ca.jx[k], cb.jx[k]}, F2{ca.jy[k], cb.jy[k]},
                                       F2{ca.jz[k], cb.jz[k]}));
        if (store) st2(hout + ((unsigned)i * NS + site), h[i]);
        if (C::shifted) h[i] = as_stored<S>(h[i]);
      }
      if (QT > 0) {
        const F2 At = both(ca.At);
#pragma unroll
        for (int i = 0; i < QTL; ++i) {
          f[i] = rfma(f[i], At, F2{ca.Kt[LT::cls(i)], cb.Kt[LT::cls(i)]});
          if (store) st2(fout + ((unsigned)i * NS + site), f[i]);
          if (C::shifted) f[i] = shifted<false>(rmul(P.scale[2], (float)LT::w(i)), th, as_stored<S>(f[i]));
        }
      }
    }
    gather_row<QU>(at, z, mine, h, u0, u1, u2);
    if (QT > 0) gather_row<QTL>(at, z, mine, f, t0, t1, t2);
    if (mine) {
      // FP16/BF16: the shifts w_i U0 of the arriving populations add up to U0
      const F2 su = both(P.inv_scale[1]), hu = both(P.shift_h), st = both(P.inv_scale[2]);
      if (z - 1 >= it.z0 && z - 1 < it.z1) {
        st2(Unew + (site - nx), C::shifted ? rfma(u0, su, hu) : u0);
        if (QT > 0) st2(thnew + (site - nx), C::shifted ? rmul(t0, st) : t0);
      }
      if (z == nz - 1 && z >= it.z0 && z < it.z1) {
        st2(Unew + site, C::shifted ? rfma(u1, su, hu) : u1);
        if (QT > 0) st2(thnew + site, C::shifted ? rmul(t1, st) : t1);
      }
    }
    u0 = u1;
    u1 = u2;
    u2 = both(0.0f);
    t0 = t1;
    t1 = t2;
    t2 = both(0.0f);
    cm = c;
    c = cp;
  }
}

}  // namespace lbpf
