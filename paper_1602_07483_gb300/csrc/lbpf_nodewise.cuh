// lbpf_nodewise.cuh -- the step as node-wise kernels: collisions without a halo, moments in a
// pass of their own.
//
// The tiled kernels (lbpf_dev.cuh) recompute the collisions of a one-node halo so that a step
// reads the distributions once.  Where memory bandwidth is not the limit, that is the wrong
// trade: here every node collides exactly once (k_phi_node, k_uth_node), with one thread per
// node, no shared memory and no barrier, and the next moments are summed from the stored
// populations by k_phi_moment and k_uth_moment, which read them once more.  Both forms round
// and add alike (lbpf_node.cuh, and the order of moment_sum below), so they agree bit for bit.
//
// A block of threads owns consecutive nodes of an xy plane (a work item: first node x0 of the
// plane, planes [z0, z1)) whatever the row length, so ragged edges idle no lanes and every
// access is to consecutive addresses.
#pragma once

#include "lbpf_node.cuh"
#include "lbpf_plan.h"

namespace lbpf {

// Where a thread's node lies.
template <bool HY>
struct NodeAt {
  int nx, ny, nz;
  unsigned plane, NS, p;
  int x, y;
  bool in;
  __device__ __forceinline__ NodeAt(const SimDev& sd, int x_, int y_)  // by coordinates (p and in unset)
      : nx(sd.nx), ny(sd.ny), nz(sd.nz), plane((unsigned)sd.nx * (unsigned)sd.ny), NS((unsigned)sd.nsite), p(0), x(x_),
        y(y_), in(false) {}
  __device__ __forceinline__ NodeAt(const SimDev& sd, unsigned node)
      : nx(sd.nx), ny(sd.ny), nz(sd.nz), plane((unsigned)sd.nx * (unsigned)sd.ny), NS((unsigned)sd.nsite), p(node) {
    in = p < plane;
    y = HY ? (int)(p / (unsigned)nx) : 0;
    x = (int)(p - (unsigned)y * (unsigned)nx);
  }
  // off the y and z walls (of the axes the lattice has links along): such nodes, x walls among
  // them, take the path without wall checks, in which links from beyond an x wall are chosen by
  // selects.  Most warps of short rows hold an x wall node; branching them into the general path
  // ran both paths (48-column boxes: every warp).
  __device__ __forceinline__ bool core(int z) const { return (!HY || (y >= 1 && y <= ny - 2)) && z >= 1 && z <= nz - 2; }
  __device__ __forceinline__ bool inner(int z) const { return core(z) && x >= 1 && x <= nx - 2; }
  __device__ __forceinline__ bool has(int z, int ex, int ey, int ez) const {  // x - e is inside
    const int sx = x - ex, sy = y - ey, sz = z - ez;
    return sx >= 0 && sx < nx && sy >= 0 && sy < ny && sz >= 0 && sz < nz;
  }
  __device__ __forceinline__ bool beyond(int ex) const {  // x - e_x lies beyond an x wall
    return ex > 0 ? x == 0 : (ex < 0 ? x == nx - 1 : false);
  }
  template <typename L>
  __device__ __forceinline__ unsigned back(int i) const {  // site(x) - site(x - e_i), modulo 2^32
    return (unsigned)(L::ez(i) * (int)plane + L::ey(i) * nx + L::ex(i));
  }
};

// Pulled populations of a node (bounce-back at walls) as raw stored numbers; src(i, s): called
// with the site each value was stored at.
template <int Q, typename S, bool HY, typename T, typename F>
__device__ __forceinline__ void pull(const NodeAt<HY>& at, int z, unsigned site, const S* __restrict__ pop, T (&v)[Q],
                                     F src) {
  using L = Lat<Q>;
  using C = Codec<S>;
  if (at.core(z)) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const bool out = at.beyond(L::ex(i));
      const unsigned back = out ? 0u : at.template back<L>(i);
      v[i] = C::raw(ld<false>(pop + (site + ((unsigned)(out ? L::opp(i) : i) * at.NS - back))));
      src(i, site - back);
    }
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const bool inside = at.has(z, L::ex(i), L::ey(i), L::ez(i));
      const unsigned s = inside ? site - at.template back<L>(i) : site;
      v[i] = C::raw(ld<false>(pop + ((unsigned)(inside ? i : L::opp(i)) * at.NS + s)));
      src(i, s);
    }
  }
}

// Sum of a node's arriving populations v in the order in which a tile marching in z adds them:
// from plane z-1, then from its own plane (wall links among them), then from plane z+1; in
// each, the links with e_y = 0 first.
template <int Q, bool HY, typename T>
__device__ __forceinline__ T moment_sum(const NodeAt<HY>& at, int z, const T (&v)[Q]) {
  using L = Lat<Q>;
  T a = T(0);
  if (at.core(z)) {
#pragma unroll
    for (int ez = 1; ez >= -1; --ez)
#pragma unroll
      for (int y0 = 1; y0 >= 0; --y0)
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          if ((L::ey(i) == 0) != (y0 == 1)) continue;
          // a link from beyond an x wall counts as the own plane's
          if (L::ez(i) == ez) a = radd(a, ez != 0 && at.beyond(L::ex(i)) ? T(0) : v[i]);
          else if (ez == 0 && L::ex(i) != 0) a = radd(a, at.beyond(L::ex(i)) ? v[i] : T(0));
        }
  } else {
#pragma unroll
    for (int ez = 1; ez >= -1; --ez)
#pragma unroll
      for (int y0 = 1; y0 >= 0; --y0)
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          if ((L::ey(i) == 0) != (y0 == 1)) continue;
          const bool inside = at.has(z, L::ex(i), L::ey(i), L::ez(i));
          if (ez == 0 ? (L::ez(i) == 0 || !inside) : (L::ez(i) == ez && inside)) a = radd(a, v[i]);
        }
  }
  return a;
}

// The moment kernels take the blocks in reverse: what the collision stored last is still in L2
// (us per step, in order / reversed: 96^3 FP32 91.5 / 86.6, 160^3 FP16 260 / 253, 256^3 the same).
__device__ __forceinline__ unsigned moment_block() { return gridDim.x - 1 - blockIdx.x; }

// Resident blocks per SM (of 128 threads) that set the register budgets.  Measured, us per
// step: phi FP32 at 6 blocks (80 registers) 256^3 D3Q19 696 (5 blocks 716); phi FP16 at 5 (96
// registers) 711 (6: 777, spills); U and theta at 5 256^3 D3Q19/D3Q7 FP16 834 (4: 872, 3: 959), FP32
// 918 (4: 921); FP64 at 3 (168 registers) 128^3 921 (4: 931, spills; 2: 983), 32^3 59 (4: 64).
#ifndef LBPF_NODE_PHI_BLOCKS
#define LBPF_NODE_PHI_BLOCKS 6
#endif
#ifndef LBPF_NODE16_PHI_BLOCKS
#define LBPF_NODE16_PHI_BLOCKS 5
#endif
#ifndef LBPF_NODE_UTH_BLOCKS
#define LBPF_NODE_UTH_BLOCKS 5
#endif
#ifndef LBPF_NODE64_BLOCKS
#define LBPF_NODE64_BLOCKS 3
#endif

// phi collision; writes the post-collision populations
template <int QP, typename S>
__global__ void __launch_bounds__(NODE_THREADS, sizeof(S) == 8 ? LBPF_NODE64_BLOCKS : sizeof(S) == 2 ? LBPF_NODE16_PHI_BLOCKS : LBPF_NODE_PHI_BLOCKS)
    k_phi_node(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items, int s6) {
  using C = Codec<S>;
  using T = typename C::T;
  using L = Lat<QP>;
  constexpr bool HY = L::has_y;
  const WorkItem it = items[blockIdx.x];
  const SimDev& sd = sims[it.sim];
  const NodeAt<HY> at(sd, (unsigned)it.x0 + threadIdx.x);
  pdl_trigger();
  // held in registers in FP16/BF16 (256^3: 733 against 752 us); read where used in FP32 and FP64,
  // whose registers are full (750 against 790 us, FP64 128^3 566 against 599 us)
  typename std::conditional<C::shifted, const Consts<T>, const Consts<T>&>::type P = consts_of<T>(sd);
  const int par = s6 & 1;
  const S* __restrict__ gin = (const S*)sd.pop[par][0];
  S* __restrict__ gout = (S*)sd.pop[par ^ 1][0];
  const T* __restrict__ phin = (const T*)sd.phi[s6 % 3];
  const T* __restrict__ phim = (const T*)sd.phi[(s6 + 2) % 3];  // phi^{n-1}: the FP16/BF16 shift
  const T* __restrict__ Un = (const T*)sd.U[par];
  const T* __restrict__ thn = (const T*)sd.th[s6 % 3];
  const bool has_th = sd.q_theta != 0;
  const T theta0 = P.theta0, scale = P.scale[0];
  pdl_wait();
  if (!at.in) return;
  const int xp = at.x < at.nx - 1 ? 1 : 0, xm = at.x > 0 ? 1 : 0;  // mirror ghosts
  const int yp = HY && at.y < at.ny - 1 ? at.nx : 0, ym = HY && at.y > 0 ? at.nx : 0;
  unsigned site = (unsigned)it.z0 * at.plane + at.p;
  T cm = ld<false>(phin + (it.z0 > 0 ? site - at.plane : site)), cc = ld<false>(phin + site);
  for (int z = it.z0; z < it.z1; ++z, site += at.plane) {
    const T cp = z < at.nz - 1 ? ld<false>(phin + (site + at.plane)) : cc;
    const T dx = radd(ld<false>(phin + (site + xp)), -ld<false>(phin + (site - xm)));
    const T dy = HY ? radd(ld<false>(phin + (site + yp)), -ld<false>(phin + (site - ym))) : T(0);
    const T U = ld<false>(Un + site), th = has_th ? ld<false>(thn + site) : theta0;
    const bool wall = !at.inner(z);
    T gp[QP], gn[QP];
    T ref[C::shifted ? QP : 1];
    pull<QP, S>(at, z, site, gin, gp, [&](int i, unsigned s) {
      if (C::shifted) ref[i] = ld<false>(phim + s);
    });
    const bool flat = !has_gradient(P, dx, dy, radd(cp, -cm));
    if (!flat) {  // no non-local term in the bulk
#pragma unroll
      for (int i = 0; i < QP; ++i) gn[i] = C::raw(ld<false>(gin + ((unsigned)i * at.NS + site)));  // B = 0 at walls
    }
    if (C::shifted) {
#pragma unroll
      for (int i = 0; i < QP; ++i) gp[i] = rfma(rmul(scale, (T)L::w(i)), ref[i], gp[i]);
    }
    PhiCoef<T> co;
    phi_coef<QP, S, true>(P, cc, U, th, dx, dy, radd(cp, -cm), wall, C::shifted ? ref[0] : T(0), co);
    phi_collide<QP>(co, gp, gn);
#pragma unroll
    for (int i = 0; i < QP; ++i) gout[(unsigned)i * at.NS + site] = C::pack(gp[i]);
    cm = cc;
    cc = cp;
  }
}

// phi^{n+1} from the stored post-collision populations
template <int QP, typename S>
__global__ void __launch_bounds__(NODE_THREADS)
    k_phi_moment(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items, int s6) {
  using C = Codec<S>;
  using T = typename C::T;
  using L = Lat<QP>;
  constexpr bool HY = L::has_y;
  const WorkItem it = items[moment_block()];
  const SimDev& sd = sims[it.sim];
  const NodeAt<HY> at(sd, (unsigned)it.x0 + threadIdx.x);
  pdl_trigger();
  const Consts<T> P = consts_of<T>(sd);
  const S* __restrict__ g = (const S*)sd.pop[(s6 & 1) ^ 1][0];
  const T* __restrict__ phin = (const T*)sd.phi[s6 % 3];
  T* __restrict__ phinew = (T*)sd.phi[(s6 + 1) % 3];
  const T scale = P.scale[0], iscale = P.inv_scale[0];
  pdl_wait();
  if (!at.in) return;
  unsigned site = (unsigned)it.z0 * at.plane + at.p;
  for (int z = it.z0; z < it.z1; ++z, site += at.plane) {
    T v[QP];
    T ref[C::shifted ? QP : 1];
    pull<QP, S>(at, z, site, g, v, [&](int i, unsigned s) {
      if (C::shifted) ref[i] = ld<false>(phin + s);
    });
    if (C::shifted) {
#pragma unroll
      for (int i = 0; i < QP; ++i) v[i] = radd(v[i], shift_of<L>(scale, i, ref[i]));
    }
    const T a = moment_sum<QP>(at, z, v);
    phinew[site] = C::shifted ? rmul(a, iscale) : a;
  }
}

// U and theta collisions with phi^{n+1}; writes the post-collision populations
template <int QU, int QT, typename S>
__global__ void __launch_bounds__(NODE_THREADS, sizeof(S) == 8 ? LBPF_NODE64_BLOCKS : LBPF_NODE_UTH_BLOCKS)
    k_uth_node(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items, int s6) {
  using C = Codec<S>;
  using T = typename C::T;
  constexpr int QTL = QT > 0 ? QT : 7;
  using LT = Lat<QTL>;
  constexpr bool HY = Lat<QU>::has_y;
  const WorkItem it = items[blockIdx.x];
  const SimDev& sd = sims[it.sim];
  const NodeAt<HY> at(sd, (unsigned)it.x0 + threadIdx.x);
  pdl_trigger();
  const Consts<T> P = consts_of<T>(sd);
  const int par = s6 & 1;
  const S* __restrict__ hin = (const S*)sd.pop[par][1];
  S* __restrict__ hout = (S*)sd.pop[par ^ 1][1];
  const S* __restrict__ fin = (const S*)sd.pop[par][2];
  S* __restrict__ fout = (S*)sd.pop[par ^ 1][2];
  const T* __restrict__ phin = (const T*)sd.phi[s6 % 3];
  const T* __restrict__ phi1 = (const T*)sd.phi[(s6 + 1) % 3];
  const T* __restrict__ Un = (const T*)sd.U[par];
  const T* __restrict__ thn = (const T*)sd.th[s6 % 3];
  const T* __restrict__ thm = (const T*)sd.th[(s6 + 2) % 3];  // theta^{n-1}: the FP16/BF16 shift of f
  const bool at_on = sd.antitrapping != 0;
  pdl_wait();
  if (!at.in) return;
  const int xp = at.x < at.nx - 1 ? 1 : 0, xm = at.x > 0 ? 1 : 0;  // mirror ghosts
  const int yp = HY && at.y < at.ny - 1 ? at.nx : 0, ym = HY && at.y > 0 ? at.nx : 0;
  unsigned site = (unsigned)it.z0 * at.plane + at.p;
  T cm = ld<false>(phi1 + (it.z0 > 0 ? site - at.plane : site)), cc = ld<false>(phi1 + site);
  for (int z = it.z0; z < it.z1; ++z, site += at.plane) {
    const T cp = z < at.nz - 1 ? ld<false>(phi1 + (site + at.plane)) : cc;
    const T pxp = ld<false>(phi1 + (site + xp)), pxm = ld<false>(phi1 + (site - xm));
    const T pyp = HY ? ld<false>(phi1 + (site + yp)) : cc, pym = HY ? ld<false>(phi1 + (site - ym)) : cc;
    const T U = ld<false>(Un + site), phn = ld<false>(phin + site), th = QT > 0 ? ld<false>(thn + site) : T(0);
    T h[QU];
    T f[QTL];
    T ref[C::shifted && QT > 0 ? QTL : 1];
    pull<QU, S>(at, z, site, hin, h, [](int, unsigned) {});
    if (QT > 0) {
      pull<QTL, S>(at, z, site, fin, f, [&](int i, unsigned s) {
        if (C::shifted) ref[i] = ld<false>(thm + s);
      });
      if (C::shifted) {
#pragma unroll
        for (int i = 0; i < QT; ++i) f[i] = rfma(rmul(P.scale[2], (T)LT::w(i)), ref[i], f[i]);
      }
    }
    UthCoef<T> co;
    uth_coef<QU, QT, S>(P, at_on, U, th, phn, cc, pxp, pxm, pyp, pym, cp, cm, co);
    u_collide<QU>(co, h);
#pragma unroll
    for (int i = 0; i < QU; ++i) hout[(unsigned)i * at.NS + site] = C::pack(h[i]);
    if (QT > 0) {
#pragma unroll
      for (int i = 0; i < QT; ++i)
        fout[(unsigned)i * at.NS + site] = C::pack(rfma(f[i], co.At, co.Kt[LT::cls(i)]));
    }
    cm = cc;
    cc = cp;
  }
}

// U^{n+1} and theta^{n+1} from the stored post-collision populations
template <int QU, int QT, typename S>
__global__ void __launch_bounds__(NODE_THREADS)
    k_uth_moment(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items, int s6) {
  using C = Codec<S>;
  using T = typename C::T;
  constexpr int QTL = QT > 0 ? QT : 7;
  using LT = Lat<QTL>;
  constexpr bool HY = Lat<QU>::has_y;
  const WorkItem it = items[moment_block()];
  const SimDev& sd = sims[it.sim];
  const NodeAt<HY> at(sd, (unsigned)it.x0 + threadIdx.x);
  pdl_trigger();
  const Consts<T> P = consts_of<T>(sd);
  const int par = s6 & 1;
  const S* __restrict__ h = (const S*)sd.pop[par ^ 1][1];
  const S* __restrict__ f = (const S*)sd.pop[par ^ 1][2];
  T* __restrict__ Unew = (T*)sd.U[par ^ 1];
  const T* __restrict__ thn = (const T*)sd.th[s6 % 3];
  T* __restrict__ thnew = (T*)sd.th[(s6 + 1) % 3];
  pdl_wait();
  if (!at.in) return;
  unsigned site = (unsigned)it.z0 * at.plane + at.p;
  for (int z = it.z0; z < it.z1; ++z, site += at.plane) {
    {
      T v[QU];
      pull<QU, S>(at, z, site, h, v, [](int, unsigned) {});
      const T a = moment_sum<QU>(at, z, v);
      // FP16/BF16: the shifts w_i U0 of the arriving populations add up to U0
      Unew[site] = C::shifted ? rfma(a, P.inv_scale[1], P.shift_h) : a;
    }
    if (QT > 0) {
      T v[QTL];
      T ref[C::shifted ? QTL : 1];
      pull<QTL, S>(at, z, site, f, v, [&](int i, unsigned s) {
        if (C::shifted) ref[i] = ld<false>(thn + s);
      });
      if (C::shifted) {
#pragma unroll
        for (int i = 0; i < QTL; ++i) v[i] = radd(v[i], shift_of<LT>(P.scale[2], i, ref[i]));
      }
      const T a = moment_sum<QTL>(at, z, v);
      thnew[site] = C::shifted ? rmul(a, P.inv_scale[2]) : a;
    }
  }
}

}  // namespace lbpf
