// lbpf_nodepair.cuh -- the node-wise step with two x-adjacent nodes per thread (FP32, FP16, BF16).
//
// The node-wise kernels (lbpf_nodewise.cuh) are bound by instructions and by the loads a warp
// has in flight more than by memory.  With a pair of nodes per thread the populations that
// move along y and z only, the non-local values, the scalars and all stores are one access of
// twice the width, address arithmetic is shared, and the collisions run on Blackwell's packed
// FP32 operations (two nodes per instruction, each rounded as the scalar operation).  It needs
// rows of even length, so that a pair never straddles a row and every pair is aligned.  Results
// agree bit for bit with the other forms of the step.
#pragma once

#include "lbpf_nodewise.cuh"

namespace lbpf {

struct alignas(8) F2 {
  float x, y;
};
__device__ __forceinline__ F2 both(float a) { return F2{a, a}; }
__device__ __forceinline__ F2 as_f2(float2 a) { return F2{a.x, a.y}; }
__device__ __forceinline__ float2 as_v(F2 a) { return make_float2(a.x, a.y); }
// Packed operations.  A sum of a packed product would be contracted, so no routine adds one.
__device__ __forceinline__ F2 rmul(F2 a, F2 b) { return as_f2(__fmul2_rn(as_v(a), as_v(b))); }
__device__ __forceinline__ F2 radd(F2 a, F2 b) { return as_f2(__fadd2_rn(as_v(a), as_v(b))); }
__device__ __forceinline__ F2 rfma(F2 a, F2 b, F2 c) { return as_f2(__ffma2_rn(as_v(a), as_v(b), as_v(c))); }
// a - b
__device__ __forceinline__ F2 rsub(F2 a, F2 b) { return rfma(b, both(-1.0f), a); }

// Two consecutive stored numbers (the first at an even index), as raw FP32 values and back.
template <bool RO>
__device__ __forceinline__ F2 ld2(const float* p) {
  return as_f2(ld<RO>(reinterpret_cast<const float2*>(p)));
}
template <bool RO>
__device__ __forceinline__ F2 ld2(const __half* p) {
  return as_f2(__half22float2(ld<RO>(reinterpret_cast<const __half2*>(p))));
}
template <bool RO>
__device__ __forceinline__ F2 ld2(const __nv_bfloat16* p) {
  return as_f2(__bfloat1622float2(ld<RO>(reinterpret_cast<const __nv_bfloat162*>(p))));
}
__device__ __forceinline__ void st2(float* p, F2 v) { *reinterpret_cast<float2*>(p) = make_float2(v.x, v.y); }
__device__ __forceinline__ void st2(__half* p, F2 v) { *reinterpret_cast<__half2*>(p) = __floats2half2_rn(v.x, v.y); }
__device__ __forceinline__ void st2(__nv_bfloat16* p, F2 v) {
  *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(v.x, v.y);
}

// Where a thread's pair lies: nodes a and a + 1 of a row.
template <bool HY>
struct PairAt {
  NodeAt<HY> a, b;
  __device__ __forceinline__ PairAt(const SimDev& sd, const WorkItem& it)
      : a(sd, (unsigned)it.x0 + 2 * threadIdx.x), b(a) {
    b.x += 1;
    b.p += 1;
  }
  __device__ __forceinline__ PairAt(const SimDev& sd, int x, int y) : a(sd, x, y), b(sd, x + 1, y) {}
  __device__ __forceinline__ bool core(int z) const { return a.core(z); }
};

// The FP16/BF16 shift on a raw stored number: fused for the pulled populations of a collision, rounded
// on its own (shift_of) for the moments; there the products are scalar, since a packed product and
// sum are contracted whatever their rounding says.
template <bool FUSED>
__device__ __forceinline__ float shifted(float ws, float ref, float raw) {
  return FUSED ? rfma(ws, ref, raw) : radd(raw, rmul(ws, ref));
}
template <bool FUSED>
__device__ __forceinline__ F2 shifted(float ws, F2 ref, F2 raw) {
  if (FUSED) return rfma(both(ws), ref, raw);
  return radd(raw, F2{rmul(ws, ref.x), rmul(ws, ref.y)});
}

// Pulled populations of a pair; with REF, the raw stored number G plus the shift S w ref(source)
// (FP16/BF16; ref: phi or theta of the step that stored it).  Off the y and z walls a link from
// beyond an x wall is chosen by selects (NodeAt::core).
template <int Q, typename S, bool HY, bool REF, bool FUSED, bool RO>
__device__ __forceinline__ void pull2(const PairAt<HY>& at, int z, unsigned site, const S* __restrict__ pop,
                                      const float* __restrict__ ref, float scale, F2 (&v)[Q]) {
  using L = Lat<Q>;
  using C = Codec<S>;
  if (at.core(z)) {
    const bool wl = at.a.x == 0, wr = at.b.x == at.b.nx - 1;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const unsigned in = (unsigned)i * at.a.NS - (unsigned)(L::ez(i) * (int)at.a.plane + L::ey(i) * at.a.nx);
      const unsigned out = (unsigned)L::opp(i) * at.a.NS;
      if (L::ex(i) == 0) v[i] = ld2<RO>(pop + (site + in));
      else if (L::ex(i) > 0)
        v[i] = F2{C::raw(ld<RO>(pop + (site + (wl ? out : in - 1)))), C::raw(ld<RO>(pop + (site + in)))};
      else
        v[i] = F2{C::raw(ld<RO>(pop + (site + (in + 1)))), C::raw(ld<RO>(pop + (site + (wr ? out + 1 : in + 2))))};
    }
    if (REF) {
      const F2 own = ld2<RO>(ref + site);
      // the rows (e_y, e_z) that the lattice pulls from, each read once
#pragma unroll
      for (int ez = -1; ez <= 1; ++ez)
#pragma unroll
        for (int ey = -1; ey <= 1; ++ey) {
          bool any = false, left = false, right = false;
#pragma unroll
          for (int i = 0; i < Q; ++i)
            if (L::ey(i) == ey && L::ez(i) == ez) {
              any = true;
              left = left || L::ex(i) > 0;
              right = right || L::ex(i) < 0;
            }
          if (!any) continue;
          const unsigned row = site - (unsigned)(ez * (int)at.a.plane + ey * at.a.nx);
          const F2 m = ey == 0 && ez == 0 ? own : ld2<RO>(ref + row);
          const float l = left ? ld<RO>(ref + (wl ? site : row - 1)) : 0.0f;
          const float r = right ? ld<RO>(ref + (wr ? site + 1 : row + 2)) : 0.0f;
#pragma unroll
          for (int i = 0; i < Q; ++i)
            if (L::ey(i) == ey && L::ez(i) == ez)
              v[i] = shifted<FUSED>(rmul(scale, (float)L::w(i)),
                                    L::ex(i) == 0 ? m : (L::ex(i) > 0 ? F2{l, m.x} : F2{m.y, r}), v[i]);
        }
    }
  } else {
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      const NodeAt<HY>& at1 = n == 0 ? at.a : at.b;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const bool inside = at1.has(z, L::ex(i), L::ey(i), L::ez(i));
        const unsigned s = inside ? site + n - at1.template back<L>(i) : site + n;
        float g = C::raw(ld<RO>(pop + ((unsigned)(inside ? i : L::opp(i)) * at1.NS + s)));
        if (REF) g = shifted<FUSED>(rmul(scale, (float)L::w(i)), ld<RO>(ref + s), g);
        (n == 0 ? v[i].x : v[i].y) = g;
      }
    }
  }
}

// Moments of a pair, in the order of moment_sum.
template <int Q, bool HY>
__device__ __forceinline__ F2 moment_sum2(const PairAt<HY>& at, int z, const F2 (&v)[Q]) {
  using L = Lat<Q>;
  F2 s = both(0.0f);
  if (at.core(z)) {
    const bool wl = at.a.x == 0, wr = at.b.x == at.b.nx - 1;
#pragma unroll
    for (int ez = 1; ez >= -1; --ez)
#pragma unroll
      for (int y0 = 1; y0 >= 0; --y0)
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          if ((L::ey(i) == 0) != (y0 == 1)) continue;
          const int ex = L::ex(i);
          // a link from beyond an x wall counts as the own plane's
          if (L::ez(i) == ez) {
            F2 t = v[i];
            if (ez != 0 && ex > 0 && wl) t.x = 0.0f;
            if (ez != 0 && ex < 0 && wr) t.y = 0.0f;
            s = radd(s, t);
          } else if (ez == 0 && ex != 0) {
            if (ex > 0) s.x = radd(s.x, wl ? v[i].x : 0.0f);
            else s.y = radd(s.y, wr ? v[i].y : 0.0f);
          }
        }
  } else {
    float one[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) one[i] = v[i].x;
    s.x = moment_sum<Q>(at.a, z, one);
#pragma unroll
    for (int i = 0; i < Q; ++i) one[i] = v[i].y;
    s.y = moment_sum<Q>(at.b, z, one);
  }
  return s;
}

// Resident blocks per SM (of 128 threads) that set the register budgets.  Measured, us per step:
// phi FP32 256^3 D3Q19 at 4 blocks 639 (3: 673, 5: 676); FP16 at 3 545 (4: 590); U and theta
// 96^3 FP32 at 4 58 (3: 61), 256^3 D3Q19/D3Q7 FP16 677 (3: 693, 5: 708).
#ifndef LBPF_PAIR_PHI_BLOCKS
#define LBPF_PAIR_PHI_BLOCKS 4
#endif
#ifndef LBPF_PAIR16_PHI_BLOCKS
#define LBPF_PAIR16_PHI_BLOCKS 3
#endif
#ifndef LBPF_PAIR_UTH_BLOCKS
#define LBPF_PAIR_UTH_BLOCKS 4
#endif
#ifndef LBPF_PAIR16_UTH_BLOCKS
#define LBPF_PAIR16_UTH_BLOCKS 4
#endif
#ifndef LBPF_PAIR_MOMENT_BLOCKS
#define LBPF_PAIR_MOMENT_BLOCKS 8
#endif
#ifndef LBPF_PAIR16_MOMENT_BLOCKS
#define LBPF_PAIR16_MOMENT_BLOCKS 6
#endif

// phi collision (k_phi_node)
template <int QP, typename S>
__global__ void __launch_bounds__(NODE_THREADS, sizeof(S) == 2 ? LBPF_PAIR16_PHI_BLOCKS : LBPF_PAIR_PHI_BLOCKS)
    k_phi_pair(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items, int s6) {
  using C = Codec<S>;
  using L = Lat<QP>;
  constexpr bool HY = L::has_y;
  const WorkItem it = items[blockIdx.x];
  const SimDev& sd = sims[it.sim];
  const PairAt<HY> at(sd, it);
  const NodeAt<HY>& a = at.a;
  pdl_trigger();
  const Consts<float>& P = sd.c32;
  const int par = s6 & 1;
  const S* __restrict__ gin = (const S*)sd.pop[par][0];
  S* __restrict__ gout = (S*)sd.pop[par ^ 1][0];
  const float* __restrict__ phin = (const float*)sd.phi[s6 % 3];
  const float* __restrict__ phim = (const float*)sd.phi[(s6 + 2) % 3];
  const float* __restrict__ Un = (const float*)sd.U[par];
  const float* __restrict__ thn = (const float*)sd.th[s6 % 3];
  const bool has_th = sd.q_theta != 0;
  const F2 theta0 = both(P.theta0);
  const float scale = P.scale[0];
  pdl_wait();
  if (!a.in) return;
  const int xr = a.x < a.nx - 2 ? 2 : 1, xl = a.x > 0 ? 1 : 0;  // mirror ghosts
  const int yp = HY && a.y < a.ny - 1 ? a.nx : 0, ym = HY && a.y > 0 ? a.nx : 0;
  unsigned site = (unsigned)it.z0 * a.plane + a.p;
  F2 cm = ld2<false>(phin + (it.z0 > 0 ? site - a.plane : site)), cc = ld2<false>(phin + site);
  for (int z = it.z0; z < it.z1; ++z, site += a.plane) {
    const F2 cp = z < a.nz - 1 ? ld2<false>(phin + (site + a.plane)) : cc;
    const float l = ld<false>(phin + (site - xl)), r = ld<false>(phin + (site + xr));
    const F2 dx = rsub(F2{cc.y, r}, F2{l, cc.x});
    const F2 dy = HY ? rsub(ld2<false>(phin + (site + yp)), ld2<false>(phin + (site - ym))) : both(0.0f);
    const F2 dz = rsub(cp, cm);
    const F2 U = ld2<false>(Un + site), th = has_th ? ld2<false>(thn + site) : theta0;
    F2 g[QP];
    pull2<QP, S, HY, C::shifted, true, false>(at, z, site, gin, phim, scale, g);
    const bool fa = !has_gradient(P, dx.x, dy.x, dz.x), fb = !has_gradient(P, dx.y, dy.y, dz.y);
    if (fa && fb) {  // bulk: no non-local term
      PhiCoef<float> ca, cb;
      phi_coef<QP, S, true>(P, cc.x, U.x, th.x, dx.x, dy.x, dz.x, false, 0.0f, ca);
      phi_coef<QP, S, true>(P, cc.y, U.y, th.y, dx.y, dy.y, dz.y, false, 0.0f, cb);
#pragma unroll
      for (int i = 0; i < QP; ++i)
        st2(gout + ((unsigned)i * a.NS + site), rfma(g[i], F2{ca.omw, cb.omw}, F2{ca.K[L::cls(i)], cb.K[L::cls(i)]}));
    } else {
      F2 gn[QP];
      const bool wa = !a.inner(z), wb = !at.b.inner(z);
      F2 ref = both(0.0f);
      if (C::shifted) ref = ld2<false>(phim + site);
      PhiCoef<float> ca, cb;
      phi_coef<QP, S, false>(P, cc.x, U.x, th.x, dx.x, dy.x, dz.x, wa, ref.x, ca);
      phi_coef<QP, S, false>(P, cc.y, U.y, th.y, dx.y, dy.y, dz.y, wb, ref.y, cb);
      // the non-local values after the coefficients, whose arithmetic then has the registers: before
      // them they spilled (56 bytes), and FP32 512^3 with a gradient at most nodes took 15.03 ms per
      // step, 14.71 so (14.77 as tiles)
#pragma unroll
      for (int i = 0; i < QP; ++i) gn[i] = ld2<false>(gin + ((unsigned)i * a.NS + site));  // B = 0 at walls
      const F2 omw{ca.omw, cb.omw}, noma2{-ca.oma2, -cb.oma2}, inv_a2{ca.inv_a2, cb.inv_a2};
#pragma unroll
      for (int i = 0; i < QP; ++i) {
        const int k = L::cls(i);
        const F2 eq = eq_of<L>(i, F2{ca.K[k], cb.K[k]}, F2{ca.nx[k], cb.nx[k]}, F2{ca.ny[k], cb.ny[k]},
                               F2{ca.nz[k], cb.nz[k]});
        st2(gout + ((unsigned)i * a.NS + site), rmul(rfma(noma2, gn[i], rfma(g[i], omw, eq)), inv_a2));
      }
    }
    cm = cc;
    cc = cp;
  }
}

// phi^{n+1} from the stored post-collision populations (k_phi_moment)
template <int QP, typename S>
__global__ void __launch_bounds__(NODE_THREADS, sizeof(S) == 2 ? LBPF_PAIR16_MOMENT_BLOCKS : LBPF_PAIR_MOMENT_BLOCKS)
    k_phi_moment2(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items, int s6) {
  using C = Codec<S>;
  constexpr bool HY = Lat<QP>::has_y;
  const WorkItem it = items[moment_block()];
  const SimDev& sd = sims[it.sim];
  const PairAt<HY> at(sd, it);
  pdl_trigger();
  const S* __restrict__ g = (const S*)sd.pop[(s6 & 1) ^ 1][0];
  const float* __restrict__ phin = (const float*)sd.phi[s6 % 3];
  float* __restrict__ phinew = (float*)sd.phi[(s6 + 1) % 3];
  const float scale = sd.c32.scale[0], iscale = sd.c32.inv_scale[0];
  pdl_wait();
  if (!at.a.in) return;
  unsigned site = (unsigned)it.z0 * at.a.plane + at.a.p;
  for (int z = it.z0; z < it.z1; ++z, site += at.a.plane) {
    F2 v[QP];
    pull2<QP, S, HY, C::shifted, false, false>(at, z, site, g, phin, scale, v);
    const F2 m = moment_sum2<QP>(at, z, v);
    st2(phinew + site, C::shifted ? rmul(m, both(iscale)) : m);
  }
}

// U and theta collisions with phi^{n+1} (k_uth_node)
template <int QU, int QT, typename S>
__global__ void __launch_bounds__(NODE_THREADS, sizeof(S) == 2 ? LBPF_PAIR16_UTH_BLOCKS : LBPF_PAIR_UTH_BLOCKS)
    k_uth_pair(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items, int s6) {
  using C = Codec<S>;
  constexpr int QTL = QT > 0 ? QT : 7;
  using L = Lat<QU>;
  using LT = Lat<QTL>;
  constexpr bool HY = L::has_y;
  const WorkItem it = items[blockIdx.x];
  const SimDev& sd = sims[it.sim];
  const PairAt<HY> at(sd, it);
  const NodeAt<HY>& a = at.a;
  pdl_trigger();
  const Consts<float>& P = sd.c32;
  const int par = s6 & 1;
  const S* __restrict__ hin = (const S*)sd.pop[par][1];
  S* __restrict__ hout = (S*)sd.pop[par ^ 1][1];
  const S* __restrict__ fin = (const S*)sd.pop[par][2];
  S* __restrict__ fout = (S*)sd.pop[par ^ 1][2];
  const float* __restrict__ phin = (const float*)sd.phi[s6 % 3];
  const float* __restrict__ phi1 = (const float*)sd.phi[(s6 + 1) % 3];
  const float* __restrict__ Un = (const float*)sd.U[par];
  const float* __restrict__ thn = (const float*)sd.th[s6 % 3];
  const float* __restrict__ thm = (const float*)sd.th[(s6 + 2) % 3];
  const bool at_on = sd.antitrapping != 0;
  pdl_wait();
  if (!a.in) return;
  const int xr = a.x < a.nx - 2 ? 2 : 1, xl = a.x > 0 ? 1 : 0;  // mirror ghosts
  const int yp = HY && a.y < a.ny - 1 ? a.nx : 0, ym = HY && a.y > 0 ? a.nx : 0;
  unsigned site = (unsigned)it.z0 * a.plane + a.p;
  F2 cm = ld2<false>(phi1 + (it.z0 > 0 ? site - a.plane : site)), cc = ld2<false>(phi1 + site);
  for (int z = it.z0; z < it.z1; ++z, site += a.plane) {
    const F2 cp = z < a.nz - 1 ? ld2<false>(phi1 + (site + a.plane)) : cc;
    const float l = ld<false>(phi1 + (site - xl)), r = ld<false>(phi1 + (site + xr));
    const F2 yu = HY ? ld2<false>(phi1 + (site + yp)) : cc, yd = HY ? ld2<false>(phi1 + (site - ym)) : cc;
    const F2 U = ld2<false>(Un + site), pn = ld2<false>(phin + site), th = QT > 0 ? ld2<false>(thn + site) : both(0.0f);
    F2 h[QU], f[QTL];
    pull2<QU, S, HY, false, true, false>(at, z, site, hin, nullptr, 0.0f, h);
    if (QT > 0) pull2<QTL, S, HY, C::shifted, true, false>(at, z, site, fin, thm, P.scale[2], f);
    UthCoef<float> ca, cb;
    uth_coef<QU, QT, S>(P, at_on, U.x, th.x, pn.x, cc.x, cc.y, l, yu.x, yd.x, cp.x, cm.x, ca);
    uth_coef<QU, QT, S>(P, at_on, U.y, th.y, pn.y, cc.y, r, cc.x, yu.y, yd.y, cp.y, cm.y, cb);
    const F2 A = both(ca.A);
#pragma unroll
    for (int i = 0; i < QU; ++i) {
      const int k = L::cls(i);
      st2(hout + ((unsigned)i * a.NS + site),
          rfma(h[i], A, eq_of<L>(i, F2{ca.K[k], cb.K[k]}, F2{ca.jx[k], cb.jx[k]}, F2{ca.jy[k], cb.jy[k]},
                                 F2{ca.jz[k], cb.jz[k]})));
    }
    if (QT > 0) {
      const F2 At = both(ca.At);
#pragma unroll
      for (int i = 0; i < QT; ++i)
        st2(fout + ((unsigned)i * a.NS + site), rfma(f[i], At, F2{ca.Kt[LT::cls(i)], cb.Kt[LT::cls(i)]}));
    }
    cm = cc;
    cc = cp;
  }
}

// U^{n+1} and theta^{n+1} from the stored post-collision populations (k_uth_moment)
template <int QU, int QT, typename S>
__global__ void __launch_bounds__(NODE_THREADS, sizeof(S) == 2 ? LBPF_PAIR16_MOMENT_BLOCKS : LBPF_PAIR_MOMENT_BLOCKS)
    k_uth_moment2(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items, int s6) {
  using C = Codec<S>;
  constexpr int QTL = QT > 0 ? QT : 7;
  constexpr bool HY = Lat<QU>::has_y;
  const WorkItem it = items[moment_block()];
  const SimDev& sd = sims[it.sim];
  const PairAt<HY> at(sd, it);
  pdl_trigger();
  const Consts<float>& P = sd.c32;
  const int par = s6 & 1;
  const S* __restrict__ h = (const S*)sd.pop[par ^ 1][1];
  const S* __restrict__ f = (const S*)sd.pop[par ^ 1][2];
  float* __restrict__ Unew = (float*)sd.U[par ^ 1];
  const float* __restrict__ thn = (const float*)sd.th[s6 % 3];
  float* __restrict__ thnew = (float*)sd.th[(s6 + 1) % 3];
  pdl_wait();
  if (!at.a.in) return;
  unsigned site = (unsigned)it.z0 * at.a.plane + at.a.p;
  for (int z = it.z0; z < it.z1; ++z, site += at.a.plane) {
    {
      F2 v[QU];
      pull2<QU, S, HY, false, false, false>(at, z, site, h, nullptr, 0.0f, v);
      const F2 m = moment_sum2<QU>(at, z, v);
      st2(Unew + site, C::shifted ? rfma(m, both(P.inv_scale[1]), both(P.shift_h)) : m);
    }
    if (QT > 0) {
      F2 v[QTL];
      pull2<QTL, S, HY, C::shifted, false, false>(at, z, site, f, thn, P.scale[2], v);
      const F2 m = moment_sum2<QTL>(at, z, v);
      st2(thnew + site, C::shifted ? rmul(m, both(P.inv_scale[2])) : m);
    }
  }
}

}  // namespace lbpf
