// lbpf_node.cuh -- the collisions of one node (Sec. 3.2-3.4), shared by every step kernel.
//
// Each routine turns a node's scalars into the coefficients of its collision; the kernels
// apply them to the populations.  All arithmetic is spelled out in fused or separately rounded
// operations, so that every kernel (a tile's owner and its halo, the tiled, the node-wise and the
// one-launch step) rounds a node alike, whatever the compiler makes of its surroundings, and
// their results agree bit for bit.  The FP32 routines (FP32, FP16 and BF16 storage) and the FP64
// routines differ: FP64 is bound by its arithmetic and arranged for few operations.
#pragma once

#include "lbpf_lattice.cuh"

namespace lbpf {

// Products and sums that the compiler does not contract.
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }

__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double rsub(double a, double b) { return __dsub_rn(a, b); }

// 1/x: IEEE division in FP64, the hardware approximate reciprocal in FP32
__device__ __forceinline__ double rcp(double x) { return 1.0 / x; }
__device__ __forceinline__ float rcp(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ double rsq(double x) { return rsqrt(x); }

// Read-only (non-coherent) load, for kernels that start after the kernels before them have ended
// (the tiles, the planes and the one-launch step): what they read this way is never written by the
// same launch.
template <typename S>
__device__ __forceinline__ S ldro(const S* p) { return __ldg(p); }

// Programmatic dependent launch: the node-wise kernels are launched so that the next one may
// start while the last blocks of this one still run.  pdl_trigger() allows that; pdl_wait()
// returns once the kernels before have finished and their writes are visible, and comes
// before the first access to what they write (or read, where this kernel writes it).
//
// Such a kernel reads what is still being written when it starts.  A non-coherent load is for data
// that nobody writes during the whole kernel, and the compiler may move it up across the wait, so
// these kernels use plain loads, which stay behind it.  They cost next to nothing: over 170 grids
// of all storage types a step takes 0.95 to 1.02 of the time with non-coherent loads (geometric mean
// 0.997).  The tiles and planes keep non-coherent loads (FP16 planes of 4000^2: 508 us per step, 536
// with plain ones) and start after the kernel ahead has ended; starting early did not pay there
// either: waiting blocks fill the SMs unevenly (841^2 FP16 tiles 64.6 us per step, 49.9 without).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// RO: by ldro, otherwise a plain load.
template <bool RO, typename S>
__device__ __forceinline__ S ld(const S* p) {
  if constexpr (RO) return ldro(p);
  else return *p;
}

// Index of the first population of weight class c (0 rest, 1 axis, 2 diagonal).
template <int Q>
__host__ __device__ constexpr int class_rep(int c) {
  return c == 0 ? 0 : (c == 1 ? 1 : Lat<Q>::diag0);
}

// Which links a collision computes: all of them, or (the tiles' halo rows) those wanted(e_y).
struct AllLinks {
  __device__ __forceinline__ constexpr bool operator()(int) const { return true; }
};

// Coefficients of a node's collisions (FP32 and FP64 arithmetic have their own).
template <typename T>
struct PhiCoef;
template <typename T>
struct UthCoef;

// ================================================================ FP32 arithmetic
// ---------------------------------------------------------------- phase field
// a_s(n) and N = |grad phi|^2 a_s d a_s / d(grad phi) (Eq. TermesAnisotropes),
// written with n = grad phi / |grad phi| so that FP32 stays in range for small
// gradients.  kind 0: Eq. (Anisotropic-Function_As), derivatives of
// Eq. (Derivees_As); kind 1: Eq. (As_K41-K61) with its analytic derivatives.
__device__ __forceinline__ float sum_squares(float a, float b, float c) { return rfma(c, c, rfma(a, a, rmul(b, b))); }
__device__ __forceinline__ float aniso_N(int kind, float e1, float e2, float gx, float gy, float gz, float G2, float& Nx,
                                         float& Ny, float& Nz) {
  using T = float;
  const T iG = rsqrtf(G2);
  const T nx = rmul(gx, iG), ny = rmul(gy, iG), nz = rmul(gz, iG);
  const T x2 = rmul(nx, nx), y2 = rmul(ny, ny), z2 = rmul(nz, nz);
  const T s4 = sum_squares(x2, y2, z2);
  T as, dx, dy, dz;  // dx = G * d a_s / d(d_x phi)
  if (kind == 0) {
    as = rfma(rmul(T(4), e1), s4, rfma(T(-3), e1, T(1)));
    const T c = rmul(T(16), e1);
    dx = rmul(rmul(c, nx), rsub(x2, s4));
    dy = rmul(rmul(c, ny), rsub(y2, s4));
    dz = rmul(rmul(c, nz), rsub(z2, s4));
  } else {
    const T p3 = rmul(rmul(x2, y2), z2);
    const T e2_part = rsub(rfma(T(66), p3, rmul(T(3), s4)), T(17.0 / 7.0));
    as = rfma(e2, e2_part, rfma(e1, rsub(s4, T(0.6)), T(1)));
    const T cs = rmul(T(4), rfma(T(3), e2, e1));
    const T cp = rmul(T(132), e2);
    auto slope = [&](T n, T n2, T b2, T c2) {  // cs n (n2 - s4) + cp n b2 c2 (1 - 3 n2)
      return rfma(rmul(rmul(rmul(cp, n), b2), c2), rfma(T(-3), n2, T(1)), rmul(rmul(cs, n), rsub(n2, s4)));
    };
    dx = slope(nx, x2, y2, z2);
    dy = slope(ny, y2, x2, z2);
    dz = slope(nz, z2, x2, y2);
  }
  const T f = rmul(rmul(G2, iG), as);  // |grad phi|^2 a_s / |grad phi|
  Nx = rmul(f, dx);
  Ny = rmul(f, dy);
  Nz = rmul(f, dz);
  return as;
}

// |grad phi|^2 from the differences of phi across the node; below grad2_min n and N are taken as
// 0 and a_s = 1
__device__ __forceinline__ bool has_gradient(const Consts<float>& P, float dx, float dy, float dz) {
  return sum_squares(rmul(dx, P.inv2dx), rmul(dy, P.inv2dx), rmul(dz, P.inv2dx)) >= P.grad2_min;
}

// g*_i = [g_i (1 - 1/eta) - (1 - a^2) g_i(x + e_i) + K_c + e_i . n_c] / a^2, c the weight class of link
// i, with K_c + e_i . n_c = g0/eta + w Q dt/tau0 and g0 = w (phi - e.N c_N).
// FP16/BF16: the same in the stored units G = (g - w phi_ref) S, phi_ref the phi^{n-1} of the
// node that stored the value; with the pulled G' = G + S w phi_ref(src) and
// G* = (g* - w phi^n) S only K changes, by -w (oma2 phi_ref(x) + a^2 phi^n), and the value
// gathered for phi^{n+1} is G* + S w phi^n (shift_of).
template <>
struct PhiCoef<float> {
  float omw, oma2, inv_a2, K[3], nx[3], ny[3], nz[3];
  bool flat;  // no gradient: a_s = 1 and N = 0, so oma2 and n_c vanish and a^2 = 1 (these are not
              // set), which spares most nodes of a run (bulk solid and melt) the anisotropy and
              // the non-local term
};

// ph, U, th: the node's values; dx, dy, dz: differences of phi across the node (twice the
// gradient in units of 1/dx, mirror ghosts at walls); wall: standard collision (a^2 := 1 in
// the prefactor and the non-local term); phr: phi_ref(x) (FP16/BF16).
// BRANCH: nodes without a gradient return early with `flat` set; otherwise `flat` stays false and
// they take the general form, to the same bits.
template <int QP, typename S, bool BRANCH>
__device__ __forceinline__ void phi_coef(const Consts<float>& P, float ph, float U, float th, float dx, float dy, float dz,
                                         bool wall, float phr, PhiCoef<float>& c) {
  using T = float;
  using L = Lat<QP>;
  constexpr bool SH = Codec<S>::shifted;
  const T gx = rmul(dx, P.inv2dx), gy = rmul(dy, P.inv2dx), gz = rmul(dz, P.inv2dx);
  const T G2 = sum_squares(gx, gy, gz);
  const bool grad = G2 >= P.grad2_min;
  T as = 1, Nx = 0, Ny = 0, Nz = 0;
  if (grad) as = aniso_N(P.aniso != T(0) ? 1 : 0, P.eps1, P.eps2, gx, gy, gz, G2, Nx, Ny, Nz);
  const T as2 = rmul(as, as);
  const T inv_eta = rcp(rfma(P.c_eta, as2, T(0.5)));
  const T omp2 = rfma(-ph, ph, T(1));
  const T Qdt = rmul(rmul(rfma(-rfma(P.lamM, U, rmul(P.lam, th)), omp2, ph), omp2), P.dt_tau0);
  const T kph = radd(rmul(inv_eta, ph), Qdt);
  c.omw = rsub(T(1), inv_eta);
  c.flat = BRANCH && !grad;
  if (c.flat) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const T wc = (T)L::w(class_rep<QP>(k));
      c.K[k] = rmul(wc, kph);
      if (SH) c.K[k] = rmul(P.scale[0], radd(c.K[k], -rmul(wc, ph)));
    }
    return;
  }
  const T a2 = wall ? T(1) : as2;
  c.inv_a2 = wall ? T(1) : rcp(a2);
  c.oma2 = rsub(T(1), a2);
  const T ncN = rmul(inv_eta, P.c_N);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const T wc = (T)L::w(class_rep<QP>(k));
    c.K[k] = rmul(wc, kph);
    const T nc = rmul(-wc, ncN);
    c.nx[k] = rmul(nc, Nx);
    c.ny[k] = rmul(nc, Ny);
    c.nz[k] = rmul(nc, Nz);
    if (SH) {
      c.K[k] = rmul(P.scale[0], radd(c.K[k], -rmul(wc, radd(rmul(c.oma2, phr), rmul(a2, ph)))));
      c.nx[k] = rmul(P.scale[0], c.nx[k]);
      c.ny[k] = rmul(P.scale[0], c.ny[k]);
      c.nz[k] = rmul(P.scale[0], c.nz[k]);
    }
  }
}

// K + e_i . n, the components added in x, y, z order
template <typename L, typename T>
__device__ __forceinline__ T eq_of(int i, T K, T ax, T ay, T az) {
  T eq = K;
  if (L::ex(i)) eq = L::ex(i) > 0 ? radd(eq, ax) : rsub(eq, ax);
  if (L::ey(i)) eq = L::ey(i) > 0 ? radd(eq, ay) : rsub(eq, ay);
  if (L::ez(i)) eq = L::ez(i) > 0 ? radd(eq, az) : rsub(eq, az);
  return eq;
}

// Post-collision populations of the links wanted(e_y) in place of the pulled ones (in the
// stored units, before the conversion to the storage type).
template <int QP, typename W = AllLinks>
__device__ __forceinline__ void phi_collide(const PhiCoef<float>& c, float (&gp)[QP], const float (&gn)[QP],
                                            W wanted = W()) {
  using L = Lat<QP>;
  if (c.flat) {
#pragma unroll
    for (int i = 0; i < QP; ++i)
      if (wanted(L::ey(i))) gp[i] = rfma(gp[i], c.omw, c.K[L::cls(i)]);
    return;
  }
#pragma unroll
  for (int i = 0; i < QP; ++i) {
    if (!wanted(L::ey(i))) continue;
    const int k = L::cls(i);
    const float eq = eq_of<L>(i, c.K[k], c.nx[k], c.ny[k], c.nz[k]);
    gp[i] = rmul(rfma(-c.oma2, gn[i], rfma(gp[i], c.omw, eq)), c.inv_a2);
  }
}

// The FP16/BF16 shift S w ref of a stored population of link i.
template <typename L>
__device__ __forceinline__ float shift_of(float scale, int i, float ref) {
  return rmul(rmul(scale, (float)L::w(i)), ref);  // scale is a power of two
}

// ---------------------------------------------------------------- U and theta
// h*_i = A h_i + K_c + e_i . j_c: h (1 - 1/eta_U) + h0/eta_U + w (S + Q_U/zeta) dt with
// h0 = A U + B (q/zeta U + e.J c_J).  FP16/BF16: in the stored units H = (h - w U0) S.
// f*_i = At f_i + Kt_c: f (1 - 1/eta_T) + w (theta/eta_T + dphi/2).  FP16/BF16: F is stored as
// (f - w theta_ref) S, theta_ref the theta^{n-1} of the storing node; with the pulled
// F' = F + S w theta_ref(src) and F* = (f* - w theta^n) S, Kt = S w (dphi/2 - theta^n (1 - 1/eta_T))
// and the value gathered for theta^{n+1} is F* + S w theta^n (shift_of).
template <>
struct UthCoef<float> {
  float A, K[3], jx[3], jy[3], jz[3];
  float At, Kt[3];
};

// phn: phi^n; pc and the six neighbours: phi^{n+1} (mirror ghosts at walls); U, th: U^n, theta^n.
template <int QU, int QT, typename S>
__device__ __forceinline__ void uth_coef(const Consts<float>& P, bool at_on, float U, float th, float phn, float pc,
                                         float pxp, float pxm, float pyp, float pym, float pzp, float pzm,
                                         UthCoef<float>& c) {
  using T = float;
  using LU = Lat<QU>;
  using LT = Lat<(QT > 0 ? QT : 7)>;
  constexpr bool SH = Codec<S>::shifted;
  const T inv2dx = P.inv2dx;
  const T opk = radd(T(1), P.k), omk = rsub(T(1), P.k);
  // q(phi) = (1 - phi)/2, zeta(phi) = ((1+k) - (1-k) phi)/2
  auto qf = [&](T p) { return rmul(T(0.5), rsub(T(1), p)); };
  // 1/zeta at the node and its six neighbours with one division (batch inversion):
  // 2 zeta = (1+k) - (1-k) phi
  auto zeta2 = [&](T p) { return rfma(-omk, p, opk); };
  const T d0 = zeta2(pc), d1 = zeta2(pxp), d2 = zeta2(pxm), d3 = zeta2(pyp), d4 = zeta2(pym), d5 = zeta2(pzp),
          d6 = zeta2(pzm);
  const T p1 = rmul(d0, d1), p2 = rmul(p1, d2), p3 = rmul(p2, d3), p4 = rmul(p3, d4), p5 = rmul(p4, d5);
  T rr = rmul(T(2), rcp(rmul(p5, d6)));  // 2 / (d0 ... d6)
  const T iz_zm = rmul(rr, p5);
  rr = rmul(rr, d6);
  const T iz_zp = rmul(rr, p4);
  rr = rmul(rr, d5);
  const T iz_ym = rmul(rr, p3);
  rr = rmul(rr, d4);
  const T iz_yp = rmul(rr, p2);
  rr = rmul(rr, d3);
  const T iz_xm = rmul(rr, p1);
  rr = rmul(rr, d2);
  const T iz_xp = rmul(rr, d0);
  const T izc = rmul(rr, d1);
  const T qc = qf(pc), qzc = rmul(qc, izc);
  const T gpx = rmul(rsub(pxp, pxm), inv2dx), gpy = rmul(rsub(pyp, pym), inv2dx), gpz = rmul(rsub(pzp, pzm), inv2dx);
  const T Fx = rmul(rsub(iz_xp, iz_xm), inv2dx), Fy = rmul(rsub(iz_yp, iz_ym), inv2dx),
          Fz = rmul(rsub(iz_zp, iz_zm), inv2dx);
  // grad(q/zeta)
  auto grad_qz = [&](T pp, T izp, T pm, T izm) { return rmul(rfma(qf(pp), izp, -rmul(qf(pm), izm)), inv2dx); };
  const T gqzx = grad_qz(pxp, iz_xp, pxm, iz_xm), gqzy = grad_qz(pyp, iz_yp, pym, iz_ym),
          gqzz = grad_qz(pzp, iz_zp, pzm, iz_zm);
  // div(D q grad(1/zeta)) in compact face form, face q = mean of nodal q
  auto face = [&](T p) { return rmul(T(0.5), radd(qc, qf(p))); };
  T dv = rfma(face(pxp), rsub(iz_xp, izc), -rmul(face(pxm), rsub(izc, iz_xm)));
  dv = rfma(face(pyp), rsub(iz_yp, izc), dv);
  dv = rfma(-face(pym), rsub(izc, iz_ym), dv);
  dv = rfma(face(pzp), rsub(iz_zp, izc), dv);
  dv = rfma(-face(pzm), rsub(izc, iz_zm), dv);
  const T divDqF = rmul(P.D_dx2, dv);
  const T dphi = rsub(pc, phn);  // phi^{n+1} - phi^n
  const T dphidt = rmul(dphi, P.inv_dt);
  const T fU = rfma(omk, U, T(1));
  T jx = 0, jy = 0, jz = 0;
  const T G2 = sum_squares(gpx, gpy, gpz);
  if (at_on && G2 >= P.grad2_min) {
    const T amp = rmul(rmul(rmul(-P.at_amp, fU), dphidt), rsqrtf(G2));
    jx = rmul(amp, gpx);
    jy = rmul(amp, gpy);
    jz = rmul(amp, gpz);
  }
  const T DqU = rmul(P.D, U);
  const T Jx = rfma(DqU, rfma(qc, Fx, gqzx), rmul(jx, izc));
  const T Jy = rfma(DqU, rfma(qc, Fy, gqzy), rmul(jy, izc));
  const T Jz = rfma(DqU, rfma(qc, Fz, gqzz), rmul(jz, izc));
  const T Ssrc = rfma(U, divDqF, rfma(jz, Fz, rfma(jx, Fx, rmul(jy, Fy))));
  const T src_dt = rmul(rfma(rmul(rmul(fU, T(0.5)), dphidt), izc, Ssrc), P.dt);
  const T qzU = rmul(qzc, U);
  c.A = rsub(T(1), P.inv_etaU);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int ic = class_rep<QU>(k);
    const T wc = (T)LU::w(ic), Bc = (T)LU::B(ic);
    c.K[k] = radd(rmul(P.inv_etaU, radd(k == 0 ? U : T(0), rmul(Bc, qzU))), rmul(wc, src_dt));
    const T jc = rmul(rmul(P.inv_etaU, Bc), P.c_J);
    c.jx[k] = rmul(jc, Jx);
    c.jy[k] = rmul(jc, Jy);
    c.jz[k] = rmul(jc, Jz);
    if (SH) {
      c.K[k] = rmul(P.scale[1], radd(c.K[k], -rmul(rmul(wc, P.shift_h), P.inv_etaU)));
      c.jx[k] = rmul(P.scale[1], c.jx[k]);
      c.jy[k] = rmul(P.scale[1], c.jy[k]);
      c.jz[k] = rmul(P.scale[1], c.jz[k]);
    }
  }
  if (QT > 0) {
    c.At = rsub(T(1), P.inv_etaT);
    T kT = radd(rmul(P.inv_etaT, th), rmul(T(0.5), dphi));
    if (SH) kT = rmul(P.scale[2], radd(rmul(T(0.5), dphi), -rmul(th, c.At)));
#pragma unroll
    for (int k = 0; k < 3; ++k) c.Kt[k] = rmul((T)LT::w(class_rep<(QT > 0 ? QT : 7)>(k)), kT);
  }
}

template <int QU, typename W = AllLinks>
__device__ __forceinline__ void u_collide(const UthCoef<float>& c, float (&h)[QU], W wanted = W()) {
  using L = Lat<QU>;
#pragma unroll
  for (int i = 0; i < QU; ++i) {
    if (!wanted(L::ey(i))) continue;
    const int k = L::cls(i);
    h[i] = rfma(h[i], c.A, eq_of<L>(i, c.K[k], c.jx[k], c.jy[k], c.jz[k]));
  }
}

// ================================================================ FP64 arithmetic
// The collisions arranged for few operations: two FMAs and one addition per population for phi,
// one FMA and one addition for U, one FMA for theta, the e_i part of the equilibrium once per
// pair of opposite links, and short forms for nodes of the bulk.
// Signed sum of the components of (ax, ay, az) along link i, added in x, y, z order: the
// value for the opposite link is its exact negative.  Never called for the rest link.
template <typename L, typename T>
__device__ __forceinline__ T along(int i, T ax, T ay, T az) {
  const int ex = L::ex(i), ey = L::ey(i), ez = L::ez(i);
  T d = T(0);
  bool any = false;
  if (ex) { d = ex > 0 ? ax : -ax; any = true; }
  if (ey) { const T v = ey > 0 ? ay : -ay; d = any ? radd(d, v) : v; any = true; }
  if (ez) { const T v = ez > 0 ? az : -az; d = any ? radd(d, v) : v; }
  return d;
}

// ---------------------------------------------------------------- phase field
// g*_i = A g_i(x) + B g_i(x + e_i) + K_c + e_i . n_c, c the weight class of link i:
// [g (1 - 1/eta) - (1 - a^2) g_nl + g0/eta + w Q dt/tau0] / a^2 with
// g0 = w (phi - e.N c_N), the division by a^2 multiplied into every coefficient.
template <>
struct PhiCoef<double> {
  double A, B, K[3], nx[3], ny[3], nz[3];
  bool flat;  // no gradient: a_s = 1 and N = 0, so B and n_c vanish (and are not set), which spares
              // most nodes of a run (bulk solid and melt) the anisotropy and the non-local term
};

__device__ __forceinline__ bool has_gradient(const Consts<double>& P, double dx, double dy, double dz) {
  return rmul(rfma(dx, dx, rfma(dy, dy, rmul(dz, dz))), P.inv2dx2) >= P.grad2_min;
}

template <int QP, typename S, bool BRANCH>  // FP64 steps node-wise only, and always branches
__device__ __forceinline__ void phi_coef(const Consts<double>& P, double ph, double U, double th, double dx, double dy,
                                         double dz, bool wall, double, PhiCoef<double>& c) {
  using T = double;
  using L = Lat<QP>;
  const T omp2 = rfma(-ph, ph, T(1));
  const T Q = rmul(rmul(rfma(-rfma(P.lamM, U, rmul(P.lam, th)), omp2, ph), omp2), P.dt_tau0);
  static_assert(BRANCH, "FP64 has no form without the branch");
  c.flat = !has_gradient(P, dx, dy, dz);
  if (c.flat) {
    const T kk = rfma(P.inv_eta1, ph, Q);
    c.A = radd(T(1), -P.inv_eta1);
#pragma unroll
    for (int k = 0; k < 3; ++k) c.K[k] = rmul((T)L::w(class_rep<QP>(k)), kk);
    return;
  }
  // a_s(n) = a0 + a4 sum n^4 + a6 nx^2 ny^2 nz^2 covers Eq. (Anisotropic-Function_As) and
  // Eq. (As_K41-K61); N = |grad phi|^2 a_s d a_s / d(grad phi) (Eq. TermesAnisotropes)
  const T s2 = rfma(dx, dx, rfma(dy, dy, rmul(dz, dz)));
  const T iG = rsq(s2);
  const T nx = rmul(dx, iG), ny = rmul(dy, iG), nz = rmul(dz, iG);
  const T x2 = rmul(nx, nx), y2 = rmul(ny, ny), z2 = rmul(nz, nz);
  const T s4 = rfma(x2, x2, rfma(y2, y2, rmul(z2, z2)));
  const T c4 = rmul(T(4), P.a4);
  T as = rfma(P.a4, s4, P.a0);
  T px = rmul(c4, radd(x2, -s4)), py = rmul(c4, radd(y2, -s4)), pz = rmul(c4, radd(z2, -s4));
  if (P.a6 != T(0)) {
    const T yz = rmul(y2, z2), xz = rmul(x2, z2), xy = rmul(x2, y2);
    const T c6 = rmul(T(2), P.a6);
    as = rfma(P.a6, rmul(x2, yz), as);
    px = rfma(rmul(c6, yz), rfma(T(-3), x2, T(1)), px);
    py = rfma(rmul(c6, xz), rfma(T(-3), y2, T(1)), py);
    pz = rfma(rmul(c6, xy), rfma(T(-3), z2, T(1)), pz);
  }
  const T f = rmul(rmul(rmul(s2, iG), P.inv2dx), as);  // |grad phi| a_s
  T Nx = rmul(f, rmul(nx, px));
  T Ny = rmul(f, rmul(ny, py));
  T Nz = rmul(f, rmul(nz, pz));
  const T as2 = rmul(as, as);
  const T eta = rfma(P.c_eta, as2, T(0.5));
  const T a2 = wall ? T(1) : as2;
  const T r = rcp(rmul(eta, as2));  // one division for both
  const T inv_eta = rmul(r, as2), inv_a2 = wall ? T(1) : rmul(r, eta);
  const T oma2 = radd(T(1), -a2);
  const T kk = rmul(rfma(inv_eta, ph, Q), inv_a2);
  const T nn = -rmul(rmul(inv_eta, P.c_N), inv_a2);
  Nx = rmul(nn, Nx);
  Ny = rmul(nn, Ny);
  Nz = rmul(nn, Nz);
  c.A = rmul(radd(T(1), -inv_eta), inv_a2);
  c.B = -rmul(oma2, inv_a2);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const T w = (T)L::w(class_rep<QP>(k));
    c.K[k] = rmul(w, kk);
    c.nx[k] = rmul(w, Nx);
    c.ny[k] = rmul(w, Ny);
    c.nz[k] = rmul(w, Nz);
  }
}

template <int QP>
__device__ __forceinline__ void phi_collide(const PhiCoef<double>& c, double (&gp)[QP], const double (&gn)[QP]) {
  using T = double;
  using L = Lat<QP>;
  if (c.flat) {
#pragma unroll
    for (int i = 0; i < QP; ++i) gp[i] = rfma(c.A, gp[i], c.K[L::cls(i)]);
    return;
  }
  gp[0] = rfma(c.A, gp[0], rfma(c.B, gn[0], c.K[0]));
#pragma unroll
  for (int i = 1; i < QP; ++i) {
    const int j = L::opp(i);
    if (j < i) continue;
    const int k = L::cls(i);
    const T d = along<L>(i, c.nx[k], c.ny[k], c.nz[k]);
    gp[i] = rfma(c.A, gp[i], rfma(c.B, gn[i], radd(c.K[k], d)));
    gp[j] = rfma(c.A, gp[j], rfma(c.B, gn[j], radd(c.K[k], -d)));
  }
}

// ---------------------------------------------------------------- U and theta
template <>
struct UthCoef<double> {
  double A, K[3], jx[3], jy[3], jz[3];
  bool flat;  // phi^{n+1} is the same at the node and its six neighbours: J = S = 0, so j_c vanish
              // (and are not set)
  double At, Kt[3];
};

template <int QU, int QT, typename S>
__device__ __forceinline__ void uth_coef(const Consts<double>& P, bool at_on, double U, double th, double phn, double pc,
                                         double pxp, double pxm, double pyp, double pym, double pzp, double pzm,
                                         UthCoef<double>& c) {
  using T = double;
  using LU = Lat<QU>;
  using LT = Lat<(QT > 0 ? QT : 7)>;
  constexpr bool HY = LU::has_y;
  // 2 zeta = (1+k) - (1-k) phi; 1/zeta at the node and its neighbours with one division
  const T opk = radd(T(1), P.k), omk = radd(T(1), -P.k);
  auto zeta2 = [&](T p) { return rfma(-omk, p, opk); };
  const T dphi = radd(pc, -phn);
  const T rate = rmul(dphi, P.inv_dt);
  const T fU = rfma(omk, U, T(1));
  const T tc = radd(T(1), -pc);  // t = 2 q = 1 - phi
  c.A = radd(T(1), -P.inv_etaU);
  if (QT > 0) {
    c.At = radd(T(1), -P.inv_etaT);
    const T kt = rfma(P.inv_etaT, th, rmul(T(0.5), dphi));
#pragma unroll
    for (int k = 0; k < 3; ++k) c.Kt[k] = rmul((T)LT::w(class_rep<(QT > 0 ? QT : 7)>(k)), kt);
  }
  // K_c from q/zeta U and (S + Q_U/zeta) dt
  auto set_K = [&](T qzU, T src) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const T w = (T)LU::w(class_rep<QU>(k)), b = (T)LU::B(class_rep<QU>(k));
      const T eq = k == 0 ? rfma(b, qzU, U) : rmul(b, qzU);
      c.K[k] = rfma(P.inv_etaU, eq, rmul(w, src));
    }
  };
  c.flat = pxp == pc && pxm == pc && pyp == pc && pym == pc && pzp == pc && pzm == pc;
  if (c.flat) {
    const T izc = rmul(T(2), rcp(zeta2(pc)));
    set_K(rmul(rmul(rmul(T(0.5), tc), izc), U), rmul(rmul(rmul(rmul(T(0.5), fU), rate), izc), P.dt));
    return;
  }
  const T d0 = zeta2(pc), d1 = zeta2(pxp), d2 = zeta2(pxm), d5 = zeta2(pzp), d6 = zeta2(pzm);
  T izc, iz_xp, iz_xm, iz_yp, iz_ym, iz_zp, iz_zm;
  {
    const T p1 = rmul(d0, d1), p2 = rmul(p1, d2);
    T rr;
    if constexpr (HY) {
      const T d3 = zeta2(pyp), d4 = zeta2(pym);
      const T p3 = rmul(p2, d3), p4 = rmul(p3, d4), p5 = rmul(p4, d5);
      rr = rmul(T(2), rcp(rmul(p5, d6)));
      iz_zm = rmul(rr, p5);
      rr = rmul(rr, d6);
      iz_zp = rmul(rr, p4);
      rr = rmul(rr, d5);
      iz_ym = rmul(rr, p3);
      rr = rmul(rr, d4);
      iz_yp = rmul(rr, p2);
      rr = rmul(rr, d3);
    } else {
      const T p5 = rmul(p2, d5);
      rr = rmul(T(2), rcp(rmul(p5, d6)));
      iz_zm = rmul(rr, p5);
      rr = rmul(rr, d6);
      iz_zp = rmul(rr, p2);
      rr = rmul(rr, d5);
    }
    iz_xm = rmul(rr, p1);
    rr = rmul(rr, d2);
    iz_xp = rmul(rr, d0);
    izc = rmul(rr, d1);
    if constexpr (!HY) iz_yp = iz_ym = izc;
  }
  // unscaled differences (the factors 1/(2 dx) and 1/2 come in at the end)
  auto t2 = [&](T p) { return radd(T(1), -p); };
  const T txp = t2(pxp), txm = t2(pxm), tzp = t2(pzp), tzm = t2(pzm);
  const T tyc_p = HY ? t2(pyp) : tc, tyc_m = HY ? t2(pym) : tc;
  const T gx = radd(pxp, -pxm), gy = HY ? radd(pyp, -pym) : T(0), gz = radd(pzp, -pzm);
  const T Fx = radd(iz_xp, -iz_xm), Fy = HY ? radd(iz_yp, -iz_ym) : T(0), Fz = radd(iz_zp, -iz_zm);
  const T qx = rfma(txp, iz_xp, -rmul(txm, iz_xm)), qz = rfma(tzp, iz_zp, -rmul(tzm, iz_zm));
  const T qy = HY ? rfma(tyc_p, iz_yp, -rmul(tyc_m, iz_ym)) : T(0);
  // div(D q grad(1/zeta)) in compact face form, face q = mean of nodal q: 1/4 of this sum
  T dv = rmul(radd(tc, txp), radd(iz_xp, -izc));
  dv = rfma(radd(tc, txm), radd(iz_xm, -izc), dv);
  if (HY) {
    dv = rfma(radd(tc, tyc_p), radd(iz_yp, -izc), dv);
    dv = rfma(radd(tc, tyc_m), radd(iz_ym, -izc), dv);
  }
  dv = rfma(radd(tc, tzp), radd(iz_zp, -izc), dv);
  dv = rfma(radd(tc, tzm), radd(iz_zm, -izc), dv);
  const T divDqF = rmul(rmul(T(0.25), P.D_dx2), dv);
  T jx = T(0), jy = T(0), jz = T(0);
  const T s2 = rfma(gx, gx, rfma(gy, gy, rmul(gz, gz)));
  if (at_on && rmul(s2, P.inv2dx2) >= P.grad2_min) {  // Eq. (AntiTrapping_Current), n = grad phi / |grad phi|
    const T amp = rmul(rmul(rmul(-P.at_amp, fU), rate), rsq(s2));
    jx = rmul(amp, gx);
    jy = rmul(amp, gy);
    jz = rmul(amp, gz);
  }
  const T DU = rmul(rmul(rmul(T(0.5), P.D), P.inv2dx), U);
  const T Jx = rfma(DU, rfma(tc, Fx, qx), rmul(jx, izc));
  const T Jy = rfma(DU, rfma(tc, Fy, qy), rmul(jy, izc));
  const T Jz = rfma(DU, rfma(tc, Fz, qz), rmul(jz, izc));
  const T jF = rmul(P.inv2dx, rfma(jx, Fx, rfma(jy, Fy, rmul(jz, Fz))));
  const T Ssrc = rfma(U, divDqF, jF);
  const T src = rmul(rfma(rmul(rmul(T(0.5), fU), rate), izc, Ssrc), P.dt);
  set_K(rmul(rmul(rmul(T(0.5), tc), izc), U), src);
  const T cj = rmul(P.inv_etaU, P.c_J);
  const T jsx = rmul(cj, Jx), jsy = rmul(cj, Jy), jsz = rmul(cj, Jz);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const T b = (T)LU::B(class_rep<QU>(k));
    c.jx[k] = rmul(b, jsx);
    c.jy[k] = rmul(b, jsy);
    c.jz[k] = rmul(b, jsz);
  }
}

template <int QU>
__device__ __forceinline__ void u_collide(const UthCoef<double>& c, double (&h)[QU]) {
  using T = double;
  using L = Lat<QU>;
  if (c.flat) {
#pragma unroll
    for (int i = 0; i < QU; ++i) h[i] = rfma(c.A, h[i], c.K[L::cls(i)]);
    return;
  }
  h[0] = rfma(c.A, h[0], c.K[0]);
#pragma unroll
  for (int i = 1; i < QU; ++i) {
    const int j = L::opp(i);
    if (j < i) continue;
    const int k = L::cls(i);
    const T d = along<L>(i, c.jx[k], c.jy[k], c.jz[k]);
    h[i] = rfma(c.A, h[i], radd(c.K[k], d));
    h[j] = rfma(c.A, h[j], radd(c.K[k], -d));
  }
}

}  // namespace lbpf
