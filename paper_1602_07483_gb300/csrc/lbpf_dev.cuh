// lbpf_dev.cuh -- device code of the lattice-Boltzmann phase-field step for sm_103a.
//
// The tiled step: the distributions are read once, at the price of halo collisions
// (lbpf_nodewise.cuh is the form without a halo).  One time step (Sec. 3.4, "Algorithm implementation") on D3Q7/D3Q15/D3Q19, or on
// D2Q5/D2Q9 over an nz = 1 grid, is two kernels:
//   k_phi : phi collision (Eq. collision stage, non-local term) + streaming with
//           bounce-back, using phi^n, U^n, theta^n; writes the post-collision
//           populations and phi^{n+1}.
//   k_uth : U collision (Eq. LBE_Eq_Transport with the equilibrium of
//           Eq. Feq_Transport) and theta collision (Eq. LBE_Eq_Temp) with
//           phi^{n+1}, dphi/dt = (phi^{n+1} - phi^n)/dt; writes the post-collision
//           populations, U^{n+1} and theta^{n+1}.
//
// Storage ("pull" layout): buffer A holds, at node x, the post-collision value
// g*_i(x) of the previous step.  The population entering the collision at x is
// g_i(x,t) = A_i(x - e_i), or A_{i'}(x) when x - e_i is outside the domain
// (halfway bounce-back).  The non-local term g_i(x + e_i, t) of the phase-field
// collision is then A_i(x) itself for every non-boundary node.
//
// Each thread block owns a 30 x (BY-2) column of the xy plane and marches in z
// over a chunk of planes; a block is 32 x BY threads, one node per thread and
// plane.  For every plane the block recomputes the
// collisions on a one-node halo (32 x BY nodes) and gathers the streamed
// populations of its interior nodes into the zeroth moment of the next step:
// populations with e_y = 0 come from the thread itself or its x-neighbour lane
// by warp shuffle, the others through a double-buffered shared-memory plane, so
// each plane needs a single barrier.  The moment fields cost one scalar write
// per node and the distributions are read once and written once.
#pragma once

#include "lbpf_node.cuh"
#include "lbpf_plan.h"

namespace lbpf {

#ifndef LBPF_MAX_BLOCK_ROWS
#define LBPF_MAX_BLOCK_ROWS 8
#endif
constexpr int MAX_BLOCK_ROWS = LBPF_MAX_BLOCK_ROWS;  // blocks of at most 32 x 8 threads

// Resident blocks per SM the step kernels are compiled for (register budget:
// 65536 / (256 x blocks) registers per thread).  Measured on 512^3: k_phi runs
// best at three blocks (80 registers); k_uth at two (at 80 registers it spills).
#ifndef LBPF_PHI_MIN_BLOCKS
#define LBPF_PHI_MIN_BLOCKS 3
#endif
#ifndef LBPF_UTH_MIN_BLOCKS
#define LBPF_UTH_MIN_BLOCKS 2
#endif
// The 2D lattices run one-warp blocks; their launch bounds (counted in 256-thread
// blocks) set the register budget that decides how many warps an SM holds.  Measured
// on 8192^2 FP32: 64 registers (four 256-thread blocks) for both kernels, 21.2 -> 26.4
// GLUPS.
#ifndef LBPF_PHI2D_MIN_BLOCKS
#define LBPF_PHI2D_MIN_BLOCKS 4
#endif
#ifndef LBPF_UTH2D_MIN_BLOCKS
#define LBPF_UTH2D_MIN_BLOCKS 4
#endif
inline __device__ int slot4(int z) { return (z + 4) & 3; }  // z >= -1

// Scalar-field ring: four planes of (BY + 2) x 34 values around the block
// region (mirror ghosts by clamping).  Each thread owns up to RPT elements of a
// plane; their in-plane offsets are computed once, and the plane two ahead of
// the collision plane is fetched into registers one iteration early.
constexpr int RPT = 2;  // 34 x (BY + 2) <= RPT x 32 x BY for BY >= 3

struct RingMap {
  int off[RPT];  // in-plane offset (y * nx + x), or -1 when the slot is unused
  __device__ __forceinline__ void init(int x0, int y0, int nx, int ny, int RW, int RS, int tid, int nthr) {
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
      const int idx = tid + r * nthr;
      off[r] = -1;
      if (idx < RS) {
        const int ly = idx / RW;
        const int lx = idx - ly * RW;
        const int gx = min(max(x0 - 2 + lx, 0), nx - 1);
        const int gy = min(max(y0 - 2 + ly, 0), ny - 1);
        off[r] = gy * nx + gx;
      }
    }
  }
};

template <typename T>
struct RingRegs {
  T v[RPT];
  // CG: through L2 (ld.global.cg) instead of the read-only path, for data written earlier
  // in the same launch
  template <bool CG = false>
  __device__ __forceinline__ void fetch(const RingMap& m, const T* __restrict__ src, int z, int nz, long long plane) {
    const T* p = src + (long long)min(max(z, 0), nz - 1) * plane;
#pragma unroll
    for (int r = 0; r < RPT; ++r)
      if (m.off[r] >= 0) v[r] = CG ? __ldcg(p + m.off[r]) : ldro(p + m.off[r]);
  }
  __device__ __forceinline__ void store(const RingMap& m, T* __restrict__ dst, int tid, int nthr) const {
#pragma unroll
    for (int r = 0; r < RPT; ++r)
      if (m.off[r] >= 0) dst[tid + r * nthr] = v[r];
  }
};

// ---------------------------------------------------------------- phase field
// One tile of the phase-field phase: the block's 30 x (BY-2) columns over planes [z0, z1).
// BYC: the block height BY when fixed at compile time (its index arithmetic then folds into
// constants), 0 to take it from blockDim.y.
template <int QP, typename S, int BYC>
__device__ __forceinline__ void phi_tile(const SimDev* __restrict__ sims, const WorkItem it, int s6) {
  using C = Codec<S>;
  using T = typename C::T;
  using L = Lat<QP>;
  using YS = YSlots<QP>;
  constexpr int NY = NYOf<QP>::value;
  const SimDev& sd = sims[it.sim];
  const int nx = sd.nx, ny = sd.ny, nz = sd.nz;
  const int BY = BYC > 0 ? BYC : (int)blockDim.y;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int tid = ty * 32 + tx, nthr = 32 * BY;
  const int x = it.x0 - 1 + tx;
  const int par = s6 & 1;
  // element offsets fit in 32 bits (Q * nsite < 2^32 is checked at create)
  const unsigned NS = (unsigned)sd.nsite;
  const unsigned plane = (unsigned)ny * (unsigned)nx;
  const S* __restrict__ gin = (const S*)sd.pop[par][0];
  S* __restrict__ gout = (S*)sd.pop[par ^ 1][0];
  const T* __restrict__ phin = (const T*)sd.phi[s6 % 3];
  const T* __restrict__ phim = (const T*)sd.phi[(s6 + 2) % 3];
  T* __restrict__ phinew = (T*)sd.phi[(s6 + 1) % 3];
  const T* __restrict__ Un = (const T*)sd.U[par];
  const T* __restrict__ thn = (const T*)sd.th[s6 % 3];
  const bool has_th = sd.q_theta != 0;

  constexpr bool HY = L::has_y;  // false: 2D lattice, one-row blocks without y halo
  const int RW = 34, RS = HY ? RW * (BY + 2) : RW, PS = BY * 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* ring = reinterpret_cast<T*>(smem_raw);  // phi^n     [4][BY+2][34]
  T* ringm = ring + 4 * RS;                  // phi^{n-1} [4][BY+2][34] (codec shift only)
  T* sG = ring + (C::shifted ? 8 : 4) * RS;  // [2][NY][BY][32]

  const Consts<T> P = consts_of<T>(sd);
  const T theta0 = P.theta0, scale = P.scale[0], iscale = P.inv_scale[0];

  const int zlo = max(it.z0 - 1, 0), zhi = min(it.z1, nz - 1);
  RingMap rm;
  rm.init(it.x0, it.y0, nx, ny, RW, RS, tid, nthr);
  {
    RingRegs<T> a;
    for (int z = zlo - 1; z <= zlo + 1; ++z) {
      a.fetch(rm, phin, z, nz, plane);
      a.store(rm, ring + slot4(z) * RS, tid, nthr);
      if (C::shifted) {
        a.fetch(rm, phim, z, nz, plane);
        a.store(rm, ringm + slot4(z) * RS, tid, nthr);
      }
    }
  }
  RingRegs<T> pf, pfm;
  if (zlo + 2 <= zhi + 1) {
    pf.fetch(rm, phin, zlo + 2, nz, plane);
    if (C::shifted) pfm.fetch(rm, phim, zlo + 2, nz, plane);
  }
  T a0A = 0, a1A = 0, a2A = 0;  // moments of planes zc-1, zc, zc+1
  int buf = 0;
  __syncthreads();

  for (int zc = zlo; zc <= zhi; ++zc) {
    T* sGb = sG + buf * NY * PS;
    const T* R0 = ring + slot4(zc) * RS;
    const T* Rp = ring + slot4(zc + 1) * RS;
    const T* Rm = ring + slot4(zc - 1) * RS;
    auto collide_row = [&](auto row_kind, T& acc0, T& acc1, T& acc2) {
      constexpr int KIND = decltype(row_kind)::value;  // 0 interior row, 1 top halo, 2 bottom halo
      auto row_needs = [](int ey) { return KIND == 0 || (KIND == 1 && ey == 1) || (KIND == 2 && ey == -1); };
      const int ly = ty;
      const int y = HY ? it.y0 - 1 + ly : it.y0 + ly;  // row 0 is a halo row except in one-row blocks
      const bool in_xy = x >= 0 && x < nx && y >= 0 && y < ny;
      const bool icol = in_xy && tx >= 1 && tx <= TILE_X && (!HY || (ly >= 1 && ly <= BY - 2));
      const int rc = HY ? (ly + 1) * RW + (tx + 1) : tx + 1;
      const unsigned site = ((unsigned)zc * (unsigned)ny + (unsigned)y) * (unsigned)nx + (unsigned)x;
      // wall node (standard collision): on a wall the lattice has links through
      // wall node (standard collision) on a face the lattice has links through; for the 3D
      // lattices the predicate keeps the order of the 3D-only kernels (the compiler's
      // schedule of the step kernels is sensitive to it)
      const bool bnd = L::has_y ? (x == 0 || y == 0 || zc == 0 || x == nx - 1 || y == ny - 1 || zc == nz - 1)
                                : (x == 0 || zc == 0 || x == nx - 1 || zc == nz - 1);
      T gs[QP];
#pragma unroll
      for (int i = 0; i < QP; ++i) gs[i] = T(0);
      if (in_xy) {
        const T Usite = ldro(Un + site);
        const T thsite = has_th ? ldro(thn + site) : theta0;
        // pulled populations g_i(x,t) and non-local values g_i(x+e_i,t), all loads first
        T gpull[QP], gnl[QP];
        if (!bnd) {
#pragma unroll
          for (int i = 0; i < QP; ++i) {
            const int ex = L::ex(i), ey = L::ey(i), ez = L::ez(i);
            if (!row_needs(ey)) continue;
            const unsigned own = (unsigned)i * NS + site;
            const unsigned off = (unsigned)(ez * (int)plane + ey * nx + ex);
            gpull[i] = C::raw(ldro(gin + (own - off)));
            if (C::shifted)  // stored units with the source's shift: Gp + S w phi_ref(src)
              gpull[i] = rfma(rmul(scale, (T)L::w(i)), (ringm + slot4(zc - ez) * RS)[rc - ey * RW - ex], gpull[i]);
            gnl[i] = C::raw(ldro(gin + own));
          }
        } else {
          // wall node: bounce-back for links from outside, standard collision (no non-local term)
#pragma unroll
          for (int i = 0; i < QP; ++i) {
            const int ex = L::ex(i), ey = L::ey(i), ez = L::ez(i);
            if (!row_needs(ey)) continue;
            const int sx = x - ex, sy = y - ey, sz = zc - ez;
            const bool inside = sx >= 0 && sx < nx && sy >= 0 && sy < ny && sz >= 0 && sz < nz;
            const unsigned src = inside ? site - (unsigned)(ez * (int)plane + ey * nx + ex) : site;
            const int ii = inside ? i : L::opp(i);
            gpull[i] = C::raw(ldro(gin + ((unsigned)ii * NS + src)));
            if (C::shifted)
              gpull[i] = rfma(rmul(scale, (T)L::w(i)), (ringm + slot4(inside ? sz : zc) * RS)[inside ? rc - ey * RW - ex : rc],
                             gpull[i]);
            gnl[i] = T(0);
          }
        }
        const T ph = R0[rc];
        // centred differences with mirror ghosts (clamped ring)
        const T dy = HY ? radd(R0[rc + RW], -R0[rc - RW]) : T(0);
        PhiCoef<T> co;
        phi_coef<QP, S, false>(P, ph, Usite, thsite, radd(R0[rc + 1], -R0[rc - 1]), dy, radd(Rp[rc], -Rm[rc]), bnd,
                           C::shifted ? (ringm + slot4(zc) * RS)[rc] : T(0), co);
        phi_collide<QP>(co, gpull, gnl, row_needs);
        const bool store = icol && zc >= it.z0 && zc < it.z1;
#pragma unroll
        for (int i = 0; i < QP; ++i) {
          const int ey = L::ey(i);
          if (!row_needs(ey)) continue;
          const auto enc = C::pack(gpull[i]);
          if (store) gout[(unsigned)i * NS + site] = enc;
          gs[i] = C::shifted ? radd(C::raw(enc), shift_of<L>(scale, i, ph)) : gpull[i];
          if (ey != 0) sGb[YS::slot(i) * PS + ly * 32 + tx] = gs[i];
        }
      }
      if (KIND == 0) {
        // populations with e_y = 0: from this lane or the x-neighbour lane (all lanes shuffle)
        T sv[QP];
  #pragma unroll
        for (int i = 0; i < QP; ++i) {
          const int ex = L::ex(i), ey = L::ey(i);
          sv[i] = gs[i];
          if (ey == 0 && ex > 0) sv[i] = __shfl_up_sync(0xffffffffu, gs[i], 1);
          if (ey == 0 && ex < 0) sv[i] = __shfl_down_sync(0xffffffffu, gs[i], 1);
        }
        if (icol) {
          if (!bnd) {
  #pragma unroll
            for (int i = 0; i < QP; ++i) {
              const int ey = L::ey(i), ez = L::ez(i);
              if (ey != 0) continue;
              if (ez < 0) acc0 += sv[i];
              else if (ez > 0) acc2 += sv[i];
              else acc1 += sv[i];
            }
          } else {
  #pragma unroll
            for (int i = 0; i < QP; ++i) {
              const int ex = L::ex(i), ey = L::ey(i), ez = L::ez(i);
              if (!row_needs(ey)) continue;
              if (ey != 0) continue;
              const int sx = x - ex, sz = zc - ez;
              const bool sin = sx >= 0 && sx < nx;
              if (sin) {
                if (ez < 0) acc0 += sv[i];
                else if (ez > 0) acc2 += sv[i];
                else acc1 += sv[i];
              }
              if (!sin || sz < 0 || sz >= nz) acc1 += gs[L::opp(i)];
            }
          }
        }
      }
    };
    // rows 0 and BY-1 are halo rows: they only feed the e_y = +1 / -1 populations to the block
    if (!HY) collide_row(std::integral_constant<int, 0>{}, a0A, a1A, a2A);
    else if (ty == 0) collide_row(std::integral_constant<int, 1>{}, a0A, a1A, a2A);
    else if (ty == BY - 1) collide_row(std::integral_constant<int, 2>{}, a0A, a1A, a2A);
    else collide_row(std::integral_constant<int, 0>{}, a0A, a1A, a2A);
    // ring plane zc+2 (its slot last held plane zc-2), then prefetch zc+3
    if (zc + 2 <= zhi + 1) {
      pf.store(rm, ring + slot4(zc + 2) * RS, tid, nthr);
      if (C::shifted) pfm.store(rm, ringm + slot4(zc + 2) * RS, tid, nthr);
    }
    if (zc + 3 <= zhi + 1) {
      pf.fetch(rm, phin, zc + 3, nz, plane);
      if (C::shifted) pfm.fetch(rm, phim, zc + 3, nz, plane);
    }
    __syncthreads();
    // populations with e_y != 0: from the neighbouring rows through shared memory
    auto gather_row = [&](const int r, T& acc0, T& acc1, T& acc2) {
      const int ly = ty;
      const int y = HY ? it.y0 - 1 + ly : it.y0 + ly;  // row 0 is a halo row except in one-row blocks
      const bool icol = x >= 0 && x < nx && y >= 0 && y < ny && tx >= 1 && tx <= TILE_X && (!HY || (ly >= 1 && ly <= BY - 2));
      if (icol) {
        const bool inner = L::has_y ? (x >= 1 && y >= 1 && zc >= 1 && x <= nx - 2 && y <= ny - 2 && zc <= nz - 2)
                                    : (x >= 1 && zc >= 1 && x <= nx - 2 && zc <= nz - 2);
        if (inner) {
#pragma unroll
          for (int i = 0; i < QP; ++i) {
            const int ex = L::ex(i), ey = L::ey(i), ez = L::ez(i);
            if (ey == 0) continue;
            const T v = sGb[YS::slot(i) * PS + (ly - ey) * 32 + tx - ex];
            if (ez < 0) acc0 += v;
            else if (ez > 0) acc2 += v;
            else acc1 += v;
          }
        } else {
#pragma unroll
          for (int i = 0; i < QP; ++i) {
            const int ex = L::ex(i), ey = L::ey(i), ez = L::ez(i);
            if (ey == 0) continue;
            const int sx = x - ex, sy = y - ey, sz = zc - ez;
            const bool sin = sx >= 0 && sx < nx && sy >= 0 && sy < ny;
            if (sin) {
              const T v = sGb[YS::slot(i) * PS + (ly - ey) * 32 + tx - ex];
              if (ez < 0) acc0 += v;
              else if (ez > 0) acc2 += v;
              else acc1 += v;
            }
            if (!sin || sz < 0 || sz >= nz) acc1 += sGb[YS::slot(L::opp(i)) * PS + ly * 32 + tx];
          }
        }
        const int zw = zc - 1;
        // FP16/BF16: the gathered values are in stored units (scale is a power of two)
        auto mP = [&](T a) { return C::shifted ? rmul(a, iscale) : a; };
        if (zw >= it.z0 && zw < it.z1 && zw >= 0) phinew[((unsigned)zw * ny + y) * (unsigned)nx + x] = mP(acc0);
        if (zc == nz - 1 && zc >= it.z0 && zc < it.z1) phinew[((unsigned)zc * ny + y) * (unsigned)nx + x] = mP(acc1);
      }
      acc0 = acc1;
      acc1 = acc2;
      acc2 = 0;
    };
    gather_row(0, a0A, a1A, a2A);
    buf ^= 1;
  }
}

template <int QP, typename S, int BYC>
__global__ void __launch_bounds__(32 * MAX_BLOCK_ROWS, Lat<QP>::has_y ? LBPF_PHI_MIN_BLOCKS : LBPF_PHI2D_MIN_BLOCKS)
    k_phi(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items, int s6) {
  const WorkItem it = items[blockIdx.x];
  phi_tile<QP, S, BYC>(sims, it, s6);
}

// ---------------------------------------------------------------- U and theta
// One tile of the U/theta phase.  COH: phi^{n+1} is read through L2 (ld.global.cg), for
// launches in which other blocks of the same launch write it.  BYC as for phi_tile.
template <int QU, int QT, typename S, bool COH, int BYC>
__device__ __forceinline__ void uth_tile(const SimDev* __restrict__ sims, const WorkItem it, int s6) {
  using C = Codec<S>;
  using T = typename C::T;
  using LU = Lat<QU>;
  using LT = Lat<(QT > 0 ? QT : 7)>;
  using YU = YSlots<QU>;
  using YT = YSlots<(QT > 0 ? QT : 7)>;
  constexpr int NYU = NYOf<QU>::value;
  constexpr int NYT = NYOf<QT>::value;
  constexpr int QTA = QT > 0 ? QT : 1;
  const SimDev& sd = sims[it.sim];
  const int nx = sd.nx, ny = sd.ny, nz = sd.nz;
  const int BY = BYC > 0 ? BYC : (int)blockDim.y;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int tid = ty * 32 + tx, nthr = 32 * BY;
  const int x = it.x0 - 1 + tx;
  const int par = s6 & 1;
  const unsigned NS = (unsigned)sd.nsite;
  const unsigned plane = (unsigned)ny * (unsigned)nx;
  const S* __restrict__ hin = (const S*)sd.pop[par][1];
  S* __restrict__ hout = (S*)sd.pop[par ^ 1][1];
  const S* __restrict__ fin = (const S*)sd.pop[par][2];
  S* __restrict__ fout = (S*)sd.pop[par ^ 1][2];
  const T* __restrict__ phin = (const T*)sd.phi[s6 % 3];
  const T* __restrict__ phi1 = (const T*)sd.phi[(s6 + 1) % 3];
  const T* __restrict__ Un = (const T*)sd.U[par];
  T* __restrict__ Unew = (T*)sd.U[par ^ 1];
  const T* __restrict__ thn = (const T*)sd.th[s6 % 3];
  T* __restrict__ thnew = (T*)sd.th[(s6 + 1) % 3];
  const T* __restrict__ thm = (const T*)sd.th[(s6 + 2) % 3];  // theta^{n-1}: the FP16/BF16 shift of f

  constexpr bool HY = LU::has_y;  // false: 2D lattices, one-row blocks without y halo
  const int RW = 34, RS = HY ? RW * (BY + 2) : RW, PS = BY * 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* ring = reinterpret_cast<T*>(smem_raw);  // phi^{n+1} [4][BY+2][34]
  // FP16/BF16 with theta evolving: theta^{n-1} [4][BY+2][34], the shift of each stored f
  constexpr bool TSH = C::shifted && QT > 0;
  T* ringt = ring + 4 * RS;
  T* sH = ring + (TSH ? 8 : 4) * RS;         // [2][NYU + NYT][BY][32]
  constexpr int NYA = NYU + NYT;

  const Consts<T> P = consts_of<T>(sd);
  const T sh_h = P.shift_h, isc_h = P.inv_scale[1], sc_f = P.scale[2], isc_f = P.inv_scale[2];
  const bool at_on = sd.antitrapping != 0;

  const int zlo = max(it.z0 - 1, 0), zhi = min(it.z1, nz - 1);
  RingMap rm;
  rm.init(it.x0, it.y0, nx, ny, RW, RS, tid, nthr);
  {
    RingRegs<T> a;
    for (int z = zlo - 1; z <= zlo + 1; ++z) {
      a.template fetch<COH>(rm, phi1, z, nz, plane);
      a.store(rm, ring + slot4(z) * RS, tid, nthr);
      if (TSH) {
        a.fetch(rm, thm, z, nz, plane);
        a.store(rm, ringt + slot4(z) * RS, tid, nthr);
      }
    }
  }
  RingRegs<T> pf, pft;
  if (zlo + 2 <= zhi + 1) {
    pf.template fetch<COH>(rm, phi1, zlo + 2, nz, plane);
    if (TSH) pft.fetch(rm, thm, zlo + 2, nz, plane);
  }
  T u0A = 0, u1A = 0, u2A = 0, t0A = 0, t1A = 0, t2A = 0;
  int buf = 0;
  __syncthreads();

  for (int zc = zlo; zc <= zhi; ++zc) {
    T* sHb = sH + buf * NYA * PS;
    T* sFb = sHb + NYU * PS;
    const T* R0 = ring + slot4(zc) * RS;
    const T* Rp = ring + slot4(zc + 1) * RS;
    const T* Rm = ring + slot4(zc - 1) * RS;
    auto collide_row = [&](auto row_kind, T& u0, T& u1, T& u2, T& t0, T& t1, T& t2) {
      constexpr int KIND = decltype(row_kind)::value;  // 0 interior row, 1 top halo, 2 bottom halo
      auto row_needs = [](int ey) { return KIND == 0 || (KIND == 1 && ey == 1) || (KIND == 2 && ey == -1); };
      const int ly = ty;
      const int y = HY ? it.y0 - 1 + ly : it.y0 + ly;  // row 0 is a halo row except in one-row blocks
      const bool in_xy = x >= 0 && x < nx && y >= 0 && y < ny;
      const bool icol = in_xy && tx >= 1 && tx <= TILE_X && (!HY || (ly >= 1 && ly <= BY - 2));
      const int rc = HY ? (ly + 1) * RW + (tx + 1) : tx + 1;
      const unsigned site = ((unsigned)zc * (unsigned)ny + (unsigned)y) * (unsigned)nx + (unsigned)x;
      const bool inner = LU::has_y ? (x >= 1 && y >= 1 && zc >= 1 && x <= nx - 2 && y <= ny - 2 && zc <= nz - 2)
                                   : (x >= 1 && zc >= 1 && x <= nx - 2 && zc <= nz - 2);
      T hs[QU], fs[QTA];
#pragma unroll
      for (int i = 0; i < QU; ++i) hs[i] = T(0);
#pragma unroll
      for (int i = 0; i < QTA; ++i) fs[i] = T(0);
      if (in_xy) {
        const T U = ldro(Un + site);
        const T phn = ldro(phin + site);
        const T th = QT > 0 ? ldro(thn + site) : T(0);
        // pulled populations, all loads first; interior nodes need no wall checks
        if (inner) {
#pragma unroll
          for (int i = 0; i < QU; ++i) {
            const int ex = LU::ex(i), ey = LU::ey(i), ez = LU::ez(i);
            if (!row_needs(ey)) continue;
            hs[i] = C::raw(ldro(hin + ((unsigned)i * NS + site - (unsigned)(ez * (int)plane + ey * nx + ex))));
          }
#pragma unroll
          for (int i = 0; i < QT; ++i) {
            const int ex = LT::ex(i), ey = LT::ey(i), ez = LT::ez(i);
            if (!row_needs(ey)) continue;
            fs[i] = C::raw(ldro(fin + ((unsigned)i * NS + site - (unsigned)(ez * (int)plane + ey * nx + ex))));
            if (TSH)  // stored units with the source's shift: F + S w theta^{n-1}(src)
              fs[i] = rfma(rmul(sc_f, (T)LT::w(i)), (ringt + slot4(zc - ez) * RS)[rc - ey * RW - ex], fs[i]);
          }
        } else {
#pragma unroll
          for (int i = 0; i < QU; ++i) {
            const int ex = LU::ex(i), ey = LU::ey(i), ez = LU::ez(i);
            if (!row_needs(ey)) continue;
            const int sx = x - ex, sy = y - ey, sz = zc - ez;
            const bool inside = sx >= 0 && sx < nx && sy >= 0 && sy < ny && sz >= 0 && sz < nz;
            const unsigned src = inside ? site - (unsigned)(ez * (int)plane + ey * nx + ex) : site;
            const int ii = inside ? i : LU::opp(i);
            hs[i] = C::raw(ldro(hin + ((unsigned)ii * NS + src)));
          }
#pragma unroll
          for (int i = 0; i < QT; ++i) {
            const int ex = LT::ex(i), ey = LT::ey(i), ez = LT::ez(i);
            if (!row_needs(ey)) continue;
            const int sx = x - ex, sy = y - ey, sz = zc - ez;
            const bool inside = sx >= 0 && sx < nx && sy >= 0 && sy < ny && sz >= 0 && sz < nz;
            const unsigned src = inside ? site - (unsigned)(ez * (int)plane + ey * nx + ex) : site;
            const int ii = inside ? i : LT::opp(i);
            fs[i] = C::raw(ldro(fin + ((unsigned)ii * NS + src)));
            if (TSH)
              fs[i] = rfma(rmul(sc_f, (T)LT::w(i)), (ringt + slot4(inside ? sz : zc) * RS)[inside ? rc - ey * RW - ex : rc],
                          fs[i]);
          }
        }
        // phi^{n+1} at the node and its six neighbours (mirror ghosts)
        const T pc = R0[rc];
        const T pxp = R0[rc + 1], pxm = R0[rc - 1], pyp = HY ? R0[rc + RW] : pc, pym = HY ? R0[rc - RW] : pc, pzp = Rp[rc], pzm = Rm[rc];
        UthCoef<T> co;
        uth_coef<QU, QT, S>(P, at_on, U, th, phn, pc, pxp, pxm, pyp, pym, pzp, pzm, co);
        const bool store = icol && zc >= it.z0 && zc < it.z1;
        u_collide<QU>(co, hs, row_needs);
#pragma unroll
        for (int i = 0; i < QU; ++i) {
          const int ey = LU::ey(i);
          if (!row_needs(ey)) continue;
          const auto enc = C::pack(hs[i]);
          if (store) hout[(unsigned)i * NS + site] = enc;
          hs[i] = C::raw(enc);
          if (ey != 0) sHb[YU::slot(i) * PS + ly * 32 + tx] = hs[i];
        }
        if (QT > 0) {
#pragma unroll
          for (int i = 0; i < QT; ++i) {
            const int ey = LT::ey(i);
            if (!row_needs(ey)) continue;
            const auto enc = C::pack(rfma(fs[i], co.At, co.Kt[LT::cls(i)]));
            if (store) fout[(unsigned)i * NS + site] = enc;
            fs[i] = C::shifted ? radd(C::raw(enc), shift_of<LT>(sc_f, i, th)) : C::raw(enc);
            if (ey != 0) sFb[YT::slot(i) * PS + ly * 32 + tx] = fs[i];
          }
        }
      }
      if (KIND == 0) {
        // populations with e_y = 0: from this lane or the x-neighbour lane (all lanes shuffle)
        T hv[QU], fv[QTA];
  #pragma unroll
        for (int i = 0; i < QU; ++i) {
          const int ex = LU::ex(i), ey = LU::ey(i);
          hv[i] = hs[i];
          if (ey == 0 && ex > 0) hv[i] = __shfl_up_sync(0xffffffffu, hs[i], 1);
          if (ey == 0 && ex < 0) hv[i] = __shfl_down_sync(0xffffffffu, hs[i], 1);
        }
  #pragma unroll
        for (int i = 0; i < QT; ++i) {
          const int ex = LT::ex(i), ey = LT::ey(i);
          fv[i] = fs[i];
          if (ey == 0 && ex > 0) fv[i] = __shfl_up_sync(0xffffffffu, fs[i], 1);
          if (ey == 0 && ex < 0) fv[i] = __shfl_down_sync(0xffffffffu, fs[i], 1);
        }
        if (icol) {
          if (inner) {
  #pragma unroll
            for (int i = 0; i < QU; ++i) {
              const int ey = LU::ey(i), ez = LU::ez(i);
              if (ey != 0) continue;
              if (ez < 0) u0 += hv[i];
              else if (ez > 0) u2 += hv[i];
              else u1 += hv[i];
            }
  #pragma unroll
            for (int i = 0; i < QT; ++i) {
              const int ey = LT::ey(i), ez = LT::ez(i);
              if (ey != 0) continue;
              if (ez < 0) t0 += fv[i];
              else if (ez > 0) t2 += fv[i];
              else t1 += fv[i];
            }
          } else {
  #pragma unroll
            for (int i = 0; i < QU; ++i) {
              const int ex = LU::ex(i), ey = LU::ey(i), ez = LU::ez(i);
              if (!row_needs(ey)) continue;
              if (ey != 0) continue;
              const int sx = x - ex, sz = zc - ez;
              const bool sin = sx >= 0 && sx < nx;
              if (sin) {
                if (ez < 0) u0 += hv[i];
                else if (ez > 0) u2 += hv[i];
                else u1 += hv[i];
              }
              if (!sin || sz < 0 || sz >= nz) u1 += hs[LU::opp(i)];
            }
  #pragma unroll
            for (int i = 0; i < QT; ++i) {
              const int ex = LT::ex(i), ey = LT::ey(i), ez = LT::ez(i);
              if (!row_needs(ey)) continue;
              if (ey != 0) continue;
              const int sx = x - ex, sz = zc - ez;
              const bool sin = sx >= 0 && sx < nx;
              if (sin) {
                if (ez < 0) t0 += fv[i];
                else if (ez > 0) t2 += fv[i];
                else t1 += fv[i];
              }
              if (!sin || sz < 0 || sz >= nz) t1 += fs[LT::opp(i)];
            }
          }
        }
      }
    };
    // rows 0 and BY-1 are halo rows: they only feed the e_y = +1 / -1 populations to the block
    if (!HY) collide_row(std::integral_constant<int, 0>{}, u0A, u1A, u2A, t0A, t1A, t2A);
    else if (ty == 0) collide_row(std::integral_constant<int, 1>{}, u0A, u1A, u2A, t0A, t1A, t2A);
    else if (ty == BY - 1) collide_row(std::integral_constant<int, 2>{}, u0A, u1A, u2A, t0A, t1A, t2A);
    else collide_row(std::integral_constant<int, 0>{}, u0A, u1A, u2A, t0A, t1A, t2A);
    if (zc + 2 <= zhi + 1) {
      pf.store(rm, ring + slot4(zc + 2) * RS, tid, nthr);
      if (TSH) pft.store(rm, ringt + slot4(zc + 2) * RS, tid, nthr);
    }
    if (zc + 3 <= zhi + 1) {
      pf.template fetch<COH>(rm, phi1, zc + 3, nz, plane);
      if (TSH) pft.fetch(rm, thm, zc + 3, nz, plane);
    }
    __syncthreads();
    auto gather_row = [&](const int r, T& u0, T& u1, T& u2, T& t0, T& t1, T& t2) {
      const int ly = ty;
      const int y = HY ? it.y0 - 1 + ly : it.y0 + ly;  // row 0 is a halo row except in one-row blocks
      const bool icol = x >= 0 && x < nx && y >= 0 && y < ny && tx >= 1 && tx <= TILE_X && (!HY || (ly >= 1 && ly <= BY - 2));
      if (icol) {
        const bool inner = LU::has_y ? (x >= 1 && y >= 1 && zc >= 1 && x <= nx - 2 && y <= ny - 2 && zc <= nz - 2)
                                     : (x >= 1 && zc >= 1 && x <= nx - 2 && zc <= nz - 2);
        if (inner) {
#pragma unroll
          for (int i = 0; i < QU; ++i) {
            const int ex = LU::ex(i), ey = LU::ey(i), ez = LU::ez(i);
            if (ey == 0) continue;
            const T v = sHb[YU::slot(i) * PS + (ly - ey) * 32 + tx - ex];
            if (ez < 0) u0 += v;
            else if (ez > 0) u2 += v;
            else u1 += v;
          }
#pragma unroll
          for (int i = 0; i < QT; ++i) {
            const int ex = LT::ex(i), ey = LT::ey(i), ez = LT::ez(i);
            if (ey == 0) continue;
            const T v = sFb[YT::slot(i) * PS + (ly - ey) * 32 + tx - ex];
            if (ez < 0) t0 += v;
            else if (ez > 0) t2 += v;
            else t1 += v;
          }
        } else {
#pragma unroll
          for (int i = 0; i < QU; ++i) {
            const int ex = LU::ex(i), ey = LU::ey(i), ez = LU::ez(i);
            if (ey == 0) continue;
            const int sx = x - ex, sy = y - ey, sz = zc - ez;
            const bool sin = sx >= 0 && sx < nx && sy >= 0 && sy < ny;
            if (sin) {
              const T v = sHb[YU::slot(i) * PS + (ly - ey) * 32 + tx - ex];
              if (ez < 0) u0 += v;
              else if (ez > 0) u2 += v;
              else u1 += v;
            }
            if (!sin || sz < 0 || sz >= nz) u1 += sHb[YU::slot(LU::opp(i)) * PS + ly * 32 + tx];
          }
#pragma unroll
          for (int i = 0; i < QT; ++i) {
            const int ex = LT::ex(i), ey = LT::ey(i), ez = LT::ez(i);
            if (ey == 0) continue;
            const int sx = x - ex, sy = y - ey, sz = zc - ez;
            const bool sin = sx >= 0 && sx < nx && sy >= 0 && sy < ny;
            if (sin) {
              const T v = sFb[YT::slot(i) * PS + (ly - ey) * 32 + tx - ex];
              if (ez < 0) t0 += v;
              else if (ez > 0) t2 += v;
              else t1 += v;
            }
            if (!sin || sz < 0 || sz >= nz) t1 += sFb[YT::slot(LT::opp(i)) * PS + ly * 32 + tx];
          }
        }
        const int zw = zc - 1;
        // FP16/BF16: the gathered sums are in stored units; the shifts w_i U0 (w_i theta0)
        // of the populations arriving at a node add up to U0 (theta0)
        auto mU = [&](T a) { return C::shifted ? rfma(a, isc_h, sh_h) : a; };
        auto mT = [&](T a) { return C::shifted ? rmul(a, isc_f) : a; };
        if (zw >= it.z0 && zw < it.z1 && zw >= 0) {
          const unsigned sw = ((unsigned)zw * ny + y) * (unsigned)nx + x;
          Unew[sw] = mU(u0);
          if (QT > 0) thnew[sw] = mT(t0);
        }
        if (zc == nz - 1 && zc >= it.z0 && zc < it.z1) {
          const unsigned sw = ((unsigned)zc * ny + y) * (unsigned)nx + x;
          Unew[sw] = mU(u1);
          if (QT > 0) thnew[sw] = mT(t1);
        }
      }
      u0 = u1;
      u1 = u2;
      u2 = 0;
      t0 = t1;
      t1 = t2;
      t2 = 0;
    };
    gather_row(0, u0A, u1A, u2A, t0A, t1A, t2A);
    buf ^= 1;
  }
}

template <int QU, int QT, typename S, int BYC>
__global__ void __launch_bounds__(32 * MAX_BLOCK_ROWS, Lat<QU>::has_y ? LBPF_UTH_MIN_BLOCKS : LBPF_UTH2D_MIN_BLOCKS)
    k_uth(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items, int s6) {
  const WorkItem it = items[blockIdx.x];
  uth_tile<QU, QT, S, false, BYC>(sims, it, s6);
}

// ---------------------------------------------------------------- one launch per step
// Both phases of a step in one persistent launch, so that tiles of the phase-field phase
// (bound by instruction issue) run beside tiles of the U/theta phase (bound by memory
// latency) on the same SMs.  Blocks draw tickets in order from a counter; ticket t names
// the phase-field tile or the U/theta tile of one work item.  The U/theta tile of an item
// reads phi^{n+1} over its ring (two nodes around its columns and rows, two planes around
// its z-chunk), so it waits for the done flags of the phase-field tiles that write that
// region; the host orders the tickets so that those tiles always come earlier, and a
// block draws a ticket only while it runs, so no wait depends on a tile that has not
// started.  The U/theta tiles read nothing else that the launch writes (the phase-field
// tiles write g at the other buffer parity and the new phi level; the U/theta tiles write
// h, f, U and theta at levels the phase-field tiles do not read).  The waits are bounded
// all the same: after about a second a wait gives up, sets *err (host-visible) and the tile
// goes ahead; the host then reports the step as failed.
struct StepSched {
  const int* order;    // ticket -> j >= 0: phase-field tile of item j; ~j: U/theta tile of item j
  const int* dep_off;  // the U/theta tile of item j waits for the phase-field tiles dep[dep_off[j] .. dep_off[j+1])
  const int* dep;
  unsigned* ctl;       // ctl[0]: next ticket; ctl[1 + j]: phase-field tile of item j done (zeroed before each launch)
  int* err;            // set to 1 when a wait gave up
  int ntickets;
  unsigned polls;      // bound of each wait (rounds of about 0.25 us)
};


__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_gpu(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// One full warp waits until done[dep[k]] != 0 for every k < n, each lane polling a share
// of the flags; false when `polls` rounds passed without that.
__device__ __forceinline__ bool wait_done(const unsigned* done, const int* dep, int n, unsigned polls) {
  const int lane = threadIdx.x & 31;
  for (unsigned r = 0; r < polls; ++r) {
    bool ok = true;
    for (int k = lane; k < n; k += 32) ok = ok && ld_acquire_gpu(done + __ldg(dep + k)) != 0u;
    if (__all_sync(0xffffffffu, ok)) return true;
    __nanosleep(200);
  }
  return false;
}

template <int QP, int QU, int QT, typename S>
__global__ void __launch_bounds__(32 * MAX_BLOCK_ROWS, Lat<QU>::has_y ? LBPF_UTH_MIN_BLOCKS : LBPF_UTH2D_MIN_BLOCKS) k_step(const SimDev* __restrict__ sims, const WorkItem* __restrict__ items,
                                                const StepSched sc, int s6) {
  __shared__ int s_ticket;
  const bool lead = threadIdx.x == 0 && threadIdx.y == 0;
  for (;;) {
    if (lead) s_ticket = (int)atomicAdd(sc.ctl, 1u);
    __syncthreads();
    const int t = s_ticket;
    if (t >= sc.ntickets) return;  // the same for every thread of the block
    const int w = __ldg(sc.order + t);
    if (w >= 0) {
      phi_tile<QP, S, 0>(sims, items[w], s6);
      __threadfence();  // this thread's phi^{n+1} stores are visible before the flag
      __syncthreads();
      if (lead) st_release_gpu(sc.ctl + 1 + w, 1u);
    } else {
      const int j = ~w;
      if (threadIdx.y == 0) {
        const int b = __ldg(sc.dep_off + j), n = __ldg(sc.dep_off + j + 1) - b;
        if (!wait_done(sc.ctl + 1, sc.dep + b, n, sc.polls) && threadIdx.x == 0) atomicExch(sc.err, 1);
      }
      __syncthreads();
      uth_tile<QU, QT, S, true, 0>(sims, items[j], s6);
      __syncthreads();  // the next tile reuses the shared memory
    }
  }
}

}  // namespace lbpf
