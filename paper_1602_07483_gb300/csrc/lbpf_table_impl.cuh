// lbpf_table_impl.cuh -- builds the KernelTable of one storage type.  Included by
// one translation unit per storage type so the template instantiations compile
// in parallel.
#pragma once

#include "lbpf_aux.cuh"
#include "lbpf_nodepair.cuh"
#include "lbpf_nodewise.cuh"
#include "lbpf_plane.cuh"
#include "lbpf_table.h"

namespace lbpf {

constexpr int AUX_THREADS = 256;

inline int aux_blocks(long long n) {
  long long b = (n + AUX_THREADS - 1) / AUX_THREADS;
  if (b > 152LL * 32) b = 152LL * 32;
  return (int)(b < 1 ? 1 : b);
}

// Launch that may overlap the end of the kernel before it in the stream (pdl_wait): node-wise kernels.
inline cudaError_t launch_pdl(void (*fn)(const SimDev*, const WorkItem*, int), dim3 g, dim3 b, size_t smem,
                              cudaStream_t st, const SimDev* sims, const WorkItem* items, int s6) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = g;
  cfg.blockDim = b;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, sims, items, s6);
}

template <int QP, typename S, int BYC>
cudaError_t launch_phi(dim3 g, dim3 b, size_t smem, cudaStream_t st, const SimDev* sims, const WorkItem* items,
                       int s6) {
  k_phi<QP, S, BYC><<<g, b, smem, st>>>(sims, items, s6);
  return cudaGetLastError();
}

template <int QU, int QT, typename S, int BYC>
cudaError_t launch_uth(dim3 g, dim3 b, size_t smem, cudaStream_t st, const SimDev* sims, const WorkItem* items,
                       int s6) {
  k_uth<QU, QT, S, BYC><<<g, b, smem, st>>>(sims, items, s6);
  return cudaGetLastError();
}

template <int QP, typename S>
cudaError_t launch_phi_plane(dim3 g, dim3 b, size_t smem, cudaStream_t st, const SimDev* sims, const WorkItem* items,
                             int s6) {
  k_phi_plane<QP, S><<<g, b, smem, st>>>(sims, items, s6);
  return cudaGetLastError();
}
template <int QU, int QT, typename S>
cudaError_t launch_uth_plane(dim3 g, dim3 b, size_t smem, cudaStream_t st, const SimDev* sims, const WorkItem* items,
                             int s6) {
  k_uth_plane<QU, QT, S><<<g, b, smem, st>>>(sims, items, s6);
  return cudaGetLastError();
}

// V nodes per thread (1 or 2; FP64 has no pairs)
template <int QP, typename S, int V>
cudaError_t launch_phi_node(dim3 g, dim3 b, size_t smem, cudaStream_t st, const SimDev* sims, const WorkItem* items,
                            int s6) {
  if constexpr (V == 2) return launch_pdl(k_phi_pair<QP, S>, g, b, smem, st, sims, items, s6);
  else return launch_pdl(k_phi_node<QP, S>, g, b, smem, st, sims, items, s6);
}
template <int QP, typename S, int V>
cudaError_t launch_phi_moment(dim3 g, dim3 b, size_t smem, cudaStream_t st, const SimDev* sims, const WorkItem* items,
                              int s6) {
  if constexpr (V == 2) return launch_pdl(k_phi_moment2<QP, S>, g, b, smem, st, sims, items, s6);
  else return launch_pdl(k_phi_moment<QP, S>, g, b, smem, st, sims, items, s6);
}
template <int QU, int QT, typename S, int V>
cudaError_t launch_uth_node(dim3 g, dim3 b, size_t smem, cudaStream_t st, const SimDev* sims, const WorkItem* items,
                            int s6) {
  if constexpr (V == 2) return launch_pdl(k_uth_pair<QU, QT, S>, g, b, smem, st, sims, items, s6);
  else return launch_pdl(k_uth_node<QU, QT, S>, g, b, smem, st, sims, items, s6);
}
template <int QU, int QT, typename S, int V>
cudaError_t launch_uth_moment(dim3 g, dim3 b, size_t smem, cudaStream_t st, const SimDev* sims, const WorkItem* items,
                              int s6) {
  if constexpr (V == 2) return launch_pdl(k_uth_moment2<QU, QT, S>, g, b, smem, st, sims, items, s6);
  else return launch_pdl(k_uth_moment<QU, QT, S>, g, b, smem, st, sims, items, s6);
}

// The U and theta pairings of one dimension.
#define LBPF_UTH_PAIRS(M)                     \
  M(7, 0) M(7, 7) M(7, 15) M(7, 19)           \
  M(15, 0) M(15, 7) M(15, 15) M(15, 19)       \
  M(19, 0) M(19, 7) M(19, 15) M(19, 19)       \
  M(5, 0) M(5, 5) M(5, 9) M(9, 0) M(9, 5) M(9, 9)

// The node-wise step's kernels with V nodes per thread, in translation units of their own.
template <typename S, int V>
void fill_node_kernels(KernelTable& t) {
#define LBPF_N(q) t.phi_node[lattice_slot(q)][V - 1] = launch_phi_node<q, S, V>;
  LBPF_N(7) LBPF_N(15) LBPF_N(19) LBPF_N(5) LBPF_N(9)
#undef LBPF_N
#define LBPF_N(qa, qb) t.uth_node[lattice_slot(qa)][lattice_slot(qb)][V - 1] = launch_uth_node<qa, qb, S, V>;
  LBPF_UTH_PAIRS(LBPF_N)
#undef LBPF_N
}
template <typename S>
void fill_plane_kernels(KernelTable& t) {
  t.phi_plane[lattice_slot(5)] = launch_phi_plane<5, S>;
  t.phi_plane[lattice_slot(9)] = launch_phi_plane<9, S>;
#define LBPF_N(qa, qb) t.uth_plane[lattice_slot(qa)][lattice_slot(qb)] = launch_uth_plane<qa, qb, S>;
  LBPF_N(5, 0) LBPF_N(5, 5) LBPF_N(5, 9) LBPF_N(9, 0) LBPF_N(9, 5) LBPF_N(9, 9)
#undef LBPF_N
}
template <typename S, int V>
void fill_moment_kernels(KernelTable& t) {
#define LBPF_N(q) t.phi_moment[lattice_slot(q)][V - 1] = launch_phi_moment<q, S, V>;
  LBPF_N(7) LBPF_N(15) LBPF_N(19) LBPF_N(5) LBPF_N(9)
#undef LBPF_N
#define LBPF_N(qa, qb) t.uth_moment[lattice_slot(qa)][lattice_slot(qb)][V - 1] = launch_uth_moment<qa, qb, S, V>;
  LBPF_UTH_PAIRS(LBPF_N)
#undef LBPF_N
}

template <int QP, int QU, int QT, typename S>
cudaError_t launch_step_one(dim3 g, dim3 b, size_t smem, cudaStream_t st, const SimDev* sims, const WorkItem* items,
                            const StepSched& sc, int s6) {
  k_step<QP, QU, QT, S><<<g, b, smem, st>>>(sims, items, sc, s6);
  return cudaGetLastError();
}

// The lattice triples with a one-launch step kernel: the paper's 3D benchmarks (D3Q19 for
// phi and U with theta frozen, on D3Q7 or on D3Q19) and its 2D set (D2Q9, D2Q5, D2Q5).
template <typename S>
void fill_step_kernels(KernelTable& t) {
#define LBPF_STEP(qa, qb, qc)                                                                     \
  t.step[lattice_slot(qa)][lattice_slot(qb)][lattice_slot(qc)] = launch_step_one<qa, qb, qc, S>; \
  t.step_fn[lattice_slot(qa)][lattice_slot(qb)][lattice_slot(qc)] = (const void*)k_step<qa, qb, qc, S>;
  LBPF_STEP(19, 19, 0) LBPF_STEP(19, 19, 7) LBPF_STEP(19, 19, 19) LBPF_STEP(9, 5, 5)
#undef LBPF_STEP
}

template <typename S>
struct AuxImpl {
  using T = typename Codec<S>::T;
  static cudaError_t init_scalar(cudaStream_t st, int nx, int ny, int nz, const double* cen, const double* rad,
                                 int nseed, double c, void* out) {
    const long long n = (long long)nx * ny * nz;
    k_init_scalar<T><<<aux_blocks(n), AUX_THREADS, 0, st>>>(nx, ny, nz, cen, rad, nseed, c, (T*)out);
    return cudaGetLastError();
  }
  static cudaError_t init_pop(cudaStream_t st, const SimDev& sd, const LatRT& Lp, const LatRT& Lu, const LatRT& Lt,
                              const void* phi0, double U0, double theta0) {
    k_init_pop<S><<<aux_blocks(sd.nsite), AUX_THREADS, 0, st>>>(sd, Lp, Lu, Lt, (const T*)phi0, U0, theta0);
    return cudaGetLastError();
  }
  static cudaError_t pack(cudaStream_t st, const SimDev& sd, int field, int par, const LatRT& L, int i,
                          const double* gi, const double* gj, const void* prev) {
    k_pack<S><<<aux_blocks(sd.nsite), AUX_THREADS, 0, st>>>(sd, field, par, L, i, gi, gj, (const T*)prev);
    return cudaGetLastError();
  }
  static cudaError_t unpack(cudaStream_t st, const SimDev& sd, int field, int par, const LatRT& L, int i, double* gi,
                            double* gj, const void* prev) {
    k_unpack<S><<<aux_blocks(sd.nsite), AUX_THREADS, 0, st>>>(sd, field, par, L, i, gi, gj, (const T*)prev);
    return cudaGetLastError();
  }
  static cudaError_t to_double(cudaStream_t st, double* out, const void* in, long long n) {
    k_to_double<T><<<aux_blocks(n), AUX_THREADS, 0, st>>>(out, (const T*)in, n);
    return cudaGetLastError();
  }
  static cudaError_t from_double(cudaStream_t st, void* out, const double* in, long long n) {
    k_from_double<T><<<aux_blocks(n), AUX_THREADS, 0, st>>>((T*)out, in, n);
    return cudaGetLastError();
  }
  static cudaError_t sums(cudaStream_t st, const void* phi, const void* U, const void* th, double theta0, double k,
                          long long n, double* part, int nblk) {
    k_sums<T><<<nblk, 256, 0, st>>>((const T*)phi, (const T*)U, (const T*)th, theta0, k, n, part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_sums_final<<<1, 128, 0, st>>>(part, nblk, part + 4 * nblk, k, n, th == nullptr, theta0);
    return cudaGetLastError();
  }
  static cudaError_t tip(cudaStream_t st, const void* phi, int nx, int ny, int nz, int axis, int cx, int cy, int cz,
                         double* out) {
    k_tip<T><<<1, dim3(32, 17), 0, st>>>((const T*)phi, nx, ny, nz, axis, cx, cy, cz, out);
    return cudaGetLastError();
  }
};

// The tiled step's one-row kernels of the 2D lattices (FP32, FP16, BF16; FP64 always steps
// node-wise).
template <typename S>
void fill_tile_kernels_2d(KernelTable& t) {
#define LBPF_PHI2(q)                                                                       \
  t.phi[lattice_slot(q)][0] = t.phi[lattice_slot(q)][1] = launch_phi<q, S, 1>;              \
  t.phi_fn[lattice_slot(q)][0] = t.phi_fn[lattice_slot(q)][1] = (const void*)k_phi<q, S, 1>;
  LBPF_PHI2(5) LBPF_PHI2(9)
#undef LBPF_PHI2
#define LBPF_UTH2(qa, qb)                                                                              \
  t.uth[lattice_slot(qa)][lattice_slot(qb)][0] = t.uth[lattice_slot(qa)][lattice_slot(qb)][1] =         \
      launch_uth<qa, qb, S, 1>;                                                                        \
  t.uth_fn[lattice_slot(qa)][lattice_slot(qb)][0] = t.uth_fn[lattice_slot(qa)][lattice_slot(qb)][1] =   \
      (const void*)k_uth<qa, qb, S, 1>;
  LBPF_UTH2(5, 0) LBPF_UTH2(5, 5) LBPF_UTH2(5, 9)
  LBPF_UTH2(9, 0) LBPF_UTH2(9, 5) LBPF_UTH2(9, 9)
#undef LBPF_UTH2
}

// The tiled step's 3D kernels (FP32), block height compiled in (BYC rows) or any (BYC = 0): U and theta of
// 30 populations and more (with fewer the step is node-wise at every size).
template <typename S, int BYC>
void fill_tile_kernels_3d(KernelTable& t) {
  constexpr int v = BYC > 0 ? 1 : 0;
#define LBPF_PHI3(q)                                            \
  t.phi[lattice_slot(q)][v] = launch_phi<q, S, BYC>;             \
  t.phi_fn[lattice_slot(q)][v] = (const void*)k_phi<q, S, BYC>;
  LBPF_PHI3(7) LBPF_PHI3(15) LBPF_PHI3(19)
#undef LBPF_PHI3
#define LBPF_UTH3(qa, qb)                                                              \
  t.uth[lattice_slot(qa)][lattice_slot(qb)][v] = launch_uth<qa, qb, S, BYC>;            \
  t.uth_fn[lattice_slot(qa)][lattice_slot(qb)][v] = (const void*)k_uth<qa, qb, S, BYC>;
  LBPF_UTH3(15, 15) LBPF_UTH3(15, 19) LBPF_UTH3(19, 15) LBPF_UTH3(19, 19)
#undef LBPF_UTH3
}

template <typename S>
KernelTable build_table() {
  KernelTable t{};
  t.sbytes = (int)sizeof(S);
  t.tbytes = (int)sizeof(typename Codec<S>::T);
  t.shifted = Codec<S>::shifted;
  if constexpr (sizeof(S) < 8) {
    fill_tile_kernels_2d<S>(t);
    fill_plane_kernels<S>(t);
  }
  t.init_scalar = AuxImpl<S>::init_scalar;
  t.init_pop = AuxImpl<S>::init_pop;
  t.pack = AuxImpl<S>::pack;
  t.unpack = AuxImpl<S>::unpack;
  t.to_double = AuxImpl<S>::to_double;
  t.from_double = AuxImpl<S>::from_double;
  t.sums = AuxImpl<S>::sums;
  t.tip = AuxImpl<S>::tip;
  return t;
}

}  // namespace lbpf
