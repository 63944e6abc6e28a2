// kern_pair_f16.cu -- node-wise kernels of two nodes per thread with __half storage (a translation
// unit of their own so that they compile in parallel).
#include "lbpf_table_impl.cuh"

namespace lbpf {
void add_pair_kernels_f16(KernelTable& t) {
  fill_node_kernels<__half, 2>(t);
  fill_moment_kernels<__half, 2>(t);
}
}  // namespace lbpf
