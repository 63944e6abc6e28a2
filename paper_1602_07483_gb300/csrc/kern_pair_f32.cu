// kern_pair_f32.cu -- node-wise kernels of two nodes per thread with float storage (a translation
// unit of their own so that they compile in parallel).
#include "lbpf_table_impl.cuh"

namespace lbpf {
void add_pair_kernels_f32(KernelTable& t) {
  fill_node_kernels<float, 2>(t);
  fill_moment_kernels<float, 2>(t);
}
}  // namespace lbpf
