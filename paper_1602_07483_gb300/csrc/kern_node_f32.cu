// kern_node_f32.cu -- node-wise collision kernels with float storage (a translation unit of
// their own so that they compile in parallel).
#include "lbpf_table_impl.cuh"

namespace lbpf {
void add_node_kernels_f32(KernelTable& t) { fill_node_kernels<float, 1>(t); }
}  // namespace lbpf
