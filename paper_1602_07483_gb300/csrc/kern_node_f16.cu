// kern_node_f16.cu -- node-wise collision kernels with __half storage (a translation unit of
// their own so that they compile in parallel).
#include "lbpf_table_impl.cuh"

namespace lbpf {
void add_node_kernels_f16(KernelTable& t) { fill_node_kernels<__half, 1>(t); }
}  // namespace lbpf
