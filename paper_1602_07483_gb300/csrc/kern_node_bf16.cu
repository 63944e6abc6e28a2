// kern_node_bf16.cu -- node-wise collision kernels with __nv_bfloat16 storage (a translation unit of
// their own so that they compile in parallel).
#include "lbpf_table_impl.cuh"

namespace lbpf {
void add_node_kernels_bf16(KernelTable& t) { fill_node_kernels<__nv_bfloat16, 1>(t); }
}  // namespace lbpf
