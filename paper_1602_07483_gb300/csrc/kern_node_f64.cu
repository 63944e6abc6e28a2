// kern_node_f64.cu -- node-wise collision kernels with double storage (a translation unit of
// their own so that they compile in parallel).
#include "lbpf_table_impl.cuh"

namespace lbpf {
void add_node_kernels_f64(KernelTable& t) { fill_node_kernels<double, 1>(t); }
}  // namespace lbpf
