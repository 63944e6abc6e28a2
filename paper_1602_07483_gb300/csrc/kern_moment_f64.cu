// kern_moment_f64.cu -- node-wise moment kernels with double storage (a translation unit of
// their own so that they compile in parallel).
#include "lbpf_table_impl.cuh"

namespace lbpf {
void add_moment_kernels_f64(KernelTable& t) { fill_moment_kernels<double, 1>(t); }
}  // namespace lbpf
