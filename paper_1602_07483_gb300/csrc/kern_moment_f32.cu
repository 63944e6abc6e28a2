// kern_moment_f32.cu -- node-wise moment kernels with float storage (a translation unit of
// their own so that they compile in parallel).
#include "lbpf_table_impl.cuh"

namespace lbpf {
void add_moment_kernels_f32(KernelTable& t) { fill_moment_kernels<float, 1>(t); }
}  // namespace lbpf
