// kern_moment_bf16.cu -- node-wise moment kernels with __nv_bfloat16 storage (a translation unit of
// their own so that they compile in parallel).
#include "lbpf_table_impl.cuh"

namespace lbpf {
void add_moment_kernels_bf16(KernelTable& t) { fill_moment_kernels<__nv_bfloat16, 1>(t); }
}  // namespace lbpf
