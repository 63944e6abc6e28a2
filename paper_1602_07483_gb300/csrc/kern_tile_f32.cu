// kern_tile_f32.cu -- the 3D tiled step kernels with float storage for blocks of any height.
#include "lbpf_table_impl.cuh"

namespace lbpf {
void add_tile_kernels_f32(KernelTable& t) { fill_tile_kernels_3d<float, 0>(t); }
}  // namespace lbpf
