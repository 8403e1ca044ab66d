// FP32 instantiation of the tile kernels (tile_impl.cuh).
#include "tile_impl.cuh"

namespace emfuse {

template <>
int launch_tile<float>(const TileArgs<float>& a, bool zero_init, bool up, cudaStream_t st, double bytes) {
    return fused_detail::launch_tile_impl<float>(a, zero_init, up, st, bytes);
}
template <>
void tile_extent<float>(int halo, int& hx, int& hy, int& out_x, int& out_y) {
    fused_detail::tile_extent_impl<float>(halo, hx, hy, out_x, out_y);
}

}  // namespace emfuse
