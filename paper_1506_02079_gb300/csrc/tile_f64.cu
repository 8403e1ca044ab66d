// FP64 instantiation of the tile kernels (tile_impl.cuh).
#include "tile_impl.cuh"

namespace emfuse {

template <>
int launch_tile<double>(const TileArgs<double>& a, bool zero_init, bool up, cudaStream_t st, double bytes) {
    return fused_detail::launch_tile_impl<double>(a, zero_init, up, st, bytes);
}
template <>
void tile_extent<double>(int halo, int& hx, int& hy, int& out_x, int& out_y) {
    fused_detail::tile_extent_impl<double>(halo, hx, hy, out_x, out_y);
}

}  // namespace emfuse
