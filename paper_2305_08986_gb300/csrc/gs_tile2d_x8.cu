// 2D cell-tile kernel (gs_tile2d.cuh), tiles of 8 x 8 evaluated cells in CTAs of 64 threads.
//
// For meshes that fill few 32-wide tiles.  A CTA of 32 x 16 FP64 cells takes the FP64 pipe of its SM
// (2 operations per clock) some 20 us whatever the mesh, while most SMs idle; 64 cells take 3 us.  The
// halo costs 31 % (64 evaluated cells for 49 owned) against 10 %, so the larger tiles stay where they
// fill the GPU.  FP64 V-cycle of the 1280 x 224 extension mesh: 2079 -> 1957 us (32 x 8 tiles took 20 to
// 38 us per step on its 80 x 14 to 320 x 56 levels); 16 x 16 solve to 1e-11: 4 % less.
#include "gs_tile2d.cuh"

namespace gs {

template <typename T>
cudaError_t launch_tile2d_x8(int mode, int ops, const TileArgs<T>& a, cudaStream_t st) {
  return tile2d::launch_shape<T, tile2d::Shape2<8, 8>>(mode, ops, a, st);
}
template cudaError_t launch_tile2d_x8<float>(int, int, const TileArgs<float>&, cudaStream_t);
template cudaError_t launch_tile2d_x8<double>(int, int, const TileArgs<double>&, cudaStream_t);

}  // namespace gs
