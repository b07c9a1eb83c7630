// 2D cell-tile kernel (gs_tile2d.cuh), tiles of 32 x 17 evaluated cells.
#include "gs_tile2d.cuh"

namespace gs {

template <typename T>
cudaError_t launch_tile2d_e17(int mode, int ops, const TileArgs<T>& a, cudaStream_t st) {
  return tile2d::launch_shape<T, tile2d::Shape2<32, 17>>(mode, ops, a, st);
}
template cudaError_t launch_tile2d_e17<float>(int, int, const TileArgs<float>&, cudaStream_t);
template cudaError_t launch_tile2d_e17<double>(int, int, const TileArgs<double>&, cudaStream_t);

}  // namespace gs
