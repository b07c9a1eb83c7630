// 3D march kernel (gs_march3d.cuh) in double.
#include "gs_march3d_launch.cuh"

namespace gs {
template <>
cudaError_t launch_march3d<double>(int mode, int ops, const TileArgs<double>& a, cudaStream_t st) {
  return march3::dispatch<double>(mode, ops, a, st);
}
}  // namespace gs
