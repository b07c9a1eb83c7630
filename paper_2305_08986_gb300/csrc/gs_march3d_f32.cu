// 3D march kernel (gs_march3d.cuh) in float.
#include "gs_march3d_launch.cuh"

namespace gs {
template <>
cudaError_t launch_march3d<float>(int mode, int ops, const TileArgs<float>& a, cudaStream_t st) {
  return march3::dispatch<float>(mode, ops, a, st);
}
}  // namespace gs
