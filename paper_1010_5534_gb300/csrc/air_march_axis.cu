// air_march_axis.cu -- the one-band march of rays along a grid axis.
#include "air_march_kernel.cuh"

namespace air {
template cudaError_t march_axis_one<0>(const MarchLaunch &);
template cudaError_t march_axis_one<1>(const MarchLaunch &);
template cudaError_t march_axis_one<2>(const MarchLaunch &);
}  // namespace air
