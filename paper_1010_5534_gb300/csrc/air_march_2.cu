// air_march_2.cu -- the march with 2 bands per thread.
#include "air_march_kernel.cuh"

namespace air {
template cudaError_t march_general<2>(const MarchLaunch &);
}  // namespace air
