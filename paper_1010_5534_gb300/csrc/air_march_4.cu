// air_march_4.cu -- the march with 4 bands per thread.
#include "air_march_kernel.cuh"

namespace air {
template cudaError_t march_general<4>(const MarchLaunch &);
}  // namespace air
