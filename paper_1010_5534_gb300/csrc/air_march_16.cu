// air_march_16.cu -- the march with 16 bands per thread.
#include "air_march_kernel.cuh"

namespace air {
template cudaError_t march_general<16>(const MarchLaunch &);
}  // namespace air
