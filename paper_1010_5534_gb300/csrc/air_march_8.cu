// air_march_8.cu -- the march with 8 bands per thread.
#include "air_march_kernel.cuh"

namespace air {
template cudaError_t march_general<8>(const MarchLaunch &);
}  // namespace air
