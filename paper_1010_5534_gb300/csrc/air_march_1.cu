// air_march_1.cu -- the march with 1 band per thread.
#include "air_march_kernel.cuh"

namespace air {
template cudaError_t march_general<1>(const MarchLaunch &);
}  // namespace air
