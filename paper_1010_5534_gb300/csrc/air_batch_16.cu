// air_batch_16.cu -- the batched kernel with 16 bands per thread.
#include "air_batch_kernel.cuh"

namespace air {
template bool batch_fns<16>(const GridView &, int, bool, int, BatchOccFn *, BatchLaunchFn *, size_t *, int *);
}  // namespace air
