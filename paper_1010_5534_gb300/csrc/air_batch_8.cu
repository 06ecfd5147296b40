// air_batch_8.cu -- the batched kernel with 8 bands per thread.
#include "air_batch_kernel.cuh"

namespace air {
template bool batch_fns<8>(const GridView &, int, bool, int, BatchOccFn *, BatchLaunchFn *, size_t *, int *);
}  // namespace air
