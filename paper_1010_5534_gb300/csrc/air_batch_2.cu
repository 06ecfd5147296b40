// air_batch_2.cu -- the batched kernel with 2 bands per thread.
#include "air_batch_kernel.cuh"

namespace air {
template bool batch_fns<2>(const GridView &, int, bool, int, BatchOccFn *, BatchLaunchFn *, size_t *, int *);
}  // namespace air
