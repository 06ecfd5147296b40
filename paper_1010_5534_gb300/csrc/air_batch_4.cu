// air_batch_4.cu -- the batched kernel with 4 bands per thread.
#include "air_batch_kernel.cuh"

namespace air {
template bool batch_fns<4>(const GridView &, int, bool, int, BatchOccFn *, BatchLaunchFn *, size_t *, int *);
}  // namespace air
