// air_batch_1.cu -- the batched kernel with 1 band per thread.
#include "air_batch_kernel.cuh"

namespace air {
template bool batch_fns<1>(const GridView &, int, bool, int, BatchOccFn *, BatchLaunchFn *, size_t *, int *);
}  // namespace air
