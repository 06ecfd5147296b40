// air_batch_wide.cu -- the batched kernel in the wide form.
#include "air_batch_kernel.cuh"

namespace air {
template bool batch_fns<0>(const GridView &, int, bool, int, BatchOccFn *, BatchLaunchFn *, size_t *, int *);
}  // namespace air
