// cr_batched512.cu -- the batched form's kernel at 512 threads (see cr_batch.cuh).
#include "cr_batch.cuh"

namespace crs {

void (*batch_kernel512())(BatchArgs) { return k_batch<512>; }

}  // namespace crs
