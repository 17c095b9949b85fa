// Batched solve kernels: FP64 values.
#include "batch_kernel.cuh"

namespace cgk {
template const void* batch_kernel_of<false>(bool jacobi);
}
