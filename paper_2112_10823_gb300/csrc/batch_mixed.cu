// Batched solve kernels: FP32 values (mixed precision).
#include "batch_kernel.cuh"

namespace cgk {
template const void* batch_kernel_of<true>(bool jacobi);
}
