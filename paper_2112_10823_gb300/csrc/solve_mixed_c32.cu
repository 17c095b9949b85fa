// Single-system solve kernels: FP32 values (mixed precision), 32-bit columns.
#include "solve_kernel.cuh"

namespace cgk {
template const void* solve_kernel_of<true, int32_t>(bool jacobi, bool small);
}
