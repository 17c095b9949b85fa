// Single-system solve kernels: FP64 values, 32-bit columns.
#include "solve_kernel.cuh"

namespace cgk {
template const void* solve_kernel_of<false, int32_t>(bool jacobi, bool small);
}
