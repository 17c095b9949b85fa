// Single-system solve kernels: FP32 values (mixed precision), 16-bit column offsets.
#include "solve_kernel.cuh"

namespace cgk {
template const void* solve_kernel_of<true, uint16_t>(bool jacobi, bool small);
}
