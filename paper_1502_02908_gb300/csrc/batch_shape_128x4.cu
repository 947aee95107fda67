// The persistent batch kernel with 128-thread blocks, 4 resident an SM.
#include "batch_kernel.cuh"

namespace episim {

BatchKernel batch_kernel_128x4(BatchForm f) { return batch_kernel_of<128, 4>(f); }

}  // namespace episim
