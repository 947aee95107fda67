// The persistent batch kernel with list events, 256-thread blocks, 1 resident an SM.
#include "batch_kernel.cuh"

namespace episim {

BatchKernel batch_lists_256x1() { return batch_lists_of<256, 1>(); }

}  // namespace episim
