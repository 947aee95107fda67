// The persistent batch kernel with list events, 256-thread blocks, 2 resident an SM.
#include "batch_kernel.cuh"

namespace episim {

BatchKernel batch_lists_256x2() { return batch_lists_of<256, 2>(); }

}  // namespace episim
