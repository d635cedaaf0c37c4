// The persistent fit kernel for blocks of up to 256 threads, 2 resident per SM (see fit_dev.cuh).
#include "fit_dev.cuh"

namespace fitcore {

const void *fit_kernel_256(bool general, bool pre) { return fit_kernel_of<256, 2>(general, pre); }

}  // namespace fitcore
