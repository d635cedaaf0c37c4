// The persistent fit kernel for blocks of up to 128 threads, 5 resident per SM (see fit_dev.cuh).
#include "fit_dev.cuh"

namespace fitcore {

const void *fit_kernel_128x5(bool general, bool pre) { return fit_kernel_of<128, 5>(general, pre); }

}  // namespace fitcore
