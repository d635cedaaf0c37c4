// The persistent fit kernel for blocks of up to 512 threads, 1 resident per SM (see fit_dev.cuh).
#include "fit_dev.cuh"

namespace fitcore {

const void *fit_kernel_512(bool general, bool pre) { return fit_kernel_of<512, 1>(general, pre); }

}  // namespace fitcore
