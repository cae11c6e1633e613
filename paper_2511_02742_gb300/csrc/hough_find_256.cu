// hough_find_256.cu -- the fixed-point find kernel for CTAs of 256 threads and
// tiles of 32 word rows.
#include "hough_kernels.cuh"

namespace hk {

// Four CTAs per SM, 64 registers a thread.
__global__ void __launch_bounds__(256, 4) find_kernel_256(KParams p)
{
    find_body<Shape<256, 32>, false>(p);
}

}  // namespace hk
