// hough_find_128.cu -- the fixed-point find kernel for CTAs of 128 threads and
// tiles of 32 word rows.
#include "hough_kernels.cuh"

namespace hk {

// Four CTAs per SM.
__global__ void __launch_bounds__(128, 4) find_kernel_128(KParams p)
{
    find_body<Shape<128, 32>, false>(p);
}

}  // namespace hk
