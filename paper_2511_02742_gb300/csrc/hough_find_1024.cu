// hough_find_1024.cu -- the fixed-point find kernel for CTAs of 1024 threads and
// tiles of 32 word rows.
#include "hough_kernels.cuh"

namespace hk {

// One CTA per SM, 64 registers a thread.
__global__ void __launch_bounds__(1024, 1) find_kernel_1024(KParams p)
{
    find_body<Shape<1024, 32>, false>(p);
}

}  // namespace hk
