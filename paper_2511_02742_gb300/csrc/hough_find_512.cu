// hough_find_512.cu -- the fixed-point find kernel for CTAs of 512 threads and
// tiles of 32 word rows.
#include "hough_kernels.cuh"

namespace hk {

// Two CTAs per SM, 64 registers a thread.
__global__ void __launch_bounds__(512, 2) find_kernel_512(KParams p)
{
    find_body<Shape<512, 32>, false>(p);
}

}  // namespace hk
