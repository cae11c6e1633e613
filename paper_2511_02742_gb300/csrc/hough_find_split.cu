// hough_find_split.cu -- the fixed-point find kernels that spread a window
// over the CTAs of a cluster (tiles of 32 word rows).
#include "hough_kernels.cuh"

namespace hk {

__global__ void __launch_bounds__(256, 2) find_split_kernel_256(KParams p)
{
    split_body<Shape<256, 32>>(p);
}

__global__ void __launch_bounds__(512, 2) find_split_kernel_512(KParams p)
{
    split_body<Shape<512, 32>>(p);
}

}  // namespace hk
