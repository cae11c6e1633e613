// hough_find.cu -- the fixed-point find kernel for any launch shape (the find
// kernels are translation units of their own, compiled in parallel).
#include "hough_kernels.cuh"

namespace hk {

// Any CTA size up to 1024 threads (64 registers a thread), any tile.
__global__ void __launch_bounds__(1024, 1) find_kernel(KParams p)
{
    find_body<AnyShape, false>(p);
}

}  // namespace hk
