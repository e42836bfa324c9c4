// reference.cu -- the reference variant (paper Sec. 2: the plain code whose
// outputs every variant is compared with): one element per thread, plain
// loads and stores, the two hardware-rounded FP64 operations.
#include "internal.h"

namespace wx {

__global__ void wxpy_reference_kernel(const SingleArgs a) {
    // Launched, and followed by the next launch, like the family's kernels, so that
    // timings compare.
    pdl_wait();
    if (!a.late) pdl_trigger();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < a.n) {
        const double xi = a.x[i];
        const double yi = a.y[i];
        a.w[i] = __dadd_rn(__dmul_rn(a.alpha, xi), yi);
    }
    if (a.late) pdl_trigger();
}

cudaError_t launch_reference(unsigned grid, unsigned tpb, const SingleArgs &a, cudaStream_t s) {
    SingleArgs r = a;
    r.late = ends_at_once(grid, (int)tpb, kSmCount);
    return launch_pdl(&wxpy_reference_kernel, grid, tpb, s, r);
}

}  // namespace wx
