// Sliced products of complex FP64 operators (VBCSR_C128).
#include "cplx.cuh"
#include "sliced_kernel.cuh"

namespace vbcsr {

const void *slice_c128_kernel_ptr(bool trans, int64_t k) { return slice_kernel_of<double2, Cplx>(trans, k); }

cudaError_t launch_slice_product_c128(bool trans, const ProdArgs &a, const SliceArgs &q, cudaStream_t s) {
    return launch_slice<double2, Cplx>(trans, a, q, s);
}

}  // namespace vbcsr
