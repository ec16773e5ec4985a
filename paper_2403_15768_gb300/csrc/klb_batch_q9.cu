// Instantiations of the batched step for the D2Q9 lattice
// (templates in klb_kernels.cuh).

#include "klb_kernels.cuh"

namespace klb {

cudaError_t launch_batch_q9(int storage, const BatchLaunch &b, cudaStream_t s)
{
    switch (storage) {
    case KLB_FP64:
        return launch_batch_q<9, double, double>(b, s);
    case KLB_FP32:
        return launch_batch_q<9, float, float>(b, s);
    case KLB_FP16_DEV:
        return launch_batch_q<9, float, __half>(b, s);
    case KLB_BF16_DEV:
        return launch_batch_q<9, float, __nv_bfloat16>(b, s);
    default:
        return cudaErrorInvalidValue;
    }
}

}  // namespace klb
