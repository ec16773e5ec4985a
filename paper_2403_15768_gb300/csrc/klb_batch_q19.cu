// Instantiations of the batched step for the D3Q19 lattice with FP64 and FP32 storage
// (templates in klb_kernels.cuh).

#include "klb_kernels.cuh"

namespace klb {

cudaError_t launch_batch_q19(int storage, const BatchLaunch &b, cudaStream_t s)
{
    switch (storage) {
    case KLB_FP64:
        return launch_batch_q<19, double, double>(b, s);
    case KLB_FP32:
        return launch_batch_q<19, float, float>(b, s);
    default:
        return cudaErrorInvalidValue;
    }
}

}  // namespace klb
