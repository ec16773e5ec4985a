// Instantiations of the batched step for the D3Q19 lattice with 16-bit storage
// (templates in klb_kernels.cuh).

#include "klb_kernels.cuh"

namespace klb {

cudaError_t launch_batch_q19_16(int storage, const BatchLaunch &b, cudaStream_t s)
{
    switch (storage) {
    case KLB_FP16_DEV:
        return launch_batch_q<19, float, __half>(b, s);
    case KLB_BF16_DEV:
        return launch_batch_q<19, float, __nv_bfloat16>(b, s);
    default:
        return cudaErrorInvalidValue;
    }
}

}  // namespace klb
