// Instantiations of the KLB kernels for the D3Q19 lattice (templates in
// klb_kernels.cuh) with FP64 and FP32 storage; 16-bit storage in
// klb_kernels_q19_16.cu, batches in klb_batch_*.cu, so that they compile in
// parallel.

#include "klb_kernels.cuh"

namespace klb {

cudaError_t launch_q19_16(int storage, const void *args, int mode, int nblocks, int bx, cudaStream_t s);

cudaError_t launch_q19(int storage, const void *args, int mode, int nblocks, int bx, cudaStream_t s)
{
    switch (storage) {
    case KLB_FP64:
        return launch_q<19, double, double>(args, mode, nblocks, bx, s);
    case KLB_FP32:
        return launch_q<19, float, float>(args, mode, nblocks, bx, s);
    default:
        return launch_q19_16(storage, args, mode, nblocks, bx, s);
    }
}

}  // namespace klb
