// mbl_coop.cu -- the cooperative launches of the resident kernels, behind one host function.
#include <cuda_runtime.h>

#include "mbl_internal.h"

namespace mbl {

int cooperative_launch(const void *kernel, unsigned blocks, unsigned threads, size_t smem, void **args,
                       cudaStream_t st)
{
    const cudaError_t e = cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(threads), args, smem, st);
    if (e == cudaSuccess) {
        note_launch();
        return MBL_OK;
    }
    (void)cudaGetLastError();
    return e == cudaErrorCooperativeLaunchTooLarge ? kTooLarge : MBL_ERR_CUDA;
}

}  // namespace mbl
