// Instantiations of batch_kernel for maps without textures: 256 threads, 5
// CTAs per SM (exact) and 4 (learned), batch-uniform modes.
#include "rbsm_batch_kernel.cuh"

namespace rbsm {

BatchKernelFn batch_kernel_untextured(bool learned, int umode)
{
    if (learned)
        return umode == 9 ? batch_kernel<256, true, 4, 9> : batch_kernel<256, true, 4, 10>;
    switch (umode) {
    case 7: return batch_kernel<256, false, 5, 7>;
    case 8: return batch_kernel<256, false, 5, 8>;
    case 9: return batch_kernel<256, false, 5, 9>;
    case 10: return batch_kernel<256, false, 5, 10>;
    case 11: return batch_kernel<256, false, 5, 11>;
    default: return batch_kernel<256, false, 5, 12>;
    }
}

}  // namespace rbsm
