// bz_lz_stretched.cu -- the active-node kernel for stretched cells, an instance per axis length.
#include "bz_lz_kernels.h"

bzk::LzKernel bzk::lz_kernel_stretched(int N)
{
    return lz_at_length<LzKernel>(N, [](auto n) -> LzKernel {
        return k_lz<4, n(), true, lz_stream_threads(n())>;
    });
}
