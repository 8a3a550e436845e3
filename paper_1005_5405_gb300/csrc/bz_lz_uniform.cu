// bz_lz_uniform.cu -- the active-node kernel for uniform cells, an instance per axis length.
#include "bz_lz_kernels.h"

bzk::LzKernel bzk::lz_kernel_uniform(int N)
{
    return lz_at_length<LzKernel>(N, [](auto n) -> LzKernel {
        return k_lz<4, n(), false, lz_stream_threads(n())>;
    });
}
