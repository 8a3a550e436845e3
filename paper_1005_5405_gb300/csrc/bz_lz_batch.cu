// bz_lz_batch.cu -- the batches' active-node kernel, an instance per axis length.
#include "bz_lz_kernels.h"

bzk::LzBatchKernel bzk::lz_batch_kernel(int N)
{
    return lz_at_length<LzBatchKernel>(N, [](auto n) -> LzBatchKernel {
        if constexpr (n() % 4 == 0) return kbl_lz<n()>;
        else return nullptr;
    });
}
