// bz_lz_kernels.h -- the instances of the active-node kernel (bz_lazy.cuh).
//
// Every axis length that the kernel takes (multiples of four from 12, N = 2 mod 4
// from 14, up to 32) has an instance with the length as a constant, uniform and
// stretched, for the shape it runs in: groups of four cells and
// lz_stream_threads(N) streaming threads.  The constant turns the node numbers'
// divisions and the stage counts into immediates: a step of 96^2 cells with the
// length read at run time and as a constant, us: 14 nodes per axis 329 / 314, 18 396 /
// 376, 22 572 / 553, 26 1022 / 948, 30 1536 / 1530; stretched 14 348 / 324, 22 612 / 580,
// 24 662 / 627, 26 1062 / 971; the others within 2 %, none slower.
// Groups of two cells (more active nodes than 16-bit offsets reach with four) and
// thread counts forced by BZ_LAZY_ST run the instances that read the length at
// run time.  The bz_lz_*.cu files hold them, so that they compile in parallel; each
// function returns nullptr where there is no instance.
#pragma once

#include "bz_lzbatch.cuh"

namespace bzk {

using LzKernel = void (*)(Geo, LzArgs);
using LzBatchKernel = void (*)(const LzInst *, const int4 *, int, int *);

LzKernel lz_kernel_uniform(int N);
LzKernel lz_kernel_stretched(int N);
LzKernel lz_kernel_general(int G, int ST, bool stretched, int VW);
LzKernel lz_kernel_bulk(int N);            // sources by bulk copies, uniform cells
LzBatchKernel lz_batch_kernel(int N);      // uniform cells, N a multiple of four

// f's value at the axis length N (f called with it as a constant), or nullptr.
template <typename P, typename F>
P lz_at_length(int N, F f)
{
    switch (N) {
#define BZ_LZ_N(n) case n: return f(std::integral_constant<int, n>{})
    BZ_LZ_N(12);
    BZ_LZ_N(14);
    BZ_LZ_N(16);
    BZ_LZ_N(18);
    BZ_LZ_N(20);
    BZ_LZ_N(22);
    BZ_LZ_N(24);
    BZ_LZ_N(26);
    BZ_LZ_N(28);
    BZ_LZ_N(30);
    BZ_LZ_N(32);
#undef BZ_LZ_N
    }
    return nullptr;
}

}  // namespace bzk
