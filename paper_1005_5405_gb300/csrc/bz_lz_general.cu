// bz_lz_general.cu -- the active-node kernel with the axis length read at run time,
// and with the sources brought by bulk copies.
#include "bz_lz_kernels.h"

namespace bzk {

template <int G, int ST>
static LzKernel lz_general(bool stretched, int VW)
{
    if (VW == 4) return stretched ? k_lz<G, 0, true, ST> : k_lz<G, 0, false, ST>;
    return stretched ? k_lz<G, 0, true, ST, false, 2> : k_lz<G, 0, false, ST, false, 2>;
}

LzKernel lz_kernel_general(int G, int ST, bool stretched, int VW)
{
    if (ST == 512) return G == 4 ? lz_general<4, 512>(stretched, VW) : lz_general<2, 512>(stretched, VW);
    return G == 4 ? lz_general<4, 256>(stretched, VW) : lz_general<2, 256>(stretched, VW);
}

LzKernel lz_kernel_bulk(int N)
{
    return N == 32 ? k_lz<4, 32, false, 256, true> : k_lz<4, 0, false, 256, true>;
}

}  // namespace bzk
