// sweep_resident_kernel for grids up to 128 cells wide.
#include "resident_kernel.cuh"

namespace hp {

ResKernel res_kernel_128(int rows)
{
    if (rows == 4) return res_kernel<4, 4, 1>();
    if (rows == 8) return res_kernel<4, 8, 1>();
    return res_kernel<4, 16, 1>();
}

}  // namespace hp
