// sweep_resident_kernel for grids more than 512 cells wide.
#include "resident_kernel.cuh"

namespace hp {

ResKernel res_kernel_wide(int rows)
{
    if (rows == 8) return res_kernel<8, 8, 1, true>();
    return res_kernel<8, 16, 1, true>();
}

}  // namespace hp
