// sweep_resident_kernel for grids up to 256 cells wide.
#include "resident_kernel.cuh"

namespace hp {

ResKernel res_kernel_256(int rows)
{
    if (rows == 4) return res_kernel<8, 4, 1>();
    if (rows == 8) return res_kernel<8, 8, 1>();
    return res_kernel<8, 16, 1>();
}

}  // namespace hp
