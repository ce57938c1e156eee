// sweep_resident_kernel for grids up to 512 cells wide.
#include "resident_kernel.cuh"

namespace hp {

ResKernel res_kernel_512(int rows)
{
    if (rows == 4) return res_kernel<8, 4, 2>();
    if (rows == 8) return res_kernel<8, 8, 2>();
    return res_kernel<8, 16, 2>();
}

}  // namespace hp
