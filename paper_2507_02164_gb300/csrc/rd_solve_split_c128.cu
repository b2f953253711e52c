// rd_solve_split_c128.cu -- the split-register solver for complex128 coefficients.
#include "rd_solve_split_launch.cuh"

namespace rd {

int launch_solve_split_c128(int degree, const SolveArgs &a, cudaStream_t st)
{
    return launch_split_degree<double2, MODE_MIXED_FP64>(degree, a, st);
}

}  // namespace rd
