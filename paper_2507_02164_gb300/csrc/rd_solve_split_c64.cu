// rd_solve_split_c64.cu -- the split-register solver for complex64
// coefficients, and the dispatch by storage type.
#include "rd_solve_split_launch.cuh"

namespace rd {

int launch_solve_split_c128(int degree, const SolveArgs &a, cudaStream_t st);

int launch_solve_split(int degree, rd_dtype dt, const SolveArgs &a, cudaStream_t st)
{
    if (dt == RD_C64) return launch_split_degree<float2>(degree, a, st);
    return launch_solve_split_c128(degree, a, st);
}

}  // namespace rd
