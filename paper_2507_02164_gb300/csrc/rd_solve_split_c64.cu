// rd_solve_split_c64.cu -- the split-register solver for complex64
// coefficients, and the dispatch by polish and storage type.
#include "rd_solve_split_launch.cuh"

namespace rd {

int launch_solve_split_df(int degree, rd_dtype dt, const SolveArgs &a, cudaStream_t st);
int launch_solve_split_c128(int degree, const SolveArgs &a, cudaStream_t st);

int launch_solve_split(int degree, rd_dtype dt, const SolveArgs &a, cudaStream_t st)
{
    if (a.polish_mode == RD_POLISH_DF) return launch_solve_split_df(degree, dt, a, st);
    if (dt == RD_C64) return launch_split_degree<float2, MODE_MIXED_FP64>(degree, a, st);
    return launch_solve_split_c128(degree, a, st);
}

}  // namespace rd
