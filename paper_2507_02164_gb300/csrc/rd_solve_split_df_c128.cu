// rd_solve_split_df_c128.cu -- the split-register solver with the compensated
// polish for complex128 coefficients (uniform batches and degree bins).
#include "rd_solve_split_launch.cuh"

namespace rd {

int launch_solve_split_df_c128(int degree, const SolveArgs &a, cudaStream_t st)
{
    return launch_split_degree<double2, MODE_MIXED_DF>(degree, a, st);
}

int launch_uneven_split_df_c128(int degree, const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets, cudaStream_t st)
{
    return launch_uneven_split_degree<double2, MODE_MIXED_DF>(degree, a, L, offsets, st);
}

}  // namespace rd
