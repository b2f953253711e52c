// rd_solve_split_df_c64.cu -- the split-register solver with the compensated
// polish for complex64 coefficients (uniform batches and degree bins), and the
// dispatch by storage type.
#include "rd_solve_split_launch.cuh"

namespace rd {

int launch_solve_split_df_c128(int degree, const SolveArgs &a, cudaStream_t st);
int launch_uneven_split_df_c128(int degree, const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets, cudaStream_t st);

int launch_solve_split_df(int degree, rd_dtype dt, const SolveArgs &a, cudaStream_t st)
{
    if (dt == RD_C64) return launch_split_degree<float2, MODE_MIXED_DF>(degree, a, st);
    return launch_solve_split_df_c128(degree, a, st);
}

int launch_uneven_split_df(int degree, rd_dtype dt, const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets,
                           cudaStream_t st)
{
    if (dt == RD_C64) return launch_uneven_split_degree<float2, MODE_MIXED_DF>(degree, a, L, offsets, st);
    return launch_uneven_split_df_c128(degree, a, L, offsets, st);
}

}  // namespace rd
