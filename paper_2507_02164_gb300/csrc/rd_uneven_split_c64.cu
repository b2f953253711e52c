// rd_uneven_split_c64.cu -- the split-register solver (rd_solve_split.cuh) for
// the degree bins of a packed complex64 batch, and the dispatch by polish and
// storage type.
#include "rd_solve_split_launch.cuh"

namespace rd {

int launch_uneven_split_df(int degree, rd_dtype dt, const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets,
                           cudaStream_t st);
int launch_uneven_split_c128(int degree, const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets, cudaStream_t st);

int launch_uneven_split(int degree, rd_dtype dt, const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets,
                        cudaStream_t st)
{
    if (a.polish_mode == RD_POLISH_DF) return launch_uneven_split_df(degree, dt, a, L, offsets, st);
    if (dt == RD_C64) return launch_uneven_split_degree<float2, MODE_MIXED_FP64>(degree, a, L, offsets, st);
    return launch_uneven_split_c128(degree, a, L, offsets, st);
}

}  // namespace rd
