// rd_uneven_split_c128.cu -- the split-register solver for the degree bins of
// a packed complex128 batch.
#include "rd_solve_split_launch.cuh"

namespace rd {

int launch_uneven_split_c128(int degree, const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets, cudaStream_t st)
{
    return launch_uneven_split_degree<double2, MODE_MIXED_FP64>(degree, a, L, offsets, st);
}

}  // namespace rd
