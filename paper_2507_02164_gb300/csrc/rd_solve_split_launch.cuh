// rd_solve_split_launch.cuh -- host-side launch of the split-register
// warp-specialised solver (rd_solve_split.cuh).
#pragma once

#include <atomic>

#include "rd_solve_split.cuh"

namespace rd {

// Once per kernel and device: the shared-memory opt-in, and the check that
// the kernel was built with the registers per thread that its roles' shares
// were added up against (a share above what the launch holds would wait
// forever). Host calls outside any stream order, so a capture may follow.
template <int N, typename Kern>
static int split_ready(Kern kern, std::atomic<int> (&ready)[64])
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return rd_check_launch("cudaGetDevice");
    if (dev < 0 || dev >= 64) return rd_set_error(RD_EUNSUPPORTED, "device %d: at most 64 devices", dev);
    if (ready[dev].load()) return RD_OK;
    cudaFuncAttributes attr;
    if (cudaFuncGetAttributes(&attr, kern) != cudaSuccess) return rd_check_launch("cudaFuncGetAttributes(split kernel)");
    if (attr.numRegs != Split<N>::LAUNCH_REGS)
        return rd_set_error(RD_EUNSUPPORTED, "split kernel of degree %d built with %d registers per thread, %d expected", N,
                            attr.numRegs, Split<N>::LAUNCH_REGS);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)split_smem_bytes<N>()) != cudaSuccess)
        return rd_check_launch("cudaFuncSetAttribute(split kernel)");
    ready[dev].store(1);
    return RD_OK;
}

template <int N, typename In>
static int launch_split_n(const SolveArgs &a, cudaStream_t st)
{
    static std::atomic<int> ready[64];
    auto kern = solve_split_kernel<N, In>;
    int rc = split_ready<N>(kern, ready);
    if (rc) return rc;
    const int64_t tasks = (a.n + 31) / 32, sms = rd_sm_count_cached();
    kern<<<(unsigned)(tasks < sms ? tasks : sms), Split<N>::THREADS, split_smem_bytes<N>(), st>>>(a);
    return rd_check_launch("solve_split_kernel");
}

template <typename In>
static int launch_split_degree(int degree, const SolveArgs &a, cudaStream_t st)
{
    switch (degree) {
    case 4: return launch_split_n<4, In>(a, st);
    case 5: return launch_split_n<5, In>(a, st);
    case 6: return launch_split_n<6, In>(a, st);
    case 7: return launch_split_n<7, In>(a, st);
    case 8: return launch_split_n<8, In>(a, st);
    case 9: return launch_split_n<9, In>(a, st);
    case 10: return launch_split_n<10, In>(a, st);
    case 11: return launch_split_n<11, In>(a, st);
    case 12: return launch_split_n<12, In>(a, st);
    default: return rd_set_error(RD_EUNSUPPORTED, "degree %d not built (4..12)", degree);
    }
}

template <int N, typename In>
static int launch_uneven_split_n(const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets, cudaStream_t st)
{
    static std::atomic<int> ready[64];
    auto kern = uneven_split_kernel<N, In>;
    int rc = split_ready<N>(kern, ready);
    if (rc) return rc;
    kern<<<rd_sm_count_cached(), Split<N>::THREADS, split_smem_bytes<N>(), st>>>(a, L.hdr, L.perm, L.bins, offsets);
    return rd_check_launch("uneven_split_kernel");
}

template <typename In>
static int launch_uneven_split_degree(int degree, const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets,
                                      cudaStream_t st)
{
    switch (degree) {
    case 4: return launch_uneven_split_n<4, In>(a, L, offsets, st);
    case 5: return launch_uneven_split_n<5, In>(a, L, offsets, st);
    case 6: return launch_uneven_split_n<6, In>(a, L, offsets, st);
    case 7: return launch_uneven_split_n<7, In>(a, L, offsets, st);
    case 8: return launch_uneven_split_n<8, In>(a, L, offsets, st);
    case 9: return launch_uneven_split_n<9, In>(a, L, offsets, st);
    case 10: return launch_uneven_split_n<10, In>(a, L, offsets, st);
    case 11: return launch_uneven_split_n<11, In>(a, L, offsets, st);
    case 12: return launch_uneven_split_n<12, In>(a, L, offsets, st);
    default: return rd_set_error(RD_EUNSUPPORTED, "degree %d not built (4..12)", degree);
    }
}

}  // namespace rd
