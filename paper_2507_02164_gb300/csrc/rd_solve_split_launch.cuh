// rd_solve_split_launch.cuh -- host-side launch of the split-register
// warp-specialised solver (rd_solve_split.cuh).
#pragma once

#include <atomic>

#include "rd_solve_split.cuh"

namespace rd {

// Once per kernel and device: the check that the kernel was built with the
// registers per thread that its roles' shares were added up against (a share
// above what the launch holds would wait forever), and the shared-memory
// opt-in. With another count SPLIT_DECLINED: the caller takes the one-role
// kernel. Host calls outside any stream order, so a capture may follow.
template <int N, typename In, int MODE, typename Kern>
static int split_ready(Kern kern, std::atomic<int> (&ready)[64])
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return rd_check_launch("cudaGetDevice");
    if (dev < 0 || dev >= 64) return rd_set_error(RD_EUNSUPPORTED, "device %d: at most 64 devices", dev);
    const int known = ready[dev].load();
    if (known) return known > 0 ? RD_OK : SPLIT_DECLINED;
    cudaFuncAttributes attr;
    if (cudaFuncGetAttributes(&attr, kern) != cudaSuccess) return rd_check_launch("cudaFuncGetAttributes(split kernel)");
    if (attr.numRegs != Split<N, MODE>::LAUNCH_REGS) {
        ready[dev].store(-1);
        return SPLIT_DECLINED;
    }
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)split_smem_bytes<N, In, MODE>()) != cudaSuccess)
        return rd_check_launch("cudaFuncSetAttribute(split kernel)");
    ready[dev].store(1);
    return RD_OK;
}

template <int N, typename In, int MODE>
static int launch_split_n(const SolveArgs &a, cudaStream_t st)
{
    static std::atomic<int> ready[64];
    auto kern = solve_split_kernel<N, In, MODE>;
    int rc = split_ready<N, In, MODE>(kern, ready);
    if (rc) return rc;
    const int64_t tasks = (a.n + 31) / 32, sms = rd_sm_count_cached();
    kern<<<(unsigned)(tasks < sms ? tasks : sms), Split<N, MODE>::THREADS, split_smem_bytes<N, In, MODE>(), st>>>(a);
    return rd_check_launch("solve_split_kernel");
}

template <int N, typename In, int MODE>
static int launch_uneven_split_n(const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets, cudaStream_t st)
{
    static std::atomic<int> ready[64];
    auto kern = uneven_split_kernel<N, In, MODE>;
    int rc = split_ready<N, In, MODE>(kern, ready);
    if (rc) return rc;
    kern<<<rd_sm_count_cached(), Split<N, MODE>::THREADS, split_smem_bytes<N, In, MODE>(), st>>>(a, L.hdr, L.perm, L.bins, offsets);
    return rd_check_launch("uneven_split_kernel");
}

// LAUNCH<N>() for the degree, one instance for each degree that is built.
#define RD_SPLIT_CASE(D, LAUNCH, ...) \
    case D: \
        if constexpr (split_built(D, MODE)) return LAUNCH<D, In, MODE>(__VA_ARGS__); \
        break;
#define RD_SPLIT_DEGREES(LAUNCH, ...) \
    switch (degree) { \
        RD_SPLIT_CASE(4, LAUNCH, __VA_ARGS__) RD_SPLIT_CASE(5, LAUNCH, __VA_ARGS__) RD_SPLIT_CASE(6, LAUNCH, __VA_ARGS__) \
        RD_SPLIT_CASE(7, LAUNCH, __VA_ARGS__) RD_SPLIT_CASE(8, LAUNCH, __VA_ARGS__) RD_SPLIT_CASE(9, LAUNCH, __VA_ARGS__) \
        RD_SPLIT_CASE(10, LAUNCH, __VA_ARGS__) RD_SPLIT_CASE(11, LAUNCH, __VA_ARGS__) RD_SPLIT_CASE(12, LAUNCH, __VA_ARGS__) \
    } \
    return rd_set_error(RD_EUNSUPPORTED, "split solver: degree %d not built", degree);

template <typename In, int MODE>
static int launch_split_degree(int degree, const SolveArgs &a, cudaStream_t st)
{
    RD_SPLIT_DEGREES(launch_split_n, a, st)
}

template <typename In, int MODE>
static int launch_uneven_split_degree(int degree, const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets,
                                      cudaStream_t st)
{
    RD_SPLIT_DEGREES(launch_uneven_split_n, a, L, offsets, st)
}

#undef RD_SPLIT_DEGREES
#undef RD_SPLIT_CASE

}  // namespace rd
