// rd_uneven_bins.cuh -- the persistent solve kernels of the uneven-degree
// path (one per degree, tasks pulled from the bin's atomic queue) and
// launch_uneven_bins. Included only by the rd_uneven_bins_*.cu files, each
// of which instantiates it for one storage type and precision mode.
#pragma once

#include <atomic>

#include "rd_solve2.cuh"
#include "rd_solve_ws.cuh"
#include "rd_uneven.cuh"

namespace rd {


// Persistent solver for the degree-N bin: each warp takes the next task of
// the bin's queue (task = 32 consecutive slots) until the queue is empty.
// One kernel per degree keeps each degree's own register allocation.
template <int N, typename In, int MODE>
__device__ __forceinline__ void uneven_solve(const SolveArgs &A, UnevenHeader *hdr, const uint32_t *perm,
                                             const char *bins, const int64_t *offsets)
{
    using T = typename std::conditional<MODE != MODE_PLAIN, float, double>::type;
    __shared__ unsigned long long acc[ST_WORDS];
    const CtaStats S = stats_begin(acc, A.stats);
    const int lane = threadIdx.x & 31;
    const int64_t cnt = hdr->count[N];
    const unsigned tasks = (unsigned)((cnt + 31) / 32);
    const PackedMap map{{}, perm + hdr->poly_base[N], offsets};
    const void *base = bins + (size_t)hdr->coef_base[N] * sizeof(In);
    for (;;) {
        unsigned t = 0;
        if (lane == 0) t = atomicAdd(&hdr->head[N], 1u);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= tasks) break;
        solve_warp<N, T, In, MODE>(A, base, cnt, (int64_t)t * 32, map, S);
    }
    stats_end(S, A.stats);
}

template <int N, typename In, int MODE, bool TWELVE>
__global__ void __launch_bounds__(solve_threads(TWELVE), solve_ctas(N, MODE))
    uneven_solve_kernel(SolveArgs A, UnevenHeader *hdr, const uint32_t *perm, const char *bins, const int64_t *offsets)
{
    uneven_solve<N, In, MODE>(A, hdr, perm, bins, offsets);
}

// The same with two lanes per polynomial (rd_solve2.cuh): tasks of 16 slots.
template <int N, typename In, int MODE>
__global__ void __maxnreg__(two_lane_regs(N, MODE))
    uneven_solve2_kernel(SolveArgs A, UnevenHeader *hdr, const uint32_t *perm, const char *bins, const int64_t *offsets)
{
    using T = typename std::conditional<MODE != MODE_PLAIN, float, double>::type;
    __shared__ unsigned long long acc[ST_WORDS];
    const CtaStats S = stats_begin(acc, A.stats);
    const int lane = threadIdx.x & 31;
    const int64_t cnt = hdr->count[N];
    const unsigned tasks = (unsigned)((cnt + 15) / 16);
    const PackedMap map{{}, perm + hdr->poly_base[N], offsets};
    const void *base = bins + (size_t)hdr->coef_base[N] * sizeof(In);
    for (;;) {
        unsigned t = 0;
        if (lane == 0) t = atomicAdd(&hdr->head[N], 1u);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= tasks) break;
        solve_warp2<N, T, In, MODE>(A, base, cnt, (int64_t)t * 16, map, S);
    }
    stats_end(S, A.stats);
}

// The warp-specialised form (rd_solve_ws.cuh) of the degree-N bin: sweep
// warps and polish warps meet at a shared-memory ring; CTA b takes the bin's
// tasks b, b + G, ... (the bin's size is read on the device). Built for the
// degrees up to UNEVEN_WS_MAX_DEG, where the split measured faster than the
// one-role kernel.
constexpr int UNEVEN_WS_MAX_DEG = 8;

template <int N, typename In, int MAXB, int MODE>
__global__ void __launch_bounds__(MAXB, 1)
    uneven_solve_ws_kernel(SolveArgs A, UnevenHeader *hdr, const uint32_t *perm, const char *bins,
                           const int64_t *offsets, int polish_warps, int slots)
{
    const int64_t cnt = hdr->count[N];
    const PackedMap map{{}, perm + hdr->poly_base[N], offsets};
    const void *base = bins + (size_t)hdr->coef_base[N] * sizeof(In);
    ws_cta<N, In, MODE>(A, base, cnt, map, polish_warps, slots);
}

// Dynamic shared memory above 48 KB needs the kernel's opt-in, per device
// (raised once per device to the largest size asked for; host calls only).
template <int N, typename In, int MAXB, int MODE>
static int uneven_ws_allow_smem(size_t bytes)
{
    static std::atomic<size_t> allowed[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return rd_check_launch("cudaGetDevice");
    if (dev < 0 || dev >= 64) return rd_set_error(RD_EUNSUPPORTED, "device %d: at most 64 devices", dev);
    if (bytes <= 48 * 1024 || bytes <= allowed[dev].load()) return RD_OK;
    if (cudaFuncSetAttribute(uneven_solve_ws_kernel<N, In, MAXB, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)bytes) != cudaSuccess)
        return rd_check_launch("cudaFuncSetAttribute(uneven_solve_ws_kernel)");
    size_t cur = allowed[dev].load();
    while (cur < bytes && !allowed[dev].compare_exchange_weak(cur, bytes)) {
    }
    return RD_OK;
}

template <int N, typename In, int MODE>
static int launch_uneven_ws(const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets, int block,
                            int polish_warps, cudaStream_t st)
{
    constexpr int MAXB = ws_max_block(N);
    const int warps = block / 32;
    const int slots = 2 * warps < WS_MAX_SLOTS ? 2 * warps : WS_MAX_SLOTS;
    const size_t smem = ws_smem_bytes(N, slots);
    int rc = uneven_ws_allow_smem<N, In, MAXB, MODE>(smem);
    if (rc) return rc;
    auto kern = uneven_solve_ws_kernel<N, In, MAXB, MODE>;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, block, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    kern<<<per_sm * rd_sm_count_cached(), block, smem, st>>>(a, L.hdr, L.perm, L.bins, offsets, polish_warps, slots);
    return rd_check_launch("uneven_solve_ws_kernel");
}

int lanes_for(int degree, bool mixed, int polish_mode, int requested);

// The occupancy maximum is asked for once per kernel, device and block size (0.2 us
// each time, of about 5 us of host time per bin).
template <auto KERN>
static int launch_persistent(const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets, int block,
                             int ctas_per_sm, cudaStream_t st, const char *what)
{
    static std::atomic<int> known[64][9];
    int per_sm = ctas_per_sm, dev = 0;
    if (per_sm <= 0) {
        const bool keep = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 && block <= 256;
        per_sm = keep ? known[dev][block / 32].load(std::memory_order_relaxed) : 0;
        if (per_sm <= 0) {
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, KERN, block, 0) != cudaSuccess || per_sm < 1)
                per_sm = 1;
            else if (keep)
                known[dev][block / 32].store(per_sm, std::memory_order_relaxed);
        }
    }
    int grid = per_sm * rd_sm_count_cached();
    KERN<<<grid, block, 0, st>>>(a, L.hdr, L.perm, L.bins, offsets);
    return rd_check_launch(what);
}

template <int N, typename In, int MODE>
static int launch_degree_bin(const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets, int block,
                             int ctas_per_sm, int lanes, int polish_warps, cudaStream_t st)
{
    if constexpr (MODE != MODE_PLAIN) {
        if (polish_warps == UNEVEN_SPLIT) {
            const int rc = launch_uneven_split(N, std::is_same<In, float2>::value ? RD_C64 : RD_C128, a, L, offsets, st);
            if (rc != SPLIT_DECLINED) return rc;
        }
    }
    if constexpr (MODE != MODE_PLAIN && N <= UNEVEN_WS_MAX_DEG) {
        if (polish_warps > 0) return launch_uneven_ws<N, In, MODE>(a, L, offsets, block, polish_warps, st);
    }
    if constexpr (N >= 2 && MODE != MODE_MIXED_DF) {
        if (lanes_for(N, MODE != MODE_PLAIN, a.polish_mode, lanes) == 2)
            return launch_persistent<uneven_solve2_kernel<N, In, MODE>>(a, L, offsets, block, ctas_per_sm, st,
                                     "uneven_solve2_kernel");
    }
    // At most eight warps per SM whatever the bin's share of the batch: free
    // registers, as solve_kernel_for (us, all of degree 8, compensated, complex64,
    // 168 / free: 17,000 124 / 107, 34,000 123 / 110, 50,000 130 / 165; FP64 polish
    // 34,000 166 / 133, 50,000 167 / 210).
    if constexpr (solve_twelve_warps(N, MODE)) {
        if (a.n > 256 * (int64_t)rd_sm_count_cached())
            return launch_persistent<uneven_solve_kernel<N, In, MODE, true>>(a, L, offsets, block, ctas_per_sm, st,
                                     "uneven_solve_kernel");
    }
    return launch_persistent<uneven_solve_kernel<N, In, MODE, false>>(a, L, offsets, block, ctas_per_sm, st,
                             "uneven_solve_kernel");
}

template <typename In, int MODE>
int launch_uneven_bins(const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets, const int *block,
                       const int *cps, const int *lanes, const int *pw, int lowest, const cudaStream_t *chain)
{
    int rc = RD_OK;
#define RD_BIN(D) \
    if (!rc && D >= lowest) rc = launch_degree_bin<D, In, MODE>(a, L, offsets, block[D], cps[D], lanes[D], pw[D], chain[D]);
    RD_BIN(12) RD_BIN(11) RD_BIN(10) RD_BIN(9) RD_BIN(8) RD_BIN(7) RD_BIN(6) RD_BIN(5) RD_BIN(4) RD_BIN(3) RD_BIN(2) RD_BIN(1)
#undef RD_BIN
    return rc;
}

}  // namespace rd

#define RD_UNEVEN_BINS(IN, MODE)                                                                          \
    namespace rd {                                                                                      \
    template int launch_uneven_bins<IN, MODE>(const SolveArgs &, const UnevenLayout &, const int64_t *, \
                                              const int *, const int *, const int *, const int *, int,  \
                                              const cudaStream_t *);                                    \
    }
