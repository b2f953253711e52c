// rd_uneven.cuh -- workspace layout of the uneven-degree solve and the
// per-bin launcher that rd_uneven.cu calls once the batch is binned. The
// launcher is defined in rd_uneven_bins.cuh and instantiated once per
// storage type and precision mode, each in a translation unit of its own
// (rd_uneven_bins_*.cu), so that the 144 solve kernels compile in parallel.
#pragma once

#include "rd_solve.cuh"

namespace rd {

constexpr int UNEVEN_MAX_DEG = 12;

struct UnevenHeader {
    uint32_t count[16];      // polynomials per degree
    uint32_t cursor[16];     // pack cursors per degree
    uint32_t poly_base[16];  // first slot of each degree's bin in perm
    uint32_t head[16];       // task queue head of each degree's solve kernel
    uint32_t bad;            // polynomials whose offsets disagree with their degree
    uint32_t overflow;       // 1: the solvable polynomials overlap (sum of (d + 1) > n_coeffs)
    uint32_t direct;         // bit d: the group kernel solves degree d, its bin is empty
    uint32_t nothing;        // 1: nothing to pack, every bin is empty
    int64_t coef_base[16];   // first element of each degree's bin in the bins region
};
static_assert(sizeof(UnevenHeader) <= 512, "header must fit its 512-byte slot");

constexpr size_t UNEVEN_HEADER_BYTES = 512;

__host__ __device__ inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct UnevenLayout {
    UnevenHeader *hdr;
    uint32_t *perm;
    char *bins;
};

struct UnevenArgs {
    const uint8_t *degrees;
    const int64_t *offsets;
    int64_t n;
    int64_t n_coeffs;
};

// A polynomial is solvable when its offsets hold exactly degree + 1
// coefficients, its degree is 1..12, and its roots fit the packed root array
// of n_coeffs - n elements: o0 >= i keeps root 0 (at o0 - i) at or above 0,
// o1 <= n_coeffs - (n - 1 - i) keeps its last root (at o1 - i - 2) below
// n_coeffs - n. The comparisons are ordered so that no difference overflows.
// These bounds hold for each polynomial alone; polynomials whose ranges
// overlap (offsets that are not monotone) are caught by the total the scan
// kernel checks.
__device__ __forceinline__ int checked_degree(const UnevenArgs &U, int64_t i, bool &consistent)
{
    int d = __ldg(U.degrees + i);
    int64_t o0 = __ldg(U.offsets + i), o1 = __ldg(U.offsets + i + 1);
    consistent = (o0 >= i) && (o1 >= o0) && (o1 <= U.n_coeffs - (U.n - 1 - i)) && (o1 - o0 == (int64_t)d + 1);
    return (consistent && d >= 1 && d <= UNEVEN_MAX_DEG) ? d : -1;
}

// NaN roots of polynomial i (its offsets passed checked_degree's bounds).
__device__ __forceinline__ void nan_roots(const UnevenArgs &U, int64_t i, double *roots)
{
    if (!roots) return;
    const int dd = __ldg(U.degrees + i);
    const int64_t r0 = __ldg(U.offsets + i) - i;
    const double q = __longlong_as_double(0x7ff8000000000000ll);
    for (int j = 0; j < dd; ++j) reinterpret_cast<double2 *>(roots)[r0 + j] = make_double2(q, q);
}

// Largest batch the uneven path takes: n < 2^32 polynomials (32-bit slots)
// and n_coeffs <= 2^40 coefficients, so that no workspace size wraps.
constexpr int64_t UNEVEN_MAX_N = (int64_t)1 << 32;
constexpr int64_t UNEVEN_MAX_COEFFS = (int64_t)1 << 40;

inline bool uneven_sizes_ok(int64_t n, int64_t n_coeffs)
{
    return n >= 0 && n < UNEVEN_MAX_N && n_coeffs >= 0 && n_coeffs <= UNEVEN_MAX_COEFFS;
}

inline size_t uneven_bytes(int64_t n, int64_t n_coeffs, size_t elem)
{
    return UNEVEN_HEADER_BYTES + align256((size_t)n * 4) + align256((size_t)n_coeffs * elem);
}

inline UnevenLayout uneven_layout(void *ws, int64_t n)
{
    char *p = reinterpret_cast<char *>(ws);
    UnevenLayout L;
    L.hdr = reinterpret_cast<UnevenHeader *>(p);
    L.perm = reinterpret_cast<uint32_t *>(p + UNEVEN_HEADER_BYTES);
    L.bins = p + UNEVEN_HEADER_BYTES + align256((size_t)n * 4);
    return L;
}

// Fork: helper streams of the calling host thread on the current device
// (created on their first use, non-blocking) made to wait for `st`; join:
// `st` made to wait for all of them. Both only record and wait on events, so
// they can be captured into a CUDA graph (as parallel branches).
constexpr int UNEVEN_SIDES = 11;
struct UnevenFork {
    int sides;  // streams forked
    cudaStream_t side[UNEVEN_SIDES];
    cudaEvent_t join[UNEVEN_SIDES];
};
int uneven_fork(cudaStream_t st, int sides, UnevenFork *out);
int uneven_join(cudaStream_t st, const UnevenFork &f);

// The split-register solver hands tasks of 32 polynomials between warps with
// waits that give up after 2 s (WS_WAIT_NS). A warp waits for about three
// tasks at most, and a sweep takes 3 us (degree 12, 1.1e6 sweeps per polynomial
// in 3.4 s), at the largest block less than 10, so at most 4,096 sweeps per
// polynomial (the defaults: 440 at degree 12) keep every wait below 0.15 s. A
// call that allows more takes the forms that wait for nothing.
inline bool split_waits_ok(int degree, int max_iters, int fixed_sweeps)
{
    return (int64_t)(degree - 1) * (fixed_sweeps > 0 ? fixed_sweeps : max_iters) <= 4096;
}

// Large bins: the split-register solver (rd_solve_split.cuh).
int launch_uneven_split(int degree, rd_dtype dt, const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets,
                        cudaStream_t st);
constexpr int UNEVEN_SPLIT = -1;  // in launch_uneven_bins' pw[d]
constexpr int SPLIT_DECLINED = 1;  // launch_solve_split, launch_uneven_split: nothing enqueued, take the one-role kernel

// Small batches: every polynomial by a group of lanes, no bins (rd_group.cu);
// asked = true: those degrees that the scan kernel has left it (hdr->direct).
int launch_uneven_group(const SolveArgs &a, rd_dtype dt, const UnevenArgs &U, const UnevenHeader *hdr, bool mixed,
                        bool asked, cudaStream_t st);
// The form of a packed batch: the degree bins, the group kernel, or both launched
// and the scan kernel deciding by degree, `lowest` and up (below it always groups).
struct UnevenForm {
    enum { bins, group, ask } form;
    int lowest;
};
UnevenForm uneven_form(int64_t n, bool mixed, bool compensated);

// Solve the degree bins of a packed batch from degree `lowest` up (one persistent
// kernel per degree, largest degree first, degree d on stream chain[d]) with
// the per-degree launch shapes block[d], cps[d], lanes per polynomial lanes[d]
// and polish warps pw[d] (> 0: the warp-specialised form, mixed mode, degrees up
// to 8; UNEVEN_SPLIT: the split-register form, degrees 4 to 12, compensated
// polish 7 to 11).
template <typename In, int MODE>
int launch_uneven_bins(const SolveArgs &a, const UnevenLayout &L, const int64_t *offsets, const int *block,
                       const int *cps, const int *lanes, const int *pw, int lowest, const cudaStream_t *chain);

// rd_roots_uneven's argument checks and launch (rd_abi.cu); fork = false
// keeps every degree bin on `stream` and makes no helper stream.
int roots_uneven_common(const void *coeffs, rd_dtype dtype, const uint8_t *degrees, const int64_t *offsets, int64_t n,
                        int64_t n_coeffs, rd_mode mode, const rd_params *params, const rd_uneven_tuning *tuning,
                        const rd_window *window, int W, int H, uint32_t *hist, double *roots, uint8_t *status,
                        rd_stats *stats, void *ws, size_t ws_bytes, bool fork, void *stream);

}  // namespace rd
