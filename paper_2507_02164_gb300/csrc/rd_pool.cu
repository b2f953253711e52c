// rd_pool.cu -- RD_PLAIN_FP64 solver for large uniform batches: every warp
// sweeps a pool of polynomials that it keeps in shared memory.
//
// The FP64 sweeps are bound by the FP64 unit, of which each SM sub-partition
// has its own: a warp instruction takes it 67.5 cycles whatever number of lanes
// is active, and one warp keeps it busy. In the one-lane-per-polynomial kernel
// (rd_solve.cuh) a lane whose polynomial is done stays idle until the warp's
// slowest is, a lane with a small active block rides in the largest block's
// sweep, and 65,536 polynomials are 3.4 warps per sub-partition, the time of
// four. Beside that, moving a matrix is free: a sweep of a 6 x 6 block takes
// some 50,000 cycles, its load from and store to shared memory about 500.
// So there is one warp per sub-partition (two where the batch fills their pools,
// launch_pool_n), with an equal share of the batch in shared memory (up to 135
// polynomials of degree 6), and before each sweep it takes the 32 largest active
// blocks. Simulated for degree 6 and a pool of 108:
// 18.4 warp sweeps per 32 polynomials instead of 21.5 (mean of a polynomial:
// 16.8), and 0.85 of the FP64 instructions. Every polynomial takes the same
// steps in the same order as in sweep_lane: the same bits and counters.
// Measured (us, degree 6, complex128, roots drawn from the disk): 65,536 1468 ->
// 1218, 40,000 1171 -> 817, 2^18 5168 -> 4676. Two warps that share one pool by
// compare-and-swap: 1202, 922, 4716; eight on one pool per SM: 1248, 1006, 4703:
// within the FP64 time of the sweeps that they save or add.
#include "rd_solve.cuh"

namespace rd {

template <int N, int W>
struct Pool {
    static constexpr int ENTRIES = N * (N + 1) / 2 + N - 1;  // of an upper Hessenberg matrix
    static constexpr int SLOT_BYTES = 16 * ENTRIES + 8;
    static constexpr int WARPS = W;                          // of a CTA, one CTA per SM
    static constexpr int FIT = 225 * 1024 / WARPS / SLOT_BYTES;
    static constexpr int SLOTS = FIT < 160 ? FIT : 160;
};

// A polynomial's place in the iteration, beside its matrix.
constexpr int POOL_M = 0xff, POOL_NOT_CONV = 0x100, POOL_DEGENERATE = 0x200;

// The step before each sweep of sweep_lane: deflate by one if the bottom
// subdiagonal is negligible, or give it up after max_iters sweeps.
template <int N>
__device__ __forceinline__ void pool_deflate(const SolveArgs &A, const cx<double> (&h)[N][N], int &m, int &its, int &flags)
{
    if (m < 2) return;
    cx<double> ta, tb, tc, td;
    trailing<N, double>(h, m, ta, tb, tc, td);
    const bool small = deflates(A, (double)A.tol, its, ta, tc, td);
    if (small || its >= A.max_iters) {
        if (!small) flags |= POOL_NOT_CONV;
        m -= 1;
        its = 0;
    }
}

template <int N, int W, typename In>
__global__ void __launch_bounds__(32 * W, 1) pool_kernel(SolveArgs A, int slots, int rounds)
{
    extern __shared__ __align__(16) double2 pool_smem[];
    __shared__ unsigned long long acc[ST_WORDS];
    __shared__ int lists[Pool<N, W>::WARPS][32];
    const CtaStats S = stats_begin(acc, A.stats);
    const UniformMap map{{}, A.n};
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double2 *ent = pool_smem + (size_t)warp * Pool<N, W>::ENTRIES * slots;  // entry e of slot p at e * slots + p
    int *state = reinterpret_cast<int *>(pool_smem + (size_t)Pool<N, W>::WARPS * Pool<N, W>::ENTRIES * slots) + warp * 2 * slots;
    int *sweeps_made = state + slots;
    int *list = lists[warp];
    const int64_t warps = (int64_t)gridDim.x * Pool<N, W>::WARPS, w = blockIdx.x + (int64_t)gridDim.x * warp;

    auto put = [&](const cx<double> (&h)[N][N], int p, int m, int its, int flags) {
        int e = 0;
#pragma unroll
        for (int r = 0; r < N; ++r)
#pragma unroll
            for (int j = r ? r - 1 : 0; j < N; ++j) ent[e++ * slots + p] = make_double2(h[r][j].re, h[r][j].im);
        state[p] = m | flags;
        sweeps_made[p] = its;
    };

    for (int round = 0; round < rounds; ++round) {
        const int64_t base = ((int64_t)round * warps + w) * slots;
        const int count = base >= A.n ? 0 : (A.n - base < slots ? (int)(A.n - base) : slots);
        if (count == 0) break;
        // ---- the companion matrices
        for (int q = 0; q < count; q += 32) {
            const int p = q + lane;
            cx<double> b[N], h[N][N];
            const bool degenerate = load_monic<N, double, In, MODE_PLAIN>(A.coeffs, A.n, p < count ? base + p : A.n, b);
#pragma unroll
            for (int r = 0; r < N; ++r)
#pragma unroll
                for (int j = 0; j < N; ++j) h[r][j] = {0.0, 0.0};
#pragma unroll
            for (int r = 0; r + 1 < N; ++r) h[r + 1][r] = {1.0, 0.0};
#pragma unroll
            for (int r = 0; r < N; ++r) h[r][N - 1] = degenerate ? cx<double>{0.0, 0.0} : cx<double>{-b[r].re, -b[r].im};
            int m = degenerate ? 0 : N, its = 0, flags = degenerate ? POOL_DEGENERATE : 0;
            pool_deflate<N>(A, h, m, its, flags);
            if (p < count) put(h, p, m, its, flags);
        }
        __syncwarp();
        // ---- sweeps, the 32 largest active blocks at a time
        unsigned n_sweeps = 0, n_pairs = 0, n_rots = 0;
        for (;;) {
            int filled = 0, M = 0;
            for (int level = N; level >= 2 && filled < 32; --level) {
                for (int q = 0; q < count && filled < 32; q += 32) {
                    const int p = q + lane;
                    const bool is = p < count && (state[p] & POOL_M) == level;
                    const unsigned votes = __ballot_sync(0xffffffffu, is);
                    if (votes && !M) M = level;
                    const int rank = filled + __popc(votes & ((1u << lane) - 1u));
                    if (is && rank < 32) list[rank] = p;
                    filled += __popc(votes);
                }
            }
            if (filled == 0) break;
            __syncwarp();
            // lanes without a block of their own go along with the first one's
            // values (m = 0): zeros would take the slow paths of / and sqrt
            const bool own = lane < filled;
            const int p = list[own ? lane : 0];
            cx<double> h[N][N];
            int e = 0;
#pragma unroll
            for (int r = 0; r < N; ++r)
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    if (j + 1 < r) {
                        h[r][j] = {0.0, 0.0};
                    } else {
                        const double2 v = ent[e++ * slots + p];
                        h[r][j] = {v.x, v.y};
                    }
                }
            int m = own ? state[p] & POOL_M : 0, its = own ? sweeps_made[p] : 0, flags = state[p] & ~POOL_M;
            __syncwarp();
            cx<double> ta, tb, tc, td;
            trailing<N, double>(h, m >= 2 ? m : 2, ta, tb, tc, td);
            const cx<double> shift = pick_shift(A, its, ta, tb, tc, td);
            qr_sweep<N, double>(h, m, M, shift);
            if (own) {
                its += 1;
                n_sweeps += 1;
                n_pairs += (unsigned)(m * (m + 1) - 2);
                n_rots += (unsigned)(m - 1);
                pool_deflate<N>(A, h, m, its, flags);
                put(h, p, m, its, flags);
            }
            __syncwarp();
        }
        // A lane's own sums of a round fit 32 bits (at most 100,000 sweeps per
        // eigenvalue: 3.3e9 flops at degree 7), a pool's do not
        S.add_wide(ST_SWEEPS, n_sweeps);
        S.add_wide(ST_PAIRS, n_pairs);
        S.add_wide(ST_ROTS, n_rots);
        S.add_wide(ST_F64, 20u * n_pairs + 24u * n_rots + 60u * n_sweeps);
        // ---- the roots: the diagonals
        for (int q = 0; q < count; q += 32) {
            const int p = q + lane;
            cx<double> d[N];
            int e = 0;
#pragma unroll
            for (int r = 0; r < N; ++r) {
                const double2 v = p < count ? ent[(e + (r ? 1 : 0)) * slots + p] : make_double2(0.0, 0.0);
                d[r] = {v.x, v.y};
                e += r ? N - r + 1 : N;
            }
            const int flags = p < count ? state[p] : POOL_DEGENERATE;
            finish_lane<N, double, In, MODE_PLAIN>(A, A.coeffs, A.n, p < count ? base + p : A.n, map, S, d,
                                                   flags & POOL_DEGENERATE, flags & POOL_NOT_CONV);
        }
        __syncwarp();
    }
    stats_end(S, A.stats);
}

// A batch of n in equal shares: as many rounds as the slots ask for.
template <int N, int W>
static void pool_shares(int64_t n, int64_t &rounds, int64_t &slots)
{
    const int64_t warps = (int64_t)rd_sm_count_cached() * W, most = Pool<N, W>::SLOTS;
    rounds = (n + warps * most - 1) / (warps * most);
    slots = (n + warps * rounds - 1) / (warps * rounds);
}

template <int N, int W, typename In>
static int launch_pool_warps(const SolveArgs &a, cudaStream_t st)
{
    using C = Pool<N, W>;
    int64_t rounds, slots;
    pool_shares<N, W>(a.n, rounds, slots);
    auto kern = pool_kernel<N, W, In>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, W * C::SLOT_BYTES * C::SLOTS) != cudaSuccess)
        return rd_check_launch("cudaFuncSetAttribute(pool_kernel)");
    kern<<<(unsigned)rd_sm_count_cached(), 32 * W, (size_t)(W * C::SLOT_BYTES * slots), st>>>(a, (int)slots, (int)rounds);
    return rd_check_launch("pool_kernel");
}

// Two warps per sub-partition hide what a lone one waits for (selection, matrix
// moves, square roots) but halve the pools: taken where a pool still holds one and
// a half warps' worth. Measured (us, complex128, one / two): 42 to 43 slots degree
// 6 100,003 1911 / 2108, 7 2348 / 2353; 54 slots 6 65,536 1238 / 1218, 2^18 4732 /
// 4676; 80 and more 3 2^18 713 / 666, 4 100,003 614 / 564, 5 100,003 1041 / 953.
template <int N, typename In>
static int launch_pool_n(const SolveArgs &a, cudaStream_t st)
{
    int64_t rounds, slots;
    pool_shares<N, 8>(a.n, rounds, slots);
    return slots >= 48 ? launch_pool_warps<N, 8, In>(a, st) : launch_pool_warps<N, 4, In>(a, st);
}

// Degree 8 (83 polynomials fit, the sweep spills) gains less than it loses at
// the next size (2^9 per SM 2595 us against 2529), degree 9 and up lose.
template <typename In>
static int launch_pool_degree(int degree, const SolveArgs &a, cudaStream_t st)
{
    switch (degree) {
    case 3: return launch_pool_n<3, In>(a, st);
    case 4: return launch_pool_n<4, In>(a, st);
    case 5: return launch_pool_n<5, In>(a, st);
    case 6: return launch_pool_n<6, In>(a, st);
    case 7: return launch_pool_n<7, In>(a, st);
    default: return rd_set_error(RD_EUNSUPPORTED, "pool solver: degree %d not built (3..7)", degree);
    }
}

int launch_pool(int degree, rd_dtype dt, const SolveArgs &a, cudaStream_t st)
{
    return dt == RD_C64 ? launch_pool_degree<float2>(degree, a, st) : launch_pool_degree<double2>(degree, a, st);
}

}  // namespace rd
