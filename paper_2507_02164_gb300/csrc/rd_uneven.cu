// rd_uneven.cu -- polynomials of uneven degree (1..12) in one pass: bin the
// batch by degree, then solve every bin with persistent kernels that pull
// 32-polynomial tasks from atomic queues.
//
// The paper solves one degree at a time (n <= 6, Sec. II-A, Table III). A
// batch of mixed degrees would otherwise run every polynomial at the largest
// degree's cost, or diverge inside warps; binning gives each warp one
// compile-time degree, so the Hessenberg matrix stays in registers.
//
// Workspace (caller-allocated, contents overwritten, 256-byte aligned):
//   [header 512 B][perm: uint32 per polynomial][bins: the coefficients again,
//   coefficient-major within each degree bin]
// Launch sequence (graph-capturable, no allocation, no synchronisation): clear
// header -> count, then for small batches one kernel that gives every polynomial
// a group of lanes (rd_group.cu), else scan -> pack -> one persistent solve kernel
// per degree, largest degree first, each with its own register allocation and
// its own task queue, on several chains of streams; in between both are launched
// and the scan chooses by the degrees that it has counted.
#include "rd_uneven.cuh"

#include <cuda.h>

namespace rd {

int launch_clear(uint32_t *p, int64_t words, cudaStream_t st);

// Count polynomials per degree; mark the unsolvable ones DEGENERATE (NaN
// roots where the offsets are consistent, nothing written where they are not).
__global__ void __launch_bounds__(256) uneven_count_kernel(UnevenArgs U, UnevenHeader *hdr, double *roots,
                                                           uint8_t *status, rd_stats *stats)
{
    __shared__ unsigned cnt[16];
    __shared__ unsigned long long acc[ST_WORDS];
    if (threadIdx.x < 16) cnt[threadIdx.x] = 0;
    const CtaStats S = stats_begin(acc, stats);  // synchronises the CTA
    __syncthreads();
    const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t warp_id = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    unsigned bad = 0, invalid = 0;
    for (int64_t base = warp_id * 32; base < U.n; base += warps_total * 32) {
        int64_t i = base + lane;
        if (i < U.n) {
            bool consistent;
            int d = checked_degree(U, i, consistent);
            if (d > 0) {
                atomicAdd(&cnt[d], 1u);
            } else {
                invalid += 1;
                bad += consistent ? 0u : 1u;
                if (status) status[i] = RD_STATUS_DEGENERATE;
                if (consistent) nan_roots(U, i, roots);
            }
        }
    }
    S.add(ST_POLYS, invalid);
    S.add(ST_STATUS0 + RD_STATUS_DEGENERATE, invalid);
    unsigned wb = __reduce_add_sync(0xffffffffu, bad);
    if (lane == 0 && wb) atomicAdd(&hdr->bad, wb);
    __syncthreads();
    if (threadIdx.x < 16 && cnt[threadIdx.x]) atomicAdd(&hdr->count[threadIdx.x], cnt[threadIdx.x]);
    stats_end(S, stats);
}

// Bin bases: poly_base[d] = sum of count[d'] for d' < d, coef_base[d] = sum
// of count[d'] (d' + 1). One warp. When the solvable polynomials need more
// than n_coeffs coefficients in all, their ranges overlap (offsets that are
// not monotone) and the bins would not fit the workspace: the batch is then
// not packed or solved (overflow = 1, every count 0), and the pack kernel
// marks its solvable polynomials DEGENERATE instead. ask > 0: only a degree from
// `ask` up that has more than a third of the solvable polynomials keeps its bin,
// the others go to the group kernel (direct, count 0, not packed).
__global__ void uneven_scan_kernel(UnevenHeader *hdr, int64_t n_coeffs, int ask)
{
    const int lane = threadIdx.x;
    unsigned c = lane < 16 ? hdr->count[lane] : 0u;
    int64_t e = lane < 16 ? (int64_t)c * (lane + 1) : 0;
    unsigned pc = c;
    int64_t pe = e;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        unsigned oc = __shfl_up_sync(0xffffffffu, pc, off);
        int64_t oe = __shfl_up_sync(0xffffffffu, pe, off);
        if (lane >= off) {
            pc += oc;
            pe += oe;
        }
    }
    const int64_t total = __shfl_sync(0xffffffffu, pe, 31);
    const bool overflow = total > n_coeffs;
    const uint64_t solvable = __shfl_sync(0xffffffffu, pc, 31);
    const bool grouped = ask && !overflow && !(lane >= ask && 3 * (uint64_t)c > solvable);
    const unsigned direct = __ballot_sync(0xffffffffu, grouped);
    const bool any = __any_sync(0xffffffffu, c && !grouped);
    if (lane < 16) {
        hdr->poly_base[lane] = pc - c;  // exclusive
        hdr->coef_base[lane] = pe - e;
        hdr->cursor[lane] = 0;
        hdr->head[lane] = 0;
        if (overflow || grouped) hdr->count[lane] = 0;
    }
    if (lane == 0) {
        hdr->overflow = overflow ? 1u : 0u;
        hdr->direct = direct;
        hdr->nothing = any ? 0u : 1u;
    }
}

// Scatter every solvable polynomial into its degree's bin: perm[slot] = its
// index, its coefficients coefficient-major at bins[coef_base[d] + k * count[d]
// + slot]. A CTA takes PACK_POLYS polynomials at a time, ranks them by degree in
// shared memory and reserves their slots with one atomic per degree on the
// bin's cursor: one per warp and degree (131,072 on each of eleven addresses
// for 2^22 polynomials) was what bounded the kernel (321 us; the whole call
// 7.90 -> 7.86 ms, its solvers start on the helper stream meanwhile).
constexpr int PACK_ROUNDS = 4, PACK_POLYS = 256 * PACK_ROUNDS;

template <typename E>
__global__ void __launch_bounds__(256) uneven_pack_kernel(UnevenArgs U, const E *__restrict__ coeffs,
                                                          UnevenHeader *hdr, uint32_t *perm, E *bins,
                                                          double *roots, uint8_t *status, rd_stats *stats)
{
    const int lane = threadIdx.x & 31;
    if (hdr->nothing) return;
    if (hdr->overflow) {
        const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
        const int64_t warp_id = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
        // overlapping ranges: nothing is packed; the solvable polynomials are
        // reported DEGENERATE with NaN roots (their own bounds hold)
        __shared__ unsigned long long acc[ST_WORDS];
        const CtaStats S = stats_begin(acc, stats);
        unsigned marked = 0;
        for (int64_t base = warp_id * 32; base < U.n; base += warps_total * 32) {
            int64_t i = base + lane;
            bool consistent;
            if (i < U.n && checked_degree(U, i, consistent) > 0) {
                marked += 1;
                if (status) status[i] = RD_STATUS_DEGENERATE;
                nan_roots(U, i, roots);
            }
        }
        S.add(ST_POLYS, marked);
        S.add(ST_STATUS0 + RD_STATUS_DEGENERATE, marked);
        stats_end(S, stats);
        return;
    }
    __shared__ unsigned cnt[16], first[16];
    const unsigned direct = hdr->direct;
    for (int64_t base = (int64_t)blockIdx.x * PACK_POLYS; base < U.n; base += (int64_t)gridDim.x * PACK_POLYS) {
        if (threadIdx.x < 16) cnt[threadIdx.x] = 0;
        __syncthreads();
        int deg[PACK_ROUNDS];
        unsigned rank[PACK_ROUNDS];
#pragma unroll
        for (int t = 0; t < PACK_ROUNDS; ++t) {
            const int64_t i = base + t * 256 + threadIdx.x;
            bool consistent;
            deg[t] = i < U.n ? checked_degree(U, i, consistent) : -1;
            if (deg[t] > 0 && ((direct >> deg[t]) & 1u)) deg[t] = -1;
            const unsigned act = __ballot_sync(0xffffffffu, deg[t] > 0);
            if (deg[t] > 0) {
                const unsigned peers = __match_any_sync(act, deg[t]);
                const int leader = __ffs(peers) - 1;
                unsigned b = 0;
                if (lane == leader) b = atomicAdd(&cnt[deg[t]], (unsigned)__popc(peers));
                rank[t] = __shfl_sync(peers, b, leader) + __popc(peers & ((1u << lane) - 1u));
            }
        }
        __syncthreads();
        if (threadIdx.x < 16 && cnt[threadIdx.x]) first[threadIdx.x] = atomicAdd(&hdr->cursor[threadIdx.x], cnt[threadIdx.x]);
        __syncthreads();
#pragma unroll
        for (int t = 0; t < PACK_ROUNDS; ++t) {
            const int64_t i = base + t * 256 + threadIdx.x;
            const int d = deg[t];
            if (d <= 0) continue;
            const unsigned slot = first[d] + rank[t], count = hdr->count[d];
            perm[hdr->poly_base[d] + slot] = (uint32_t)i;
            const E *src = coeffs + __ldg(U.offsets + i);
            E *dst = bins + hdr->coef_base[d] + slot;
            for (int k = 0; k <= d; ++k) dst[(int64_t)k * count] = __ldg(src + k);
        }
    }
}

namespace {
// Driver entry points (looked up at run time: the library links the runtime only).
template <typename F>
F driver_entry(const char *name)
{
    void *p = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &found) != cudaSuccess ||
        found != cudaDriverEntryPointSuccess)
        return nullptr;
    return reinterpret_cast<F>(p);
}

// The current context's id, unique for the life of the process (0: none). A
// device reset gives the next context another one; the handles of the old one may
// not even be looked at then.
unsigned long long context_id()
{
    static const auto get = driver_entry<CUresult (*)(CUcontext, unsigned long long *)>("cuCtxGetId");
    unsigned long long id = 0;
    return get && get(nullptr, &id) == CUDA_SUCCESS ? id : 0;
}

bool primary_context_active(int dev)
{
    static const auto get = driver_entry<CUresult (*)(CUdevice, unsigned *, int *)>("cuDevicePrimaryCtxGetState");
    unsigned flags = 0;
    int active = 0;
    return get && get(dev, &flags, &active) == CUDA_SUCCESS && active;
}

// The helper streams, the fork event and a join event for each, per device,
// owned by one host thread and released when that thread exits, unless their
// context is gone by then (errors ignored: at process exit the runtime may
// already be gone).
struct ForkState {
    int device = -1;
    unsigned long long context = 0;
    cudaStream_t side[UNEVEN_SIDES] = {};
    cudaEvent_t fork = nullptr, join[UNEVEN_SIDES] = {};
    void release()
    {
        if (fork) cudaEventDestroy(fork);
        for (int k = 0; k < UNEVEN_SIDES; ++k) {
            if (join[k]) cudaEventDestroy(join[k]);
            if (side[k]) cudaStreamDestroy(side[k]);
        }
    }
    void forget()
    {
        fork = nullptr;
        for (int k = 0; k < UNEVEN_SIDES; ++k) {
            join[k] = nullptr;
            side[k] = nullptr;
        }
    }
    ~ForkState()
    {
        if (!fork) return;
        int current = 0;
        if (context_id() == context) {
            release();
        } else if (primary_context_active(device) && cudaGetDevice(&current) == cudaSuccess && current != device) {
            if (cudaSetDevice(device) == cudaSuccess && context_id() == context) release();
            cudaSetDevice(current);
        }
    }
};
thread_local ForkState g_fork[64];
}  // namespace

// The calling host thread's handles on the current device, made on its first call.
static int uneven_handles(ForkState **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return rd_set_error(RD_ECUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
    if (dev < 0 || dev >= 64) return rd_set_error(RD_EUNSUPPORTED, "device index %d above 63", dev);
    ForkState &f = g_fork[dev];
    const unsigned long long context = context_id();
    if (f.fork && f.context != context) f.forget();  // made before a device reset
    if (!f.fork) {
        f.device = dev;
        f.context = context;
        // all or none: a partial failure releases what it made
        e = cudaEventCreateWithFlags(&f.fork, cudaEventDisableTiming);
        for (int k = 0; k < UNEVEN_SIDES && e == cudaSuccess; ++k) {
            e = cudaStreamCreateWithFlags(&f.side[k], cudaStreamNonBlocking);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&f.join[k], cudaEventDisableTiming);
        }
        if (e != cudaSuccess) {
            f.release();
            f.forget();
            return rd_set_error(RD_ECUDA, "uneven helper streams: %s (the first call on a device from a host thread "
                                          "creates them; make that call outside stream capture)",
                                cudaGetErrorString(e));
        }
    }
    *out = &f;
    return RD_OK;
}

int uneven_fork(cudaStream_t st, int sides, UnevenFork *out)
{
    ForkState *state = nullptr;
    int rc = uneven_handles(&state);
    if (rc) return rc;
    ForkState &f = *state;
    cudaError_t e = sides ? cudaEventRecord(f.fork, st) : cudaSuccess;
    for (int k = 0; k < sides && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(f.side[k], f.fork, 0);
    if (e != cudaSuccess) return rd_set_error(RD_ECUDA, "uneven fork: %s", cudaGetErrorString(e));
    out->sides = sides;
    for (int k = 0; k < sides; ++k) {
        out->side[k] = f.side[k];
        out->join[k] = f.join[k];
    }
    return RD_OK;
}

// The other helper streams wait for what the first one has to do so far.
static int uneven_follow(const UnevenFork &f)
{
    cudaError_t e = cudaEventRecord(f.join[0], f.side[0]);
    for (int k = 1; k < f.sides && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(f.side[k], f.join[0], 0);
    return e == cudaSuccess ? RD_OK : rd_set_error(RD_ECUDA, "uneven fork: %s", cudaGetErrorString(e));
}

int uneven_join(cudaStream_t st, const UnevenFork &f)
{
    for (int k = 0; k < f.sides; ++k) {
        cudaError_t e;
        if ((e = cudaEventRecord(f.join[k], f.side[k])) != cudaSuccess || (e = cudaStreamWaitEvent(st, f.join[k], 0)) != cudaSuccess)
            return rd_set_error(RD_ECUDA, "uneven join: %s", cudaGetErrorString(e));
    }
    return RD_OK;
}

size_t uneven_workspace_bytes(int64_t n, int64_t n_coeffs, rd_dtype dt)
{
    if (!uneven_sizes_ok(n, n_coeffs)) return 0;
    return uneven_bytes(n, n_coeffs, dt == RD_C64 ? 8 : 16);
}

// The chains of the degree bins: the caller's stream and helper streams, forked
// from it and joined back (under stream capture: parallel graph branches), so that
// other bins' kernels take over the SMs one bin's kernel leaves while its queue
// drains (a call that may not fork runs them all on the caller's stream). Bins that
// do not fill the chip are bound by the slowest warp of each kernel and want all
// twelve side by side; large ones want few kernels competing. Measured (us, degrees 2..12, complex64,
// FP64 polish; 2 / 4 / 12 chains): 50,000 680 / 536 / 364, 100,000 706 / 517 / 417,
// 200,000 852 / 619 / 598, 400,000 1075 / 984 / 1003, 2^22 7865 / 7739 / 8100. Degree
// d goes to chain d mod the number of chains, launched largest first. (Where the
// scan decides between the group kernel and the bins, the former has the caller's
// stream, the packing and the bins that may be asked for, at most two of them with
// work, three helper streams. Behind one another on one stream the empty ones take
// 5 us each.)
constexpr int UNEVEN_ASK_SIDES = 3;
static int uneven_sides(int64_t n) { return n <= (int64_t)1536 * rd_sm_count_cached() ? UNEVEN_SIDES : 3; }

// Whether the degree bins 4 to 12 (compensated polish 7 to 11) take the split-register solver
// (rd_solve_split.cuh) where the caller left their launch shapes open. The
// bins' sizes exist only on the device, so the line is drawn on n; each split
// kernel takes whole SMs, so small bins lose the overlap of the chains.
// Measured (us, degrees 2..12, complex64, split / one role): 300,000 1030 / 930,
// 2^19 1560 / 1430, 2^20 2385 / 2498, 2^22 7909 / 9357 (complex128 2574 / 2621,
// 8702 / 9864). Compensated polish: 2^20 1932 / 1888, 1,500,000 2583 / 2658,
// 2^22 6683 / 7323 (complex128 2196 / 2134, 2903 / 2978, 7572 / 8327).
static bool uneven_split_takes(int64_t n, bool mixed, int polish_mode)
{
    return mixed && n >= (int64_t)(polish_mode == RD_POLISH_DF ? 9216 : 6144) * rd_sm_count_cached();
}

int launch_uneven(const SolveArgs &a, rd_dtype dt, const uint8_t *degrees, const int64_t *offsets, int64_t n,
                  int64_t n_coeffs, bool mixed, void *ws, const int *block, const int *cps, const int *lanes,
                  const int *pw, bool fork, const bool *open_shape, cudaStream_t st)
{
    UnevenLayout L = uneven_layout(ws, n);
    UnevenArgs U{degrees, offsets, n, n_coeffs};
    int rc = launch_clear(reinterpret_cast<uint32_t *>(L.hdr), UNEVEN_HEADER_BYTES / 4, st);
    if (rc) return rc;
    const int tb = 256;
    int64_t ctas = (n + tb - 1) / tb;
    int64_t cap = (int64_t)rd_sm_count_cached() * 8;
    if (ctas > cap) ctas = cap;
    if (ctas < 1) ctas = 1;
    uneven_count_kernel<<<(unsigned)ctas, tb, 0, st>>>(U, L.hdr, a.roots, a.status, a.stats);
    if ((rc = rd_check_launch("uneven_count_kernel"))) return rc;
    // Roots that go over the coefficients: the bins read their own copy, the group
    // kernel would read the caller's array while other polynomials' roots are stored
    const int64_t n_roots = n_coeffs > n ? n_coeffs - n : 0;
    const uintptr_t c0 = reinterpret_cast<uintptr_t>(a.coeffs), r0 = reinterpret_cast<uintptr_t>(a.roots);
    const bool in_place = r0 && r0 < c0 + (uint64_t)n_coeffs * (dt == RD_C64 ? 8 : 16) && c0 < r0 + (uint64_t)n_roots * 16;
    bool all_open = true;
    for (int d = 1; d <= UNEVEN_MAX_DEG; ++d) all_open &= open_shape[d];
    UnevenForm F{UnevenForm::bins, 1};
    if (all_open && !in_place) F = uneven_form(n, mixed, a.polish_mode == RD_POLISH_DF);
    if (F.form == UnevenForm::group) {
        // the first call of a host thread, or after a device reset, makes the helper
        // streams whatever its size, so that a larger batch can be captured after it
        cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
        if (fork && cudaStreamIsCapturing(st, &capturing) == cudaSuccess && capturing == cudaStreamCaptureStatusNone) {
            UnevenFork none;
            if ((rc = uneven_fork(st, 0, &none))) return rc;
        }
        return launch_uneven_group(a, dt, U, L.hdr, mixed, false, st);
    }
    int bins_pw[16];
    const bool split = uneven_split_takes(n, mixed, a.polish_mode), df = a.polish_mode == RD_POLISH_DF;
    const int first = df ? 7 : 4, last = df ? 11 : UNEVEN_MAX_DEG;
    for (int d = 0; d < 16; ++d) {
        const bool takes = split && open_shape[d] && d >= first && d <= last && split_waits_ok(d, a.max_iters, a.fixed_sweeps);
        bins_pw[d] = takes ? UNEVEN_SPLIT : pw[d];
    }
    pw = bins_pw;
    const bool ask = F.form == UnevenForm::ask;
    uneven_scan_kernel<<<1, 32, 0, st>>>(L.hdr, n_coeffs, ask ? F.lowest : 0);
    if ((rc = rd_check_launch("uneven_scan_kernel"))) return rc;
    UnevenFork f;
    f.sides = 0;
    if (ask && fork && (rc = uneven_fork(st, UNEVEN_ASK_SIDES, &f))) return rc;
    if (ask) rc = launch_uneven_group(a, dt, U, L.hdr, mixed, true, st);
    cudaStream_t pack = f.sides ? f.side[0] : st;
    if (dt == RD_C64)
        uneven_pack_kernel<float2><<<(unsigned)ctas, tb, 0, pack>>>(U, reinterpret_cast<const float2 *>(a.coeffs), L.hdr,
                                                                    L.perm, reinterpret_cast<float2 *>(L.bins), a.roots,
                                                                    a.status, a.stats);
    else
        uneven_pack_kernel<double2><<<(unsigned)ctas, tb, 0, pack>>>(U, reinterpret_cast<const double2 *>(a.coeffs),
                                                                     L.hdr, L.perm, reinterpret_cast<double2 *>(L.bins),
                                                                     a.roots, a.status, a.stats);
    if (!rc) rc = rd_check_launch("uneven_pack_kernel");
    if (!rc && ask && f.sides) rc = uneven_follow(f);
    if (!rc && !ask && fork) {
        if ((rc = uneven_fork(st, uneven_sides(n), &f))) return rc;
    }
    cudaStream_t chain[UNEVEN_MAX_DEG + 1];
    for (int d = 1; d <= UNEVEN_MAX_DEG; ++d) {
        const int k = ask ? (f.sides ? 1 + d % f.sides : 0) : d % (f.sides + 1);  // 0: the caller's stream
        chain[d] = k ? f.side[k - 1] : st;
    }
    const int mode = !mixed ? MODE_PLAIN : (a.polish_mode == RD_POLISH_DF ? MODE_MIXED_DF : MODE_MIXED_FP64);
    auto bins = [&](auto launch) { return launch(a, L, offsets, block, cps, lanes, pw, F.lowest, chain); };
    if (rc) {
    } else if (dt == RD_C64) {
        if (mode == MODE_PLAIN) rc = bins(launch_uneven_bins<float2, MODE_PLAIN>);
        else if (mode == MODE_MIXED_DF) rc = bins(launch_uneven_bins<float2, MODE_MIXED_DF>);
        else rc = bins(launch_uneven_bins<float2, MODE_MIXED_FP64>);
    } else {
        if (mode == MODE_PLAIN) rc = bins(launch_uneven_bins<double2, MODE_PLAIN>);
        else if (mode == MODE_MIXED_DF) rc = bins(launch_uneven_bins<double2, MODE_MIXED_DF>);
        else rc = bins(launch_uneven_bins<double2, MODE_MIXED_FP64>);
    }
    const int rj = f.sides ? uneven_join(st, f) : RD_OK;
    return rc ? rc : rj;
}

}  // namespace rd
