// rd_solve_split.cuh -- warp-specialised RD_MIXED solver whose two roles have
// register shares of their own (setmaxnreg).
//
// GB300's FP64 unit belongs to an SM sub-partition, takes 67.5 cycles per warp
// instruction, and one warp with a single dependent chain keeps it busy. What
// leaves it idle is a sub-partition none of whose warps is polishing. The
// sweeps want the opposite of the polish: registers (the Hessenberg matrix)
// and two warps per sub-partition for their latency, where the polish wants
// little state and enough warps to cover its FP32 part. With one register
// count for both roles (rd_solve_ws.cuh) degrees 9 and up have 8 warps per SM,
// one of each role per sub-partition, and lose to the one-role kernel.
// Here the sweep warps take the registers that the polish warps give up: the
// polish (finish_lean) keeps its polynomial's coefficients and roots in shared
// memory. The ring, its tickets and bounded waits are rd_solve_ws.cuh's; the
// arithmetic is finish_lane's, operation for operation, so roots, status,
// histogram and counters are the same bits.
#pragma once

#include "rd_solve_ws.cuh"
#include "rd_uneven.cuh"

namespace rd {

// Warps of each role, registers of a polish warp and ring slots, by degree
// (multiples of four warps: setmaxnreg works on warpgroups, and a warpgroup
// has one warp in each sub-partition); the sweep warps share what the polish
// warps leave of the launch's registers. Measured on complex64 (us, 2^19
// complex-Gaussian polynomials; degree 6 also 2^23 Littlewood), sweep warps /
// polish warps / polish registers:
//   4: 8/16/48 251, 8/12/56 260, 8/8/64 305     5: 8/12/64 378, 8/16/56 381, 8/8/64 435
//   6: 12/16/48 527, 7972; 8/12/64 542, 8232; 8/16/56 529, 9309; 8/8/80 592, 8889
//   7: 8/12/56 718, 8/8/72 773     8: 8/12/48 964, 8/8/72 996, 12/4/80 1507
//   9: 8/8/72 1254, 8/4/88 1906   10: 8/8/72 1510, 8/4/88 2343
//  11: 8/8/56 1901, 8/8/64 2007 (the sweeps spill 172 B), 8/4/88 2817
//  12: 8/8/40 with 12 slots 2817 (what shared memory leaves of L1 holds the
//      sweeps' spills), with 32 slots 3504; 8/4/72 3377
// One polish warp per sub-partition is not enough for any degree (its FP32
// part idles the FP64 unit half of the time); the sweeps need two.
struct SplitShape {
    int sweep, polish, polish_regs, slots;
};
__host__ __device__ constexpr SplitShape split_shape(int n)
{
    return n == 4   ? SplitShape{8, 16, 48, 48}
           : n == 5 ? SplitShape{8, 12, 64, 40}
           : n == 6 ? SplitShape{12, 16, 48, 32}
           : n == 7 ? SplitShape{8, 12, 56, 40}
           : n == 8 ? SplitShape{8, 12, 48, 40}
           : n <= 10 ? SplitShape{8, 8, 72, 32}
           : n == 11 ? SplitShape{8, 8, 56, 16}
                     : SplitShape{8, 8, 40, 12};
}

// The same for the compensated polish, whose work is FP32 like the sweeps':
// what the split gives it is eight sweep warps with the registers they want
// beside eight that need few, where the one-role kernel has 8 to 12 in all.
// Measured as above (2^19, complex64; one role 7 711, 8 1010, 9 1302, 10 1620,
// 11 1901, 12 2448):
//   7: 8/8/72 652, 12/8/72 716, 8/12/64 774     8: 8/8/72 875, 12/8/72 919, 8/12/64 947
//   9: 8/8/64 1069, 8/8/72 1074, 8/8/48 1088   10: 8/8/64 1286, 8/8/72 1303, 8/8/40 1347
//  11: 8/8/40 1680, 8/8/48 1709, 8/8/56 1815, 8/8/64 1960 (the sweeps spill)
// Degree 12 spills in every split (2614 the best), and 4 to 6 already have
// sixteen warps in one role: not built.
__host__ __device__ constexpr SplitShape split_shape_df(int n)
{
    return n <= 8    ? SplitShape{8, 8, 72, 24}
           : n <= 10 ? SplitShape{8, 8, 64, 24}
                     : SplitShape{8, 8, 40, 16};
}

// The degrees each polish is built for.
__host__ __device__ constexpr bool split_built(int n, int mode)
{
    return mode == MODE_MIXED_DF ? n >= 7 && n <= 11 : n >= 4 && n <= 12;
}

template <int N, int MODE>
struct Split {
    static constexpr SplitShape shape = MODE == MODE_MIXED_DF ? split_shape_df(N) : split_shape(N);
    static constexpr int SWEEP = shape.sweep, POLISH = shape.polish, POLISH_REGS = shape.polish_regs, SLOTS = shape.slots;
    static constexpr int THREADS = 32 * (SWEEP + POLISH);
    static constexpr int LAUNCH_REGS = 65536 / THREADS / 8 * 8;
    static constexpr int SWEEP_REGS = ((SWEEP + POLISH) * LAUNCH_REGS - POLISH * POLISH_REGS) / SWEEP / 8 * 8;
    static_assert(SWEEP % 4 == 0 && POLISH % 4 == 0, "whole warpgroups");
    static_assert(POLISH_REGS % 8 == 0 && POLISH_REGS <= LAUNCH_REGS && LAUNCH_REGS <= SWEEP_REGS && SWEEP_REGS <= 256, "");
    static_assert(SWEEP * SWEEP_REGS + POLISH * POLISH_REGS <= (SWEEP + POLISH) * LAUNCH_REGS,
                  "the shares must fit the registers of the launch, or setmaxnreg.inc waits forever");
    static_assert(split_built(N, MODE), "");
    static_assert(SLOTS > POLISH && SLOTS <= WS_MAX_SLOTS, "a polish warp keeps its slot until it has finished it");
};

// A polish warp's shared memory: lane-major, one 8- or 16-byte access per
// lane and value, 256 or 512 contiguous bytes per warp.
template <int N, bool LO>
struct LeanMem {
    double2 ad[N + 1][32];              // coefficients in FP64 (complex128: scaled by a power of two)
    double2 z[N][32];                   // polished roots
    float2 af[N + 1][32];               // coefficients in FP32
    float2 alo[LO ? N + 1 : 1][LO ? 32 : 1];  // what FP32 leaves of them (compensated polish, complex128)
};
template <typename In, int MODE>
constexpr bool lean_lo = MODE == MODE_MIXED_DF && !std::is_same<In, float2>::value;
template <int N, typename In, int MODE>
constexpr size_t lean_bytes = (sizeof(LeanMem<N, lean_lo<In, MODE>>) + 15) / 16 * 16;

template <int N, typename In, int MODE>
__host__ __device__ constexpr size_t split_smem_bytes()
{
    return ws_smem_bytes(N, Split<N, MODE>::SLOTS) + (size_t)Split<N, MODE>::POLISH * lean_bytes<N, In, MODE>;
}

// finish_lane (either polish) for the eigenvalues in `slot`, its
// coefficients and roots in `mem`. All 32 lanes of the warp call it together;
// the slot's eigenvalues are overwritten (by the FP32 copies of the roots).
template <int N, typename In, int MODE, class Map>
__device__ __forceinline__ void finish_lean(const SolveArgs &A, const void *coeffs, int64_t n, int64_t i,
                                            const Map &map, const CtaStats &S, WsSlot<N> &slot,
                                            LeanMem<N, lean_lo<In, MODE>> &mem, bool degenerate, bool not_conv)
{
    constexpr bool DF = MODE == MODE_MIXED_DF, LO = lean_lo<In, MODE>;
    constexpr bool C64 = std::is_same<In, float2>::value;
    const int lane = threadIdx.x & 31;
    const bool valid = i < n;
    uint8_t st = degenerate ? RD_STATUS_DEGENERATE : (not_conv ? RD_STATUS_NOT_CONVERGED : RD_STATUS_OK);
    unsigned newton = 0, extra = 0;  // extra: steps taken for any of the warp's polynomials
    const bool polish = A.polish_steps > 0 || A.polish_extra > 0;
    auto ad = [&](int k) -> cx<double> {
        const double2 v = mem.ad[k][lane];
        return {v.x, v.y};
    };
    auto af = [&](int k) -> cx<float> {
        const float2 v = mem.af[k][lane];
        return {v.x, v.y};
    };
    auto root = [&](int j) -> cx<double> {
        const double2 v = mem.z[j][lane];
        return {v.x, v.y};
    };
    auto eigenvalue = [&](int j) -> cx<float> {
        const float2 v = slot.d[j][lane];
        return {v.x, v.y};
    };
    if (!polish || __all_sync(0xffffffffu, degenerate)) {
#pragma unroll 1
        for (int j = 0; j < N; ++j) {
            const cx<double> z = f2d(eigenvalue(j));
            mem.z[j][lane] = make_double2(z.re, z.im);
        }
    } else {
        if constexpr (C64) {
#pragma unroll
            for (int k = 0; k <= N; ++k) {
                const cx<float> a = !degenerate ? InLoad<In>::ldf(coeffs, (int64_t)k * n + i) : cx<float>{k == N ? 1.0f : 0.0f, 0.0f};
                const cx<double> w = f2d(a);
                mem.af[k][lane] = make_float2(a.re, a.im);
                mem.ad[k][lane] = make_double2(w.re, w.im);
            }
        } else {
            unsigned emax = 0;
#pragma unroll
            for (int k = 0; k <= N; ++k) {
                const cx<double> a = !degenerate ? InLoad<In>::ld(coeffs, (int64_t)k * n + i) : cx<double>{k == N ? 1.0 : 0.0, 0.0};
                emax = max(emax, max(exponent_bits(a.re), exponent_bits(a.im)));
                mem.ad[k][lane] = make_double2(a.re, a.im);
            }
            const double f = pow2_scale(emax);
#pragma unroll
            for (int k = 0; k <= N; ++k) {
                cx<double> a = ad(k);
                a = {a.re * f, a.im * f};
                mem.ad[k][lane] = make_double2(a.re, a.im);
                const cx<float> h = d2f(a);
                mem.af[k][lane] = make_float2(h.re, h.im);
                if constexpr (LO) mem.alo[k][lane] = make_float2(d2f(a.re - f2d(h.re)), d2f(a.im - f2d(h.im)));
            }
        }
        const float rtol = A.residual_tol > 0 ? (float)A.residual_tol : (float)(64.0 * N * 0x1p-53);
        auto weight = [&](float az) {
            float den = abs1(af(N));
#pragma unroll
            for (int k = N - 1; k >= 0; --k) den = fmaf(den, az, abs1(af(k)));
            return den;
        };
        auto horner = [&](cx<double> z) {
            cx<double> p = ad(N);
#pragma unroll
            for (int k = N - 1; k >= 0; --k) p = cfma(p, z, ad(k));
            return p;
        };
        auto passes = [&](cx<double> p, cx<double> z) {
            const float den = weight(sqrtf(norm2(d2f(z))));
            return (sqrtf(norm2(d2f(p))) <= rtol * den) && finite_bits(z.re) && finite_bits(z.im);
        };
        unsigned failed = 0;  // bit j: root j failed the residual test
#pragma unroll 1
        for (int j = 0; j < N; ++j) {
            cx<float> zf = eigenvalue(j);
            cx<double> zj;
            bool good = false;
            if constexpr (DF) {
                cx<float> zl = {0.0f, 0.0f};
                auto lo = [&](int k) -> cx<float> {
                    if constexpr (LO) return {mem.alo[k][lane].x, mem.alo[k][lane].y};
                    return {0.0f, 0.0f};
                };
#pragma unroll 1
                for (int step = 0; step < A.polish_steps; ++step) {
                    asm volatile("" ::: "memory");  // the coefficients stay in shared memory
                    CompHorner ch(zf, af(N), lo(N));
#pragma unroll
                    for (int k = N - 1; k >= 0; --k) ch.step<LO>(af(k), lo(k));
                    if (!ch.newton(zf, zl)) break;
                    newton += 1;
                }
                zj = {f2d(zf.re) + f2d(zl.re), f2d(zf.im) + f2d(zl.im)};
            } else {
                zj = f2d(zf);
                float moved = CUDART_INF_F;
#pragma unroll 1
                for (int step = 0; step < A.polish_steps; ++step) {
                    asm volatile("" ::: "memory");  // the coefficients stay in shared memory
                    // p in FP64 and, in its shadow, p' in FP32
                    cx<double> p = ad(N);
                    cx<float> pf = af(N), dp = {0.0f, 0.0f};
#pragma unroll
                    for (int k = N - 1; k >= 0; --k) {
                        p = cfma(p, zj, ad(k));
                        dp = cfma(dp, zf, pf);
                        pf = cfma(pf, zf, af(k));
                    }
                    const cx<float> dz = cdiv(d2f(p), dp);
                    if (!finite_c(dz)) break;
                    zj = sub(zj, f2d(dz));
                    zf = sub(zf, dz);
                    moved = abs1(dz);
                    newton += 1;
                }
                const cx<float> zr = d2f(zj);
                const float az = sqrtf(norm2(zr));
                good = residual_certain(N, moved, abs1(sub(zr, zf)), az, weight(az), abs1(af(N)), rtol);
            }
            if (!__all_sync(0xffffffffu, good || degenerate)) good = passes(horner(zj), zj);
            failed |= (good ? 0u : 1u) << j;
            mem.z[j][lane] = make_double2(zj.re, zj.im);
        }
        if (degenerate) failed = 0;
        if (A.polish_extra > 0 && __any_sync(0xffffffffu, failed != 0)) {
            // Further steps with p and p' both in FP64. The failed roots of the
            // whole warp go to one lane each, whichever polynomial they belong to
            // (everything they need is in shared memory): a warp whose polynomials
            // fail on all roots takes one pass instead of N (129,600 sub-disks of
            // the full pipeline, some 100 of whose 4,050 warps have rejected
            // polynomials: the solve 484 -> 470 us, about 1 % of the whole call). The slot's eigenvalues are no longer
            // needed; it holds the list (lane, root).
            unsigned *list = reinterpret_cast<unsigned *>(&slot.d[0][0]);
            unsigned at = __popc(failed);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned v = __shfl_up_sync(0xffffffffu, at, o);
                at += lane >= o ? v : 0u;
            }
            const unsigned total = __shfl_sync(0xffffffffu, at, 31);
            const unsigned begin = at - __popc(failed);
            __syncwarp();
            at = begin;
            for (unsigned m = failed; m; m &= m - 1u) list[at++] = (unsigned)lane | ((unsigned)(__ffs(m) - 1) << 8);
            __syncwarp();
#pragma unroll 1
            for (unsigned t = lane; t < total; t += 32) {
                const int l = (int)(list[t] & 31u), j = (int)(list[t] >> 8);
                auto adl = [&](int k) -> cx<double> { return {mem.ad[k][l].x, mem.ad[k][l].y}; };
                cx<double> zj = {mem.z[j][l].x, mem.z[j][l].y};
                bool good = false;
                for (int it = 0; !good && it < A.polish_extra; ++it) {
                    cx<double> p = adl(N), dp = {0.0, 0.0};
#pragma unroll 1
                    for (int k = N - 1; k >= 0; --k) {
                        dp = cfma(dp, zj, p);
                        p = cfma(p, zj, adl(k));
                    }
                    const cx<double> dz = cdiv(p, dp);
                    if (!(finite_bits(dz.re) && finite_bits(dz.im))) break;
                    zj = sub(zj, dz);
                    extra += 1;
                    cx<double> q = adl(N);
                    const float az = sqrtf(norm2(d2f(zj)));
                    float den = abs1(cx<float>{mem.af[N][l].x, mem.af[N][l].y});
#pragma unroll 1
                    for (int k = N - 1; k >= 0; --k) {
                        q = cfma(q, zj, adl(k));
                        den = fmaf(den, az, abs1(cx<float>{mem.af[k][l].x, mem.af[k][l].y}));
                    }
                    good = (sqrtf(norm2(d2f(q))) <= rtol * den) && finite_bits(zj.re) && finite_bits(zj.im);
                }
                mem.z[j][l] = make_double2(zj.re, zj.im);
                list[t] = good ? 1u : 0u;
            }
            __syncwarp();
            at = begin;
            for (unsigned m = failed; m; m &= m - 1u) failed &= ~(list[at++] << (__ffs(m) - 1));
            __syncwarp();
        }
        bool reject = failed != 0;
        // separation: the FP32 screen, then the FP64 test where a lane needs it
#pragma unroll 1
        for (int j = 0; j < N; ++j) {
            const cx<float> z = d2f(root(j));
            slot.d[j][lane] = make_float2(z.re, z.im);
        }
        const float screen = fmaxf(1e-4f, 2.0f * (float)A.collapse_tol);
        bool near = false;
#pragma unroll 1
        for (int j = 0; j + 1 < N; ++j) {
            const cx<float> z = eigenvalue(j);
            const float lim = screen * fmaxf(1.0f, abs1(z));
            for (int k = j + 1; k < N; ++k) near |= abs1(sub(z, eigenvalue(k))) <= lim;
        }
        if (__any_sync(0xffffffffu, near) && near) {
#pragma unroll 1
            for (int j = 0; j + 1 < N; ++j) {
                const cx<double> z = root(j);
                const double lim = A.collapse_tol * fmax(1.0, fabs(z.re) + fabs(z.im));
#pragma unroll 1
                for (int k = j + 1; k < N; ++k) {
                    const cx<double> d = sub(z, root(k));
                    reject |= (fabs(d.re) + fabs(d.im)) <= lim;
                }
            }
        }
        if (reject && st == RD_STATUS_OK && !degenerate) st = RD_STATUS_REJECTED;
    }
    const unsigned nw = (degenerate ? 0u : newton) + extra, nr = (degenerate || !polish) ? 0u : (unsigned)N;
    S.add(ST_NEWTON, nw);
    if constexpr (DF) {
        S.add(ST_F64, (8u * N + 6u) * nr);
        S.add(ST_F32, (66u * N + 50u) * nw + (2u * N + 4u) * nr);
    } else {
        S.add(ST_F64, (8u * N + 2u) * nw + (8u * N + 4u) * nr);
        S.add(ST_F32, (8u * N + 3u) * nw + (2u * N + 4u) * nr);
    }
    S.add(ST_POLYS, valid ? 1u : 0u);
#pragma unroll
    for (int k = 0; k < 4; ++k) S.add(ST_STATUS0 + k, (valid && st == k) ? 1u : 0u);
    const int64_t pid = valid ? map.poly(i) : 0;
    if (valid && A.status) A.status[pid] = st;

    // ---- store and bin the roots
    cx<double> cen = {0.0, 0.0};
    int64_t my_tile = pid;
    if (A.hist && A.clip_on && valid) {
        cen = map.centre(A, pid);
        my_tile = map.tile(A, pid);
    }
    unsigned n_clipped = 0, n_binned = 0, n_oow = 0;
#pragma unroll 1
    for (int j = 0; j < N; ++j) {
        cx<double> z = root(j);
        if (degenerate) z = {__longlong_as_double(0x7ff8000000000000ll), __longlong_as_double(0x7ff8000000000000ll)};
        if (A.roots && valid) reinterpret_cast<double2 *>(A.roots)[map.root(pid, j)] = make_double2(z.re, z.im);
        if (A.hist) {
            double x = z.re, y = z.im;
            bool keep = valid;
            if (A.clip_on) {
                x = __dadd_rn(__dmul_rn(A.radius, x), cen.re);
                y = __dadd_rn(__dmul_rn(A.radius, y), cen.im);
                const int t = pixel_of(A.tiles, x, y);
                const bool in_tile = (t >= 0) && ((int64_t)t == my_tile);
                n_clipped += (valid && !in_tile) ? 1u : 0u;
                keep = keep && in_tile;
            }
            const int pix = keep ? pixel_of(A.bin, x, y) : -1;
            n_binned += (pix >= 0) ? 1u : 0u;
            n_oow += (keep && pix < 0) ? 1u : 0u;
            hist_add(A.hist, pix);
        }
    }
    if (A.hist) {
        S.add(ST_CLIPPED, n_clipped);
        S.add(ST_BINNED, n_binned);
        S.add(ST_OOW, n_oow);
    }
}

// One CTA of the split form over a coefficient-major batch (ws_cta's tasks
// and ring): warps 0 .. POLISH-1 polish, the others sweep.
template <int N, typename In, int MODE, class Map>
__device__ __forceinline__ void split_cta(const SolveArgs &A, const void *coeffs, int64_t n, const Map &map)
{
    using C = Split<N, MODE>;
    using Lean = LeanMem<N, lean_lo<In, MODE>>;
    extern __shared__ __align__(16) unsigned char ws_smem[];
    constexpr size_t lean_all = C::POLISH * lean_bytes<N, In, MODE>;
    WsCtl *ctl = reinterpret_cast<WsCtl *>(ws_smem + lean_all);
    WsSlot<N> *ring = reinterpret_cast<WsSlot<N> *>(ws_smem + lean_all + sizeof(WsCtl));
    __shared__ unsigned long long acc[ST_WORDS];
    if (threadIdx.x == 0) {
        ctl->sweep_ticket = 0;
        ctl->polish_ticket = 0;
        ctl->abort = 0;
    }
    if (threadIdx.x < WS_MAX_SLOTS) ctl->state[threadIdx.x] = 0;
    __syncthreads();
    const CtaStats S = stats_begin(acc, A.stats);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t tasks = (n + 31) / 32;
    const int64_t G = gridDim.x, b = blockIdx.x;
    const unsigned my_tasks = b < tasks ? (unsigned)((tasks - b + G - 1) / G) : 0u;
    volatile unsigned *abort_flag = &ctl->abort;

    if (warp >= C::POLISH) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(C::SWEEP_REGS));
        for (;;) {
            unsigned k = 0;
            if (lane == 0) k = atomicAdd(&ctl->sweep_ticket, 1u);
            k = __shfl_sync(0xffffffffu, k, 0);
            if (__any_sync(0xffffffffu, k >= my_tasks || *abort_flag)) break;
            const int64_t i = (b + (int64_t)k * G) * 32 + lane;
            cx<float> d[N];
            bool degenerate, not_conv;
            sweep_lane<N, float, In, MODE>(A, coeffs, n, i, S, d, degenerate, not_conv);
            if (!ws_put<N>(ctl, ring, C::SLOTS, k, d, degenerate, not_conv, abort_flag)) break;
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(C::POLISH_REGS));
        for (;;) {
            unsigned k = 0;
            if (lane == 0) k = atomicAdd(&ctl->polish_ticket, 1u);
            k = __shfl_sync(0xffffffffu, k, 0);
            if (k >= my_tasks) break;
            const int64_t i = (b + (int64_t)k * G) * 32 + lane;
            const unsigned slot = k % (unsigned)C::SLOTS, round = k / (unsigned)C::SLOTS;
            if (!ws_wait(&ctl->state[slot], 2u * round + 1u, abort_flag)) {
                ws_report_abandoned(A, map, S, i, n);
                continue;
            }
            WsSlot<N> &w = ring[slot];
            const bool degenerate = (w.degenerate >> lane) & 1u;
            const bool not_conv = (w.not_conv >> lane) & 1u;
            Lean &lean = *reinterpret_cast<Lean *>(ws_smem + warp * lean_bytes<N, In, MODE>);
            finish_lean<N, In, MODE>(A, coeffs, n, i, map, S, w, lean, degenerate, not_conv);
            ws_publish(&ctl->state[slot], 2u * round + 2u);
        }
    }
    stats_end(S, A.stats);
}

template <int N, typename In, int MODE>
__global__ void __launch_bounds__(Split<N, MODE>::THREADS, 1) solve_split_kernel(SolveArgs A)
{
    split_cta<N, In, MODE>(A, A.coeffs, A.n, UniformMap{{}, A.n});
}

// The degree-N bin of a packed batch (its size is read on the device).
template <int N, typename In, int MODE>
__global__ void __launch_bounds__(Split<N, MODE>::THREADS, 1)
    uneven_split_kernel(SolveArgs A, const UnevenHeader *hdr, const uint32_t *perm, const char *bins, const int64_t *offsets)
{
    const PackedMap map{{}, perm + hdr->poly_base[N], offsets};
    split_cta<N, In, MODE>(A, bins + (size_t)hdr->coef_base[N] * sizeof(In), hdr->count[N], map);
}

}  // namespace rd
