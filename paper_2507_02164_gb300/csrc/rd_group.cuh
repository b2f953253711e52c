// rd_group.cuh -- the solver for small batches: a group of G lanes (8 up to
// degree 8, 16 up to 12) works on one polynomial, its Hessenberg matrix in
// shared memory.
//
// A batch that does not fill the chip is bound by the latency of one warp.
// The one-thread-per-polynomial kernel (rd_solve.cuh) then runs straight-line
// code of thousands of instructions per sweep on a single warp of an SM
// (instruction fetch and dependent issue; 0.2 instructions per clock at degree
// 12) and polishes its roots one after another. Here
//   * the left rotations of a sweep run with one lane per column, the right
//     rotations with one lane per row: a lane carries one entry of its column
//     (row) from rotation to rotation in registers and reads the other from
//     shared memory ahead of the rotation that needs it;
//   * all loops are rolled (the degree is a runtime value, the code fits the
//     instruction cache), so one kernel serves every degree, and a packed
//     batch of mixed degrees needs no binning;
//   * each root is polished by a lane of its own.
// Every value goes through the operations of rd_solve.cuh in the same order,
// so roots, status, histogram and counters are the same bits; only entries
// that no result depends on (the columns right of the active block) are not
// computed. Issue slots per polynomial are 6 to 8 times the one-thread
// kernel's, so the host takes this path only while the chip has them to spare
// (rd_group.cu).
#pragma once

#include "rd_solve.cuh"
#include "rd_uneven.cuh"

namespace rd {

constexpr int GROUP_MAX_N = 12;
constexpr int GROUP_LD = GROUP_MAX_N + 1;  // odd row stride: lanes walking down a column meet different banks

// Complex numbers in shared memory, one 8- or 16-byte access each.
template <typename T>
struct alignas(2 * sizeof(T)) Packed {
    T re, im;
    __device__ __forceinline__ operator cx<T>() const { return {re, im}; }
    __device__ __forceinline__ void operator=(cx<T> v)
    {
        using V = typename std::conditional<sizeof(T) == 8, double2, float2>::type;
        V u;
        u.x = v.re;
        u.y = v.im;
        *reinterpret_cast<V *>(this) = u;
    }
};

// One polynomial's shared memory.
template <typename T>
struct GroupMem {
    Packed<T> h[GROUP_MAX_N * GROUP_LD];
    Packed<T> s[GROUP_MAX_N];
    T c[GROUP_MAX_N];
    Packed<double> z[GROUP_MAX_N];
    Packed<double> ad[GROUP_MAX_N + 1];
    Packed<float> af[GROUP_MAX_N + 1];
    Packed<float> alo[GROUP_MAX_N + 1];
};

template <typename T>
__device__ __forceinline__ cx<T> shfl_from(cx<T> v, int src)
{
    return {__shfl_sync(0xffffffffu, v.re, src), __shfl_sync(0xffffffffu, v.im, src)};
}

// Solve, finish and bin one polynomial per group of G lanes; all 32 lanes of
// the warp call it together. Coefficient k of the group's polynomial is
// element k * cstride + c0 of `coeffs`; N is its degree (1 .. 12, N <= G);
// live = false: no polynomial (N is then 1 and nothing is read or written).
template <int G, typename T, typename In, int MODE, class Map>
__device__ __forceinline__ void solve_group(const SolveArgs &A, const void *coeffs, int64_t c0, int64_t cstride,
                                            int N, int64_t pid, bool live, const Map &map, GroupMem<T> &W,
                                            const CtaStats &S)
{
    constexpr bool MIXED = MODE != MODE_PLAIN;
    constexpr bool C64 = std::is_same<In, float2>::value;
    const int lane = threadIdx.x & 31, l = lane % G, first = lane - l;
    const unsigned gmask = (G == 32 ? 0xffffffffu : ((1u << G) - 1u)) << first;
    auto group_any = [&](bool p) { return (__ballot_sync(0xffffffffu, p) & gmask) != 0; };
    Packed<T> *h = W.h;
    auto at = [](int r, int j) { return r * GROUP_LD + j; };
    __syncwarp();

    // ---- coefficients (lane l: k = l, l + G), degeneracy, the monic b, the
    // companion matrix (load_monic's operations)
    bool bad = !live;
    for (int k = l; k <= N; k += G) {
        if constexpr (C64) {
            const cx<float> a = live ? InLoad<In>::ldf(coeffs, (int64_t)k * cstride + c0) : cx<float>{0.0f, 0.0f};
            W.af[k] = a;
            bad |= !finite_c(a);
        } else {
            const cx<double> a = live ? InLoad<In>::ld(coeffs, (int64_t)k * cstride + c0) : cx<double>{0.0, 0.0};
            W.ad[k] = a;
            bad |= !finite_c(a);
        }
    }
    __syncwarp();
    if constexpr (C64)
        bad |= W.af[N].re == 0.0f && W.af[N].im == 0.0f;
    else
        bad |= W.ad[N].re == 0.0 && W.ad[N].im == 0.0;
    const bool degenerate = group_any(bad);
    for (int e = l; e < N * GROUP_LD; e += G) h[e] = cx<T>{T(0), T(0)};
    __syncwarp();
    if constexpr (MIXED && C64) {
        const cx<float> inv = cdiv(cx<float>{1.0f, 0.0f}, degenerate ? cx<float>{1.0f, 0.0f} : cx<float>(W.af[N]));
        for (int k = l; k < N; k += G) {
            const cx<float> b = mul(cx<float>(W.af[k]), inv);
            if (k >= 1) h[at(k, k - 1)] = cx<T>{T(1), T(0)};
            h[at(k, N - 1)] = degenerate ? cx<T>{T(0), T(0)} : cx<T>{-b.re, -b.im};
        }
    } else {
        cx<double> lead;
        if constexpr (C64)
            lead = {(double)W.af[N].re, (double)W.af[N].im};
        else
            lead = W.ad[N];
        const cx<double> inv = cdiv(cx<double>{1.0, 0.0}, degenerate ? cx<double>{1.0, 0.0} : lead);
        for (int k = l; k < N; k += G) {
            cx<double> a;
            if constexpr (C64)
                a = {(double)W.af[k].re, (double)W.af[k].im};
            else
                a = W.ad[k];
            const cx<double> q = mul(a, inv);
            const cx<T> b = {(T)q.re, (T)q.im};
            if (k >= 1) h[at(k, k - 1)] = cx<T>{T(1), T(0)};
            h[at(k, N - 1)] = degenerate ? cx<T>{T(0), T(0)} : cx<T>{-b.re, -b.im};
        }
    }
    __syncwarp();

    // ---- QR iteration with deflation (Alg. 1); every lane of the group decides alike
    const T tol = (T)A.tol;
    int m = degenerate ? 0 : N;
    int its = 0;
    bool not_conv = false;
    unsigned n_sweeps = 0, n_pairs = 0, n_rots = 0;
    for (;;) {
        if (m >= 2) {
            const cx<T> ta = h[at(m - 2, m - 2)], tc = h[at(m - 1, m - 2)], td = h[at(m - 1, m - 1)];
            const bool small = deflates(A, tol, its, ta, tc, td);
            if (small || its >= A.max_iters) {
                not_conv |= !small;
                m -= 1;
                its = 0;
            }
        }
        const int mm = m >= 2 ? m : 0;
        const int M = __reduce_max_sync(0xffffffffu, mm);
        if (M < 2) break;
        cx<T> shift = {T(0), T(0)};
        if (mm) {
            const cx<T> ta = h[at(m - 2, m - 2)], tb = h[at(m - 2, m - 1)], tc = h[at(m - 1, m - 2)],
                        td = h[at(m - 1, m - 1)];
            shift = pick_shift(A, its, ta, tb, tc, td);
        }
        __syncwarp();  // every lane has read the trailing block
        // left rotations: lane l holds column l; x = its entry of row r-1
        cx<T> x = l < mm ? cx<T>(h[at(0, l)]) : cx<T>{T(0), T(0)};
        if (l == 0) {
            x.re -= shift.re;
            x.im -= shift.im;
        }
        // (y: its entry of row r, read one rotation ahead)
        cx<T> y = l < mm && mm > 1 ? cx<T>(h[at(1, l)]) : cx<T>{T(0), T(0)};
        for (int r = 1; r < M; ++r) {
            const bool act = r < mm;
            cx<T> ahead = {T(0), T(0)};
            if (r + 1 < mm && l >= r && l < mm) ahead = h[at(r + 1, l)];
            if (l == r) {
                y.re -= shift.re;
                y.im -= shift.im;
            }
            T c;
            cx<T> s, top;
            givens(x, y, c, s, top);  // lane r-1's is the rotation
            c = __shfl_sync(0xffffffffu, c, first + r - 1);
            s = shfl_from(s, first + r - 1);
            // lane r-1 closes its column (top, 0), the lanes right of it rotate theirs
            const bool own = act && l == r - 1, right = act && l >= r && l < mm;
            cx<T> nx = x, ny = y;
            rot_rows(c, s, nx, ny);
            if (own || right) h[at(r - 1, l)] = own ? top : nx;
            if (own) {
                h[at(r, l)] = cx<T>{T(0), T(0)};
                W.c[r] = c;
                W.s[r] = s;
            }
            x = sel(right, ny, x);
            y = ahead;
        }
        if (mm && l == mm - 1) h[at(l, l)] = x;
        __syncwarp();
        // right rotations: lane l holds row l; x = its entry of column r-1
        x = l < mm ? cx<T>(h[at(l, l > 0 ? l - 1 : 0)]) : cx<T>{T(0), T(0)};
        const int r0 = l > 0 ? l : 1;
        if (r0 < mm) {
            y = h[at(l, r0)];
            T c = W.c[r0];
            cx<T> s = W.s[r0];
            for (int r = r0; r < mm; ++r) {
                cx<T> ya = {T(0), T(0)}, sa = {T(0), T(0)};
                T ca = T(0);
                if (r + 1 < mm) {
                    ya = h[at(l, r + 1)];
                    ca = W.c[r + 1];
                    sa = W.s[r + 1];
                }
                rot_cols(c, s, x, y);
                if (l == r - 1) {
                    x.re += shift.re;
                    x.im += shift.im;
                }
                h[at(l, r - 1)] = x;
                x = y;
                y = ya;
                c = ca;
                s = sa;
            }
        }
        if (l < mm) {
            if (l == mm - 1) {
                x.re += shift.re;
                x.im += shift.im;
            }
            h[at(l, mm - 1)] = x;
        }
        __syncwarp();
        if (mm) {
            its += 1;
            n_sweeps += 1;
            n_pairs += (unsigned)(mm * (mm + 1) - 2);
            n_rots += (unsigned)(mm - 1);
        }
    }
    const unsigned once = l == 0 ? 1u : 0u;  // counters per polynomial
    S.add(ST_SWEEPS, n_sweeps * once);
    S.add(ST_PAIRS, n_pairs * once);
    S.add(ST_ROTS, n_rots * once);
    S.add(MIXED ? ST_F32 : ST_F64, (20u * n_pairs + 24u * n_rots + 60u * n_sweeps) * once);

    // ---- this lane's root: diagonal entry l (finish_lane's operations)
    const bool mine = l < N;
    const cx<T> d = mine ? cx<T>(h[at(l, l)]) : cx<T>{T(0), T(0)};
    uint8_t st = degenerate ? RD_STATUS_DEGENERATE : (not_conv ? RD_STATUS_NOT_CONVERGED : RD_STATUS_OK);
    cx<double> zj;
    if constexpr (!MIXED) {
        zj = {(double)d.re, (double)d.im};
    } else {
        cx<float> zf = {d.re, d.im};
        unsigned newton = 0;
        const bool polish = A.polish_steps > 0 || A.polish_extra > 0;
        zj = f2d(zf);
        if (polish && !__all_sync(0xffffffffu, degenerate)) {
            constexpr bool LO = MODE == MODE_MIXED_DF && !C64;
            // the coefficients in FP64 and FP32
            if constexpr (C64) {
                for (int k = l; k <= N; k += G) {
                    if (degenerate) W.af[k] = cx<float>{k == N ? 1.0f : 0.0f, 0.0f};
                    W.ad[k] = f2d(cx<float>(W.af[k]));
                }
            } else {
                unsigned emax = 0;
                for (int k = l; k <= N; k += G) {
                    if (degenerate) W.ad[k] = cx<double>{k == N ? 1.0 : 0.0, 0.0};
                    emax = max(emax, max(exponent_bits(W.ad[k].re), exponent_bits(W.ad[k].im)));
                }
#pragma unroll
                for (int o = G / 2; o > 0; o >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
                const double f = pow2_scale(emax);
                for (int k = l; k <= N; k += G) {
                    const cx<double> a = {W.ad[k].re * f, W.ad[k].im * f};
                    W.ad[k] = a;
                    W.af[k] = d2f(a);
                    if constexpr (LO) W.alo[k] = cx<float>{d2f(a.re - f2d(W.af[k].re)), d2f(a.im - f2d(W.af[k].im))};
                }
            }
            __syncwarp();
            auto ad = [&](int k) -> cx<double> { return W.ad[k]; };
            auto af = [&](int k) -> cx<float> { return W.af[k]; };
            [[maybe_unused]] auto lo = [&](int k) -> cx<float> {
                if constexpr (LO) return W.alo[k];
                return {0.0f, 0.0f};
            };
            const float rtol = A.residual_tol > 0 ? (float)A.residual_tol : (float)(64.0 * N * 0x1p-53);
            auto weight = [&](float az) {
                float den = abs1(af(N));
                for (int k = N - 1; k >= 0; --k) den = fmaf(den, az, abs1(af(k)));
                return den;
            };
            auto horner = [&](cx<double> zz) {
                cx<double> p = ad(N);
                for (int k = N - 1; k >= 0; --k) p = cfma(p, zz, ad(k));
                return p;
            };
            auto passes = [&](cx<double> p, cx<double> zz) {
                const float den = weight(sqrtf(norm2(d2f(zz))));
                return (sqrtf(norm2(d2f(p))) <= rtol * den) && finite_bits(zz.re) && finite_bits(zz.im);
            };
            bool good = false;
            if constexpr (MODE == MODE_MIXED_DF) {
                cx<float> zl = {0.0f, 0.0f};
                for (int step = 0; step < A.polish_steps; ++step) {
                    CompHorner ch(zf, af(N), lo(N));
                    for (int k = N - 1; k >= 0; --k) ch.step<LO>(af(k), lo(k));
                    if (!ch.newton(zf, zl)) break;
                    newton += 1;
                }
                zj = {f2d(zf.re) + f2d(zl.re), f2d(zf.im) + f2d(zl.im)};
            } else {
                float moved = CUDART_INF_F;
                for (int step = 0; step < A.polish_steps; ++step) {
                    const cx<double> p = horner(zj);
                    cx<float> pf = af(N), dp = {0.0f, 0.0f};
                    for (int k = N - 1; k >= 0; --k) {
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
            if (!__all_sync(0xffffffffu, good || degenerate || !mine)) good = passes(horner(zj), zj);
            bool failed = mine && !degenerate && !good;
            for (int it = 0; failed && it < A.polish_extra; ++it) {
                cx<double> p = ad(N), dp = {0.0, 0.0};
                for (int k = N - 1; k >= 0; --k) {
                    dp = cfma(dp, zj, p);
                    p = cfma(p, zj, ad(k));
                }
                const cx<double> dz = cdiv(p, dp);
                if (!(finite_bits(dz.re) && finite_bits(dz.im))) break;
                zj = sub(zj, dz);
                newton += 1;
                if (passes(horner(zj), zj)) failed = false;
            }
            // separation (finish_lane's screen and test), pair (l, k), k > l
            if (mine) W.z[l] = zj;
            __syncwarp();
            bool near = false;
            const float screen = fmaxf(1e-4f, 2.0f * (float)A.collapse_tol);
            const cx<float> zs = d2f(zj);
            for (int k = l + 1; k < N; ++k) near |= abs1(sub(zs, d2f(cx<double>(W.z[k])))) <= screen * fmaxf(1.0f, abs1(zs));
            bool reject = failed;
            if (group_any(near)) {
                const double lim = A.collapse_tol * fmax(1.0, fabs(zj.re) + fabs(zj.im));
                for (int k = l + 1; k < N; ++k) {
                    const cx<double> dd = sub(zj, cx<double>(W.z[k]));
                    reject |= (fabs(dd.re) + fabs(dd.im)) <= lim;
                }
            }
            if (group_any(reject && mine) && st == RD_STATUS_OK) st = RD_STATUS_REJECTED;
        }
        const unsigned nw = (degenerate || !mine) ? 0u : newton, nr = (degenerate || !polish) ? 0u : (unsigned)N * once;
        S.add(ST_NEWTON, nw);
        if constexpr (MODE == MODE_MIXED_DF) {
            S.add(ST_F64, (8u * N + 6u) * nr);
            S.add(ST_F32, (66u * N + 50u) * nw + (2u * N + 4u) * nr);
        } else {
            S.add(ST_F64, (8u * N + 2u) * nw + (8u * N + 4u) * nr);
            S.add(ST_F32, (8u * N + 3u) * nw + (2u * N + 4u) * nr);
        }
    }
    if (degenerate) zj = {__longlong_as_double(0x7ff8000000000000ll), __longlong_as_double(0x7ff8000000000000ll)};
    if constexpr (!MIXED) S.add(ST_F64, degenerate ? 0u : 4u * N * once);
    const bool keeper = live && l == 0;
    S.add(ST_POLYS, keeper ? 1u : 0u);
#pragma unroll
    for (int k = 0; k < 4; ++k) S.add(ST_STATUS0 + k, (keeper && st == k) ? 1u : 0u);
    if (keeper && A.status) A.status[pid] = st;

    // ---- store and bin this lane's root
    const bool out = live && mine;
    if (A.roots && out) reinterpret_cast<double2 *>(A.roots)[map.root(pid, l)] = make_double2(zj.re, zj.im);
    if (A.hist) {
        double px = zj.re, py = zj.im;
        bool keep = out, clipped = false;
        if (A.clip_on) {
            cx<double> cen = {0.0, 0.0};
            int64_t my_tile = pid;
            if (out) {
                cen = map.centre(A, pid);
                my_tile = map.tile(A, pid);
            }
            px = __dadd_rn(__dmul_rn(A.radius, px), cen.re);
            py = __dadd_rn(__dmul_rn(A.radius, py), cen.im);
            const int t = pixel_of(A.tiles, px, py);
            const bool in_tile = (t >= 0) && ((int64_t)t == my_tile);
            clipped = out && !in_tile;
            keep = keep && in_tile;
        }
        const int pix = keep ? pixel_of(A.bin, px, py) : -1;
        hist_add(A.hist, pix);
        S.add(ST_CLIPPED, clipped ? 1u : 0u);
        S.add(ST_BINNED, pix >= 0 ? 1u : 0u);
        S.add(ST_OOW, (keep && pix < 0) ? 1u : 0u);
    }
}

constexpr int GROUP_BLOCK = 32;  // one warp per CTA: a small batch spreads over as many SMs as it has warps

// Uniform batch of A.n polynomials of degree N <= G, coefficient-major.
template <int G, typename In, int MODE>
__global__ void __launch_bounds__(GROUP_BLOCK) solve_group_kernel(SolveArgs A, int N)
{
    using T = typename std::conditional<MODE != MODE_PLAIN, float, double>::type;
    constexpr int P = 32 / G;
    __shared__ GroupMem<T> mem[P];
    __shared__ unsigned long long acc[ST_WORDS];
    const CtaStats S = stats_begin(acc, A.stats);
    const UniformMap map{{}, A.n};
    const int g = (threadIdx.x & 31) / G;
    for (int64_t base = (int64_t)blockIdx.x * P; base < A.n; base += (int64_t)gridDim.x * P) {
        const int64_t i = base + g;
        const bool live = i < A.n;
        solve_group<G, T, In, MODE>(A, A.coeffs, live ? i : 0, A.n, live ? N : 1, live ? i : 0, live, map, mem[g], S);
    }
    stats_end(S, A.stats);
}

// Packed batch of mixed degrees (rd_roots_uneven's layout and consistency
// rule), after uneven_count_kernel: it has marked the unsolvable polynomials;
// the solvable ones are solved here, or (when they need more than n_coeffs
// coefficients in all) marked DEGENERATE.
struct DirectMap : ClipFromArrays {
    const int64_t *offsets;
    __device__ int64_t root(int64_t p, int j) const { return __ldg(offsets + p) - p + j; }
};

template <typename In, int MODE>
__global__ void __launch_bounds__(GROUP_BLOCK) uneven_group_kernel(SolveArgs A, UnevenArgs U, const UnevenHeader *hdr,
                                                                   bool asked)
{
    const unsigned degrees = asked ? hdr->direct : ~0u;  // (0: the ranges overlap, nothing is solved)
    if (!degrees) return;
    using T = typename std::conditional<MODE != MODE_PLAIN, float, double>::type;
    constexpr int G = 16, P = 32 / G;
    __shared__ GroupMem<T> mem[P];
    __shared__ unsigned long long acc[ST_WORDS];
    const CtaStats S = stats_begin(acc, A.stats);
    int64_t total = 0;  // (asked: at most what the scan has checked)
    for (int d = 1; d <= UNEVEN_MAX_DEG; ++d) total += (int64_t)__ldg(hdr->count + d) * (d + 1);
    const bool overflow = total > U.n_coeffs;
    const DirectMap map{{}, U.offsets};
    const int g = (threadIdx.x & 31) / G;
    const bool first = (threadIdx.x % G) == 0;
    for (int64_t base = (int64_t)blockIdx.x * P; base < U.n; base += (int64_t)gridDim.x * P) {
        const int64_t i = base + g;
        bool consistent = false;
        const int d = i < U.n ? checked_degree(U, i, consistent) : -1;
        if (overflow) {
            const bool mark = d > 0 && first;
            if (mark) {
                if (A.status) A.status[i] = RD_STATUS_DEGENERATE;
                nan_roots(U, i, A.roots);
            }
            S.add(ST_POLYS, mark ? 1u : 0u);
            S.add(ST_STATUS0 + RD_STATUS_DEGENERATE, mark ? 1u : 0u);
            continue;
        }
        const bool live = d > 0 && ((degrees >> d) & 1u);
        if (!__any_sync(0xffffffffu, live)) continue;
        solve_group<G, T, In, MODE>(A, A.coeffs, live ? __ldg(U.offsets + i) : 0, 1, live ? d : 1, live ? i : 0, live,
                                    map, mem[g], S);
    }
    stats_end(S, A.stats);
}

}  // namespace rd
