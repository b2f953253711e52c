// rd_l2.cu -- least-squares (L2) polynomial approximation on sub-disks.
//
// Paper: Tang & Quan, arXiv 2507.02164, Sec. II: the domain is split into
// small subregions and f is approximated on each by a polynomial g; Sec. II-A:
// with <g, h> = integral over the unit disk of g conj(h), the coefficients
// solve G a = b with G_jk = <z^j, z^k>, b_j = <f, z^j>. Taking the measure as
// area (dA = r dr dtheta), G is diagonal with G_jj = pi/(j+1), so
//   a_j = (j+1)/pi * <g, w^j>.
// Quadrature: Gauss-Legendre in r on [0,1] (nr nodes, the Jacobian r folded
// into the weights), the trapezoid rule in theta (nt = 32 equispaced angles,
// exact for trigonometric degree < 32). Per sub-disk:
//   <g, w^j> ~ sum_p w_p r_p^{j+1} (2 pi / nt) sum_q g(r_p e^{i theta_q}) e^{-i j theta_q}.
//
// One warp per sub-disk; its 16 x 32 samples (8 KB) are read once.
//   * FP64 sums (l2_kernel): the FP64 pipe is the bound, so the angular sum is
//     split first. theta_{q+8t} = theta_q + t pi/2, hence e^{-i j theta} over t
//     = 0..3 is (-i)^{jt} times the value at theta_q: a 4-point transform (16
//     additions) serves every j through j mod 4, and the radial sums with
//     their real weights (2 FMA per j) run on a quarter of the terms: 30 FP64
//     operations per 4 samples at degree 6 instead of 56.
//   * double-float sums (l2_kernel_df): lane q owns angle theta_q; radial sums
//     u_j(q) = sum_p (w_p r_p^{j+1}) g_pq, then v_j = sum_q u_j(q) e^{-i j theta_q}
//     by a warp reduce-scatter.
#include <atomic>
#include <cmath>
#include <mutex>

#include "rd_common.cuh"

namespace rd {

constexpr int L2_NT = 32;
constexpr int L2_MAX_NR = 32;
constexpr int L2_MAX_DEG = 12;

struct L2Tables {
    double wr[L2_MAX_NR][L2_MAX_DEG + 1];   // w_p r_p^{j+1} * (2 pi / nt) * (j+1) / pi
    double tw[L2_MAX_DEG + 1][L2_NT][2];    // e^{-i j theta_q}
};

// Legendre P_n(x) and P_{n-1}(x) by the three-term recurrence.
static void legendre_pair(int n, double x, double &pn, double &pn1)
{
    double pm1 = 1.0, p = x;  // P_0, P_1
    if (n == 0) {
        pn = 1.0;
        pn1 = 0.0;
        return;
    }
    for (int k = 2; k <= n; ++k) {
        double next = ((2 * k - 1) * x * p - (k - 1) * pm1) / k;
        pm1 = p;
        p = next;
    }
    pn = p;
    pn1 = pm1;
}

// Gauss-Legendre on [0, 1]: nodes are the zeros of P_n mapped from [-1, 1],
// found by Newton's method from Tricomi's first-order estimate; the weights are
// 2 / ((1 - x^2) P_n'(x)^2) on [-1, 1], halved for [0, 1], with
// P_n'(x) = n (P_{n-1}(x) - x P_n(x)) / (1 - x^2).
int l2_nodes_host(int nr, double *r, double *w)
{
    const double pi = 3.14159265358979323846;
    for (int k = 1; k <= nr; ++k) {
        double x = (1.0 - (nr - 1.0) / (8.0 * nr * nr * nr)) * std::cos(pi * (4.0 * k - 1.0) / (4.0 * nr + 2.0));
        for (int it = 0; it < 60; ++it) {
            double pn, pn1;
            legendre_pair(nr, x, pn, pn1);
            double dpn = nr * (pn1 - x * pn) / ((1.0 - x) * (1.0 + x));
            double dx = pn / dpn;
            x -= dx;
            if (std::fabs(dx) < 1e-17) break;
        }
        double pn, pn1;
        legendre_pair(nr, x, pn, pn1);
        double omx2 = (1.0 - x) * (1.0 + x);
        double dpn = nr * (pn1 - x * pn) / omx2;
        double wt = 2.0 / (omx2 * dpn * dpn);
        // k = 1 is the largest node: fill from the top so r ascends
        r[nr - k] = 0.5 * (1.0 + x);
        w[nr - k] = 0.5 * wt;
    }
    return 0;
}

constexpr int L2_Q = 8;             // angle classes: theta_q, q < 8, and its three quarter turns
constexpr int L2_G = 32 / L2_Q;     // radius groups of a warp
constexpr int L2_WARPS = 8;         // warps per CTA

__device__ __forceinline__ cx<double> shfl_xor_c(cx<double> v, int o)
{
    return {__shfl_xor_sync(0xffffffffu, v.re, o), __shfl_xor_sync(0xffffffffu, v.im, o)};
}

// FP64 sums. Lane (group r = lane / 8, class q = lane % 8) takes the radii p =
// r, r + 4, ... at the angles q + 8 t: per load instruction four runs of 128
// bytes. Then, per pass of 8 coefficients j = j0 + jj: a reduce-scatter over
// the radius groups leaves group r the sums of jj = r and r + 4 (12
// additions), which it multiplies by e^{-i j theta_q} and sums over the 8
// classes (8 + 4 operations). Bound by the FP64 pipe: about 9 operations per
// sample at degree 6 (16.8 with the angles summed one by one). 50,021
// sub-disks of 16 x 32 samples: 458 us, 95 % of the FP64 rate (744 us before).
// NR > 0, DEG >= 0: a build for that node count and degree; NR = 0, DEG = -1:
// runtime bounds (the same operations in the same order).
template <int NR, int DEG>
__global__ void __launch_bounds__(L2_WARPS * 32) l2_kernel(const double2 *__restrict__ samples, int64_t n, int nr_arg,
                                                          int degree_arg, double2 *coeffs, const __grid_constant__ L2Tables T)
{
    constexpr int JMAX = DEG >= 0 ? DEG : L2_MAX_DEG;
    const int nr = NR > 0 ? NR : nr_arg;
    const int degree = DEG >= 0 ? DEG : degree_arg;
    // the lanes of a warp read the weights of four radii and the twiddles of
    // eight angles at a time: from shared memory, where the constant bank
    // would serialise them
    __shared__ double s_wr[L2_MAX_NR * (L2_MAX_DEG + 1)];
    __shared__ double2 s_tw[(L2_MAX_DEG + 1) * L2_Q];
    for (int i = threadIdx.x; i < nr * (JMAX + 1); i += blockDim.x) s_wr[i] = T.wr[i / (JMAX + 1)][i % (JMAX + 1)];
    for (int i = threadIdx.x; i < (JMAX + 1) * L2_Q; i += blockDim.x)
        s_tw[i] = make_double2(T.tw[i / L2_Q][i % L2_Q][0], T.tw[i / L2_Q][i % L2_Q][1]);
    __syncthreads();
    const int lane = threadIdx.x & 31, q = lane % L2_Q, r = lane / L2_Q;
    const int warps = blockDim.x >> 5;
    const int64_t warps_total = (int64_t)gridDim.x * warps;
    for (int64_t s = (int64_t)blockIdx.x * warps + (threadIdx.x >> 5); s < n; s += warps_total) {
        const double2 *g = samples + s * (int64_t)nr * L2_NT + q;
        cx<double> u[JMAX + 1];
        // the radial sums; returns whether a sample is 2^1021 or more (or not
        // finite), where the unweighted sums below could overflow
        auto radial = [&](auto scaled) {
            bool large = false;
#pragma unroll
            for (int j = 0; j <= JMAX; ++j) u[j] = {0.0, 0.0};
#pragma unroll(NR > 0 ? NR / L2_G : 1)
            for (int p = r; p < nr; p += L2_G) {
                cx<double> f[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const double2 v = __ldg(g + p * L2_NT + t * L2_Q);
                    large |= max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu) >= 0x7fc00000u;
                    f[t] = decltype(scaled)::value ? cx<double>{v.x * 0x1p-4, v.y * 0x1p-4} : cx<double>{v.x, v.y};
                }
                const cx<double> s02 = add(f[0], f[2]), d02 = sub(f[0], f[2]), s13 = add(f[1], f[3]), d13 = sub(f[1], f[3]);
                // G[k] = sum_t (-i)^{kt} f_t
                const cx<double> G[4] = {add(s02, s13), {d02.re + d13.im, d02.im - d13.re}, sub(s02, s13),
                                         {d02.re - d13.im, d02.im + d13.re}};
#pragma unroll
                for (int j = 0; j <= JMAX; ++j)
                    if (j <= degree) {
                        const double w = s_wr[p * (JMAX + 1) + j];
                        u[j] = {fma(w, G[j & 3].re, u[j].re), fma(w, G[j & 3].im, u[j].im)};
                    }
            }
            return large;
        };
        const bool rescaled = __any_sync(0xffffffffu, radial(std::false_type{}));
        if (rescaled) radial(std::true_type{});
#pragma unroll
        for (int j0 = 0; j0 <= JMAX; j0 += 8) {
            if (j0 > degree) break;
            cx<double> v[8];
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) v[jj] = j0 + jj <= JMAX ? u[j0 + jj] : cx<double>{0.0, 0.0};
            // over the radius groups: bit 1 of r keeps jj with that bit, then bit 0
            const bool hi = (r & 2) != 0, lo = (r & 1) != 0;
            cx<double> w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int a = (i & 1) | ((i & 2) << 1);  // jj with bit 1 clear: 0, 1, 4, 5
                w[i] = add(sel(hi, v[a + 2], v[a]), shfl_xor_c(sel(hi, v[a], v[a + 2]), 16));
            }
            cx<double> x[2];  // jj = r, r + 4
#pragma unroll
            for (int i = 0; i < 2; ++i)
                x[i] = add(sel(lo, w[2 * i + 1], w[2 * i]), shfl_xor_c(sel(lo, w[2 * i], w[2 * i + 1]), 8));
            // times e^{-i j theta_q}, then over the 8 classes: bit 2 of q keeps
            // one of the two coefficients, bit 1 its real or imaginary part
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int j = j0 + r + 4 * i;
                const double2 t = s_tw[(j <= JMAX ? j : 0) * L2_Q + q];
                x[i] = {fma(x[i].re, t.x, -x[i].im * t.y), fma(x[i].re, t.y, x[i].im * t.x)};
            }
            const bool second = (q & 4) != 0, imag = (q & 2) != 0;
            const cx<double> y = add(sel(second, x[1], x[0]), shfl_xor_c(sel(second, x[0], x[1]), 4));
            double z = (imag ? y.im : y.re) + __shfl_xor_sync(0xffffffffu, imag ? y.re : y.im, 2);
            z += __shfl_xor_sync(0xffffffffu, z, 1);
            if (rescaled) z *= 0x1p4;
            const double im = __shfl_down_sync(0xffffffffu, z, 2);
            const int j = j0 + r + (second ? 4 : 0);
            if ((q & 3) == 0 && j <= degree) coeffs[(int64_t)j * n + s] = make_double2(z, im);
        }
    }
}

// ---- double-float variant on the FP32 pipe --------------------------------
// Same sums, each term a double-float (hi + lo floats): GB300 runs FP32 64x
// faster than FP64. Samples are first scaled by a power of two per sub-disk
// (the largest exponent of its 512 samples becomes 0; sin(z^3) reaches 1e41,
// beyond FP32) and split into hi + lo floats with integer operations, then
// the scale is applied back to the FP64 coefficients exactly.

// The radial weights are stored as (w, w) pairs: the real and imaginary
// parts of a sample go through the same operations with the same weight, as
// the two halves of packed FP32 instructions (FFMA2 / FMUL2 / FADD2, each
// half rounded as its scalar form), one issue slot for both.
struct L2TablesDF {
    float2 whi[L2_MAX_NR][L2_MAX_DEG + 1], wlo[L2_MAX_NR][L2_MAX_DEG + 1];
    float thi[L2_MAX_DEG + 1][L2_NT][2], tlo[L2_MAX_DEG + 1][L2_NT][2];
};

__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(r)
        : "l"(*reinterpret_cast<const unsigned long long *>(&a)), "l"(*reinterpret_cast<const unsigned long long *>(&b)));
    return *reinterpret_cast<const float2 *>(&r);
}

// two_sum on both halves: s = a + b and its exact rounding error e
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2 &s, float2 &e)
{
    s = __fadd2_rn(a, b);
    const float2 bb = sub2(s, a);
    e = __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// NR > 0, DEG >= 0: a build for that radial node count and degree (loops of
// fixed length, arrays of DEG + 1 coefficients); NR = 0, DEG = -1: the runtime
// nr and degree, with arrays for L2_MAX_DEG. Both do the same operations in
// the same order.
template <int NR, int DEG>
__global__ void __launch_bounds__(256, 2) l2_kernel_df(const double2 *__restrict__ samples, int64_t n, int nr_arg,
                                                    int degree_arg, double2 *coeffs, const L2TablesDF T)
{
    constexpr int JMAX = DEG >= 0 ? DEG : L2_MAX_DEG;
    const int nr = NR > 0 ? NR : nr_arg;
    const int degree = DEG >= 0 ? DEG : degree_arg;
    const int lane = threadIdx.x & 31;
    const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
    dfl twr[JMAX + 1], twi[JMAX + 1];
#pragma unroll
    for (int j = 0; j <= JMAX; ++j) {
        twr[j] = {T.thi[j][lane][0], T.tlo[j][lane][0]};
        twi[j] = {T.thi[j][lane][1], T.tlo[j][lane][1]};
    }
    for (int64_t s = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); s < n; s += warps_total) {
        const double2 *g = samples + s * (int64_t)nr * L2_NT;
        // per sub-disk scale: the largest biased exponent of its samples
        unsigned emax = 0;
#pragma unroll(NR > 0 ? NR : 1)
        for (int p = 0; p < nr; ++p) {
            double2 v = __ldg(g + p * L2_NT + lane);
            unsigned ex = ((unsigned)__double2hiint(v.x) >> 20) & 0x7ffu;
            unsigned ey = ((unsigned)__double2hiint(v.y) >> 20) & 0x7ffu;
            emax = max(emax, max(ex, ey));
        }
        emax = __reduce_max_sync(0xffffffffu, emax);
        const int shift = (int)emax - 1023;
        // accumulators as (real, imaginary) pairs: ah[j] the high parts, al[j] the low
        float2 ah[JMAX + 1], al[JMAX + 1];
#pragma unroll
        for (int j = 0; j <= JMAX; ++j) ah[j] = al[j] = make_float2(0.0f, 0.0f);
        // Four samples at a time with fixed bounds; with runtime bounds one, which is
        // the faster at every node count (30,000 sub-disks, degree 12, us, one / four:
        // 4 nodes 188 / 190, 8 250 / 263, 16 371 / 409, 24 515 / 558).
#pragma unroll(NR > 0 ? 4 : 1)
        for (int p = 0; p < nr; ++p) {
            double2 v = __ldg(g + p * L2_NT + lane);
            const dfl gx = split_scaled(v.x, shift), gy = split_scaled(v.y, shift);
            const float2 gh = make_float2(gx.hi, gy.hi), gl = make_float2(gx.lo, gy.lo);
#pragma unroll
            for (int j = 0; j <= JMAX; ++j)
                if (j <= degree) {
                    const float2 wh = T.whi[p][j], wl = T.wlo[p][j];
                    // exact product hi and its error, then TwoSum into the accumulator
                    const float2 ph = __fmul2_rn(wh, gh);
                    float2 pe = __ffma2_rn(wh, gh, make_float2(-ph.x, -ph.y));
                    pe = __ffma2_rn(wh, gl, pe);
                    pe = __ffma2_rn(wl, gh, pe);
                    float2 t, te;
                    two_sum2(ah[j], ph, t, te);
                    ah[j] = t;
                    al[j] = __fadd2_rn(al[j], __fadd2_rn(te, pe));
                }
        }
        dfl ur[JMAX + 1], ui[JMAX + 1];
#pragma unroll
        for (int j = 0; j <= JMAX; ++j) {
            ur[j] = {ah[j].x, al[j].x};
            ui[j] = {ah[j].y, al[j].y};
        }
#pragma unroll
        for (int j0 = 0; j0 <= JMAX; j0 += 8) {
            if (j0 > degree) break;
            dfl val[16];
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
                const int j = j0 + jj;
                dfl vr = {0.0f, 0.0f}, vi = {0.0f, 0.0f};
                if (j <= JMAX && j <= degree) {
                    dfl a = fast_two_sum(ur[j].hi, ur[j].lo), b = fast_two_sum(ui[j].hi, ui[j].lo);
                    vr = df_add(df_mul(a, twr[j]), df_neg(df_mul(b, twi[j])));
                    vi = df_add(df_mul(a, twi[j]), df_mul(b, twr[j]));
                }
                val[2 * jj] = vr;
                val[2 * jj + 1] = vi;
            }
            // double-float reduce-scatter: level by level (offsets 16, 8, 4, 2) a
            // lane keeps one half of its values, sends the other half to its
            // partner and adds what it receives; the last level (offset 1) adds
            // the partner's copy of the same value. Lane L then holds the warp
            // sum of value (L >> 1) & 15: 16 additions per lane instead of 80
#pragma unroll
            for (int lev = 0; lev < 4; ++lev) {
                const int o = 16 >> lev, half = 16 >> (lev + 1);
                const bool upper = (lane & o) != 0;
#pragma unroll
                for (int i = 0; i < half; ++i) {
                    dfl send = upper ? val[i] : val[i + half];
                    dfl keep = upper ? val[i + half] : val[i];
                    dfl got = {__shfl_xor_sync(0xffffffffu, send.hi, o), __shfl_xor_sync(0xffffffffu, send.lo, o)};
                    val[i] = df_add(keep, got);
                }
            }
            dfl got = {__shfl_xor_sync(0xffffffffu, val[0].hi, 1), __shfl_xor_sync(0xffffffffu, val[0].lo, 1)};
            dfl sum = df_add(val[0], got);
            // back to FP64 and to the sub-disk's scale (a power of two: exact)
            double d = (f2d(sum.hi) + f2d(sum.lo)) * __longlong_as_double((long long)(shift + 1023) << 52);
            double im = __shfl_down_sync(0xffffffffu, d, 2);
            const int jj = lane >> 2;
            if ((lane & 3) == 0 && j0 + jj <= degree) coeffs[(int64_t)(j0 + jj) * n + s] = make_double2(d, im);
        }
    }
}

// The tables of a node count, built on its first use and kept (host memory,
// 24 KB per node count, at most 32 of them): building them takes 80 us at nr
// = 16 and 200 us at 24 (nodes by Newton's method, powers), more than the
// kernel takes on a few thousand sub-disks. They hold every coefficient up to
// L2_MAX_DEG; the kernels read those of their degree.
struct L2HostTables {
    L2Tables fp64;
    L2TablesDF df;
};

static const L2HostTables &l2_tables(int nr)
{
    static L2HostTables tables[L2_MAX_NR + 1];
    static std::atomic<bool> ready[L2_MAX_NR + 1];
    static std::mutex mu;
    L2HostTables *t = &tables[nr];
    if (ready[nr].load(std::memory_order_acquire)) return *t;
    std::lock_guard<std::mutex> lk(mu);
    if (!ready[nr].load(std::memory_order_relaxed)) {
        double r[L2_MAX_NR], w[L2_MAX_NR];
        l2_nodes_host(nr, r, w);
        const double pi = 3.14159265358979323846;
        for (int p = 0; p < nr; ++p)
            for (int j = 0; j <= L2_MAX_DEG; ++j) {
                const double v = w[p] * std::pow(r[p], j + 1) * (2.0 * pi / L2_NT) * (j + 1) / pi;
                const float h = (float)v, l = (float)(v - (double)h);
                t->fp64.wr[p][j] = v;
                t->df.whi[p][j] = make_float2(h, h);
                t->df.wlo[p][j] = make_float2(l, l);
            }
        for (int j = 0; j <= L2_MAX_DEG; ++j)
            for (int q = 0; q < L2_NT; ++q) {
                // e^{-i j theta_q}, theta_q = 2 pi q / nt, reduced exactly: (j q) mod nt
                const double ang = 2.0 * pi * ((j * q) % L2_NT) / L2_NT;
                const double c[2] = {std::cos(ang), -std::sin(ang)};
                for (int k = 0; k < 2; ++k) {
                    t->fp64.tw[j][q][k] = c[k];
                    t->df.thi[j][q][k] = (float)c[k];
                    t->df.tlo[j][q][k] = (float)(c[k] - (double)t->df.thi[j][q][k]);
                }
            }
        ready[nr].store(true, std::memory_order_release);
    }
    return *t;
}

int launch_l2(const double *samples, int64_t n, int nr, int degree, double *coeffs, int precision,
              cudaStream_t st)
{
    const double2 *sp = reinterpret_cast<const double2 *>(samples);
    double2 *cp = reinterpret_cast<double2 *>(coeffs);
    const int64_t sms = rd_sm_count_cached();
    if (precision == 1) {
        const L2TablesDF &T = l2_tables(nr).df;
        const int block = 256;
        int64_t ctas = (n + 7) / 8;
        if (ctas > sms * 8) ctas = sms * 8;
        if (nr == 16 && degree == 6)  // the full pipeline's 16 x 32 nodes and degree-6 fits
            l2_kernel_df<16, 6><<<(unsigned)ctas, block, 0, st>>>(sp, n, nr, degree, cp, T);
        else
            l2_kernel_df<0, -1><<<(unsigned)ctas, block, 0, st>>>(sp, n, nr, degree, cp, T);
        return rd_check_launch("l2_kernel_df");
    }
    const L2Tables &T = l2_tables(nr).fp64;
    // 8 warps per CTA; fewer while a small n would leave SMs without a CTA
    const int64_t warps = n >= sms * L2_WARPS ? L2_WARPS : (n + sms - 1) / sms;
    const int block = 32 * (int)warps;
    int64_t ctas = (n + warps - 1) / warps;
    if (ctas > sms * 8) ctas = sms * 8;
    if (nr == 16 && degree == 6)
        l2_kernel<16, 6><<<(unsigned)ctas, block, 0, st>>>(sp, n, nr, degree, cp, T);
    else
        l2_kernel<0, -1><<<(unsigned)ctas, block, 0, st>>>(sp, n, nr, degree, cp, T);
    return rd_check_launch("l2_kernel");
}

}  // namespace rd
