// rd_group.cu -- launches of the small-batch solver (rd_group.cuh) and the
// sizes that take it.
#include "rd_group.cuh"

namespace rd {

// Whether a uniform batch takes the small-batch solver when the caller left
// the launch shape open. Measured (us, 152 SMs, group / one thread per
// polynomial at 32 threads per CTA, one launch with binning):
//   mixed, n   700: degree 3 14.6 / 16.7   6 28.7 / 51.4   12  76.0 / 186.7
//             4800: degree 3 16.5 / 16.5   6 35.1 / 45.4   12 110.8 / 190.8
//             6000: degree 3 16.5 / 16.7   9 86.3 / 92.5   12 127.9 / 192.9
//             8000: degree 3 18.6 / 16.6   9  125 / 86.2   12 186.5 / 190.9
//   plain, n  1216: degree 5  250 / 234    6  338 / 347    12  1179 / 1972
//             2432: degree 5  250 / 225    6  367 / 361    12  1847 / 1908
// so the line lies at 40 polynomials per SM (mixed, from degree 3) and at 8
// (plain, from degree 6: its FP64 instructions cost the same for one active
// lane as for 32). Degree 9, the first with 16 lanes per polynomial, has the least
// to gain; with the compensated polish it ends earlier (complex64 4855 68.3 / 78.4,
// 5923 79.4 / 74.4).
bool group_takes(int degree, int64_t n, bool mixed, bool compensated)
{
    const int64_t sms = rd_sm_count_cached();
    if (!mixed) return degree >= 6 && n <= 8 * sms;
    return degree >= 3 && n <= (compensated && degree == 9 ? 36 : 40) * sms;
}

// The same for a packed batch, which this solver takes in one launch after the
// count, where the degree bins are twelve kernels side by side, as long as the
// slowest warp of them. What decides is how the degrees are spread, which only
// the device knows: half-empty kernels lose to the groups up to 144 polynomials
// per SM, one well-filled kernel of degree 5 and up wins from 56 on (us, group /
// bins):
//   degrees 2..12   fp64 8000 140 / 279   14,000 204 / 289   21,000 278 / 299
//                   df   8000 138 / 229   14,000 206 / 256   21,000 280 / 257
//   9..12           fp64 14,000 242 / 318  21,000 337 / 336   df 14,000 244 / 264
//   degree 9        fp64 14,000 175 / 154  21,000 244 / 152   df  8,000 122 / 117  12,000 152 / 119
//   degree 12       fp64 14,000 260 / 267  21,000 370 / 268   df 12,000 228 / 207
//   degree 6        fp64 17,000 121 / 128  21,000 142 / 129   df 14,000 103 / 97   21,000 142 / 97
//   plain           2..12 2000 1319 / 2172, 4000 2354 / 2351; degree 8 3600 1314 / 1060
// so up to 88 per SM (compensated 56, plain 16) the groups, from 144 (128, 24) the
// bins; in between the groups, but for a degree with more than a third of the batch
// from 7 up, above 104 (80, plain always) per SM from 5 up. The launches of the
// bins that may be asked cost a batch of degrees 2..12 2 to 5 % there, one of
// degrees 1..4 13 to 20 us of host time.
UnevenForm uneven_form(int64_t n, bool mixed, bool compensated)
{
    const int64_t sms = rd_sm_count_cached();
    const int sure = !mixed ? 16 : (compensated ? 56 : 88), high = !mixed ? 16 : (compensated ? 80 : 104),
              most = !mixed ? 24 : (compensated ? 128 : 144);
    if (n <= sure * sms) return {UnevenForm::group, 0};
    if (n <= most * sms) return {UnevenForm::ask, n <= high * sms ? 7 : 5};
    return {UnevenForm::bins, 1};
}

template <int G, typename In, int MODE>
static int launch_group_n(int degree, const SolveArgs &a, cudaStream_t st)
{
    constexpr int P = 32 / G;
    solve_group_kernel<G, In, MODE><<<(unsigned)((a.n + P - 1) / P), GROUP_BLOCK, 0, st>>>(a, degree);
    return rd_check_launch("solve_group_kernel");
}

template <int G, typename In>
static int launch_group_mode(int degree, bool mixed, const SolveArgs &a, cudaStream_t st)
{
    if (!mixed) return launch_group_n<G, In, MODE_PLAIN>(degree, a, st);
    if (a.polish_mode == RD_POLISH_DF) return launch_group_n<G, In, MODE_MIXED_DF>(degree, a, st);
    return launch_group_n<G, In, MODE_MIXED_FP64>(degree, a, st);
}

int launch_group(int degree, rd_dtype dt, bool mixed, const SolveArgs &a, cudaStream_t st)
{
    if (degree <= 8)
        return dt == RD_C64 ? launch_group_mode<8, float2>(degree, mixed, a, st)
                            : launch_group_mode<8, double2>(degree, mixed, a, st);
    return dt == RD_C64 ? launch_group_mode<16, float2>(degree, mixed, a, st)
                        : launch_group_mode<16, double2>(degree, mixed, a, st);
}

template <typename In>
static int launch_uneven_group_mode(const SolveArgs &a, const UnevenArgs &U, const UnevenHeader *hdr, bool mixed,
                                    bool asked, cudaStream_t st)
{
    const unsigned grid = (unsigned)((U.n + 1) / 2);
    if (!mixed)
        uneven_group_kernel<In, MODE_PLAIN><<<grid, GROUP_BLOCK, 0, st>>>(a, U, hdr, asked);
    else if (a.polish_mode == RD_POLISH_DF)
        uneven_group_kernel<In, MODE_MIXED_DF><<<grid, GROUP_BLOCK, 0, st>>>(a, U, hdr, asked);
    else
        uneven_group_kernel<In, MODE_MIXED_FP64><<<grid, GROUP_BLOCK, 0, st>>>(a, U, hdr, asked);
    return rd_check_launch("uneven_group_kernel");
}

int launch_uneven_group(const SolveArgs &a, rd_dtype dt, const UnevenArgs &U, const UnevenHeader *hdr, bool mixed,
                        bool asked, cudaStream_t st)
{
    return dt == RD_C64 ? launch_uneven_group_mode<float2>(a, U, hdr, mixed, asked, st)
                        : launch_uneven_group_mode<double2>(a, U, hdr, mixed, asked, st);
}

}  // namespace rd
