// graded.cuh -- entrywise accuracy of the fixed-point FP64 products.
//
// The products of pair_q.cu and pair_tc.cu (T = double) align the rows of X and
// the columns of Y to their largest magnitudes: every output carries an error
// of about 2^-58 rowmax_i colmax_j.  A floating FP64 sum errs by 2^-53 of its own
// terms |X_ik| |Y_kj|.  The transforms act on each entry alone, so where an
// entry's terms lie far below the bounds (rare transitions, chains whose far
// states are reached with small probability, a nearly triangular kernel), the
// aligned sum would lose digits that the entry's time series keeps.
//
// Such outputs are found by their exponents and summed again with every entry
// aligned by itself and every term shifted to the largest one: floating sums, but on
// the integer pipes (in FP64, at two operations per clock and SM, the inverse of a
// birth-death chain of d = 64, N = 2^12 took 25 to 32 ms, with these sums 12.8; the
// aligned sums alone, without a correct digit, 5.4; the FP64 tiles of all products 32.8).
// An output (i, j) of the frequency pair p is sound when
//   rowmax_i(p) colmax_j(p) < 2^GUARD S,
// S the larger of
//   max_k |X_ik(0)| |Y_kj(0)| / sqrt(M): a lower bound of the entry's root mean
//     square over the frequencies, which is what its error in time is relative
//     to (the FFT of a nonnegative series is largest at frequency 0, and its mean
//     square is at least 1 / M of the square of any one value), and
//   max_k |X_ik(p)| |Y_kj(p)|, its own terms;
// the sum's error then stays below about 2^(GUARD - 58) of the entry's scale (2^-44,
// 6e-14), and below 2^-53 for the entries within 2^5 of the bounds, which are most.
// Against references with 94-bit residuals, states entered with probability 1e-1 to
// 1e-8 come out within 8e-13 of their largest value with GUARD = 14 (d = 4 to 64, N = 2^12; 9e-14
// in floating FP64, whose error, like this one, grows with N) and within 2e-13 with 12.
// Up to 16 terms 12 costs ordinary models nothing beyond their first levels (Lognormal d = 16,
// N = 2^10: 0.46 -> 0.63 ms, 0.53 with 14), so they take it; an entrance with 18 x 18 blocks, N =
// 10000, has one output in ten below 2^-12 there: 2.86 -> 3.75 ms, 2.95 with 14.  Weibull and
// Lognormal models of 5 to 64 states have unsound outputs in the first few levels
// (M <= 64) alone: e0 - q has the identity on its diagonal there and very small entries
// beside it (Lognormal d = 24, N = 2^12: 1.77 -> 2.14 ms).
#pragma once
#include "kernels.cuh"
#include "q64.cuh"

// by the number of terms; the digit products have 17 or more
constexpr int GR_GUARD = 14;
__host__ __device__ constexpr int gr_guard(int m) { return m <= 16 ? 12 : GR_GUARD; }
// alignments of a row and a column below which results may be subnormal
constexpr int GR_LOW = 1150;
// Logarithms: biased exponent and four bits of mantissa of the larger part's high
// word, a lower bound of 16 (log2 |x| + 1023).  Sums of two that are negative
// stand for products that are zero or underflow.
constexpr int GR_ZERO = -32768, GR_SUBNORMAL = -16 * 51;
__device__ __forceinline__ unsigned gr_magnitude(cx<double> z) { return max(q_magnitude(z.re), q_magnitude(z.im)); }
__device__ __forceinline__ short gr_log(unsigned m)
{
    return (short)(m >= 0x100000u ? (int)(m >> 16) : (m != 0u ? GR_SUBNORMAL : GR_ZERO));
}

// Whether terms of logarithm g, log_m / 2 below, show an output of alignments ax, ay to be sound
__device__ __forceinline__ bool gr_in_range(int ax, int ay) { return min(ax, ay) > Q_EXMIN && ax + ay > GR_LOW; }
__device__ __forceinline__ bool gr_sound_by(int ax, int ay, int g, int log_m, int guard)
{
    return gr_in_range(ax, ay) && 16 * (ax + ay + 2 - guard) + 8 * log_m <= g;
}

// The whole test of output (i, j).  x0, xp: logarithms of X's row i at frequency 0
// and at the pair, y0, yp: of Y's column j, in steps of c.  (Outputs of rows and
// columns that hold an Inf or NaN are NaN in the first sum already.)
__device__ __forceinline__ bool gr_sound(const short *x0, const short *y0, const short *xp, const short *yp, int m, int c,
                                         int ax, int ay, int log_m)
{
    int g0 = 2 * GR_ZERO, gp = 2 * GR_ZERO;
    for (int k = 0; k < m; ++k) {
        g0 = max(g0, x0[k] + y0[k * c]);
        gp = max(gp, xp[k] + yp[k * c]);
    }
    if (max(ax, ay) >= Q_NONFINITE || gp < 0) return true;  // NaN, or zero
    return gr_sound_by(ax, ay, g0, log_m, gr_guard(m)) || gr_sound_by(ax, ay, gp, 0, gr_guard(m));
}

// 2 Xh(f) and 2 Xh(M - f) of an entry from its packed values, as limbs aligned to its own
// exponent l >> 4 (|re|, |im| of the packed values < 2^((l >> 4) - 1022)) at 2^GR_TOP; tiny
// values are scaled up first (exact), where their zero or subnormal parts would not
// shift out of the alignment
constexpr int GR_TOP = 56;
__device__ __forceinline__ short gr_scaled(cx<double> &za, cx<double> &zb)
{
    unsigned b = max(gr_magnitude(za), gr_magnitude(zb));
    if (b >= ((unsigned)Q_TINY << 20)) return (short)(b >> 16);
    za = c_scal(za, Q_SCALE);
    zb = c_scal(zb, Q_SCALE);
    b = max(gr_magnitude(za), gr_magnitude(zb));
    return (short)(b == 0u ? GR_ZERO : (int)(b >> 16) - 16 * Q_UP);
}
__device__ __forceinline__ void gr_split(cx<double> za, cx<double> zb, qtw w, short &l, qtw &f, qtw &g)
{
    l = gr_scaled(za, zb);
    const int e = l == GR_ZERO ? Q_EXMIN : (int)(max(gr_magnitude(za), gr_magnitude(zb)) >> 20);
    cx<q64> s, t;
    q_split(za, zb, w, e, GR_TOP, s, t);
    f = q_limbs(c_add(s, t));
    g = q_limbs({{s.re.v - t.re.v}, {t.im.v - s.im.v}});
}

// a + x y / 2^(60 + s), rounded
__device__ __forceinline__ void gr_mac(long long &re, long long &im, const qtw &x, const qtw &y, int s)
{
    const int nh = -x.ih, nl = -x.il;
    const long long half = (1ll << s) >> 1;
    long long mr = q_wide(nl, y.ih, q_wide(nh, y.il, q_wide(x.rl, y.rh, q_wide(x.rh, y.rl, 1ll << 29))));
    long long mi = q_wide(x.il, y.rh, q_wide(x.ih, y.rl, q_wide(x.rl, y.ih, q_wide(x.rh, y.il, 1ll << 29))));
    mr = q_wide(nh, y.ih, q_wide(x.rh, y.rh, q_sar30(mr)));
    mi = q_wide(x.ih, y.rh, q_wide(x.rh, y.ih, q_sar30(mi)));
    re += (mr + half) >> s;
    im += (mi + half) >> s;
}

// x 2^de with gradual underflow
__device__ __forceinline__ double gr_scale(double x, int de)
{
    const int e = ((__double2hiint(x) >> 20) & 0x7ff) + de;
    return x == 0.0 || e >= 1 ? q_scale(x, de) : (e > -120 ? q_scale(x, de + Q_UP) * (1.0 / Q_SCALE) : 0.0);
}

// An output's sum at one frequency, halved for q_merge, from gr_mac's sums with the
// largest exponent sum G
__device__ __forceinline__ cx<double> gr_value(long long re, long long im, int G)
{
    const int de = G - 2017 - 2 * GR_TOP;  // the alignments, the limbs, the split's factors 2 and the merge's 1/2
    return {gr_scale(q94_to_double(re, 0), de), gr_scale(q94_to_double(im, 0), de)};
}

// The sum from limbs and logarithms of gr_split (X's row, Y's column in steps of c).  A
// term stays below 2^60 and the sum of m <= 79 of them below 2^63 (2 top + 4 - 60 +
// log2 m with top = 56); it is rounded at 2^-50 to 2^-56 of the largest one.
__device__ __forceinline__ cx<double> gr_sum(const qtw *x, const qtw *y, const short *xl, const short *yl, int m, int c)
{
    int G = 2 * GR_ZERO;
    for (int k = 0; k < m; ++k) G = max(G, (xl[k] >> 4) + (yl[k * c] >> 4));
    long long re = 0, im = 0;
    for (int k = 0; k < m; ++k) {
        const int s = G - (xl[k] >> 4) - (yl[k * c] >> 4);
        if (s <= 61) gr_mac(re, im, x[k], y[k * c], s);
    }
    return gr_value(re, im, G);
}

// The tensor-core product leaves two bytes per pair of the launch, [pair][column / GR_BJ]:
// bit b says that rows GR_BI b .. hold an output not shown to be sound;
// mrc_pair_redo sums the unsound ones of these blocks again.
constexpr int GR_BI = 16, GR_BJ = 32;
