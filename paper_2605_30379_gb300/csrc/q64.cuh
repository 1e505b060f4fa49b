// q64.cuh -- 64-bit fixed-point arithmetic of the FP64 FFT passes.
//
// The FP64 pipe of this GPU issues two operations per clock and SM, the
// integer pipes about thirty times as many (measured: DFMA 2, IMAD.WIDE 60,
// 32-bit adds 90 per clock and SM), so a pass converts its points to
// fixed-point numbers with one exponent per CTA and entry column, runs its
// in-CTA stages in 64-bit integers and converts back on the store.
//
// Scaling.  A column's points (the R points of the pass at one entry) are
// aligned to the largest exponent among them; the inputs of every stage of
// radix 8 are kept below 2^57 (|re|, |im|; 2^59 in the last one), so that
// its sums stay below 2^60.5 and fit the next twiddle products.  The shift
// before a stage is taken from the magnitudes the previous stage left in the
// column (block floating point): none where the values did not grow.  A
// stage thus rounds at 2^-57 .. 2^-56 of the column's largest magnitude;
// against 128-bit references, passes of 512 and 1024 points err 0.4 to 0.8
// times as much (root mean square) as the same passes in FP64, for random,
// decaying and constant-plus-decaying columns alike (with fixed divisions by
// the radix instead of the measured ones: 0.7 to 7 times).
//
// Products.  A value a < 2^61 and a twiddle w <= 2^60 are split into a high
// limb and a 30-bit low limb each (nonnegative for a, balanced for w); the
// product takes the high and the two middle limb products (32 x 32 -> 64 bit
// multiply-adds), the low one is below the rounding of the result.
//
// Every rounding is unbiased: a constant offset of the points would add up in
// the zero frequency, which the inverse amplifies by N (e0 - q is singular
// there).
#pragma once
#include "arith.cuh"

struct q64 {
    long long v;
};
// twiddle factor: Q60 limbs of its real and imaginary parts
struct __align__(16) qtw {
    int rh, rl, ih, il;
};

constexpr int Q_TOP = 60;
constexpr int Q_NONFINITE = 4096;  // alignment exponent of a column or row that holds an Inf or NaN
constexpr int Q_MASK30 = (1 << 30) - 1;

// 64-bit values in two registers, with the instructions written out: from C++
// expressions the compiler made twice as many of them (a complex product 63
// instructions, with these 29)
__device__ __forceinline__ long long q_wide(int a, int b, long long c)
{
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ int q_lo(long long a) { return (int)a; }
__device__ __forceinline__ int q_hi(long long a) { return (int)(a >> 32); }
__device__ __forceinline__ long long q_join(int lo, int hi)
{
    long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
// a >> 30, as a 32-bit number and as a 64-bit one
__device__ __forceinline__ int q_top30(long long a)
{
    int r;
    asm("shf.l.clamp.b32 %0, %1, %2, 2;" : "=r"(r) : "r"(q_lo(a)), "r"(q_hi(a)));
    return r;
}
__device__ __forceinline__ long long q_sar30(long long a) { return q_join(q_top30(a), q_hi(a) >> 30); }

// x 2^(top + 1022 - ex) rounded to an integer, for |x| < 2^(ex - 1022), ex >=
// Q_EXMIN and top <= 60: the magnitude is rounded (symmetric in the sign, so that
// a column of one sign is not shortened; a tie, frequent where few bits are
// dropped, goes by a mantissa bit that is kept); neg (0 or -1) flips the sign.
// Q_EXMIN shifts zeros (and subnormals) out altogether.
constexpr int Q_EXMIN = 64;
// Values whose alignment would be near it are scaled up first (exact): below 2^-895 by 2^256
constexpr int Q_TINY = 128, Q_UP = 256;
constexpr double Q_SCALE = 0x1p256;
__device__ __forceinline__ q64 q_decode(double x, int ex, int top, int neg = 0)
{
    const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
    const int sh = min(ex + (62 - top) - (int)((hw >> 20) & 0x7ffu), 63);
    const unsigned mh = (hw & 0xfffffu) | 0x100000u;
    const long long m = q_join((int)(lw << 10), (int)__funnelshift_l(lw, mh, 10)) - (long long)(hw & 1u);
    const unsigned long long w = ((unsigned long long)m >> sh) + 1ull;
    const int s = ((int)hw >> 31) ^ neg;
    const long long r = (long long)(w >> 1);
    return {q_join(q_lo(r) ^ s, q_hi(r) ^ s) - (long long)s};
}

// n / 2^11 rounded half to even
__device__ __forceinline__ unsigned long long q_round11(unsigned long long n)
{
    const unsigned long long m = n >> 11;
    return m + (((unsigned)n & 0x7ffu) + ((unsigned)m & 1u) > 0x400u ? 1ull : 0ull);
}

// The rest of q_encode, of a magnitude (out of line: one copy of the code)
static __device__ __noinline__ double q_encode_rest(long long a, int eb)
{
    const int lz = __clzll(a);
    const int e = eb - lz, u = min(max(1 - e, 0), 54);  // a subnormal drops u bits more; what falls out is kept as one bit
    unsigned long long n = (unsigned long long)a << (lz & 63);
    n = (n >> u) | ((n & ((1ull << u) - 1ull)) != 0ull ? 1ull : 0ull);
    const unsigned long long m = q_round11(n);
    if (a == 0) return 0.0;
    if (e >= 2047) return __longlong_as_double(0x7ff0000000000000ll);
    return __hiloint2double((int)((unsigned)(m >> 32) + ((unsigned)max(e - 1, 0) << 20)), (int)(unsigned)m);
}

// v 2^(eb - 1086) rounded to a double (gradual underflow, infinity above the
// range), |v| < 2^63: a value with leading bit 63 - lz gets the biased exponent
// eb - lz.
__device__ __forceinline__ double q_encode(q64 x, int eb, unsigned sgn)
{
    const int s = q_hi(x.v) >> 31;
    const long long a = q_join(q_lo(x.v) ^ s, q_hi(x.v) ^ s) - (long long)s;
    const unsigned sg = ((unsigned)s ^ sgn) & 0x80000000u;
    // the common case: the value's high word is not zero and no exponent between
    // eb - 63 and eb leaves the range
    if (q_hi(a) != 0 && (unsigned)(eb - 64) < 2047u - 64u) {
        const int lz = __clz(q_hi(a)) - 1;  // leading bit to 62
        const unsigned hi = __funnelshift_l((unsigned)q_lo(a), (unsigned)q_hi(a), lz);
        const unsigned long long n = (unsigned long long)q_join(q_lo(a) << lz, (int)hi) + 0x200ull;
        return __hiloint2double((int)((unsigned)(n >> 42) + ((unsigned)(eb - 2 - lz) << 20) | sg), (int)(n >> 10));
    }
    const double y = q_encode_rest(a, eb);
    return __hiloint2double(__double2hiint(y) | (int)sg, __double2loint(y));
}

// a w for a real factor w <= 2^60 (Q60).  (With the mean of the low product in its
// place small values were off by up to half a unit, the positive ones all one way:
// the inverse transform of a spectrum near one added -4e-17 up over 2^10 points.)
__device__ __forceinline__ long long q_mul(long long a, long long w)
{
    const int ah = q_top30(a), al = q_lo(a) & Q_MASK30, wh = (int)(w >> 30), wl = (int)w & Q_MASK30;
    const long long mid = q_wide(al, wh, q_wide(ah, wl, (long long)(int)__umulhi((unsigned)al << 2, (unsigned)wl) + (1ll << 29)));
    return q_wide(ah, wh, q_sar30(mid));
}

template <>
struct Ar<q64> {
    static __device__ __forceinline__ q64 add(q64 a, q64 b) { return {a.v + b.v}; }
    static __device__ __forceinline__ q64 sub(q64 a, q64 b) { return {a.v - b.v}; }
    static __device__ __forceinline__ q64 add_nn(q64 a, q64 b) { return {a.v + b.v}; }
    static __device__ __forceinline__ q64 sub_nn(q64 a, q64 b) { return {a.v - b.v}; }
    static __device__ __forceinline__ q64 neg(q64 a) { return {-a.v}; }
    static __device__ __forceinline__ q64 mul(q64 a, q64 w) { return {q_mul(a.v, w.v)}; }
    static __device__ __forceinline__ q64 norm(q64 a) { return a; }
    // sqrt(1/2) 2^60
    static __device__ __forceinline__ q64 rsqrt2() { return {815238614083298888ll}; }
};

// a w / 2^s without its last shift: high + middle products as a 64-bit number
// of weight 2^-s, to be shifted right by s.  c is the middle products' start:
// q_round_start(s) rounds the result.  (A tie, which only twiddles that are powers
// of two meet, but for those with one point in 2^s, goes up; with one less it goes
// down.  The passes take the two in turn: all ties up made the zero frequency of
// e0 plus a small tail 4e-16 too large at M = 2^10.)  To it they add the mean of the low
// products that are left out (the low limbs of a are 2^29 in the mean): the same
// twiddle serves every entry of a matrix, so that the offset would add up over a
// row.
__device__ __forceinline__ long long q_round_start(int s) { return 1ll << (29 + s); }
__device__ __forceinline__ cx<q64> c_mul(cx<q64> a, qtw w, long long c = 1ll << 29)
{
    const int arh = q_top30(a.re.v), arl = q_lo(a.re.v) & Q_MASK30;
    const int aih = q_top30(a.im.v), ail = q_lo(a.im.v) & Q_MASK30;
    const int nh = -aih, nl = -ail;
    long long mr = q_wide(arh, w.rl, c + (long long)((w.rl - w.il) >> 1));
    long long mi = q_wide(arh, w.il, c + (long long)((w.rl + w.il) >> 1));
    mr = q_wide(arl, w.rh, mr);
    mi = q_wide(arl, w.ih, mi);
    mr = q_wide(nh, w.il, mr);
    mi = q_wide(aih, w.rl, mi);
    mr = q_wide(nl, w.ih, mr);
    mi = q_wide(ail, w.rh, mi);
    return {{q_wide(nh, w.ih, q_wide(arh, w.rh, q_sar30(mr)))}, {q_wide(aih, w.rh, q_wide(arh, w.ih, q_sar30(mi)))}};
}

// a / 2^s rounded half to even, s < 32
__device__ __forceinline__ long long q_shift_even(long long a, int s)
{
    const long long h = s ? (1ll << (s - 1)) - 1 + ((a >> s) & 1) : 0;
    return (a + h) >> s;
}

// a >> s, s < 32
__device__ __forceinline__ cx<q64> q_shift(cx<q64> a, int s)
{
    const int rl = (int)__funnelshift_r((unsigned)q_lo(a.re.v), (unsigned)q_hi(a.re.v), s), rh = q_hi(a.re.v) >> s;
    const int il = (int)__funnelshift_r((unsigned)q_lo(a.im.v), (unsigned)q_hi(a.im.v), s), ih = q_hi(a.im.v) >> s;
    return {{q_join(rl, rh)}, {q_join(il, ih)}};
}

// the magnitude bits of a value's high word
__device__ __forceinline__ unsigned q_bits(q64 a)
{
    const int h = (int)(a.v >> 32);
    return (unsigned)(h ^ (h >> 31));
}

// limbs with balanced 30-bit low parts
__device__ __forceinline__ qtw q_limbs(cx<q64> v)
{
    const int rl = (int)((unsigned)v.re.v << 2) >> 2, il = (int)((unsigned)v.im.v << 2) >> 2;
    return {(int)((v.re.v - rl) >> 30), rl, (int)((v.im.v - il) >> 30), il};
}

// the limbs of w / 2^s (conjugated if conj)
__device__ __forceinline__ qtw q_twiddle(cx<double> w, int s, bool conj)
{
    const long long r = q_decode(w.re, 1022 + s, Q_TOP).v, i = q_decode(w.im, 1022 + s, Q_TOP, conj ? -1 : 0).v;
    return q_limbs({{r}, {i}});
}

// (U : rest) with U < 2^63 and 32 bits of rest, rounded to a double: leading bit
// 63 - lz of U gets the biased exponent eb - lz; neg flips the sign
__device__ __forceinline__ double q_pack(unsigned long long U, unsigned rest, int eb, bool neg)
{
    const bool big = (U >> 31) != 0ull;
    const unsigned long long W = big ? U : (U << 32) | rest;
    const int lz = __clzll((long long)W);
    const unsigned long long n = (W << (lz & 63)) | (big ? ((unsigned long long)rest << lz) >> 32 : 0ull);
    const unsigned long long m = q_round11(n);
    const int e = eb - lz - (big ? 0 : 32);
    const unsigned long long b = W == 0ull ? 0ull : ((unsigned long long)(unsigned)(e - 1) << 52) + m;
    return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ull : 0ull)));
}

// H 2^32 + L rounded to a double (|H| < 2^50, |L| < 2^50): the sum of a
// product's weight groups, two halves of four
__device__ __forceinline__ double q96_to_double(long long H, long long L)
{
    const long long hi = H + (L >> 32);
    const unsigned lo = (unsigned)L;
    const bool neg = hi < 0;
    const unsigned al = neg ? 0u - lo : lo;
    const unsigned long long ah = (unsigned long long)(neg ? ~hi + (lo == 0u ? 1 : 0) : hi);
    return q_pack((ah << 13) | (al >> 19), al << 13, 1023 + 63 + 19, neg);
}

// hi 2^30 + mid rounded to a double (0 <= mid < 2^30, |hi| < 2^63)
__device__ __forceinline__ double q94_to_double(long long hi, int mid)
{
    const unsigned lo = (unsigned)mid << 2;
    const bool neg = hi < 0;
    const unsigned al = neg ? 0u - lo : lo;
    const unsigned long long ah = (unsigned long long)(neg ? ~hi + (lo == 0u ? 1 : 0) : hi);
    return q_pack(ah, al, 1023 + 63 + 30, neg);
}

// x 2^de by its exponent (zero below the normal range, infinity above it)
__device__ __forceinline__ double q_scale(double x, int de)
{
    const int hw = __double2hiint(x), e = ((hw >> 20) & 0x7ff) + de;
    const bool z = (hw & 0x7ff00000) == 0 || e < 1;
    const int sg = hw & (int)0x80000000;
    const int h = z ? sg : (e > 2046 ? sg | 0x7ff00000 : hw + (de << 20));
    return __hiloint2double(h, z || e > 2046 ? 0 : __double2loint(x));
}

// 2 Xh(f) = s + t and 2 Xh(M - f) = conj(s - t) of packed values a = Z(f),
// b = Z(M - f) as fixed-point numbers aligned to ex at 2^top (|re|, |im| < 2^top):
// s = a + conj b, t = w (-i) (a - conj b).
__device__ __forceinline__ void q_split(cx<double> za, cx<double> zb, qtw w, int ex, int top, cx<q64> &s, cx<q64> &t)
{
    const cx<q64> a = {q_decode(za.re, ex, top), q_decode(za.im, ex, top)};
    const cx<q64> b = {q_decode(zb.re, ex, top), q_decode(zb.im, ex, top)};
    s = {{a.re.v + b.re.v}, {a.im.v - b.im.v}};
    t = c_mul(cx<q64>{{a.im.v + b.im.v}, {b.re.v - a.re.v}}, w);
}

// the high word of a magnitude (nonnegative: orders like the magnitude), and
// the alignment exponent of a row or column from the largest of them: every
// magnitude below 63/64 2^(ex - 1022); Q_NONFINITE when an Inf or NaN is among them
__device__ __forceinline__ unsigned q_magnitude(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ int q_align(unsigned m)
{
    const int ex = max(Q_EXMIN, (int)((m + 0x8000u) >> 20));
    return ex >= 2047 ? Q_NONFINITE : ex;
}

// The packed spectrum of the pair f, M - f from cf = C(f) / 2, cg = C(M - f) / 2:
// ZC(f) = s + i p, ZC(M - f) = conj s + i conj p,
// s = cf + conj cg, p = conj w (cf - conj cg).
__device__ __forceinline__ void q_merge(cx<double> cf, cx<double> cg, cx<double> w, cx<double> &zf, cx<double> &zg)
{
    const double sr = cf.re + cg.re, si = cf.im - cg.im;
    const double dr = cf.re - cg.re, di = cf.im + cg.im;
    const double pr = fma(w.re, dr, w.im * di), pi = fma(w.re, di, -(w.im * dr));
    zf = {sr - pi, si + pr};
    zg = {sr + pi, pr - si};
}
