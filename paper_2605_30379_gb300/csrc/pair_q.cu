// pair_q.cu -- FP64 per-frequency complex matrix products (Eq.
// (fft-convolution): C(phi) = X(phi) Y(phi), X r x m, Y m x c) in 64-bit fixed
// point, for matrices that fit in shared memory: the square ones too small for
// the tensor-core tiles and the rectangular ones.
//
// The FP64 pipe gives two multiply-adds per clock and SM, a 32 x 32 -> 64 bit
// integer multiply-add sixty; a complex multiply-add takes sixteen of the
// latter on numbers of two limbs.  Rows of X and columns of Y are aligned to
// their largest magnitude over both frequencies of a pair (2 Xh and 2 Yh below
// 2^58 to 2^60, as m allows: a high limb and a balanced 30-bit low limb), the
// limb products
// accumulate exactly in 64 bits by weight (the lower sums are carried upward
// every eight terms), and each sum is rounded once to FP64.  (Without the low
// products, a quarter of the work, the error of a Weibull d = 16, N = 2048
// inverse rises from FP64's 1.2e-15 to 9e-15: e0 - q is singular at frequency
// zero.)  Outputs whose terms lie far below their row and column bounds are summed
// again by the same CTA (graded.cuh).
//
// One CTA takes the pairs p0 .. p0 + pp - 1 (pp so that its outputs fill the
// threads once, fewer when there are fewer pairs than SMs): it loads their
// spectra, splits both frequencies into limbs in shared memory, and every
// thread forms C(f)_ij and C(M - f)_ij of its outputs and merges them.  No work
// is done for padding.  Against the FP64-pipe tiles of 16, 24 and 32 it
// replaces: the products of a d = 16, N = 8192 inverse 1.1 -> 0.4 ms, of the
// d = 4, N = 2^15 renewal equation (a 16 x 16 tile) 3.2 -> 0.1 ms, of an
// entrance with 18 x 18 blocks, N = 10000, 6.4 -> 1.2 ms.
#include <algorithm>

#include "graded.cuh"
#include "mrc_internal.h"

namespace {

constexpr int NT = 128;
// raw values below 2^top, 2 Xh below 2^(top + 2), so that m products of two
// numbers of such moduli stay below 2^63 with their 2^60 taken off
__device__ __forceinline__ int top_for(int m) { return m <= 4 ? 58 : (m <= 31 ? 57 : 56); }
constexpr int PAIR_MAX = 200 * 1024, SMEM_MAX = 213 * 1024;  // of a pair; of a CTA, with the logarithms

// t / d for t, d < 2^16 by a multiplication (a division by a run-time number
// takes some 25 instructions, and every entry and output is indexed by three)
struct FastDiv {
    unsigned m, d;
    __device__ __forceinline__ explicit FastDiv(int d_) : m(0xffffffffu / (unsigned)d_ + 1u), d((unsigned)d_) {}
    __device__ __forceinline__ int div(int t) const { return d == 1u ? t : (int)__umulhi((unsigned)t, m); }
};

// accumulators of one complex sum: 2^60 h + 2^30 m + l
struct acc {
    long long hr, hi, mr, mi, lr, li;
};

__device__ __forceinline__ void mac(acc &a, const qtw &x, const qtw &y)
{
    const int nh = -x.ih, nl = -x.il;
    a.hr = q_wide(nh, y.ih, q_wide(x.rh, y.rh, a.hr));
    a.hi = q_wide(x.ih, y.rh, q_wide(x.rh, y.ih, a.hi));
    a.mr = q_wide(nl, y.ih, q_wide(nh, y.il, q_wide(x.rl, y.rh, q_wide(x.rh, y.rl, a.mr))));
    a.mi = q_wide(x.il, y.rh, q_wide(x.ih, y.rl, q_wide(x.rl, y.ih, q_wide(x.rh, y.il, a.mi))));
    a.lr = q_wide(nl, y.il, q_wide(x.rl, y.rl, a.lr));
    a.li = q_wide(x.il, y.rl, q_wide(x.rl, y.il, a.li));
}

__device__ __forceinline__ void fold(acc &a)
{
    a.mr += a.lr >> 30;
    a.mi += a.li >> 30;
    a.lr &= Q_MASK30;
    a.li &= Q_MASK30;
    a.hr += a.mr >> 30;
    a.hi += a.mi >> 30;
    a.mr &= Q_MASK30;
    a.mi &= Q_MASK30;
}

size_t pair_bytes(int r, int m, int c)
{
    return 2 * sizeof(qtw) * ((size_t)r * m + (size_t)m * c) + sizeof(qtw) + sizeof(int) * ((size_t)r + c);
}
// shared memory of a CTA of pp pairs: theirs and the logarithms at frequency 0 of
// X's diagonal and Y
size_t cta_bytes(int pp, int r, int m, int c) { return pp * pair_bytes(r, m, c) + sizeof(short) * ((size_t)r + (size_t)m * c); }

// The CTA's shared memory
struct Smem {
    qtw *sf, *sg, *stw;  // per pair: X then Y entries at f and g, twiddle
    unsigned *bnd;       // per pair: r row and c column bounds
    short *x0, *y0;      // logarithms at frequency 0: X_ii (column 0 where X has one), Y
    __device__ __forceinline__ Smem(unsigned char *p, int pp, int ex2, int r, int c)
        : sf(reinterpret_cast<qtw *>(p)), sg(sf + pp * ex2), stw(sg + pp * ex2),
          bnd(reinterpret_cast<unsigned *>(stw + pp)), x0(reinterpret_cast<short *>(bnd + pp * (r + c))), y0(x0 + r)
    {
    }
};

// A lower bound of a term's size from the limbs' high parts (2 Xh and 2 Yh: at most
// four times the packed values that gr_sound compares), over 2^60
__device__ __forceinline__ float term_size(const qtw &a, const qtw &b, const qtw &u, const qtw &v)
{
    return (float)max(max(abs(a.rh), abs(a.ih)), max(abs(b.rh), abs(b.ih))) *
           (float)max(max(abs(u.rh), abs(u.ih)), max(abs(v.rh), abs(v.ih)));
}

// The logarithm of the largest term of an output from its row of X and its column of Y
// in global memory: packed values at rows f and g
__device__ __forceinline__ int largest_term(const cx<double> *xf, const cx<double> *xg, const cx<double> *yf,
                                            const cx<double> *yg, int m, int c)
{
    int l = 2 * GR_ZERO;
    for (int k = 0; k < m; ++k)
        l = max(l, gr_log(max(gr_magnitude(xf[k]), gr_magnitude(xg[k]))) +
                       gr_log(max(gr_magnitude(yf[k * c]), gr_magnitude(yg[k * c]))));
    return l;
}

// One unsound output by one warp, with every entry aligned by itself, its terms
// across the lanes: for CTAs with a few of them (one output in a thousand of an
// entrance with 18 x 18 blocks, N = 10000, is 2^-14 below its bounds; splitting the whole
// pairs again for it took the call from 2.86 to 3.02 ms)
__device__ __forceinline__ void redo_one(const PairArgs &a, int64_t f, int i, int j, qtw w)
{
    const int r = a.r, m = a.m, c = a.c, lane = threadIdx.x & 31;
    const int64_t g = (a.M - f) & (a.M - 1), EX = (int64_t)r * m, EY = (int64_t)m * c, EC = (int64_t)r * c;
    const cx<double> *X = reinterpret_cast<const cx<double> *>(a.zx) + i * m;
    const cx<double> *Y = reinterpret_cast<const cx<double> *>(a.zy) + j;
    int G = 2 * GR_ZERO;
    for (int k = lane; k < m; k += 32) {
        cx<double> xf = X[f * EX + k], xg = X[g * EX + k], yf = Y[f * EY + k * c], yg = Y[g * EY + k * c];
        G = max(G, (gr_scaled(xf, xg) >> 4) + (gr_scaled(yf, yg) >> 4));
    }
    G = __reduce_max_sync(0xffffffffu, G);
    long long v[4] = {0, 0, 0, 0};
    for (int k = lane; k < m; k += 32) {
        short lx, ly;
        qtw xf, xg, yf, yg;
        gr_split(X[f * EX + k], X[g * EX + k], w, lx, xf, xg);
        gr_split(Y[f * EY + k * c], Y[g * EY + k * c], w, ly, yf, yg);
        const int s = G - (lx >> 4) - (ly >> 4);
        if (s > 61) continue;
        gr_mac(v[0], v[1], xf, yf, s);
        gr_mac(v[2], v[3], xg, yg, s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] += __shfl_xor_sync(0xffffffffu, v[u], o);
    if (lane != 0) return;
    cx<double> *ZC = reinterpret_cast<cx<double> *>(a.zc) + (int64_t)i * c + j;
    const cx<double> *tw = reinterpret_cast<const cx<double> *>(a.tw);
    cx<double> zf, zg;
    q_merge(gr_value(v[0], v[1], G), gr_value(v[2], v[3], G), tw[f << (a.tw_log - a.logM - 1)], zf, zg);
    ZC[f * EC] = zf;
    if (g != f) ZC[g * EC] = zg;
}

// All unsound outputs of the CTA's pairs.  One frequency after the other, so that
// the limbs of the first sum leave room for the entries' logarithms; C(f) waits in
// the output.
__device__ __forceinline__ void pairq_redo(const PairArgs *ap, int64_t p0)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const PairArgs &a = *ap;
    const int r = a.r, m = a.m, c = a.c, EX = r * m, EC = r * c, ex2 = EX + m * c;
    const int np = (int)min((int64_t)a.pp, a.npairs - p0);
    const Smem s(smem, a.pp, ex2, r, c);
    short *const lp = reinterpret_cast<short *>(s.sg), *const l0 = lp + np * ex2;  // of the pairs' entries, of those at frequency 0
    const cx<double> *ZX = reinterpret_cast<const cx<double> *>(a.zx), *ZY = reinterpret_cast<const cx<double> *>(a.zy);
    cx<double> *ZC = reinterpret_cast<cx<double> *>(a.zc);
    const cx<double> *tw = reinterpret_cast<const cx<double> *>(a.tw);
    auto packed = [&](int64_t row, int e) { return e < EX ? ZX[row * EX + e] : ZY[row * (ex2 - EX) + e - EX]; };
    for (int t = threadIdx.x; t < np * ex2; t += NT) {
        const int q = t / ex2, e = t - q * ex2;
        const int64_t f = p0 + q, g = (a.M - f) & (a.M - 1);
        lp[t] = gr_log(max(gr_magnitude(packed(f, e)), gr_magnitude(packed(g, e))));
        if (q == 0) l0[e] = gr_log(gr_magnitude(packed(0, e)));
    }
    __syncthreads();
    for (int phase = 0; phase < 2; ++phase) {
        for (int t = threadIdx.x; t < np * ex2; t += NT) {
            const int q = t / ex2, e = t - q * ex2;
            const int64_t f = p0 + q, g = (a.M - f) & (a.M - 1);
            qtw vf, vg;
            gr_split(packed(f, e), packed(g, e), s.stw[q], lp[t], vf, vg);
            s.sf[t] = phase == 0 ? vf : vg;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < np * EC; t += NT) {
            const int q = t / EC, e = t - q * EC, i = e / c, j = e - i * c, xo = q * ex2 + i * m, yo = q * ex2 + EX + j;
            const unsigned *b = s.bnd + q * (r + c);
            if (gr_sound(l0 + i * m, l0 + EX + j, lp + xo, lp + yo, m, c, q_align(b[i]), q_align(b[r + j]), a.logM)) continue;
            const cx<double> v = gr_sum(s.sf + xo, s.sf + yo, lp + xo, lp + yo, m, c);
            const int64_t f = p0 + q, g = (a.M - f) & (a.M - 1);
            if (phase == 0) {
                ZC[f * EC + e] = v;
                continue;
            }
            cx<double> zf, zg;
            q_merge(ZC[f * EC + e], v, tw[f << (a.tw_log - a.logM - 1)], zf, zg);
            ZC[f * EC + e] = zf;
            if (g != f) ZC[g * EC + e] = zg;
        }
        __syncthreads();
    }
}

__device__ __forceinline__ void pairq_body(const PairArgs &a, int64_t p0)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int LIST = 64;
    __shared__ int nredo;  // unsound outputs, the first of them
    __shared__ unsigned short redo[LIST];
    const int r = a.r, m = a.m, c = a.c, EX = r * m, EY = m * c, EC = r * c, ex2 = EX + EY;
    const int np = (int)min((int64_t)a.pp, a.npairs - p0);
    const Smem sm(smem, a.pp, ex2, r, c);
    qtw *sf = sm.sf, *sg = sm.sg, *stw = sm.stw;
    unsigned *bnd = sm.bnd;
    const cx<double> *ZX = reinterpret_cast<const cx<double> *>(a.zx), *ZY = reinterpret_cast<const cx<double> *>(a.zy);
    cx<double> *ZC = reinterpret_cast<cx<double> *>(a.zc);
    const cx<double> *tw = reinterpret_cast<const cx<double> *>(a.tw);
    const int64_t M = a.M;
    const int tws = a.tw_log - a.logM - 1;
    const int tid = threadIdx.x, top = top_for(m);
    const FastDiv dex2(ex2), dm(m), dc(c), dEC(EC);

    if (tid == 0) nredo = 0;
    for (int t = tid; t < np * (r + c); t += NT) bnd[t] = 0u;
    for (int t = tid; t < np; t += NT) stw[t] = q_twiddle(tw[(p0 + t) << tws], 0, false);
    overlap_release();
    overlap_wait();
    __syncthreads();
    // raw spectra of both rows of every pair, and the row and column bounds
    for (int t = tid; t < np * ex2; t += NT) {
        const int q = dex2.div(t), e = t - q * ex2;
        const int64_t f = p0 + q, g = (M - f) & (M - 1);
        const bool x = e < EX;
        const int ee = x ? e : e - EX;
        const cx<double> za = x ? ZX[f * EX + ee] : ZY[f * EY + ee], zb = x ? ZX[g * EX + ee] : ZY[g * EY + ee];
        reinterpret_cast<cx<double> *>(sf)[t] = za;
        reinterpret_cast<cx<double> *>(sg)[t] = zb;
        const int rc = x ? dm.div(ee) : ee - dc.div(ee) * c;
        // frequency 0: Y and X's diagonal
        if (q == 0 && !x) sm.y0[ee] = gr_log(gr_magnitude(ZY[ee]));
        if (q == 0 && x && ee == rc * m + min(rc, m - 1)) sm.x0[rc] = gr_log(gr_magnitude(ZX[ee]));
        atomicMax(&bnd[q * (r + c) + (x ? rc : r + rc)], max(gr_magnitude(za), gr_magnitude(zb)));
    }
    __syncthreads();
    // the split of both frequencies, in place (every thread its own entries)
    for (int t = tid; t < np * ex2; t += NT) {
        const int q = dex2.div(t), e = t - q * ex2;
        const bool x = e < EX;
        const int ee = x ? e : e - EX;
        cx<q64> s, u;
        q_split(reinterpret_cast<cx<double> *>(sf)[t], reinterpret_cast<cx<double> *>(sg)[t], stw[q],
                q_align(bnd[q * (r + c) + (x ? dm.div(ee) : r + ee - dc.div(ee) * c)]), top, s, u);
        sf[t] = q_limbs(c_add(s, u));
        sg[t] = q_limbs({{s.re.v - u.re.v}, {u.im.v - s.im.v}});
    }
    __syncthreads();
    const int guard = gr_guard(m);
    const float own_min = exp2f((float)(2 * top - 60 - guard + 4));  // term_size of an output sound by its own terms
    for (int t = tid; t < np * EC; t += NT) {
        const int q = dEC.div(t), e = t - q * EC, i = dc.div(e), j = e - i * c;
        const int xo = q * ex2 + i * m, yo = q * ex2 + EX + j;
        acc af{}, ag{};
        for (int k0 = 0; k0 < m; k0 += 8) {
            const int kn = min(8, m - k0);
#pragma unroll 4
            for (int k = k0; k < k0 + kn; ++k) {
                mac(af, sf[xo + k], sf[yo + k * c]);
                mac(ag, sg[xo + k], sg[yo + k * c]);
            }
            fold(af);
            fold(ag);
        }
        const int ax = q_align(bnd[q * (r + c) + i]), ay = q_align(bnd[q * (r + c) + r + j]);
        // gr_sound, the likely reasons first: the term k = i at frequency 0, the terms k = i
        // and k = j of the pair itself, all terms at frequency 0
        const int ki = min(i, m - 1), kj = min(j, m - 1);
        if (!gr_sound_by(ax, ay, sm.x0[i] + sm.y0[ki * c + j], a.logM, guard)) {
            const float s = fmaxf(term_size(sf[xo + ki], sg[xo + ki], sf[yo + ki * c], sg[yo + ki * c]),
                                  term_size(sf[xo + kj], sg[xo + kj], sf[yo + kj * c], sg[yo + kj * c]));
            if (!gr_in_range(ax, ay) || s < own_min) {
                int g0 = 2 * GR_ZERO;
                for (int k = 0; k < m; ++k) g0 = max(g0, gr_log(gr_magnitude(ZX[i * m + k])) + sm.y0[k * c + j]);
                if (!gr_sound_by(ax, ay, g0, a.logM, guard) && max(ax, ay) < Q_NONFINITE) {
                    const int64_t f = p0 + q, g = (M - f) & (M - 1);
                    const int gp = largest_term(ZX + f * EX + i * m, ZX + g * EX + i * m, ZY + f * EY + j, ZY + g * EY + j, m, c);
                    if (gp >= 0 && !gr_sound_by(ax, ay, gp, 0, guard)) {
                        const int n = atomicAdd(&nredo, 1);
                        if (n < LIST) redo[n] = (unsigned short)t;
                    }
                }
            }
        }
        const int de = ax + ay - 2017 - 2 * top;  // the alignments, the limbs, the split's factors 2 and the merge's 1/2
        cx<double> cf = {q_scale(q94_to_double(af.hr, (int)af.mr), de), q_scale(q94_to_double(af.hi, (int)af.mi), de)};
        cx<double> cg = {q_scale(q94_to_double(ag.hr, (int)ag.mr), de), q_scale(q94_to_double(ag.hi, (int)ag.mi), de)};
        if (max(ax, ay) >= Q_NONFINITE) cf.re = cf.im = cg.re = cg.im = __longlong_as_double(0x7ff8000000000000ll);
        const int64_t f = p0 + q, g = (M - f) & (M - 1);
        cx<double> zf, zg;
        q_merge(cf, cg, tw[f << tws], zf, zg);
        ZC[f * EC + e] = zf;
        if (g != f) ZC[g * EC + e] = zg;
    }
    __syncthreads();
    if (nredo > LIST) pairq_redo(&a, p0);
    else
        for (int n = tid >> 5; n < nredo; n += NT / 32) {
            const int t = redo[n], q = dEC.div(t), e = t - q * EC, i = dc.div(e);
            redo_one(a, p0 + q, i, e - i * c, stw[q]);
        }
}

// Product with a diagonal right factor, C(f)_ij = X(f)_ij Y(f)_j: a complex
// product per entry, with each pair of packed values aligned by itself and
// merged in fixed point.  The 56 FP64 operations per pair of entries were what
// bound it (1.1 ms at d = 32, M = 2^14, where its bytes take 0.08 ms; now
// 0.21).  CTA:
// the pairs p0 .. p0 + pp - 1; Y's factors once per column.
__global__ void __launch_bounds__(NT) pairdiagq_kernel(const PairArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int r = a.r, c = a.c, E = r * c;
    const int64_t p0 = (int64_t)blockIdx.x * a.pp, M = a.M;
    const int np = (int)min((int64_t)a.pp, a.npairs - p0), tws = a.tw_log - a.logM - 1, tid = threadIdx.x;
    qtw *yf = reinterpret_cast<qtw *>(smem), *yg = yf + a.pp * c, *stw = yg + a.pp * c;
    int *yex = reinterpret_cast<int *>(stw + a.pp);
    const cx<double> *ZX = reinterpret_cast<const cx<double> *>(a.zx), *ZY = reinterpret_cast<const cx<double> *>(a.zy);
    cx<double> *ZC = reinterpret_cast<cx<double> *>(a.zc);
    const cx<double> *tw = reinterpret_cast<const cx<double> *>(a.tw);
    // the alignment; tiny values are scaled up by 2^up for it
    auto align = [](cx<double> &za, cx<double> &zb, int &up) {
        unsigned b = max(gr_magnitude(za), gr_magnitude(zb));
        up = 0;
        if (b < ((unsigned)Q_TINY << 20) && b != 0u) {
            up = Q_UP;
            za = c_scal(za, Q_SCALE);
            zb = c_scal(zb, Q_SCALE);
            b = max(gr_magnitude(za), gr_magnitude(zb));
        }
        return q_align(b);
    };
    // 2 Xh(f) and 2 Xh(M - f), moduli below 2^60
    auto split = [](cx<double> za, cx<double> zb, qtw w, int ex, cx<q64> &xf, cx<q64> &xg) {
        cx<q64> s, t;
        q_split(za, zb, w, ex, Q_TOP - 2, s, t);
        xf = c_add(s, t);
        xg = {{s.re.v - t.re.v}, {t.im.v - s.im.v}};
    };
    for (int t = tid; t < np * c; t += NT) {
        const int q = t / c, j = t - q * c;
        const int64_t f = p0 + q, g = (M - f) & (M - 1);
        const qtw w = q_twiddle(tw[f << tws], 0, false);
        if (j == 0) stw[q] = q_twiddle(c_conj(tw[f << tws]), 0, false);
        cx<double> za = ZY[f * c + j], zb = ZY[g * c + j];
        int up;
        const int ex = align(za, zb, up);
        cx<q64> vf, vg;
        split(za, zb, w, ex, vf, vg);
        yf[t] = q_limbs(vf);
        yg[t] = q_limbs(vg);
        yex[t] = ex - up;
    }
    __syncthreads();
    for (int t = tid; t < np * E; t += NT) {
        const int q = t / E, e = t - q * E, j = e % c;
        const int64_t f = p0 + q, g = (M - f) & (M - 1);
        cx<double> za = ZX[f * E + e], zb = ZX[g * E + e];
        int up;
        const int ex = align(za, zb, up), ey = yex[q * c + j];
        const qtw wc = stw[q];  // conj w
        cx<q64> xf, xg;
        split(za, zb, qtw{wc.rh, wc.rl, -wc.ih, -wc.il}, ex, xf, xg);
        const cx<q64> cf = c_mul(xf, yf[q * c + j]), cg = c_mul(xg, yg[q * c + j]);
        // s = cf + conj cg, p = conj w (cf - conj cg); ZC(f) = s + i p, ZC(M - f) = conj s + i conj p
        const cx<q64> s = {{cf.re.v + cg.re.v}, {cf.im.v - cg.im.v}};
        const cx<q64> p = c_mul(cx<q64>{{cf.re.v - cg.re.v}, {cf.im.v + cg.im.v}}, wc);
        // cf = 4 C(f) 2^(2 1080 - 60 - ex - ey); the merge halves
        const int eb = ex - up + ey - 2 * (Q_TOP - 2 + 1022) + Q_TOP - 3 + 1086;
        cx<double> zf = {q_encode({s.re.v - p.im.v}, eb, 0u), q_encode({s.im.v + p.re.v}, eb, 0u)};
        cx<double> zg = {q_encode({s.re.v + p.im.v}, eb, 0u), q_encode({p.re.v - s.im.v}, eb, 0u)};
        if (max(ex, ey) >= Q_NONFINITE) zf.re = zf.im = zg.re = zg.im = __longlong_as_double(0x7ff8000000000000ll);
        ZC[f * E + e] = zf;
        if (g != f) ZC[g * E + e] = zg;
    }
}

__global__ void __launch_bounds__(NT) pairq_kernel(const __grid_constant__ PairArgs a) { pairq_body(a, (int64_t)blockIdx.x * a.pp); }

__global__ void __launch_bounds__(NT) pairq_seg_kernel(const __grid_constant__ SegParams<PairArgs> P)
{
    const int s = seg_find(P, blockIdx.x);
    pairq_body(P.a[s], (int64_t)(blockIdx.x - P.first[s]) * P.a[s].pp);
}

} // namespace

// Besides the shared memory: sums of up to 79 terms stay below 2^63 (gr_sum; the limb
// sums 127), and outputs are counted in 16 bits (FastDiv, the list of unsound ones)
bool mrc_pairq_supported(int r, int m, int c)
{
    return m <= 79 && (int64_t)r * c < 65536 && pair_bytes(r, m, c) <= (size_t)PAIR_MAX;
}

// Pairs per CTA: outputs for every thread, but no fewer CTAs than SMs where the
// pairs allow, and at most 48 KB of shared memory when one pair needs less
// (several CTAs per SM hide the loads of each other)
int mrc_pairq_pp(int64_t npairs, int r, int m, int c)
{
    const int64_t fill = std::max(1, NT / (r * c)), spread = std::max<int64_t>(1, npairs / 152);
    const int64_t fit = std::max<int64_t>(1, (int64_t)(48 * 1024 / pair_bytes(r, m, c)));
    return (int)std::min(std::min(fill, spread), fit);
}

cudaError_t mrc_pairq_init(void)
{
    cudaError_t e = cudaFuncSetAttribute(pairq_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(pairq_seg_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
}

cudaError_t mrc_pairq(const PairArgs &a0, int kclass, cudaStream_t st)
{
    PairArgs a = a0;
    a.pp = mrc_pairq_pp(a.npairs, a.r, a.m, a.c);
    const double by = (double)a.M * ((double)a.r * a.m + (double)a.m * a.c + (double)a.r * a.c) * 16.0;
    mrc_prof_pre(kclass, st);
    const unsigned grid = (unsigned)((a.npairs + a.pp - 1) / a.pp);
    const size_t smem = cta_bytes(a.pp, a.r, a.m, a.c);
    if (grid <= MRC_OVERLAP_CTAS) {
        const cudaError_t e = mrc_launch_overlapped(pairq_kernel, dim3(grid), NT, smem, st, a);
        if (e != cudaSuccess) return e;
    } else {
        pairq_kernel<<<grid, NT, smem, st>>>(a);
    }
    mrc_prof_post(kclass, st, by, 8.0 * a.r * a.m * a.c * (double)(a.M + 1));
    return cudaGetLastError();
}

cudaError_t mrc_pairdiagq(const PairArgs &a0, int kclass, cudaStream_t st)
{
    PairArgs a = a0;
    const int64_t fill = std::max(1, 2 * NT / (a.r * a.c)), spread = std::max<int64_t>(1, a.npairs / 304);
    a.pp = (int)std::min(fill, spread);
    const size_t sm = a.pp * (2 * sizeof(qtw) * a.c + sizeof(qtw) + sizeof(int) * a.c);
    mrc_prof_pre(kclass, st);
    pairdiagq_kernel<<<(unsigned)((a.npairs + a.pp - 1) / a.pp), NT, sm, st>>>(a);
    mrc_prof_post(kclass, st, (double)a.M * (2.0 * a.r * a.c + a.c) * 16.0, 6.0 * a.r * a.c * (double)(a.M + 1));
    return cudaGetLastError();
}

cudaError_t mrc_pairq_seg(const SegParams<PairArgs> &P, unsigned nctas, double bytes, double flops, int kclass,
                          cudaStream_t st)
{
    if (P.nseg <= 0 || nctas == 0) return cudaSuccess;
    size_t sm = 0;
    for (int s = 0; s < P.nseg; ++s) sm = std::max(sm, cta_bytes(P.a[s].pp, P.a[s].r, P.a[s].m, P.a[s].c));
    mrc_prof_pre(kclass, st);
    pairq_seg_kernel<<<nctas, NT, sm, st>>>(P);
    mrc_prof_post(kclass, st, bytes, flops);
    return cudaGetLastError();
}
