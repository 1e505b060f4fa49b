// fftq.cuh -- FFT passes of the FP64 path in 64-bit block floating point
// (q64.cuh), over the same data, layout and pass structure as the passes of
// kernels.cuh.
//
// What bounds them: integer instructions (about 330 per point and pass of radix
// 2^9, against the 60 FP64 operations per point of a two-pass transform that kept
// the FP64 pipe busy ten times as long), and in small launches the instruction
// caches: with every point's conversion unrolled in registers the first launch of
// a radix took 20 to 25 us where the next took 5, and warps waited for
// instructions 13 of 18 cycles.  So the points live in shared memory between
// the phases: asynchronous copies bring them in, rolled loops convert them (one
// copy of the code), one loop body serves every radix-8 stage after the first,
// and the inverse transform is the forward one with real and imaginary parts
// exchanged on the way in and out (whole inverse d = 3, N = 2^11 270 -> 190 us,
// d = 16, N = 2^13 1.31 -> 1.09 ms; large launches as before, 16 ps per point of a
// radix-2^7 pass).
#pragma once
#include "kernels.cuh"
#include "q64.cuh"

template <int LOGR, int EC>
struct QPlan {
    static constexpr int R = 1 << LOGR;
    static constexpr int FIRST = (LOGR < 3) ? LOGR : ((LOGR % 3) == 0 ? 3 : (LOGR % 3));
    static constexpr int NSTAGE = (LOGR < 3) ? 1 : 1 + (LOGR - FIRST) / 3;
    static constexpr int EPT = (LOGR < 3) ? R : 8;  // points per thread
    static constexpr int NT = R * EC / EPT;         // at most 1024 (R = 2^10, 8 entries)
    static constexpr int LEC = EC == 1 ? 0 : EC == 4 ? 2 : 3;
    // resident CTAs per SM asked of the compiler: 1024 threads of 64 registers
    static constexpr int MINB = NT < 64 ? 1 : 1024 / NT;
};

__device__ __forceinline__ void q_copy(unsigned dst, const void *src, bool ok, int bytes)
{
    // bytes past the valid rows and entries are zero-filled, nothing is read for them
    if (bytes == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(ok ? 8 : 0) : "memory");
}

// the OR (or maximum) of a thread's value over its entry column, to smem[e]
template <int EC, int NT, bool MAX>
__device__ __forceinline__ void q_column(unsigned m, unsigned *dst, int tid)
{
    constexpr int NL = NT < 32 ? NT : 32;  // lanes of a warp in use
    constexpr unsigned mask = NL == 32 ? 0xffffffffu : (1u << (NL & 31)) - 1u;
#pragma unroll
    for (int o = EC; o < NL; o <<= 1) {
        const unsigned w = __shfl_xor_sync(mask, m, o);
        m = MAX ? max(m, w) : m | w;
    }
    if ((tid & 31) < EC) {
        if (MAX) atomicMax(&dst[tid & (EC - 1)], m);
        else atomicOr(&dst[tid & (EC - 1)], m);
    }
}

template <int LOGR, int EC>
__device__ __forceinline__ void fftq_body(const FftArgs &a, int64_t j, int e0)
{
    using P = QPlan<LOGR, EC>;
    constexpr int R = P::R, NT = P::NT, EPT = P::EPT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<q64> *sm = reinterpret_cast<cx<q64> *>(smem_raw);  // [R][EC]: point rho, entry e at rho EC + e
    qtw *stw = reinterpret_cast<qtw *>(sm + R * EC);      // [R]  W_R^t
    qtw *spt = stw + R;                                   // [R]  inter-pass twiddles / 2^FIRST
    __shared__ unsigned smax[EC];                         // largest magnitude (high word) per entry
    __shared__ unsigned sor[3 * EC];                      // magnitude bits after each stage but the last
    const cx<double> *tw = reinterpret_cast<const cx<double> *>(a.tw);
    const int tid = threadIdx.x, e = tid & (EC - 1);
    const bool live = e < a.E - e0, swap = a.dir > 0;
    const int64_t jm = j & (a.Ns - 1);
    for (int t = tid; t < 3 * EC; t += NT) {
        sor[t] = 0u;
        if (t < EC) smax[t] = 0u;
    }
    auto fill = [&]() {
        if constexpr (P::NSTAGE > 1)
            for (int t = tid; t < R; t += NT) stw[t] = q_twiddle(tw[(int64_t)t << (a.tw_log - LOGR)], 0, false);
        if (a.Ns > 1) {
            const int sh = a.tw_log - (a.logNs + LOGR);
            for (int t = tid; t < R; t += NT) spt[t] = q_twiddle(tw[(jm * t) << sh], P::FIRST, false);
        }
    };
    // beside its predecessor's end a small launch fills its tables; otherwise
    // the copies go first
    if (a.pdl) {
        overlap_release();
        fill();
    }
    overlap_wait();

    // A thread's points are i = 0 .. EPT - 1 at tid + i NT: entry e, rho = that >> LEC;
    // the points of its first-stage butterflies are among them.
    {
        const int64_t S = a.M >> LOGR, k0 = j + (tid >> P::LEC) * S, dk = (NT >> P::LEC) * S;
        const unsigned dst = (unsigned)__cvta_generic_to_shared(sm) + 16u * tid;
        const int64_t off = (a.src_row0 + (a.src_mode == SRC_CPLX ? k0 : 2 * k0)) * a.src_ld + e0 + e;
        // valid points: i < n (zero-filled beyond; the last real point may be half)
        const int64_t left = (a.src_mode == SRC_CPLX ? a.src_nvalid : (a.src_nvalid + 1) / 2) - k0;
        const int n = !live || left <= 0 ? 0 : (int)min((int64_t)EPT, (left + dk - 1) / dk);
        if (a.src_mode == SRC_CPLX) {
            const cx<double> *z = reinterpret_cast<const cx<double> *>(a.src), *p = z + off;
            const int64_t dp = dk * a.src_ld;
#pragma unroll
            for (int i = 0; i < EPT; ++i, p += dp) q_copy(dst + 16u * NT * i, i < n ? p : z, i < n, 16);
        } else {
            const double *z = reinterpret_cast<const double *>(a.src), *p = z + off;
            const int64_t dp = 2 * dk * a.src_ld;
            const int odd = (int)(a.src_nvalid & 1) && n > 0 && k0 + (n - 1) * dk == a.src_nvalid / 2 ? n - 1 : -1;
#pragma unroll
            for (int i = 0; i < EPT; ++i, p += dp) {
                const bool ok0 = i < n, ok1 = ok0 && i != odd;
                q_copy(dst + 16u * NT * i, ok0 ? p : z, ok0, 8);
                q_copy(dst + 16u * NT * i + 8u, ok1 ? p + a.src_ld : z, ok1, 8);
            }
        }
    }
    if (!a.pdl) fill();
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    // the entry's largest magnitude over the CTA's R points, and the conversion
    auto raw = [&](int i) -> cx<double> {
        return {__longlong_as_double(sm[i].re.v), __longlong_as_double(sm[i].im.v)};
    };
    {
        unsigned m = 0;
#pragma unroll 2
        for (int i = 0; i < EPT; ++i) {
            const cx<double> x = raw(tid + i * NT);
            m = max(m, max(q_magnitude(x.re), q_magnitude(x.im)));
        }
        q_column<EC, NT, true>(m, smax, tid);
    }
    __syncthreads();
    // |re|, |im| <= 2^(ex - 1022) (1 + 2^-20): a largest value of one, the diagonal of e0 - q and
    // of its inverse, does not cost its columns a bit
    int ex = (int)((smax[e] - min(smax[e], 1u)) >> 20);
    // columns below 2^-895 (not zero) are scaled up first, where their zeros and
    // subnormals would not shift out of the alignment
    const bool tiny = ex < Q_TINY && smax[e] != 0u;
    if (tiny) {
#pragma unroll 1
        for (int i = tid; i < R * EC; i += NT) {
            const cx<double> x = raw(i);
            sm[i] = {{__double_as_longlong(x.re * Q_SCALE)}, {__double_as_longlong(x.im * Q_SCALE)}};
        }
        ex = max(ex, 1) + Q_UP;
    }
    ex = smax[e] >= 0x7ff00000u ? Q_NONFINITE : max(ex, Q_EXMIN);
    {
        // with inter-pass twiddles (stored as w / 2^FIRST) the points come in at
        // 2^60, else already divided by the first radix
        const int top = a.Ns > 1 ? Q_TOP : Q_TOP - P::FIRST, neg = a.src_neg ? -1 : 0, odd = tid >> P::LEC & 1;
#pragma unroll 2
        for (int i = 0; i < EPT; ++i) {
            const cx<double> x = raw(tid + i * NT);
            cx<q64> v = {q_decode(swap ? x.im : x.re, ex, top, neg), q_decode(swap ? x.re : x.im, ex, top, neg)};
            if (a.Ns > 1) v = c_mul(v, spt[(tid + i * NT) >> P::LEC], (1ll << 29) - (NT >> P::LEC & i ? odd ^ 1 : odd));
            sm[tid + i * NT] = v;
        }
    }
    if (tiny) ex -= Q_UP;
    // first stage (radix 2^FIRST, no twiddles)
    {
        constexpr int r = 1 << P::FIRST, UPT = EPT / r;
        cx<q64> v[UPT][r];
#pragma unroll
        for (int u = 0; u < UPT; ++u)
#pragma unroll
            for (int q = 0; q < r; ++q) v[u][q] = sm[tid + NT * (u + q * UPT)];
        __syncthreads();
        unsigned m = 0;
#pragma unroll
        for (int u = 0; u < UPT; ++u) {
            dft_r<q64, false, P::FIRST>(v[u]);
            const int b = (tid + u * NT) >> P::LEC;
#pragma unroll
            for (int q = 0; q < r; ++q) {
                sm[(b * r + q) * EC + e] = v[u][q];
                m |= q_bits(v[u][q].re) | q_bits(v[u][q].im);
            }
        }
        if constexpr (P::NSTAGE > 1) q_column<EC, NT, false>(m, sor, tid);
        __syncthreads();
    }
    // radix-8 stages S = 1 .. NSTAGE - 1; the shift before each leaves it its
    // growth (|re|, |im| of its inputs below 2^57, 2^59 in the last one, whose
    // outputs meet no more products)
#pragma unroll 1
    for (int S = 1; S < P::NSTAGE; ++S) {
        const int lns = P::FIRST + 3 * (S - 1);
        const bool last = S == P::NSTAGE - 1;
        const int b = tid >> P::LEC, bm = b & ((1 << lns) - 1);
        const int qs = max(0, 64 - __clz((int)sor[(S - 1) * EC + e]) - (last ? Q_TOP - 1 : Q_TOP - 3));
        // (unit twiddles, b = 0 mod 2^lns: see q_round_start)
        const int odd = (b >> lns) & 1;
        const long long qc = q_round_start(qs) - odd, qd = q_round_start(qs) - (odd ^ 1);
        ex += qs;
        cx<q64> v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = sm[tid + NT * q];
        __syncthreads();  // every read done before the in-place writes
        v[0] = {{q_shift_even(v[0].re.v, qs)}, {q_shift_even(v[0].im.v, qs)}};
#pragma unroll
        for (int q = 1; q < 8; ++q) v[q] = q_shift(c_mul(v[q], stw[(bm * q) << (LOGR - lns - 3)], q & 1 ? qd : qc), qs);
        dft8<q64, false>(v);
        const int ob = ((b >> lns) << (lns + 3)) + bm;
        unsigned m = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            sm[(ob + (q << lns)) * EC + e] = v[q];
            m |= q_bits(v[q].re) | q_bits(v[q].im);
        }
        if (!last) q_column<EC, NT, false>(m, &sor[S * EC], tid);
        __syncthreads();
    }

    // back to floating point and out: point f goes to row base_out + f Ns; the
    // exponent takes the alignment, the shifts and the output scale (a signed
    // power of two)
    const unsigned hs = (unsigned)__double2hiint(a.dst_scale), sgn = hs & 0x80000000u;
    const int eb = ex + P::FIRST + 4 + (int)((hs >> 20) & 0x7ffu) - 1023;
    const int64_t base_out = (j >> a.logNs << (a.logNs + LOGR)) + jm, ld = a.dst_ld;
    const int64_t k0 = base_out + (int64_t)(tid >> P::LEC) * a.Ns, dk = (NT >> P::LEC) * a.Ns;
    auto value = [&](int i, double &y0, double &y1) {
        const cx<q64> v = sm[tid + i * NT];
        y0 = q_encode(swap ? v.im : v.re, eb, sgn);
        y1 = q_encode(swap ? v.re : v.im, eb, sgn);
        if (ex >= Q_NONFINITE) y0 = y1 = __longlong_as_double(0x7ff8000000000000ll);  // an Inf or NaN in the column
    };
    if (!live) return;
    if (a.dst_mode == DST_CPLX) {
        cx<double> *p = reinterpret_cast<cx<double> *>(a.dst) + k0 * ld + e0 + e;
        const int64_t dp = dk * ld;
#pragma unroll 2
        for (int i = 0; i < EPT; ++i, p += dp) {
            double y0, y1;
            value(i, y0, y1);
            *p = {y0, y1};
        }
    } else {
        double *p = reinterpret_cast<double *>(a.dst) + (a.dst_row0 - a.dst_lo + 2 * k0) * ld + e0 + e;
        const int64_t dp = 2 * dk * ld;
        const bool eye_e = a.dst_eye_d > 0 && (e0 + e) % max(a.dst_eye_d + 1, 1) == 0;
        const int lo = (int)a.dst_lo, hi = (int)a.dst_hi;  // real rows: at most 2^21
        int rr = (int)(2 * k0);
#pragma unroll 1
        for (int i = 0; i < EPT; ++i, p += dp, rr += (int)(2 * dk)) {
            double y0, y1;
            value(i, y0, y1);
            if (eye_e && rr == 0) y0 += 1.0;
            const bool in0 = rr >= lo && rr < hi, in1 = rr + 1 >= lo && rr + 1 < hi;
            if (a.dst_mode == DST_REAL64_ADD) {
                if (in0) p[0] += y0;
                if (in1) p[ld] += y1;
            } else {
                if (in0) p[0] = y0;
                if (in1) p[ld] = y1;
            }
        }
    }
}

template <int LOGR, int EC>
__global__ void __launch_bounds__(QPlan<LOGR, EC>::NT, QPlan<LOGR, EC>::MINB) fftq_pass_kernel(FftArgs a)
{
    fftq_body<LOGR, EC>(a, blockIdx.y, blockIdx.x * EC);
}

// CTA b of a segmented launch: see fft_seg_run in kernels.cuh
template <int LOGR, int EC>
__global__ void __launch_bounds__(QPlan<LOGR, EC>::NT, QPlan<LOGR, EC>::MINB)
    fftq_seg_kernel(const __grid_constant__ SegParams<FftArgs> P)
{
    const int s = seg_find(P, blockIdx.x);
    const FftArgs &a = P.a[s];
    const unsigned loc = blockIdx.x - P.first[s], nchunk = (unsigned)((a.E + EC - 1) / EC), j = loc / nchunk;
    fftq_body<LOGR, EC>(a, j, (int)(loc - j * nchunk) * EC);
}

// Launch table: 8, 4 and (from radix 2^8) 1 entries per CTA
template <int OFF, int... L>
void fftq_fill(FftEntry (*t)[11], FftSegEntry *ts, std::integer_sequence<int, L...>)
{
    ((t[0][OFF + L] = FftEntry{fftq_pass_kernel<OFF + L, 8>, QPlan<OFF + L, 8>::NT}), ...);
    ((t[1][OFF + L] = FftEntry{fftq_pass_kernel<OFF + L, 4>, QPlan<OFF + L, 4>::NT}), ...);
    if constexpr (OFF >= 8) ((t[2][OFF + L] = FftEntry{fftq_pass_kernel<OFF + L, 1>, QPlan<OFF + L, 1>::NT}), ...);
    ((ts[OFF + L] = FftSegEntry{fftq_seg_kernel<OFF + L, 8>, QPlan<OFF + L, 8>::NT}), ...);
}
