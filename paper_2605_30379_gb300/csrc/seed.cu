// seed.cu -- the start of the Newton doubling: psi(0) = A(0)^(-1) by
// Gauss-Jordan elimination with partial pivoting (Theorem 2.2, Eq. (newton))
// and, for d <= 32, the first m0 coefficients by Newton doubling with direct
// sums, in one launch of one thread-block cluster per model.
//
// What bounds it is latency: every column of the elimination and every level
// waits for the one before.  One CTA on global memory took 23 us for d = 3,
// 0.5 ms for d = 64 and 12 ms for d = 256, and the direct recursion that
// followed 120 us for 32 coefficients at d = 3 (one dependent sum after the
// other).  Here the data live in shared memory; for d > 32 the CTAs own the rows
// i = rank mod CL and exchange pivots and pivot rows through distributed shared
// memory with one cluster barrier per column, and a level m -> 2m takes two
// barriers, its sums spread over all threads of the cluster (whole inverse d = 3,
// N = 128 in FP64 262 -> 37 us, mixed d = 256, N = 4096 183 -> 172 ms).
#include <cooperative_groups.h>

#include <float.h>

#include <algorithm>
#include <atomic>
#include <initializer_list>

#include "mrc_internal.h"

namespace cg = cooperative_groups;

namespace {

constexpr int NT = 256;
constexpr int CLMAX = 16;
constexpr int SMEM_MAX = 216 * 1024;
constexpr int DSMALL = MRC_SEED_DMAX;  // up to here every CTA eliminates by itself and the levels run

struct Pivot {
    double v;
    int i;
};

__device__ __forceinline__ bool better(double v, int i, const Pivot &p) { return v > p.v || (v == p.v && i < p.i); }

// argmax over the warp, on every lane
__device__ __forceinline__ Pivot warp_pivot(Pivot p)
{
    for (int o = 16; o > 0; o >>= 1) {
        const double v = __shfl_xor_sync(0xffffffffu, p.v, o);
        const int i = __shfl_xor_sync(0xffffffffu, p.i, o);
        if (better(v, i, p)) p = {v, i};
    }
    return p;
}

// a / p from r = 1 / p: the quotient corrected by its remainder (three FP64
// operations per element instead of a division's twenty; the FP64 pipe takes
// 17 cycles per warp and operation)
__device__ __forceinline__ double quot(double a, double p, double r)
{
    const double q = a * r;
    const double e = fma(-q, p, a);
    return fabs(e) <= DBL_MAX ? fma(e, r, q) : a / p;  // 1 / p or the product out of range
}

__device__ double max_abs(const double *__restrict__ A0, int n)
{
    __shared__ double sv[NT / 32];
    double m = 0.0;
    for (int t = threadIdx.x; t < n; t += NT) m = fmax(m, fabs(A0[t]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) sv[threadIdx.x >> 5] = m;
    __syncthreads();
    for (int w = 0; w < NT / 32; ++w) m = fmax(m, sv[w]);
    return m;
}

// Elimination on [A0 | I] (d x 2d in shared memory, d <= 32), every CTA by
// itself.  Returns false (on every thread) if a pivot is not above tol.
__device__ bool gj_small(const double *__restrict__ A0, double *W, int d, double tol)
{
    __shared__ double fac[DSMALL], rp;
    __shared__ Pivot sp;
    const int n2 = 2 * d, tid = threadIdx.x;
    for (int t = tid; t < d * n2; t += NT) {
        const int i = t / n2, j = t - i * n2;
        W[t] = j < d ? A0[i * d + j] : (j - d == i ? 1.0 : 0.0);
    }
    __syncthreads();
    for (int col = 0; col < d; ++col) {
        if (tid < 32) {
            Pivot p = {-1.0, 0x7fffffff};
            if (tid >= col && tid < d && better(fabs(W[tid * n2 + col]), tid, p)) p = {fabs(W[tid * n2 + col]), tid};
            p = warp_pivot(p);
            if (tid == 0) {
                sp = p;
                rp = p.v > tol ? 1.0 / W[p.i * n2 + col] : 0.0;
            }
        }
        __syncthreads();
        if (!(sp.v > tol)) return false;
        const int piv = sp.i;
        const double pv = W[piv * n2 + col];
        double a = 0.0, b = 0.0;
        if (tid < n2) {
            a = W[piv * n2 + tid];
            b = W[col * n2 + tid];
        }
        if (tid < d) fac[tid] = tid == piv ? W[col * n2 + col] : W[tid * n2 + col];  // after the exchange
        __syncthreads();
        if (tid < n2) {
            W[piv * n2 + tid] = b;
            W[col * n2 + tid] = quot(a, pv, rp);
        }
        __syncthreads();
        for (int t = tid; t < d * n2; t += NT) {
            const int i = t / n2, j = t - i * n2;
            if (i != col) W[t] = fma(-fac[i], W[col * n2 + j], W[t]);
        }
        __syncthreads();
    }
    return true;
}

// The same elimination for d > 32 with the rows spread over the cluster, in
// place: a finished column of the left block keeps the column of the right
// block that its pivot row started, so that after the last step
// A0^(-1)[c][perm[c']] = S[perm[c]][c'], perm[c] the pivot row of column c (rows
// are not moved).  S: this CTA's rows rank + t CL.  GLOBAL: the rows are those of
// `out` instead, for matrices whose rows do not fit the cluster's shared memory (8
// CTAs: d > 460), and S holds only the pivot rows; the cluster barriers order
// those accesses too.
template <bool GLOBAL>
__device__ bool gj_cluster(cg::cluster_group &cl, const double *__restrict__ A0, double *out, double *S, int d, double tol,
                           int CL, int rank)
{
    __shared__ Pivot slot[2][CLMAX];
    __shared__ int perm[512];
    __shared__ double pr[2];
    __shared__ unsigned char used[512 / 8];  // of this CTA's rows (d / CL <= 64)
    const int nr = (d - rank + CL - 1) / CL, tid = threadIdx.x;
    double *buf = S + (GLOBAL ? 0 : (size_t)((d + CL - 1) / CL) * d);  // [2][d] normalised pivot rows
    auto row = [&](int r) { return GLOBAL ? out + (size_t)(rank + r * CL) * d : S + (size_t)r * d; };
    for (int t = tid; t < nr * d; t += NT) {
        const int r = t / d;
        row(r)[t - r * d] = A0[(size_t)(rank + r * CL) * d + (t - r * d)];
    }
    if (tid < 64) used[tid] = 0;
    __syncthreads();
    int prow = -1;  // this CTA's row that was the last pivot, still to be replaced by buf
    for (int col = 0; col < d; ++col) {
        const int b = col & 1;
        if (tid < 32) {
            Pivot p = {-1.0, 0x7fffffff};
            for (int r = tid; r < nr; r += 32)
                if (!used[r] && better(fabs(row(r)[col]), rank + r * CL, p)) p = {fabs(row(r)[col]), rank + r * CL};
            p = warp_pivot(p);
            if (tid < CL) cl.map_shared_rank(&slot[0][0], tid)[b * CLMAX + rank] = p;
        }
        cl.sync();
        Pivot p = slot[b][0];
        for (int r = 1; r < CL; ++r)
            if (better(slot[b][r].v, slot[b][r].i, p)) p = slot[b][r];
        if (!(p.v > tol)) return false;
        // every CTA has read the last pivot row: its owner may now replace it
        if (prow >= 0)
            for (int j = tid; j < d; j += NT) row(prow)[j] = buf[(b ^ 1) * d + j];
        const int owner = p.i % CL, lr = p.i / CL;
        const double *src = GLOBAL ? out + (size_t)p.i * d : cl.map_shared_rank(S, owner) + (size_t)lr * d;
        if (tid == 0) {
            pr[0] = src[col];
            pr[1] = 1.0 / pr[0];
        }
        double x[2];  // NT threads take two elements each of up to 512
#pragma unroll
        for (int q = 0; q < 2; ++q) x[q] = tid + q * NT < d ? (tid + q * NT == col ? 1.0 : src[tid + q * NT]) : 0.0;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (tid + q * NT < d) buf[b * d + tid + q * NT] = quot(x[q], pr[0], pr[1]);
        prow = owner == rank ? lr : -1;
        if (tid == 0) {
            perm[col] = p.i;
            if (prow >= 0) used[prow] = 1;
        }
        __syncthreads();
        // one warp per row: f is read before any lane changes it
        for (int r = tid >> 5; r < nr; r += NT / 32) {
            if (r == prow) continue;
            double *s = row(r);
            const double f = s[col];
            __syncwarp();
            for (int j = tid & 31; j < d; j += 32) s[j] = fma(-f, buf[b * d + j], j == col ? 0.0 : s[j]);
        }
        __syncthreads();
    }
    cl.sync();  // no CTA leaves while its rows are still read
    if (prow >= 0)
        for (int j = tid; j < d; j += NT) row(prow)[j] = buf[((d - 1) & 1) * d + j];
    __syncthreads();
    if (!GLOBAL) {
        for (int c = 0; c < d; ++c)
            if (perm[c] % CL == rank) {
                const double *s = row(perm[c] / CL);
                for (int j = tid; j < d; j += NT) out[(size_t)c * d + perm[j]] = s[j];
            }
        return true;
    }
    // the columns of the own rows, then the rows column by column, in place
    for (int r = 0; r < nr; ++r) {
        double *s = row(r);
        for (int j = tid; j < d; j += NT) buf[j] = s[j];
        __syncthreads();
        for (int j = tid; j < d; j += NT) s[perm[j]] = buf[j];
        __syncthreads();
    }
    cl.sync();
    for (int j = rank; j < d; j += CL) {
        for (int i = tid; i < d; i += NT) buf[i] = out[(size_t)i * d + j];
        __syncthreads();
        for (int c = tid; c < d; c += NT) out[(size_t)c * d + j] = buf[perm[c]];
        __syncthreads();
    }
    return true;
}

// One sum per group of tpo lanes: sum over t in [0, nt) of X(x0 - t) Y(t) at
// (i, j), both in shared memory (E entries per coefficient).
__device__ __forceinline__ double conv_sum(const double *X, const double *Y, int x0, int nt, int i, int j, int d, int E,
                                           int lane, int tpo)
{
    double s0 = 0.0, s1 = 0.0;
    for (int t = lane; t < nt; t += tpo) {
        const double *x = X + (x0 - t) * E + i * d, *y = Y + t * E + j;
        int u = 0;
        for (; u + 1 < d; u += 2) {
            s0 = fma(x[u], y[u * d], s0);
            s1 = fma(x[u + 1], y[(u + 1) * d], s1);
        }
        if (u < d) s0 = fma(x[u], y[u * d], s0);
    }
    s0 += s1;
    for (int o = tpo >> 1; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    return s0;
}

// Levels m -> 2m up to n (Eq. (newton) with direct sums): R = -(A B)[m, 2m),
// B[m, 2m) = (B R)[0, m).  Small levels are computed by every CTA for itself,
// the others by the cluster, each sum sent to all its CTAs.
__device__ void levels(cg::cluster_group &cl, const double *As, double *Bs, double *Rs, double *__restrict__ psi, int d,
                       int n, int CL, int rank)
{
    const int E = d * d, tid = threadIdx.x;
    bool local = false;  // the last level was computed by each CTA for itself
    for (int m = 1; m < n; m *= 2) {
        const int rows = min(2 * m, n) - m, outs = rows * E;
        const bool own = (long long)outs * m * d <= 6144;
        if (!own && local) cl.sync();  // before any CTA writes to another that may still read
        local = own;
        const int nc = own ? 1 : CL, me = own ? 0 : rank;
        int tpo = 1;
        while (tpo < 32 && tpo < m && outs * tpo < nc * NT) tpo <<= 1;
        const int lane = tid & (tpo - 1), grp = tid / tpo, ng = NT / tpo;
        for (int ph = 0; ph < 2; ++ph) {
            double *dst = ph == 0 ? Rs : Bs + (size_t)m * E;
            // whole warps take every round (the sums use shuffles)
            for (int o0 = 0; o0 < outs; o0 += nc * ng) {
                const int o = o0 + me * ng + grp;
                const bool in = o < outs;
                const int s = in ? o / E : 0, e = in ? o - s * E : 0, i = e / d, j = e - i * d;
                double v;
                if (ph == 0) v = -conv_sum(As, Bs, m + s, in ? m : 0, i, j, d, E, lane, tpo);
                else v = conv_sum(Bs, Rs, s, in ? s + 1 : 0, i, j, d, E, lane, tpo);
                if (!in) continue;
                if (own) {
                    if (lane == 0) dst[o] = v;
                } else {
                    for (int r = lane; r < CL; r += tpo) cl.map_shared_rank(dst, r)[o] = v;
                }
                if (ph == 1 && lane == 0 && (!own || rank == 0)) psi[(size_t)m * E + o] = v;
            }
            if (own) __syncthreads();
            else cl.sync();
        }
    }
}

// shared memory of a CTA's rows and two pivot rows (d > DSMALL), and whether a CTA has it
__host__ __device__ inline size_t cluster_smem(int d, int CL) { return sizeof(double) * ((size_t)((d + CL - 1) / CL) * d + 2 * d); }
__host__ __device__ inline bool cluster_fits(int d, int CL) { return cluster_smem(d, CL) <= (size_t)SMEM_MAX; }

template <bool GLOBAL>
__device__ __forceinline__ void seed_run(const SeedArgs &g)
{
    extern __shared__ __align__(16) unsigned char smem[];
    cg::cluster_group cl = cg::this_cluster();
    const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank(), d = g.d, E = d * d, tid = threadIdx.x;
    double *S = reinterpret_cast<double *>(smem);
    const double tol = (double)d * 0x1p-52 * max_abs(g.A, E);
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    if (d > DSMALL) {
        cl.sync();  // every CTA of the cluster runs before any writes to another's shared memory
        bool ok;
        if (GLOBAL && !cluster_fits(d, CL)) ok = gj_cluster<true>(cl, g.A, g.psi, S, d, tol, CL, rank);
        else ok = gj_cluster<false>(cl, g.A, g.psi, S, d, tol, CL, rank);
        if (!ok) {
            if (rank == 0 && tid == 0) atomicExch(g.status, 2);
            for (int t = rank * NT + tid; t < E; t += CL * NT) g.psi[t] = nan;
            cl.sync();
        }
        return;
    }
    double *As = S + 2 * E, *Bs = As + (size_t)g.m0 * E, *Rs = Bs + (size_t)g.m0 * E;
    for (int t = tid; t < g.m0 * E; t += NT) As[t] = g.A[t];
    const bool ok = gj_small(g.A, S, d, tol);
    __syncthreads();
    if (!ok && rank == 0 && tid == 0) atomicExch(g.status, 2);
    for (int t = tid; t < E; t += NT) {
        const int i = t / d, j = t - i * d;
        const double v = ok ? S[i * 2 * d + d + j] : nan;
        Bs[t] = v;
        if (rank == 0) g.psi[t] = v;
    }
    cl.sync();
    levels(cl, As, Bs, Rs, g.psi, d, g.m0, CL, rank);
    cl.sync();  // no CTA leaves while others still write to its shared memory
}

// GLOBAL: a model of the launch does not fit
template <bool GLOBAL>
__global__ void __launch_bounds__(NT) seed_kernel(const __grid_constant__ SegParams<SeedArgs> P, int CL)
{
    seed_run<GLOBAL>(P.a[blockIdx.x / CL]);
}

size_t seed_smem(int d, int m0, int CL)
{
    const size_t E = (size_t)d * d;
    if (d > DSMALL) return cluster_fits(d, CL) ? cluster_smem(d, CL) : sizeof(double) * 2 * d;
    return sizeof(double) * E * (2 + 2 * (size_t)m0 + std::max(1, m0 / 2));
}

// 16 CTAs where the current device can place such a cluster, else the portable 8.
// Function attributes and the answer belong to a device: every one is set up and
// asked by itself (mrc_seed_init, or the first launch there).
int query_cluster()
{
    for (auto k : {seed_kernel<false>, seed_kernel<true>})
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX) != cudaSuccess ||
            cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
            cudaGetLastError();
            return 8;
        }
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CLMAX;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(CLMAX);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = SMEM_MAX;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nc = 0;
    if (cudaOccupancyMaxActiveClusters(&nc, seed_kernel<false>, &cfg) != cudaSuccess || nc < 1) {
        cudaGetLastError();
        return 8;
    }
    return CLMAX;
}

std::atomic<int> device_cluster[64];  // by device, 0: not asked yet

int cluster_size()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return query_cluster();
    int n = device_cluster[dev].load();
    if (n == 0) device_cluster[dev].store(n = query_cluster());
    return n;
}

} // namespace

// The first coefficients, by powers of two: while a level's direct sums (1.5
// m^2 d^3 multiply-adds, 1.9 per clock and SM, 16 SMs: 13 us for 8e5) take less
// than the seven launches of a level by FFT (about 30 us); two for d > 32 (psi(1) by
// base_case_kernel).  The mixed path's FP32 levels start after 32, 8 or 2: their
// rounding decides its last digits, and stays what it was.
int64_t mrc_base_size(int d, int64_t N, bool f32)
{
    int64_t m0 = 2;
    if (f32) m0 = d <= 8 ? 32 : (d <= 32 ? 8 : 2);
    else if (d <= DSMALL)
        while (m0 < 256 && 1.5 * (double)(m0 * m0) * d * d * d <= 8e5) m0 *= 2;
    return std::min<int64_t>(m0, N);
}

cudaError_t mrc_seed_init(void)
{
    int dev = 0;
    const int n = query_cluster();
    if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64) device_cluster[dev].store(n);
    const cudaError_t e = cudaFuncSetAttribute(seed_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(seed_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
}

cudaError_t mrc_seed(const SegParams<SeedArgs> &P, cudaStream_t st, int cluster)
{
    if (P.nseg <= 0) return cudaSuccess;
    const int CL = cluster ? cluster : cluster_size();
    size_t sm = 0;
    bool fits = true;
    for (int s = 0; s < P.nseg; ++s) {
        sm = std::max(sm, seed_smem(P.a[s].d, P.a[s].m0, CL));
        fits = fits && (P.a[s].d <= DSMALL || cluster_fits(P.a[s].d, CL));
    }
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CL;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(CL * P.nseg));
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    mrc_prof_pre(7, st);
    cudaError_t e = cudaLaunchKernelEx(&cfg, fits ? seed_kernel<false> : seed_kernel<true>, P, CL);
    mrc_prof_post(7, st, 0, 0);
    return e != cudaSuccess ? e : cudaGetLastError();
}
