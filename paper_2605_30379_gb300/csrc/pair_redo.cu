// pair_redo.cu -- the second sum of the FP64 digit products' outputs that lie far
// below their row and column bounds (graded.cuh): blocks of 16 x 32 outputs of a
// frequency pair that the product has marked.
//
// A marked block is taken by one CTA, its unsound outputs one by one from a list, so
// that a kernel with a few small entries pays for those alone; a launch without marks
// reads two bytes per pair.  What bounds a graded product is the integer pipes (some
// 70 instructions per term of an output at both frequencies).
#include <algorithm>

#include "graded.cuh"
#include "mrc_internal.h"

namespace {

constexpr int NT = 256;
constexpr int XN = GR_BI * 64, YN = 64 * GR_BJ;

struct Smem {
    qtw xf[XN], xg[XN], yf[YN], yg[YN];         // limbs [i][k] and [k][j] at f and M - f
    short x0[XN], xp[XN], y0[YN], yp[YN];       // logarithms at frequency 0 and of the pair
    unsigned bx[GR_BI], by[GR_BJ];              // row and column bounds of the pair
    unsigned char rowuse[GR_BI], coluse[GR_BJ];
    unsigned short list[GR_BI * GR_BJ];
    unsigned todo[NT];
    int nlist, ntodo;
};

__device__ void block_redo(const PairArgs &a, Smem &s, int64_t p, int i0, int j0)
{
    const int d = a.r, tid = threadIdx.x;
    const int64_t E = (int64_t)d * d, f = p, g = (a.M - p) & (a.M - 1);
    const cx<double> *ZX = reinterpret_cast<const cx<double> *>(a.zx), *ZY = reinterpret_cast<const cx<double> *>(a.zy);
    cx<double> *ZC = reinterpret_cast<cx<double> *>(a.zc);
    const int rows = min(GR_BI, d - i0), cols = min(GR_BJ, d - j0);
    __syncthreads();  // the block before is done
    if (tid < GR_BI) s.bx[tid] = 0u, s.rowuse[tid] = 0;
    if (tid < GR_BJ) s.by[tid] = 0u, s.coluse[tid] = 0;
    if (tid == 0) s.nlist = 0;
    __syncthreads();
    for (int t = tid; t < XN; t += NT) {
        const int i = t >> 6, k = t & 63;
        if (i >= rows || k >= d) continue;
        const int64_t e = (int64_t)(i0 + i) * d + k;
        const unsigned b = max(gr_magnitude(ZX[f * E + e]), gr_magnitude(ZX[g * E + e]));
        s.xp[t] = gr_log(b);
        s.x0[t] = gr_log(gr_magnitude(ZX[e]));
        atomicMax(&s.bx[i], b);
    }
    for (int t = tid; t < YN; t += NT) {
        const int k = t / GR_BJ, j = t % GR_BJ;
        if (j >= cols || k >= d) continue;
        const int64_t e = (int64_t)k * d + j0 + j;
        const unsigned b = max(gr_magnitude(ZY[f * E + e]), gr_magnitude(ZY[g * E + e]));
        s.yp[t] = gr_log(b);
        s.y0[t] = gr_log(gr_magnitude(ZY[e]));
        atomicMax(&s.by[j], b);
    }
    __syncthreads();
    for (int t = tid; t < GR_BI * GR_BJ; t += NT) {
        const int i = t / GR_BJ, j = t % GR_BJ;
        if (i >= rows || j >= cols) continue;
        if (gr_sound(s.x0 + i * 64, s.y0 + j, s.xp + i * 64, s.yp + j, d, GR_BJ, q_align(s.bx[i]), q_align(s.by[j]), a.logM))
            continue;
        s.rowuse[i] = s.coluse[j] = 1;
        s.list[atomicAdd(&s.nlist, 1)] = (unsigned short)t;
    }
    __syncthreads();
    const cx<double> *tw = reinterpret_cast<const cx<double> *>(a.tw);
    const cx<double> w = tw[f << (a.tw_log - a.logM - 1)];
    const qtw wq = q_twiddle(w, 0, false);
    for (int t = tid; t < XN; t += NT) {
        const int i = t >> 6, k = t & 63;
        if (i >= rows || k >= d || !s.rowuse[i]) continue;
        const int64_t e = (int64_t)(i0 + i) * d + k;
        gr_split(ZX[f * E + e], ZX[g * E + e], wq, s.xp[t], s.xf[t], s.xg[t]);
    }
    for (int t = tid; t < YN; t += NT) {
        const int k = t / GR_BJ, j = t % GR_BJ;
        if (j >= cols || k >= d || !s.coluse[j]) continue;
        const int64_t e = (int64_t)k * d + j0 + j;
        gr_split(ZY[f * E + e], ZY[g * E + e], wq, s.yp[t], s.yf[t], s.yg[t]);
    }
    __syncthreads();
    for (int n = tid; n < s.nlist; n += NT) {
        const int t = s.list[n], i = t / GR_BJ, j = t % GR_BJ;
        cx<double> zf, zg;
        q_merge(gr_sum(s.xf + i * 64, s.yf + j, s.xp + i * 64, s.yp + j, d, GR_BJ),
                gr_sum(s.xg + i * 64, s.yg + j, s.xp + i * 64, s.yp + j, d, GR_BJ), w, zf, zg);
        const int64_t e = (int64_t)(i0 + i) * d + j0 + j;
        ZC[f * E + e] = zf;
        if (g != f) ZC[g * E + e] = zg;
    }
}

// nrb x ncb blocks per product and pair; the CTA looks at blocks blockIdx.x + u gridDim.x,
// NT of them at a time, and takes the marked ones
__global__ void __launch_bounds__(NT) redo_kernel(const __grid_constant__ SegParams<PairArgs> P, unsigned nblocks, int nrb,
                                                  int ncb)
{
    extern __shared__ __align__(16) unsigned char smem[];
    Smem &s = *reinterpret_cast<Smem *>(smem);
    overlap_release();
    overlap_wait();
    const unsigned npairs = (unsigned)P.a[0].npairs, nb = (unsigned)(nrb * ncb);
    for (uint64_t b0 = blockIdx.x; b0 < nblocks; b0 += (uint64_t)NT * gridDim.x) {
        __syncthreads();
        if (threadIdx.x == 0) s.ntodo = 0;
        __syncthreads();
        const uint64_t b = b0 + (uint64_t)threadIdx.x * gridDim.x;
        if (b < nblocks) {
            const unsigned gp = (unsigned)(b / nb), q = (unsigned)(b % nb);
            if (P.a[0].marks[2 * (int64_t)gp + q % ncb] >> (q / ncb) & 1) s.todo[atomicAdd(&s.ntodo, 1)] = (unsigned)b;
        }
        __syncthreads();
        const int n = s.ntodo;
        for (int u = 0; u < n; ++u) {
            const unsigned gp = s.todo[u] / nb, q = s.todo[u] % nb;
            block_redo(P.a[gp / npairs], s, gp % npairs, GR_BI * (int)(q / ncb), GR_BJ * (int)(q % ncb));
        }
    }
}

} // namespace

cudaError_t mrc_redo_init(void)
{
    return cudaFuncSetAttribute(redo_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
}

cudaError_t mrc_pair_redo(const SegParams<PairArgs> &P, int kclass, cudaStream_t st)
{
    const int d = P.a[0].r, nrb = (d + GR_BI - 1) / GR_BI, ncb = nrb <= 2 ? 1 : 2;  // (every product has the same ceil(d / 16))
    const uint64_t nblocks = (uint64_t)P.a[0].npairs * P.nseg * nrb * ncb;
    if (!P.a[0].marks || nblocks >> 32) return cudaErrorInvalidValue;
    const unsigned grid = (unsigned)std::min<uint64_t>(nblocks, 304);  // two CTAs fit an SM
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = sizeof(Smem);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    mrc_prof_pre(kclass, st);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, redo_kernel, P, (unsigned)nblocks, nrb, ncb);
    mrc_prof_post(kclass, st, 0, 0);
    return e != cudaSuccess ? e : cudaGetLastError();
}
