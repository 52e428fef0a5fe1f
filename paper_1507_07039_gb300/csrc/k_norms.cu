// What every path's iteration shares after its products: the norms of W'
// and h (k_reduce_wnorms), then the diagonals of Eq. 6, the norms of P' and C', the
// counter and the stop test (k_fin), for one network or a set.  Every
// reduction has a fixed order, so an iteration is deterministic.  Also the
// FP32 FMA rate of the device (measurement support).
#include "panda_internal.cuh"

namespace panda {

namespace {

// Slot sums for 32 consecutive rows per block, 8 threads per row: thread
// (g, x) adds slots g, g + 8, g + 16, ... of row x, then the 8 partial sums
// are added in FP64 in group order (a fixed order, so the result is
// deterministic).  The per-thread sums are compensated FP32 (each addition's
// rounding error recovered exactly by Knuth's TwoSum and carried along), about
// as accurate as FP64 additions of the FP32 slots but on the FP32 pipe, which
// on this GPU is far wider than the FP64 one.
constexpr int RS_ROWS = 32, RS_GROUPS = 8;

// This thread's slots g, g + 8, ... inside [lo, hi), in ascending order
template <int NV>
__device__ __forceinline__ void slot_range(const float *const (&src)[NV], int lo, int hi, int ld, int x,
                                           float (&s)[NV], float (&c)[NV])
{
    const int g = threadIdx.x / RS_ROWS;
    int b = lo + (((g - lo) % RS_GROUPS) + RS_GROUPS) % RS_GROUPS;
    // four slots' loads in flight at a time; the additions keep the order
    for (; b + 3 * RS_GROUPS < hi; b += 4 * RS_GROUPS) {
        float t[NV][4];
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int u = 0; u < 4; ++u)
                t[v][u] = src[v][(size_t)(b + u * RS_GROUPS) * ld + x];
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int u = 0; u < 4; ++u)
                two_sum_add(s[v], c[v], t[v][u]);
    }
    for (; b < hi; b += RS_GROUPS)
#pragma unroll
        for (int v = 0; v < NV; ++v)
            two_sum_add(s[v], c[v], src[v][(size_t)b * ld + x]);
}

// Sums over the slots in [lo0, hi0) and [lo1, hi1) (lo1 >= hi0): slots outside
// them hold zeros, whose additions would change nothing.
template <int NV>
__device__ __forceinline__ void slot_sums(const float *const (&src)[NV], int lo0, int hi0, int lo1, int hi1, int ld,
                                          int x, bool ok, double (&out)[NV], double (*sh)[RS_GROUPS][RS_ROWS])
{
    const int lx = threadIdx.x & (RS_ROWS - 1), g = threadIdx.x / RS_ROWS;
    float s[NV], c[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v)
        s[v] = c[v] = 0.0f;
    if (ok) {
        slot_range<NV>(src, lo0, hi0, ld, x, s, c);
        slot_range<NV>(src, lo1, hi1, ld, x, s, c);
    }
#pragma unroll
    for (int v = 0; v < NV; ++v)
        sh[v][g][lx] = (double)s[v] + (double)c[v];
    __syncthreads();
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        double t = 0.0;
        for (int q = 0; q < RS_GROUPS; ++q)
            t += sh[v][q][lx];
        out[v] = t;
    }
}

// The largest of one warp's values into *slot (float bits of non-negative
// values order like the values, so an unsigned maximum is exact and the
// result does not depend on the order of the warps).
__device__ __forceinline__ void fp8_norm_max(unsigned *slot, float v)
{
    unsigned u = __float_as_uint(fmaxf(v, 0.0f));
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1)
        u = max(u, __shfl_xor_sync(0xffffffffu, u, off));
    if ((threadIdx.x & 31) == 0)
        atomicMax(slot, u);
}

// h (Eq. 7) of the iteration under way from phase 1's partial sums, in FP64 in a fixed order.
__device__ __forceinline__ void sum_h(const Dev &d)
{
    __shared__ double sh[8];
    const int n = d.nbT * d.nwr;
    double s = 0.0;
    for (int q = threadIdx.x; q < n; q += RS_ROWS * RS_GROUPS)
        s += d.hpart[q];
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1)
        s += __shfl_xor_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0)
        sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < 8; ++q)
            s += sh[q];
        d.ctl->h_next = s / ((double)d.T * (double)d.G);
    }
}

// rsqW[i] = sum_b wrow_part[b][i], csqW[j] = sum_b wcol_part[b][j] (FP64): block b of one network's
// launch, b < ceil(T/32) rows of W, then its columns, the last one h
__device__ __forceinline__ void reduce_wnorms_block(const Dev &d, int b)
{
    if (!d.ctl->active)
        return;
    __shared__ double sh[1][RS_GROUPS][RS_ROWS];
    const int bT = ceil_div(d.T, RS_ROWS);
    if (b == bT + ceil_div(d.G, RS_ROWS)) {
        sum_h(d);
        return;
    }
    const bool rows = b < bT;
    const int x = ((rows ? b : b - bT) * RS_ROWS) + (threadIdx.x & (RS_ROWS - 1));
    const bool ok = x < (rows ? d.T : d.G);
    const float *const src[1] = {rows ? d.wrow_part : d.wcol_part};
    double out[1];
    slot_sums<1>(src, 0, rows ? d.nwr : d.nbT, 0, 0, rows ? d.Tp : d.Gp, x, ok, out, sh);
    if (threadIdx.x >= RS_ROWS)
        return;
    if (ok)
        (rows ? d.rsqW : d.csqW)[x] = (float)out[0];
    if (d.fp8)
        fp8_norm_max(&d.f8n[rows ? 2 : 3], ok ? (float)out[0] : 0.0f);
}

__global__ void __launch_bounds__(RS_ROWS * RS_GROUPS) k_reduce_wnorms(const __grid_constant__ Dev d)
{
    reduce_wnorms_block(d, blockIdx.x);
}

// a set of networks: blocks[blockIdx.x] = (network, its block)
__global__ void __launch_bounds__(RS_ROWS * RS_GROUPS) k_reduce_wnorms_set(const Dev *devs, const int2 *blocks)
{
    const int2 w = blocks[blockIdx.x];
    reduce_wnorms_block(devs[w.x], w.y);
}

// The history, the counter and the stop test, by one thread of a network's last k_fin block to
// finish (a kernel of its own cost every iteration about 3 us at the smallest networks).
__device__ __forceinline__ void tail(const Dev &d)
{
    Ctl *ctl = d.ctl;
    const double h = ctl->h_next;
    const int t = ctl->iters + 1;
    if (t - 1 < HIST_CAP)
        d.hist[t - 1] = h;
    ctl->iters = t;
    ctl->h_last = h;
    ctl->converged = h < ctl->tol;
    if (d.fp8) {  // the new state's norm maxima, and the scale of the next W' (Eq. 2)
        for (int q = 0; q < 4; ++q) {
            d.f8n[4 + q] = *(volatile unsigned *)&d.f8n[q];
            d.f8n[q] = 0u;
        }
        d.f8[3] = e4m3_scale(fp8_bound_w(__uint_as_float(d.f8n[4]), __uint_as_float(d.f8n[5]),
                                         __uint_as_float(d.f8n[6]), __uint_as_float(d.f8n[7])));
    }
    ctl->fin_blocks = 0;
    int status = *(volatile int *)&ctl->status;  // the other blocks' findings
    if (!isfinite(h))
        ctl->status = status |= ST_NONFINITE;
    if (ctl->converged || t >= ctl->stop_at || status)
        ctl->active = 0;
}

// ---------------------------------------------------------------------------
// Eq. 6 diagonals and the squared norms of P' and C' (32 rows per block, the
// row partial sums added by 8 threads per row).  Blocks [0, ceil(T/32)) take
// rows of P, the rest rows of C.
// ---------------------------------------------------------------------------
// block b of one network's launch: b < ceil(T/32) rows of P, the rest rows of C
__device__ __forceinline__ void fin_block(const Dev &d, int b)
{
    const Ctl *ctl = d.ctl;
    if (!ctl->active)  // (the network's last block clears it once every other block has passed here)
        return;
    if (b == ceil_div(d.T, RS_ROWS) + ceil_div(d.G, RS_ROWS))  // (h's block in a set's list: done)
        return;
    __shared__ double sh[3][RS_GROUPS][RS_ROWS];
    const int bT = ceil_div(d.T, RS_ROWS);
    const bool isP = b < bT;
    const int i = ((isP ? b : b - bT) * RS_ROWS) + (threadIdx.x & (RS_ROWS - 1));
    const int n = isP ? d.T : d.G;       // network size
    const bool ok = i < n;
    // what the end needs besides the sums is fetched with them
    const double alpha = (double)ctl->alpha;
    const int t = ctl->iters + 1;
    const double growth = d.e2tab[t < HIST_CAP ? t : HIST_CAP];
    double *dg = isP ? d.pd : d.cd;
    const double old = threadIdx.x < RS_ROWS && ok ? dg[i] : 0.0;
    const int ld = isP ? d.Tp : d.Gp;
    const float *const src[3] = {isP ? d.ps_sum : d.cs_sum, isP ? d.ps_sq : d.cs_sq, isP ? d.ps_vsq : d.cs_vsq};
    double sums[3];
    if (d.narrow) {
        // 128 x 64 tiles: a row of 64-block b has row-role partials in slots [2 (b / 2), nb) and
        // column-role partials in [nb, nb + b / 2 + 1)
        const int nb = ceil_div(ld, 64), b64 = ((isP ? b : b - bT) * RS_ROWS) >> 6;
        slot_sums<3>(src, b64 & ~1, nb, nb, nb + b64 / 2 + 1, ld, i, ok, sums, sh);
    } else {
        // 256 x 256 tiles: a row of 256-block b has row-role partials in slots [b, nb) (tiles
        // (b, bn >= b)) and column-role partials in [nb, nb + 2 b + 2) (tiles (bm <= b, b), one per
        // CTA of the pair)
        const int nb = ceil_div(ld, 256), b256 = ((isP ? b : b - bT) * RS_ROWS) >> 8;
        slot_sums<3>(src, b256, nb, nb, nb + 2 * b256 + 2, ld, i, ok, sums, sh);
    }
    float nrm = 0.0f;  // the row's new squared norm (0 past the network)
    if (threadIdx.x < RS_ROWS && ok) {
        const double s1 = sums[0], s2 = sums[1], sv = sums[2], inv = isP ? d.inv_n1P : d.inv_n1C;
        double sigma = 0.0;  // population std of the n - 1 off-diagonal entries (0 for one entry)
        if (n > 2) {
            const double m = s1 * inv;
            const double var = s2 * inv - m * m;
            sigma = var > 0.0 ? sqrt(var) : 0.0;
        }
        const double gain = d.diag == 1 ? 1.0 : alpha;  // PANDA_DIAG_D0_LITERAL has no alpha
        const double mult = isP ? (double)d.G : (double)d.T;  // N_a with P, N_e with C
        const double nd = (1.0 - alpha) * old + gain * mult * sigma * growth;
        dg[i] = nd;
        const float ndf = (float)nd;
        nrm = (float)(sv + nd * nd);
        (isP ? d.pdf : d.cdf)[i] = ndf;
        (isP ? d.rsqP : d.csqC)[i] = nrm;
        if (!isfinite(ndf) || !isfinite(nrm))
            atomicOr(&d.ctl->status, ST_NONFINITE);
    }
    if (d.fp8 && threadIdx.x < RS_ROWS)  // the whole first warp, past the network too
        fp8_norm_max(&d.f8n[isP ? 0 : 1], nrm);
    if (threadIdx.x < RS_ROWS) {  // the first warp did the work
        __threadfence();
        __syncwarp();
        if (threadIdx.x == 0 &&
            atomicAdd(&d.ctl->fin_blocks, 1u) + 1u == (unsigned)(bT + ceil_div(d.G, RS_ROWS))) {
            __threadfence();
            tail(d);
        }
    }
}

__global__ void __launch_bounds__(RS_ROWS * RS_GROUPS) k_fin(const __grid_constant__ Dev d)
{
    fin_block(d, blockIdx.x);
}

__global__ void __launch_bounds__(RS_ROWS * RS_GROUPS) k_fin_set(const Dev *devs, const int2 *blocks)
{
    const int2 w = blocks[blockIdx.x];
    fin_block(devs[w.x], w.y);
}

}  // namespace

cudaError_t launch_reduce_wnorms(const Dev &d, cudaStream_t s)
{
    return launch(k_reduce_wnorms, set_norm_blocks(d.T, d.G) + 1, RS_ROWS * RS_GROUPS, 0, s, d);
}

cudaError_t launch_reduce_wnorms_set(const Dev *devs, const int2 *blocks, int nblocks, cudaStream_t s)
{
    return launch(k_reduce_wnorms_set, nblocks, RS_ROWS * RS_GROUPS, 0, s, devs, blocks);
}

cudaError_t launch_fin_set(const Dev *devs, const int2 *blocks, int nblocks, cudaStream_t s)
{
    return launch(k_fin_set, nblocks, RS_ROWS * RS_GROUPS, 0, s, devs, blocks);
}

int set_norm_blocks(int T, int G) { return ceil_div(T, RS_ROWS) + ceil_div(G, RS_ROWS); }

cudaError_t launch_fin(const Dev &d, cudaStream_t s, KernelEvents &ke)
{
    cudaError_t e = launch(k_fin, set_norm_blocks(d.T, d.G), RS_ROWS * RS_GROUPS, 0, s, d);
    ke.mark(s);
    return e;
}

}  // namespace panda

// ---- FP32 FFMA throughput of the device (measurement support) -------------
namespace panda {
namespace {

constexpr int FFMA_CHAINS = 8, FFMA_LOOP = 4096, FFMA_THREADS = 512;

// Every thread runs FFMA_CHAINS independent chains x <- x * a + b for
// FFMA_LOOP rounds (a, b are launch arguments, so nothing is folded); the
// store is taken only if a chain lands on `never`, which the host makes
// unreachable, so the loop is not removed.
__global__ void __launch_bounds__(FFMA_THREADS) k_ffma_loop(float a, float b, float never, float *out)
{
    float x[FFMA_CHAINS];
#pragma unroll
    for (int c = 0; c < FFMA_CHAINS; ++c)
        x[c] = (float)(threadIdx.x + c) * 1e-3f;
#pragma unroll 32  // 256 FMAs per trip through the loop: its counter and branch are noise
    for (int it = 0; it < FFMA_LOOP; ++it)
#pragma unroll
        for (int c = 0; c < FFMA_CHAINS; ++c)
            x[c] = fmaf(x[c], a, b);
    float s = 0.0f;
#pragma unroll
    for (int c = 0; c < FFMA_CHAINS; ++c)
        s += x[c];
    if (s == never)
        out[blockIdx.x] = s;
}

}  // namespace

cudaError_t measure_ffma_peak(double *tflops)
{
    int dev = 0, nsm = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)))
        return e;
    float *out = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if ((e = cudaMalloc(&out, sizeof(float) * 4 * nsm)))
        return e;
    const int blocks = 4 * nsm;  // 4 x 16 warps per SM: 16 per scheduler
    double best_ms = 1e30;
    if (!(e = cudaEventCreate(&e0)) && !(e = cudaEventCreate(&e1))) {
        for (int rep = 0; rep < 12 && !e; ++rep) {
            cudaEventRecord(e0);
            k_ffma_loop<<<blocks, FFMA_THREADS>>>(0.999f, 1e-4f, -1.0f, out);
            cudaEventRecord(e1);
            if (!(e = cudaEventSynchronize(e1))) {
                float ms = 0.0f;
                cudaEventElapsedTime(&ms, e0, e1);
                if (rep >= 2 && ms < best_ms)  // the first launches warm up the clocks
                    best_ms = ms;
            }
        }
        if (!e)
            e = cudaGetLastError();
    }
    if (e0)
        cudaEventDestroy(e0);
    if (e1)
        cudaEventDestroy(e1);
    cudaFree(out);
    if (e)
        return e;
    const double flop = 2.0 * FFMA_CHAINS * FFMA_LOOP * (double)FFMA_THREADS * blocks;
    *tflops = flop / (best_ms * 1e-3) / 1e12;
    return cudaSuccess;
}

}  // namespace panda
