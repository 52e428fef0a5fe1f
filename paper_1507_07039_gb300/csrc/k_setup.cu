// State in and out: input validation, the Z-score of each network (Section
// II-A, NormalizeNetwork) with FP64 statistics, the diagonals of P and C into
// FP64 vectors, every copy that the iteration reads, the initial squared
// norms; and the networks back into dense arrays.
//
// Every reduction here runs with a fixed grid and a fixed summation order, so
// results are identical from run to run.
#include <algorithm>

#include "panda_internal.cuh"

namespace panda {

namespace {

constexpr int RED_BLOCKS = 1024;
constexpr int RED_THREADS = 256;

__device__ double block_sum_fixed(double v, double *sh)
{
    // fixed-shape tree: the result does not depend on scheduling
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    double r = sh[0];
    __syncthreads();
    return r;
}

// The FP32 pairs the element kernels use, stored after the FP64 statistics:
// stats[0] = mean, stats[1] = population std, then as floats (16-byte
// aligned) mean = mh + ml and 1 / std = rh + rl, each to about 2^-48.
__device__ __forceinline__ float4 *stats_pairs(double *stats) { return reinterpret_cast<float4 *>(stats + 2); }
__device__ __forceinline__ float4 stats_pairs(const double *stats)
{
    return *reinterpret_cast<const float4 *>(stats + 2);
}

// x - (mh + ml) = s + t: s = fl(x - mh) and t its rounding error minus ml
__device__ __forceinline__ void centre(float x, float mh, float ml, float &s, float &t)
{
    float e;
    two_sum(x, -mh, s, e);
    t = __fsub_rn(e, ml);
}

// Adds the terms of one element to a compensated pair: mode 0 adds x; mode 1
// adds (x - mean)^2 = (s + t)^2 = p + (pe + 2 s t + t^2), with s^2 = p + pe
// exact.
template <int MODE>
__device__ __forceinline__ void stats_term(float x, float mh, float ml, float &acc, float &cmp)
{
    if (MODE == 0) {
        two_sum_add(acc, cmp, x);
    } else {
        float s, t, p, pe;
        centre(x, mh, ml, s, t);
        two_prod(s, s, p, pe);
        two_sum_add(acc, cmp, p);
        cmp = __fadd_rn(cmp, __fmaf_rn(t, t, __fmaf_rn(__fmul_rn(2.0f, s), t, pe)));
    }
}

// Partial sums for the Z-score in a fixed order.  Block b takes rows b,
// b + gridDim.x, ...; thread x takes the 4-wide column groups x, x + 256, ...
// of each (rows start 16-byte aligned), then the ragged columns.  A thread's
// terms within one row go into a compensated FP32 pair (TwoSum), the pair
// into the thread's FP64 total at the row's end, and the block's totals
// through a fixed tree.  Mode 0: sum of x.  Mode 1: sum of (x - mean)^2,
// mean from stats (the difference kept as an FP32 pair, its square from
// two_prod).  About as accurate as FP64 sums of the FP32 entries, on the FP32
// pipe.
// Rows that are not 16-byte aligned (a caller's array, read where it lies) are
// read as scalars in the same groups and order: the same sums to the bit.
__device__ __forceinline__ float4 load4(const float *x, int c4, bool aligned)
{
    if (aligned)
        return __ldcs(reinterpret_cast<const float4 *>(x) + c4);
    const float *p = x + 4 * (size_t)c4;
    return make_float4(__ldcs(p), __ldcs(p + 1), __ldcs(p + 2), __ldcs(p + 3));
}

template <int MODE>
__global__ void k_stats_partial(const float *__restrict__ X, int rows, int cols, int ld, bool aligned,
                                const double *stats, double *partials)
{
    __shared__ double sh[RED_THREADS];
    float mh = 0.0f, ml = 0.0f;
    if (MODE == 1) {
        const float4 q = stats_pairs(stats);
        mh = q.x;
        ml = q.y;
    }
    const int c4n = cols >> 2;
    double tot = 0.0;
    for (int r = blockIdx.x; r < rows; r += gridDim.x) {
        const float *x = X + (size_t)r * ld;
        float acc = 0.0f, cmp = 0.0f;
#pragma unroll 2
        for (int c = threadIdx.x; c < c4n; c += RED_THREADS) {
            const float4 v = load4(x, c, aligned);
            stats_term<MODE>(v.x, mh, ml, acc, cmp);
            stats_term<MODE>(v.y, mh, ml, acc, cmp);
            stats_term<MODE>(v.z, mh, ml, acc, cmp);
            stats_term<MODE>(v.w, mh, ml, acc, cmp);
        }
        for (int c = (c4n << 2) + threadIdx.x; c < cols; c += RED_THREADS)
            stats_term<MODE>(x[c], mh, ml, acc, cmp);
        tot += (double)acc + (double)cmp;
    }
    double s = block_sum_fixed(tot, sh);
    if (threadIdx.x == 0)
        partials[blockIdx.x] = s;
}

// Mode 0: stats[0] = mean and its FP32 pair.  Mode 1: stats[1] = population
// std and the FP32 pair of its reciprocal (zero when std is not positive).
__global__ void k_stats_final(const double *partials, int n, double count, int mode, double *stats)
{
    __shared__ double sh[RED_THREADS];
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        acc += partials[i];
    double s = block_sum_fixed(acc, sh);
    if (threadIdx.x == 0) {
        float4 *q = stats_pairs(stats);
        if (mode == 0) {
            const double m = s / count;
            stats[0] = m;
            const float mh = (float)m;
            q->x = mh;
            q->y = (float)(m - (double)mh);
        } else {
            const double sd = sqrt(s / count);
            stats[1] = sd;
            const double r = sd > 0.0 ? 1.0 / sd : 0.0;
            const float rh = (float)r;
            q->z = rh;
            q->w = (float)(r - (double)rh);
        }
    }
}

// z = (x - mean) / std (Section II-A, NormalizeNetwork) from the FP32 pairs:
// (s + t) (rh + rl) = s rh + (its exact rounding error + s rl + t rh), the
// terms left out being below 2^-44 of z; the final FP32 addition rounds that
// sum once.  The FP32 result therefore equals the correctly rounded quotient
// except when that lies within about 2^-44 relative of a rounding midpoint.
__device__ __forceinline__ float zscore_one(float x, float4 q)
{
    float s, t, p, pe;
    centre(x, q.x, q.y, s, t);
    two_prod(s, q.z, p, pe);
    return __fadd_rn(p, __fmaf_rn(t, q.z, __fmaf_rn(s, q.w, pe)));
}

// ---- a state from its networks ------------------------------------------------
// One pass over each network where it lies (the caller's device array, or the
// buffer it was copied into): entries checked, Z-scored on the way when `stats`
// is given, and written in every form the iteration reads.  The former
// sequence (copy into a padded FP32 matrix, check, Z-score in place, strip the
// diagonal, split) passed over C six to ten times and staged it in a matrix of
// its own: panda_set_state at 1000 x 17000 took 3.5 ms under BF16X3.

// BF16 parts of four values (N = 2: hi, lo; 3: h, m, l), each the nearest to
// what the ones before leave
template <int N>
__device__ __forceinline__ void parts4(const float (&v)[4], uint2 (&p)[N])
{
    float x[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
    for (int q = 0; q < N; ++q) {
        uint32_t w[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            asm("cvt.rn.satfinite.bf16x2.f32 %0, %2, %1;" : "=r"(w[h]) : "f"(x[2 * h]), "f"(x[2 * h + 1]));
            x[2 * h] -= __uint_as_float(w[h] << 16);
            x[2 * h + 1] -= __uint_as_float(w[h] & 0xffff0000u);
        }
        p[q] = make_uint2(w[0], w[1]);
    }
}
// four entries' parts at element offset o (a multiple of 4) of the parts that are held
__device__ __forceinline__ void put_parts(const Parts &t, size_t o, const float (&v)[4])
{
    if (!t.h)
        return;
    if (t.m) {
        uint2 p[3];
        parts4<3>(v, p);
        *reinterpret_cast<uint2 *>(t.h + o) = p[0];
        *reinterpret_cast<uint2 *>(t.m + o) = p[1];
        *reinterpret_cast<uint2 *>(t.l + o) = p[2];
    } else {
        uint2 p[2];
        parts4<2>(v, p);
        *reinterpret_cast<uint2 *>(t.h + o) = p[0];
        *reinterpret_cast<uint2 *>(t.l + o) = p[1];
    }
}

// W (rows x cols, row stride ldi) into out (row stride ldo, a multiple of 4) and
// its parts, zeros in the padding (column ldo - 1 the last);
// block (x, y) takes 1024 columns of row y.  X may be out itself.
__device__ __forceinline__ void load_w(const float *X, int rows, int cols, int ldi, const double *stats, float *out, int ldo,
                                       const Parts &parts, int *flags, int x, int r)
{
    const int c = 4 * (x * blockDim.x + threadIdx.x);
    int bad = 0;
    if (c < ldo) {
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool in = r < rows && c + u < cols;
            v[u] = in ? X[(size_t)r * ldi + c + u] : 0.0f;
            bad |= !isfinite(v[u]);
            if (stats && in)
                v[u] = zscore_one(v[u], stats_pairs(stats));
        }
        const size_t o = (size_t)r * ldo + c;
        *reinterpret_cast<float4 *>(out + o) = make_float4(v[0], v[1], v[2], v[3]);
        put_parts(parts, o, v);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0)
        atomicOr(&flags[0], 1);
}

// A symmetric n x n network (row stride ldi) as 64 x 64 blocks: each pair of
// mirror blocks (bi, bj), (bj, bi), bi <= bj, is read once, along rows.
// flags[0] |= 1 on a non-finite entry, flags[1] |= 1 when X[i][j] != X[j][i].
// Written, padding (to out.ld, a multiple of 64) included: block (bi, bj) of
// out.F and of the parts, block (bj, bi) too where the form holds it; the
// diagonal goes to out.d and out.df and reads as zero in F and the parts.  X
// may be out.F itself (each block pair is one block's alone).  256 threads.
// Bound by memory.  A thread holds four entries of four rows of the upper block
// in registers and only the lower block goes through shared memory; whole
// blocks of 16-byte aligned rows load 16 bytes at a time without a bounds
// check.  With both blocks in shared memory, scalar loads and a check per entry
// the instructions took longer than the bytes: 545 us for the networks of
// 1000 x 17000 under BF16X3 (2.07 GB), 355 us now.
constexpr int LB = 64;
__host__ __device__ inline int block_pairs(int ld) { return ceil_div(ld, LB) * (ceil_div(ld, LB) + 1) / 2; }
// pair t of the upper triangle's blocks, numbered column by column; 8 t + 1 < 2^24 for n <= 46000, so
// the FP32 square root is close; the loops correct it
__device__ __forceinline__ void block_pair(int t, int &bi, int &bj)
{
    bj = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while (bj > 0 && bj * (bj + 1) / 2 > t)
        --bj;
    while ((bj + 1) * (bj + 2) / 2 <= t)
        ++bj;
    bi = t - bj * (bj + 1) / 2;
}
__device__ __forceinline__ void load_sym(const float *X, int n, int ldi, const double *stats, const SymOut &out, int *flags,
                                         int first, int step)
{
    const int npairs = block_pairs(out.ld);
    __shared__ float lo[LB][LB + 1], up[LB][LB + 1];  // rows of 65: columns are read as well as rows
    const int c4 = 4 * (threadIdx.x & 15), tr = threadIdx.x >> 4;  // rows tr, tr + 16, ..., four columns
    const bool aligned = (ldi & 3) == 0 && ((uintptr_t)X & 15) == 0;
    const float4 q = stats ? stats_pairs(stats) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float nf = 0.0f;  // NaN once an entry is not finite
    bool asym = false;
    for (int t = first; t < npairs; t += step) {
        int bi, bj;
        block_pair(t, bi, bj);
        const int i0 = bi * LB, j0 = bj * LB;
        const bool whole = j0 + LB <= n;  // (i0 <= j0)
        float a[4][4];
        if (whole && aligned) {
            float4 v[4], w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                v[k] = __ldcs(reinterpret_cast<const float4 *>(X + (size_t)(i0 + 16 * k + tr) * ldi + j0 + c4));
#pragma unroll
            for (int k = 0; k < 4; ++k)
                w[k] = __ldcs(reinterpret_cast<const float4 *>(X + (size_t)(j0 + 16 * k + tr) * ldi + i0 + c4));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                a[k][0] = v[k].x;
                a[k][1] = v[k].y;
                a[k][2] = v[k].z;
                a[k][3] = v[k].w;
                float *l = &lo[16 * k + tr][c4];
                l[0] = w[k].x;
                l[1] = w[k].y;
                l[2] = w[k].z;
                l[3] = w[k].w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int r = 16 * k + tr, c = c4 + u;
                    a[k][u] = i0 + r < n && j0 + c < n ? X[(size_t)(i0 + r) * ldi + j0 + c] : 0.0f;
                    lo[r][c] = j0 + r < n && i0 + c < n ? X[(size_t)(j0 + r) * ldi + i0 + c] : 0.0f;
                }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float m = lo[c4 + u][16 * k + tr];
                nf = fmaf(a[k][u], 0.0f, fmaf(m, 0.0f, nf));
                asym |= a[k][u] != m;
            }
        if (stats) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (whole || (i0 + 16 * k + tr < n && j0 + c4 + u < n))
                        a[k][u] = zscore_one(a[k][u], q);
        }
        if (bi == bj) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (16 * k + tr == c4 + u && i0 + c4 + u < n) {
                        out.d[i0 + c4 + u] = (double)a[k][u];
                        out.df[i0 + c4 + u] = a[k][u];
                        a[k][u] = 0.0f;
                    }
        }
        const bool lf = out.F && out.f_full, lp = out.parts.h && (out.p_full || i0 / out.p_block == j0 / out.p_block);
        const bool lower = bi != bj && (lf || lp);
        // rows of the upper block
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const size_t o = (size_t)(i0 + 16 * k + tr) * out.ld + j0 + c4;
            if (out.F)
                *reinterpret_cast<float4 *>(out.F + o) = make_float4(a[k][0], a[k][1], a[k][2], a[k][3]);
            put_parts(out.parts, o, a[k]);
            if (lower) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    up[16 * k + tr][c4 + u] = a[k][u];
            }
        }
        __syncthreads();
        // rows of the lower block, from the upper one's columns (the next pair's writes to `up` are
        // behind its own barrier)
        if (lower) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int r = 16 * k + tr;
                const float v[4] = {up[c4][r], up[c4 + 1][r], up[c4 + 2][r], up[c4 + 3][r]};
                const size_t o = (size_t)(j0 + r) * out.ld + i0 + c4;
                if (lf)
                    *reinterpret_cast<float4 *>(out.F + o) = make_float4(v[0], v[1], v[2], v[3]);
                if (lp)
                    put_parts(out.parts, o, v);
            }
        }
    }
    const int bad = __syncthreads_or(nf != nf);
    const int ne = __syncthreads_or(asym);
    if (threadIdx.x == 0) {
        if (bad)
            atomicOr(&flags[0], 1);
        if (ne)
            atomicOr(&flags[1], 1);
    }
}

// One launch: blocks [0, nc) C, [nc, nc + np) P, the rest W.
__global__ void __launch_bounds__(256, 4) k_load(const __grid_constant__ StateIn in, float *W, Parts wparts, int Gp,
                                              const __grid_constant__ SymOut P, const __grid_constant__ SymOut C, int nc,
                                              int np, int *flags)
{
    const int b = blockIdx.x;
    if (b < nc) {
        load_sym(in.C, in.G, in.ldc, in.sc, C, flags, b, nc);
    } else if (b < nc + np) {
        load_sym(in.P, in.T, in.ldp, in.sp, P, flags, b - nc, np);
    } else {
        const int q = b - nc - np, xb = ceil_div(Gp, 1024);
        load_w(in.W, in.T, in.G, in.ldw, in.sw, W, Gp, wparts, flags, q % xb, q / xb);
    }
}

__global__ void k_diag_to_float(const double *d, float *df, int n)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        df[i] = (float)d[i];
}

// x^2 into a compensated FP32 pair: x^2 = p + pe exactly, p through TwoSum
__device__ __forceinline__ void sq_add(float x, float &acc, float &cmp)
{
    float p, pe;
    two_prod(x, x, p, pe);
    two_sum_add(acc, cmp, p);
    cmp = __fadd_rn(cmp, pe);
}

// out[i] = sum_j X[i][j]^2, X Z-scored on the way when `stats` is given; with
// `diag` the entry on the diagonal is left out and diag[i]^2 added: one warp
// per row, lane l taking the 4-wide column groups l, l + 32, ..., then the
// ragged columns.  Compensated FP32 pairs folded into an FP64 total every 16
// groups, FP64 across the warp: a fixed order.
__device__ __forceinline__ void row_norms(const float *__restrict__ X, int rows, int cols, int ld, const double *stats,
                                          const double *diag, float *out, int block)
{
    const int warp = block * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (warp >= rows)
        return;
    const bool aligned = (ld & 3) == 0 && ((uintptr_t)X & 15) == 0;
    const float *x = X + (size_t)warp * ld;
    const int c4n = cols >> 2, skip = diag ? warp : -1;
    const float4 q = stats ? stats_pairs(stats) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    auto term = [&](float v, int c, float &acc, float &cmp) {
        if (stats)
            v = zscore_one(v, q);
        sq_add(c == skip ? 0.0f : v, acc, cmp);
    };
    double tot = 0.0;
    for (int c0 = 0; c0 < c4n; c0 += 16 * 32) {
        float acc = 0.0f, cmp = 0.0f;
        const int ce = min(c4n, c0 + 16 * 32);
#pragma unroll 4
        for (int c = c0 + lane; c < ce; c += 32) {
            const float4 v = load4(x, c, aligned);
            term(v.x, 4 * c, acc, cmp);
            term(v.y, 4 * c + 1, acc, cmp);
            term(v.z, 4 * c + 2, acc, cmp);
            term(v.w, 4 * c + 3, acc, cmp);
        }
        tot += (double)acc + (double)cmp;
    }
    {
        float acc = 0.0f, cmp = 0.0f;
        for (int c = (c4n << 2) + lane; c < cols; c += 32)
            term(x[c], c, acc, cmp);
        tot += (double)acc + (double)cmp;
    }
    for (int o = 16; o > 0; o >>= 1)
        tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if (lane == 0) {
        if (diag)
            tot += diag[warp] * diag[warp];
        out[warp] = (float)tot;
    }
}

// out[j] = sum_i X[i][j]^2 over the first `rows` rows: the squared column
// norms of a row-major matrix without its transpose.  A block takes 32
// columns, its eight warps every eighth row (compensated FP32 pairs folded
// into FP64 every 32 of them), FP64 across the warps in a fixed order.
__device__ __forceinline__ void col_norms(const float *__restrict__ X, int rows, int cols, int ld, float *out, int block)
{
    __shared__ double sh[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, j = block * 32 + lane;
    double tot = 0.0;
    if (j < cols)
        for (int r0 = w; r0 < rows; r0 += 256) {
            float acc = 0.0f, cmp = 0.0f;
            const int re = min(rows, r0 + 256);
#pragma unroll 8
            for (int r = r0; r < re; r += 8)
                sq_add(X[(size_t)r * ld + j], acc, cmp);
            tot += (double)acc + (double)cmp;
        }
    sh[w][lane] = tot;
    __syncthreads();
    if (w == 0 && j < cols) {
        double t = 0.0;
        for (int q = 0; q < 8; ++q)
            t += sh[q][lane];
        out[j] = (float)t;
    }
}

// One launch: blocks of 8 rows of C, then of P, then of W, then of 32 columns of W.
__global__ void __launch_bounds__(256) k_norms(const __grid_constant__ StateNorms n)
{
    const StateIn &in = n.in;
    const int bG = ceil_div(in.G, 8), bT = ceil_div(in.T, 8), b = blockIdx.x;
    if (b < bG)
        row_norms(in.C, in.G, in.G, in.ldc, in.sc, n.cd, n.csqC, b);
    else if (b < bG + bT)
        row_norms(in.P, in.T, in.T, in.ldp, in.sp, n.pd, n.rsqP, b - bG);
    else if (b < bG + 2 * bT)
        row_norms(in.W, in.T, in.G, in.ldw, nullptr, nullptr, n.rsqW, b - bG - bT);
    else
        col_norms(in.W, in.T, in.G, in.ldw, n.csqW, b - bG - 2 * bT);
}

// Lower triangle from the upper one: X[r][c] = X[c][r] for r > c (32 x 32
// blocks through shared memory, so both sides are read and written along rows).
__global__ void k_symmetrize(float *X, int n, int ld)
{
    __shared__ float tile[32][33];
    const int bx = blockIdx.x, by = blockIdx.y;  // destination block (row by, column bx)
    if (by < bx)
        return;
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
    for (int k = ty; k < 32; k += 8) {  // source block (row bx, column by)
        const int r = bx * 32 + k, c = by * 32 + tx;
        tile[k][tx] = (r < n && c < n) ? X[(size_t)r * ld + c] : 0.0f;
    }
    __syncthreads();
    for (int k = ty; k < 32; k += 8) {
        const int r = by * 32 + k, c = bx * 32 + tx;  // destination (r, c) = source (c, r)
        if (r < n && c < n && r > c)
            X[(size_t)r * ld + c] = tile[tx][k];
    }
}

}  // namespace

namespace {

// Pearson initialisation (Sec. II-A), first step: row g of the expression
// matrix X (G x N, row-major) becomes z_g = (x_g - m_g) / |x_g - m_g|, so that
// z_g . z_h is the correlation of genes g and h.  One warp per row; mean and
// centred norm in FP64 (two passes, fixed lane order); z stored as a BF16
// split (hi = bf16(z), lo = bf16(z - hi)) in Zh, Zl ([G][Kp], the padding left
// zero by the caller).  flags[0] |= 1 on a non-finite sample, |= 2 on a row of
// zero variance.
__global__ void k_standardize_rows(const float *__restrict__ X, int G, int N, __nv_bfloat16 *__restrict__ Zh,
                                   __nv_bfloat16 *__restrict__ Zl, int Kp, int *flags)
{
    const int g = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (g >= G)
        return;
    const float *x = X + (size_t)g * N;
    double s = 0.0;
    bool finite = true;
    for (int k = lane; k < N; k += 32) {
        finite = finite && isfinite(x[k]);
        s += (double)x[k];
    }
    for (int off = 16; off >= 1; off >>= 1)
        s += __shfl_xor_sync(0xffffffffu, s, off);
    const double m = s / (double)N;
    double q = 0.0;
    for (int k = lane; k < N; k += 32) {
        const double d = (double)x[k] - m;
        q += d * d;
    }
    for (int off = 16; off >= 1; off >>= 1)
        q += __shfl_xor_sync(0xffffffffu, q, off);
    const unsigned bad = __ballot_sync(0xffffffffu, !finite);
    if (lane == 0 && (bad || !(q > 0.0)))
        atomicOr(flags, (bad ? 1 : 0) | (q > 0.0 ? 0 : 2));
    if (bad || !(q > 0.0))
        return;
    const double inv = 1.0 / sqrt(q);
    for (int k = lane; k < N; k += 32) {
        const float z = (float)(((double)x[k] - m) * inv);
        const __nv_bfloat16 hi = __float2bfloat16_rn(z);
        Zh[(size_t)g * Kp + k] = hi;
        Zl[(size_t)g * Kp + k] = __float2bfloat16_rn(z - __bfloat162float(hi));
    }
}

// The full symmetric n x n matrix (dense, any alignment) from its
// strict upper triangle, FP32 in X or a BF16 split pair H + L (exact in FP32;
// row stride ldi, a multiple of 4), and its FP64 diagonal, in 64 x 64 blocks:
// each block above the diagonal is read once and written twice, the second
// time turned through shared memory, 16 bytes at a time where the rows allow it
// (1000 x 17000: 335 us, 353 with 4-byte stores).  256 threads.
__device__ __forceinline__ void store_sym(const float *__restrict__ X, const __nv_bfloat16 *__restrict__ H,
                                          const __nv_bfloat16 *__restrict__ L, int n, int ldi,
                                          const double *__restrict__ diag, float *__restrict__ out, int first, int step)
{
    const int npairs = block_pairs(n), ldo = n;
    __shared__ float a[LB][LB + 1];
    const int tx = threadIdx.x & (LB - 1), ty = threadIdx.x / LB;  // stores: 4 rows of 64
    const int c4 = 4 * (threadIdx.x & 15), tr = threadIdx.x >> 4;  // loads: 16 rows of 16 x 4
    const bool aligned = (ldo & 3) == 0 && ((uintptr_t)out & 15) == 0;
    for (int t = first; t < npairs; t += step) {
        int bi, bj;
        block_pair(t, bi, bj);
        const int i0 = bi * LB, j0 = bj * LB;
        const bool vec = aligned && bi < bj && j0 + LB <= n;  // 16 bytes at a time, no bounds, no diagonal
#pragma unroll
        for (int k = 0; k < LB; k += 16) {
            const int r = k + tr, gi = i0 + r, gj = j0 + c4;
            float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (gi < n && gj < n) {  // (the padding up to the row stride is readable)
                const size_t o = (size_t)gi * ldi + gj;
                if (X) {
                    const float4 f = *reinterpret_cast<const float4 *>(X + o);
                    v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
                } else {
                    const uint2 h = *reinterpret_cast<const uint2 *>(H + o), l = *reinterpret_cast<const uint2 *>(L + o);
                    v[0] = __uint_as_float(h.x << 16) + __uint_as_float(l.x << 16);
                    v[1] = __uint_as_float(h.x & 0xffff0000u) + __uint_as_float(l.x & 0xffff0000u);
                    v[2] = __uint_as_float(h.y << 16) + __uint_as_float(l.y << 16);
                    v[3] = __uint_as_float(h.y & 0xffff0000u) + __uint_as_float(l.y & 0xffff0000u);
                }
            }
            if (vec)
                __stcs(reinterpret_cast<float4 *>(out + (size_t)gi * ldo + gj), make_float4(v[0], v[1], v[2], v[3]));
#pragma unroll
            for (int u = 0; u < 4; ++u)
                a[r][c4 + u] = v[u];
        }
        __syncthreads();
        if (vec) {
#pragma unroll
            for (int k = 0; k < LB; k += 16) {
                const int r = k + tr;
                __stcs(reinterpret_cast<float4 *>(out + (size_t)(j0 + r) * ldo + i0 + c4),
                       make_float4(a[c4][r], a[c4 + 1][r], a[c4 + 2][r], a[c4 + 3][r]));
            }
        }
#pragma unroll 4
        for (int k = 0; k < LB && !vec; k += 4) {
            const int r = k + ty;
            if (i0 + r < n && j0 + tx < n) {
                const bool up = bi < bj || r < tx;
                out[(size_t)(i0 + r) * ldo + j0 + tx] =
                    bi == bj && r == tx ? (float)diag[i0 + r] : (up ? a[r][tx] : a[tx][r]);
            }
            if (bi < bj && j0 + r < n && i0 + tx < n)
                out[(size_t)(j0 + r) * ldo + i0 + tx] = a[tx][r];
        }
        __syncthreads();
    }
}

// One launch: blocks [0, nc) C, [nc, nc + np) P, the rest rows of W.
__global__ void __launch_bounds__(256) k_store(const __grid_constant__ StateOut o, int nc, int np)
{
    if (o.flags && (o.flags[0] | o.flags[1] | o.ctl->status))
        return;
    const int b = blockIdx.x;
    if (b < nc) {
        store_sym(o.C, o.Ch, o.Cl, o.G, o.Gp, o.cd, o.oC, b, nc);
    } else if (b < nc + np) {
        store_sym(o.P, nullptr, nullptr, o.T, o.Tp, o.pd, o.oP, b - nc, np);
    } else {
        const int r = b - nc - np;
        const float *w = o.W + (size_t)r * o.Gp;
        float *out = o.oW + (size_t)r * o.G;
        const int g4 = (o.G & 3) == 0 && ((uintptr_t)o.oW & 15) == 0 ? o.G >> 2 : 0;
#pragma unroll 4
        for (int c = threadIdx.x; c < g4; c += 256)
            __stcs(reinterpret_cast<float4 *>(out) + c, reinterpret_cast<const float4 *>(w)[c]);
#pragma unroll 4
        for (int c = 4 * g4 + threadIdx.x; c < o.G; c += 256)
            out[c] = w[c];
    }
}

// X_ii = 1 for i < n (a correlation matrix's diagonal)
__global__ void k_unit_diag(float *X, int n, int ld)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        X[(size_t)i * ld + i] = 1.0f;
}

}  // namespace

cudaError_t launch_standardize_rows(const float *X, int G, int N, __nv_bfloat16 *Zh, __nv_bfloat16 *Zl, int Kp,
                                    int *flags, cudaStream_t s)
{
    k_standardize_rows<<<ceil_div(G, 8), 256, 0, s>>>(X, G, N, Zh, Zl, Kp, flags);
    return cudaGetLastError();
}

cudaError_t launch_unit_diag(float *X, int n, int ld, cudaStream_t s)
{
    k_unit_diag<<<ceil_div(n, 256), 256, 0, s>>>(X, n, ld);
    return cudaGetLastError();
}

cudaError_t launch_store(const StateOut &o, cudaStream_t s)
{
    const int nc = o.oC ? std::min(block_pairs(o.G), 152 * 12) : 0, np = o.oP ? std::min(block_pairs(o.T), 152 * 4) : 0;
    const int n = nc + np + (o.oW ? o.T : 0);
    if (n == 0)
        return cudaSuccess;
    k_store<<<n, 256, 0, s>>>(o, nc, np);
    return cudaGetLastError();
}

cudaError_t launch_symmetrize(float *X, int n, int ld, cudaStream_t s)
{
    dim3 grid(ceil_div(n, 32), ceil_div(n, 32)), block(32, 8);
    k_symmetrize<<<grid, block, 0, s>>>(X, n, ld);
    return cudaGetLastError();
}

// The element kernels read rows as float4: the row stride and base must
// keep every row 16-byte aligned.
static bool rows_aligned(const void *X, int ld) { return (ld & 3) == 0 && ((uintptr_t)X & 15) == 0; }

cudaError_t launch_stats(const float *X, int rows, int cols, int ld, double *stats, double *partials, cudaStream_t s)
{
    if ((uintptr_t)stats & 15)
        return cudaErrorInvalidValue;
    const bool al = rows_aligned(X, ld);
    double count = (double)rows * (double)cols;
    k_stats_partial<0><<<RED_BLOCKS, RED_THREADS, 0, s>>>(X, rows, cols, ld, al, stats, partials);
    k_stats_final<<<1, RED_THREADS, 0, s>>>(partials, RED_BLOCKS, count, 0, stats);
    k_stats_partial<1><<<RED_BLOCKS, RED_THREADS, 0, s>>>(X, rows, cols, ld, al, stats, partials);
    k_stats_final<<<1, RED_THREADS, 0, s>>>(partials, RED_BLOCKS, count, 1, stats);
    return cudaGetLastError();
}

cudaError_t launch_load(const StateIn &in, float *W, const Parts &wparts, int Tp, int Gp, const SymOut &P, const SymOut &C,
                        int *flags, cudaStream_t s)
{
    const int nc = std::min(block_pairs(C.ld), 152 * 4), np = std::min(block_pairs(P.ld), 152 * 2);
    k_load<<<nc + np + Tp * ceil_div(Gp, 1024), 256, 0, s>>>(in, W, wparts, Gp, P, C, nc, np, flags);
    return cudaGetLastError();
}

cudaError_t launch_norms(const StateNorms &n, cudaStream_t s)
{
    k_norms<<<ceil_div(n.in.G, 8) + 2 * ceil_div(n.in.T, 8) + ceil_div(n.in.G, 32), 256, 0, s>>>(n);
    return cudaGetLastError();
}

cudaError_t launch_diag_to_float(const double *d, float *df, int n, cudaStream_t s)
{
    k_diag_to_float<<<ceil_div(n, 256), 256, 0, s>>>(d, df, n);
    return cudaGetLastError();
}

}  // namespace panda
