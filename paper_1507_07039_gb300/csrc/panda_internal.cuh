// Internal declarations of libpanda_gb300 (not part of the C ABI).
//
// Device layout (all row-major, every dimension padded with zeros to a
// multiple of 128, or 256 on the tensor-core path, so that GEMM tiles never
// need bounds checks in their main loops; the epilogues mask by the true T
// and G):
//   W[2]   Tp x Gp  fp32   regulatory network, ping-pong (current / next)
//   Poff   Tp x Tp  fp32   P with a zero diagonal (diagonal kept in pd)
//   Coff   Gp x Gp  fp32   C with a zero diagonal (diagonal kept in cd); in the
//                          BF16X3 and BF16X2 modes only while a create or
//                          set_state derives the state, which is then held as
//                          the split pair Ch + Cl alone
//   pd, cd          fp64   diagonals of P and C
//   rsqP, csqC      fp32   |P_i.|^2 and |C_.j|^2, diagonal included
//   rsqW, csqW      fp32   |W_i.|^2 and |W_.j|^2 of the current W
// plus per-tile partial sums (scratch) and a small control block.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cmath>
#include <vector>
#include <cuda_bf16.h>
#include <stdint.h>

namespace panda {

constexpr int TILE = 128;          // padding granule
constexpr int HIST_CAP = 1 << 16;  // iterations whose h is kept on the device

// Device control block, read by every kernel of an iteration.
struct Ctl {
    int active;     // kernels of an iteration do their work only while 1
    int iters;      // iterations done so far (the next one uses t = iters + 1)
    int stop_at;    // iteration count at which the current run stops
    int status;     // bit 0: non-finite state; bit 1: device wait timed out
    int converged;  // 1 when the last iteration gave h < tol
    float alpha;
    unsigned fin_blocks;  // k_fin: blocks done in this iteration (the last one runs the tail)
    double tol;
    double h_last;
    double h_next;  // h of the iteration under way (k_reduce_wnorms)
};

enum : int { ST_NONFINITE = 1, ST_TIMEOUT = 2 };

// Pointers and shapes handed to kernels by value.
struct Dev {
    int T, G, Tp, Gp, nbT, nbG;  // true sizes, padded sizes, 128-blocks
    int diag;                    // panda_diag
    double inv_n1P, inv_n1C;     // 1 / (T - 1), 1 / (G - 1) (0 for one node)
    float *W[2];
    float *Poff, *Coff;
    double *pd, *cd;
    float *pdf, *cdf;            // FP32 copies of the diagonals for epilogues
    float *rsqP, *csqC, *rsqW, *csqW;
    // scratch
    int nwr;                     // phase 1's column tiles: slots of the next two arrays
    float *wrow_part;            // nwr x Tp
    float *wcol_part;            // nbT x Gp
    double *hpart;               // nwr x nbT
    float *ps_sum, *ps_sq, *ps_vsq;  // slots x Tp  row partials of P'
    float *cs_sum, *cs_sq, *cs_vsq;  // slots x Gp  row partials of C'
    int narrow;                      // layout of those slots, row roles first, then column roles:
                                     // 0: 256-column tiles of CTA pairs; 1: FP32's 64-column tiles
    Ctl *ctl;
    double *hist;                // HIST_CAP
    double *e2tab;               // HIST_CAP + 1: e^{2 alpha t}, computed on the host
    // BF16 split copies (tensor-core path only; NULL otherwise)
    __nv_bfloat16 *Wh[2], *Wl[2];  // W^T operands are read from these MN-major
    __nv_bfloat16 *Ph, *Pl, *Ch, *Cl;
    // FP32 path: the middle parts of the three-way splits (h, m, l) of W, P_off and C_off
    __nv_bfloat16 *Wm[2], *Pm, *Cm;
    void *f32_host;              // host-side tensor maps and work lists (FP32 path)
    // 1: C is held only as its split pair Ch + Cl (BF16X3, BF16X2): its upper
    // triangle and diagonal 256-blocks are the state, Coff is NULL between
    // calls (a staging buffer while a create or set_state derives the state)
    int c_split;
    // 1: B operands carry their lo halves too (BF16X3, hi.hi + hi.lo + lo.hi);
    // 0: B operands are BF16 hi only (BF16X2, hi.hi + lo.hi; C's lo half is never made)
    int split_b;
    // FP8MIX: E4M3 copies (one byte per entry) for W.C and W^T.W, and their scales
    int fp8;
    uint8_t *W8[2], *Wt8[2];     // W [Tp][Gp] and W^T [Gp][Tp], entries times f8[b]
    uint8_t *C8;                 // C_off [Gp][Gp], both triangles, entries times f8[2]
    float *f8;                   // [0], [1]: scale of W8/Wt8 buffer b; [2]: of C8; [3]: for the next W'
    unsigned *f8n;               // squared-norm maxima (float bits): [0..3] this iteration's
                                 // (rsqP, csqC, rsqW, csqW), [4..7] the state's, latched
    void *tc_host;               // host-side tensor maps of the split copies (tensor-core path)
    float *p1_acc;               // phase 1: per CTA of its grid, a tile's slot: the running sum of the
                                 // availability numerator's chunks; FP32: an uncut tile's R-num
    float *p1_fix;               // slots where a cut tile's parts meet: per tile cut between two CTA
                                 // pairs one per CTA rank; FP32: one per part and rank
    int *p1_flag;                // per cut tile and CTA rank: its head's adds have landed (FP32: the
                                 // parts that have arrived)
    int p1_cuts;                 // cut tiles (slots and flag pairs above)
};

// Largest power of two s with s * bound <= 448 (the largest finite E4M3 value):
// bound >= every |x| that is scaled by s, so no entry saturates.
__host__ __device__ inline float e4m3_scale(float bound)
{
    if (!(bound > 0.0f) || !(bound < 3.0e38f))
        return 1.0f;
    const float x = 448.0f / bound;
    union { float f; unsigned u; } v{x};
    int e = (int)((v.u >> 23) & 0xffu) - 127;  // floor(log2 x) for normal x
    e = e < -100 ? -100 : (e > 100 ? 100 : e);
    v.u = (unsigned)(e + 127) << 23;
    return v.f;
}

// The alpha-free bounds behind the scales.  |Tan(x, y)| <= sqrt(|x| |y|) (Eq. 1);
// the damped updates are convex combinations, so |W'| <= max(|W|, (|R| + |A|) / 2)
// and |C'| <= max(|C|, |Tan|).  An entry is at most its row's norm.  The factor
// 1.25 covers E4M3 numerators, which may exceed the exact products by ~2^-4 per term.
__host__ __device__ inline float fp8_bound_w(float mrP, float mcC, float mrW, float mcW)
{
    const float t = 1.25f * 0.5f * (sqrtf(sqrtf(mrP) * sqrtf(mcW)) + sqrtf(sqrtf(mrW) * sqrtf(mcC)));
    return 1.001f * fmaxf(sqrtf(mrW), t);
}
__host__ __device__ inline float fp8_bound_c(float mcC, float mcW)
{
    return 1.001f * fmaxf(sqrtf(mcC), 1.25f * sqrtf(mcW));
}

// A kernel launch that returns its error.
template <class... P, class... A>
inline cudaError_t launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A &...args)
{
    kernel<<<grid, block, smem, s>>>(static_cast<P>(args)...);
    return cudaGetLastError();
}

// Where a caller's array lies: in memory that kernels on `device` may read and write (HERE), in
// another GPU's (ELSEWHERE: only copies reach it, whether or not peer access is on), or on the host.
enum class Where { HOST, HERE, ELSEWHERE };
inline Where where_is(const void *p, int device)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return Where::HOST;
    }
    if (a.type == cudaMemoryTypeManaged)
        return Where::HERE;
    return a.type != cudaMemoryTypeDevice ? Where::HOST : a.device == device ? Where::HERE : Where::ELSEWHERE;
}

__host__ __device__ inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
__host__ __device__ inline int round_up(int a, int b) { return ceil_div(a, b) * b; }

// ---- FP32 error-free transforms --------------------------------------------
// This GPU's FP64 pipe issues about two operations per clock per SM, the FP32
// pipe 128, so sums and products that want more than FP32 accuracy run as
// FP32 pairs whose rounding errors are recovered exactly.

// Knuth's TwoSum: s + x = s' + e exactly (round to nearest, no overflow),
// s' = fl(s + x); the error e is added into the compensation c.
__device__ __forceinline__ void two_sum_add(float &s, float &c, float x)
{
    const float t = s + x;
    const float z = t - s;
    c += (s - (t - z)) + (x - z);
    s = t;
}

// a + b = s + e exactly
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float z = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
}

// a * b = p + e exactly (the product's rounding error from one FMA), barring
// underflow of e
__device__ __forceinline__ void two_prod(float a, float b, float &p, float &e)
{
    p = __fmul_rn(a, b);
    e = __fmaf_rn(a, b, -p);
}

// ---- launchers (k_setup.cu) ------------------------------------------------
// Z-score statistics of X (read only): stats[0] = mean, stats[1] = population std, then the
// FP32 pairs that the loads below apply; 4 doubles, 16-byte aligned
cudaError_t launch_stats(const float *X, int rows, int cols, int ld, double *stats, double *partials, cudaStream_t s);
// BF16 parts of a matrix: h, l (two-way split) or h, m, l (three-way, exact); h NULL: none
struct Parts {
    __nv_bfloat16 *h, *m, *l;
};
// What a symmetric network becomes: its FP32 matrix F (NULL: not held) with a zero diagonal,
// both triangles if f_full, else the upper one and the diagonal 64-blocks; its parts, both
// triangles if p_full, else the upper one and the diagonal blocks of p_block; its diagonal.
struct SymOut {
    float *F;
    int f_full;
    Parts parts;
    int p_full, p_block;
    int ld;  // row stride of F and the parts
    double *d;
    float *df;
};
// The networks of a state where they lie (device memory, any alignment, row strides ld*), each
// Z-scored by its stats (NULL: as it is)
struct StateIn {
    const float *W, *P, *C;
    int T, G, ldw, ldp, ldc;
    const double *sw, *sp, *sc;
};
// Checked (flags[0] |= 1: a non-finite entry, flags[1] |= 1: P or C not symmetric) and written in
// those forms, the padding up to Tp x Gp, Tp x Tp and Gp x Gp as zeros
cudaError_t launch_load(const StateIn &in, float *W, const Parts &wparts, int Tp, int Gp, const SymOut &P, const SymOut &C,
                        int *flags, cudaStream_t s);
// Squared norms: rows and columns of W (as loaded, row stride Gp), rows of P and C from where
// they lie, the diagonal entry left out and pd, cd added; P and C Z-scored by their stats
struct StateNorms {
    StateIn in;       // (in.W, in.ldw: W as loaded; in.sw unused)
    const double *pd, *cd;
    float *rsqW, *csqW, *rsqP, *csqC;
};
cudaError_t launch_norms(const StateNorms &n, cudaStream_t s);
cudaError_t launch_diag_to_float(const double *d, float *df, int n, cudaStream_t s);
// X[r][c] = X[c][r] for r > c: the full matrix from its upper triangle
cudaError_t launch_symmetrize(float *X, int n, int ld, cudaStream_t s);
// The state back into dense device arrays (each may be NULL): W (row stride Gp) and the symmetric
// matrices with these strict upper triangles (FP32 X, or X NULL and the BF16 split pair H + L)
// and diagonals.  With guard.flags: nothing is written if the checks or the iteration found a fault.
struct StateOut {
    int T, G, Tp, Gp;
    const float *W, *P, *C;
    const __nv_bfloat16 *Ch, *Cl;
    const double *pd, *cd;
    float *oW, *oP, *oC;
    const int *flags;
    const Ctl *ctl;
};
cudaError_t launch_store(const StateOut &o, cudaStream_t s);
// Pearson initialisation (Sec. II-A): unit-norm centred rows of X (G x N) as a
// BF16 split [G][Kp]; flags[0] |= 1 (non-finite) / 2 (zero variance)
cudaError_t launch_standardize_rows(const float *X, int G, int N, __nv_bfloat16 *Zh, __nv_bfloat16 *Zl, int Kp,
                                    int *flags, cudaStream_t s);
cudaError_t launch_unit_diag(float *X, int n, int ld, cudaStream_t s);

// Optional per-kernel timing: when ev is not NULL, ev[0] is recorded before the
// first kernel of the iteration and ev[k + 1] after kernel k.
struct KernelEvents {
    cudaEvent_t *ev;
    int n;  // events recorded so far
    bool capturing;  // a graph is being captured: the record becomes an event-record node
    void mark(cudaStream_t s)
    {
        if (ev)
            cudaEventRecordWithFlags(ev[n++], s, capturing ? cudaEventRecordExternal : cudaEventRecordDefault);
    }
};

// ---- after the products (k_norms.cu) ----------------------------------------
// Diagonals, norms of P and C, h, counter, stop test
cudaError_t launch_fin(const Dev &d, cudaStream_t s, KernelEvents &ke);
// FP64 sums of the per-tile norm partials of W', and h
cudaError_t launch_reduce_wnorms(const Dev &d, cudaStream_t s);
// The same kernels over a set of networks (device arrays): blocks[b] = (network,
// that network's block), set_norm_blocks(T, G) + 1 blocks per network.
cudaError_t launch_reduce_wnorms_set(const Dev *devs, const int2 *blocks, int nblocks, cudaStream_t s);
cudaError_t launch_fin_set(const Dev *devs, const int2 *blocks, int nblocks, cudaStream_t s);
int set_norm_blocks(int T, int G);
// FP32 FFMA throughput of the current device in TFLOP/s (best of several
// timed launches of a loop of independent FMAs on every SM)
cudaError_t measure_ffma_peak(double *tflops);

// ---- tensor-core path (k_tc.cu) --------------------------------------------
constexpr int TC_KERNELS = 4;
extern const char *const TC_KERNEL_NAMES[TC_KERNELS];
bool tc_supported();
// Tensor maps and schedules (at the first call) and FP8MIX's E4M3 copies of the state in W[cur],
// Coff.  restored: the state came back from a checkpoint, so its BF16 split copies are made here
// too and the FP8MIX scales are kept; else the scales are derived from the state's norms.
cudaError_t tc_prepare(Dev &d, int cur, cudaStream_t s, bool restored);
void tc_release(Dev &d);
// Tiles of one network's phase 1 cut between two CTA pairs (each needs a
// running-sum slot per CTA rank and a flag per rank); -1 on a CUDA error.
int tc_phase1_cuts(const Dev &d);
// The phase-1 launch of a prepared tensor-core context: CTA pairs, resident
// two-CTA clusters; returns its cut tiles (-1: not prepared).
int tc_phase1_layout(const Dev &d, int *pairs, int *clusters);
// The phase-1 pieces of one network (Dev needs Tp, Gp, fp8, split_b) for
// `pairs` CTA pairs: per pair p, items[off[p] .. off[p + 1]) of (mt, nt,
// c0 | c1 << 16, cut or -1); returns the number of cut tiles.  Host only.
int tc_phase1_plan(const Dev &d, int pairs, bool cut_ok, std::vector<int> &off, std::vector<int4> &items);
cudaError_t launch_iteration_tc(const Dev &d, int cur, cudaStream_t s, KernelEvents &ke);

// A set of networks (tensor-core modes, same options) iterated by one launch
// per phase: phases 1 and 2 persistent over LPT schedules of every network's
// tiles, the norm and stop kernels over all their rows.  Each network's W
// buffer is (parity + its iteration count) & 1.  A tile's result does not
// depend on which pair computes it or when, so every schedule gives the same
// bits and the fastest can be picked by timing real iterations.
// C (Gp x Gp, FP32, row stride Gp) = Z . Z^T with the three-term BF16 split of
// Z ([Gp][Kp] hi and lo, Gp a multiple of 256, Kp of 64) on CTA pairs; a
// timed-out wait sets ST_TIMEOUT in ctl (device memory).
cudaError_t tc_gram(const __nv_bfloat16 *Zh, const __nv_bfloat16 *Zl, int Gp, int Kp, float *C, Ctl *ctl,
                    cudaStream_t s);

// Row-major BF16 matrix rows x cols as a tensor map: boxes of 64 columns (128
// bytes, the swizzle span) by box_rows rows; what lies outside reads as zero.
cudaError_t tc_make_map(CUtensorMap *m, const void *base, int rows, int cols, int box_rows);

// ---- FP32 path (k_f32.cu) ----------------------------------------------------
constexpr int F32_KERNELS = 4;
extern const char *const F32_KERNEL_NAMES[F32_KERNELS];
// The work lists of a network (Dev needs its sizes), kept in d.f32_host, and the
// scratch they need: floats of the per-CTA slots and of the cut tiles' slots,
// cut tiles (two counters each), the tile shape.
void f32_plan(Dev &d, int nsm, size_t *slot_floats, size_t *fix_floats, int *fixes, bool *pair);
// That plan's tile shape, and per phase its CTAs, items and cut tiles.  Host only.
void f32_plan_info(const Dev &d, int nsm, bool *pair, int *ctas, int *items, int *cuts);
// Tensor maps and device lists at the first call; restored: also the split copies of W[cur], Poff, Coff.
cudaError_t f32_prepare(Dev &d, int cur, cudaStream_t s, bool restored);
// Edge of the diagonal blocks inside which phase 2 keeps both triangles of C's split copy.
int f32_diag_block(const Dev &d);
void f32_release(Dev &d);
cudaError_t launch_iteration_f32(const Dev &d, int cur, cudaStream_t s, KernelEvents &ke);
// panda_step_static's single iteration: whole tiles, one per CTA, so at most F32_STATIC_ITEMS of
// them a phase for 512 x 512.  f32_static_lists writes both phases' lists to `lists` (device,
// F32_STATIC_LIST_BYTES), arms *d.ctl for one iteration at growth factors e2[0], e2[1], and clears
// flags[0..3]; f32_static_host returns the tensor maps of a Dev whose arrays lie at `d` (kept per
// device and padded shape by the caller).
constexpr int F32_STATIC_ITEMS = 40;
constexpr size_t F32_STATIC_LIST_BYTES = 2 * (F32_STATIC_ITEMS * 16 + 256);
constexpr size_t F32_STATIC_SLOT_BYTES = (size_t)F32_STATIC_ITEMS * 128 * 64 * sizeof(float);
cudaError_t f32_static_host(const Dev &d, void *lists, void **host);
cudaError_t f32_static_lists(const Dev &d, float alpha, double e2, void *lists, int *flags, cudaStream_t s);

struct TcSet;
// Schedule candidates of the set engine's autotuner: phase 1 (the order of each
// network's tiles in the persistent pairs' LPT lists) and phase 2 (cost model,
// epilogue weight, order of the LPT lists); TC_*_NAMES describe them.
constexpr int TC_P1_CANDS = 2, TC_P2_CANDS = 6;
extern const char *const TC_P1_NAMES[TC_P1_CANDS];
extern const char *const TC_P2_NAMES[TC_P2_CANDS];
// s: the stream that every other call of the set is given
cudaError_t tc_set_create(const std::vector<const Dev *> &ds, cudaStream_t s, TcSet **out);
cudaError_t tc_set_parity(TcSet *t, const std::vector<int> &parity, cudaStream_t s);
// one iteration of every active network with phase-1 schedule p1 and phase-2
// schedule p2; events (each may be NULL) before phase 1, before phase 2, after phase 2
cudaError_t tc_set_launch(TcSet *t, int p1, int p2, cudaStream_t s, cudaEvent_t ev0, cudaEvent_t ev1,
                          cudaEvent_t ev2);
cudaError_t tc_set_gather(TcSet *t, Ctl *host, cudaStream_t s);  // all control blocks to host (async)
void tc_set_destroy(TcSet *t);
// D (M x N, row-major) = A (M x K) . B (N x K)^T through the tcgen05 pipeline,
// host buffers; terms = 1 (hi only) or 3 (split).  *status: device status bits.
// stall_kb >= 0 plants a stage whose loads are never issued (timeout test).
cudaError_t tc_selftest_gemm(int M, int N, int K, const float *A, const float *B, float *D, int terms,
                             int pair, int stall_kb, int *status);

}  // namespace panda
