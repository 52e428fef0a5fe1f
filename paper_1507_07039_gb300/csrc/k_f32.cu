// FP32 path of one PANDA iteration on the tensor cores (sm_103a).
//
//   k_f32_phase1  per tile of W': R-num = P_off . W (K = TFs) and A-num =
//                 W . C_off (K = genes), then the fused epilogue of Eqs. 1-4:
//                 W', its three-way split, h and norm partials
//   k_reduce_wnorms  (k_norms.cu)
//   k_f32_phase2  upper-triangle tiles of W'.W'^T (P, K = genes) and
//                 W'^T.W' (C, K = TFs) with the damped update of Eq. 5, the
//                 FP32 upper triangle, split copies, partial sums for Eq. 6
//   k_fin (k_norms.cu): diagonals, norms, h, stop test
//
// Every FP32 operand is held beside its value as three BF16 parts, h = bf16(x),
// m = bf16(x - h), l = x - h - m: 3 x 8 significant bits, so h + m + l = x
// exactly for |x| above 2^-110 (below, l leaves BF16's range and x keeps fewer
// bits, to a spacing of 2^-133).  A product takes the six part products of
// weight down to 2^-16 (h.h, h.m, m.h, m.m, h.l, l.h; the three left out are
// below 2^-23 of |a||b| together, of either sign).  What the tensor core does
// lose is its accumulation: FP32, but truncated toward zero at every MMA
// (measured: -1.9e-8 of the running sum per MMA), where the former FFMA kernel
// rounded to nearest at every product.  So no chain is long: each K = 64
// stage starts a fresh accumulator, the small part products go first, while
// the accumulator is still 2^-8 of its final size, the four h.h MMAs last, and
// the stages are added up in FP32 registers, rounding to nearest.  Four
// truncations and one rounding per 64 products, where FFMA rounded 64 times:
// W after 3 iterations at 1000 x 17000 is 6e-8 from FP64 (2-norm), FFMA
// 5.0e-7.  The two TMEM buffers alternate between stages, so the epilogue
// warps drain one (and add it up) while the tensor core fills the other.
//
// Bound: the tensor pipe, 6 x the algorithmic flops (FFMA: 78 TFLOP/s
// measured, 49 reached).  A stage's operands are 96 KB per CTA for 24 MMAs,
// three quarters of BF16X3's bytes per MMA (64 KB for 12).
//
// Two tile shapes, the same code: 256 x 256 on a CTA pair (cta_group::2), and
// 128 x 64 on one CTA for networks with too few tiles to fill the chip with
// pairs (operand bytes per flop are three times a pair's, but more SMs work, a
// tile's epilogue is a quarter as long, and a third operand stage fits).
// Against 128 x 128 on one CTA the narrow tile took phases 1 + 2 from 94 to
// 85 us at 1000 x 1000, 97 to 78 us at 250 x 2100 and 44 to 38 us at 125 x 125
// (with the timing events' own 5 us each).
//
// Tiles that would leave workers idle are cut along K (f32_plan): every part
// but the last to arrive leaves its sums in slots in L2; the last one adds all
// parts in part order, so the result does not depend on who that is, and
// nobody waits.
//
// On pairs phase 2 (1.51 ms at 1000 x 17000, 1.07 of it MMAs at the rate of
// phase 1) waits for a tile's epilogue, 13 us beside 16 stages of 1.9 us, but
// for the two stages that the buffers hold.  Slower or no faster: the sums
// handed to four epilogue warps of their own through L2 (1.45-1.47 ms here, 215
// instead of 174 us at 1000 x 5200), the epilogue a chunk at a time between the
// next tile's stages (1.66 ms: too few registers beside the sums), the sums
// through L2 instead of TMEM so that both buffers are free (1.64 ms).
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <queue>
#include <vector>

#include "panda_internal.cuh"
#include "tc_common.cuh"

namespace panda {

namespace {

using namespace tc;

constexpr int EPI = 8;                         // epilogue warps: two per TMEM lane quarter
constexpr int NTHREADS = 128 + 32 * EPI;       // warpgroup 0: TMA, MMA (two warps idle); then the epilogue

struct F32Maps {
    CUtensorMap P[3];       // P_off parts [Tp][Tp], boxes of 64 x 128
    CUtensorMap W[2][3];    // W parts [Tp][Gp], both buffers
    CUtensorMap Wm[2][3];   // the same arrays in boxes of 64 x 64: W^T operands, MN-major
    CUtensorMap C[3];       // C_off parts [Gp][Gp]
    CUtensorMap Cm[3];      // in boxes of 64 x 64
};

// A work item: part `part` of `nparts` of a tile, stages [s0, s1) of its K.
// Phase 1: a = mt | nt << 16 (row and column tile), and stages run over R-num
// (TFs) first, then A-num (genes); part 0 holds all of R-num.  Phase 2: a =
// bm | bn << 15 (row and column tile), bit 31 set for a P tile.  fix (cut tiles): its arrival counter, slot: its first slot.
struct __align__(16) Item {
    uint32_t a;
    uint16_t s0, s1;
    uint16_t part, nparts;
    uint16_t fix, slot;
};
static_assert(sizeof(Item) == 16, "one 16-byte load");

template <bool PAIR>
struct Tile {
    static constexpr int M = PAIR ? 256 : 128, N = PAIR ? 256 : 64;  // tile rows and columns
    static constexpr int BROWS = PAIR ? 128 : 64;                    // B rows that one CTA loads
    static constexpr uint32_t B_PART = BROWS * BK * 2;
    static constexpr uint32_t STAGE = 3 * A_BYTES + 3 * B_PART;      // per CTA: A h, m, l and B h, m, l
    // accumulators per stage: a narrow MMA is over before the one before it on the same
    // accumulator has written back, so one CTA's K slices alternate between two
    static constexpr int NACC = PAIR ? 1 : 2;
    static constexpr int NCH = N / 32;             // 16-column chunks of one epilogue warp
    static constexpr int SLOT = 128 * N;           // floats of one CTA's tile sums
    static constexpr uint32_t COLS = 512;          // TMEM columns held
};

constexpr int MAX_ST = 3;
struct Sync {
    uint64_t full[MAX_ST], empty[MAX_ST];
    uint64_t done[2], free_[2];  // a stage's accumulator is complete / drained
    uint64_t fin;                // every MMA of this CTA (pair) is complete
    uint32_t tmem;
    int abort, issued, consumed, last;
};
constexpr size_t sync_bytes() { return (sizeof(Sync) + 15) & ~size_t(15); }

// Operand stages, and the rows that a warp stages at a time for its mirrored
// stores: what fits beside the sums (three under D2)
template <bool PAIR, bool SIM>
constexpr int stages_of() { return PAIR || SIM ? 2 : 3; }
template <bool PAIR, bool SIM>
constexpr int mirror_rows() { return PAIR && !SIM ? 16 : 8; }
// stages, barriers; c_j, |W_.j|^2, |C_.j|^2 of the columns, the column sums [quarter], row sums [half], h
template <bool PAIR>
constexpr size_t p1_smem()
{
    return 1024 + (size_t)stages_of<PAIR, false>() * Tile<PAIR>::STAGE + sync_bytes() +
           (7 * Tile<PAIR>::N + 2 * 128) * sizeof(float) + EPI * sizeof(double);
}
// stages, barriers; the column norms, column sums [quarter][sum], row sums [half][sum], staging blocks
template <bool PAIR, bool SIM>
constexpr size_t p2_smem()
{
    constexpr int N = Tile<PAIR>::N, NS = SIM ? 3 : 2;
    return 1024 + (size_t)stages_of<PAIR, SIM>() * Tile<PAIR>::STAGE + sync_bytes() +
           (N + 4 * NS * N + 2 * NS * 128 + EPI * mirror_rows<PAIR, SIM>() * 17) * sizeof(float);
}
static_assert(p1_smem<true>() <= 232448 && p2_smem<true, false>() <= 232448 && p2_smem<true, true>() <= 232448 &&
                  p1_smem<false>() <= 232448 && p2_smem<false, false>() <= 232448 && p2_smem<false, true>() <= 232448,
              "fits in the shared memory of a CTA");

__device__ __forceinline__ uint8_t *align1024(uint8_t *p)
{
    return reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// h, m, l of two values, packed as BF16 pairs (first value in the low half).
// Saturating, so that a value above the largest BF16 still splits into finite parts.
__device__ __forceinline__ uint32_t cvt2(float x0, float x1)
{
    uint32_t r;
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %2, %1;" : "=r"(r) : "f"(x0), "f"(x1));
    return r;
}
__device__ __forceinline__ void split3(float x0, float x1, uint32_t (&p)[3])
{
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        p[q] = cvt2(x0, x1);
        x0 -= __uint_as_float(p[q] << 16);
        x1 -= __uint_as_float(p[q] & 0xffff0000u);
    }
}

// Eq. 1 from the numerator and the squared norms: rsqrtf with one Newton step
// (about 1 ulp) over the whole range of floats.  The denominator is at least
// (|x|^2 + |y|^2) / 2, so only two zero vectors meet the lower clamp (numerator
// 0, result 0); the upper one keeps the Newton step finite where a norm has
// overflowed (y = 0, result 0).  (With the denominator clamped at the smallest
// normal float, entries of 2^-66 gave W off by 4e-2 of its largest one; rsqrtf's
// care of subnormal arguments costs 0.5% to 2%: 125 x 125 to h < 1e-3 784 -> 801
// us, 1000 x 17000, three iterations, 11.63 -> 11.70 ms.)
__device__ __forceinline__ float tanimoto_newton(float num, float nx, float ny)
{
    const float den = fmaxf((nx + ny) - fabsf(num), 1.401298464e-45f);
    const float y = rsqrtf(den), s = num * y;
    return fmaf(0.5f * s, fmaf(-fminf(den, 3.402823466e38f) * y, y, 1.0f), s);
}

// Eqs. 2 and 5: (1 - alpha) x + alpha y, y the mean of n similarities given as their sum.  Below
// alpha = 1/2 as x + alpha (y - x), which does not round 1 - alpha; from there on, where 1 - alpha is
// exact, as it stands: alpha = 1 gives y, where the first form would leave a rounding of x's size in
// it (2-norm of one update's error at alpha = 0.1, 0.5, 0.9, 1, first form and second: 2.6e-8, 3.9e-8,
// 4.6e-8, 4.0e-8 and 4.3e-8, 2.8e-8, 2.5e-8, 0).
struct Damp {
    float a, keep, minus;
    __device__ __forceinline__ Damp(float alpha, float n)
        : a(alpha / n), keep(alpha < 0.5f ? 1.0f : 1.0f - alpha), minus(alpha < 0.5f ? -n : 0.0f)
    {
    }
    __device__ __forceinline__ float operator()(float x, float sum) const
    {
        return fmaf(a, fmaf(minus, x, sum), keep * x);
    }
};

// ---- one CTA or a CTA pair ----------------------------------------------------------
template <bool PAIR>
__device__ __forceinline__ void load_box(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y)
{
    if (PAIR)  // counted on the even CTA's barrier
        tma_load_2d_pair(dst, map, mapa_shared(smem_u32(bar), 0), x, y);
    else
        tma_load_2d(dst, map, bar, x, y);
}
template <bool PAIR>
__device__ __forceinline__ void group_sync()  // the CTA, or both of the pair
{
    if (PAIR)
        cluster_sync();
    else
        __syncthreads();
}
__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 2, %0;" ::"n"(32 * EPI) : "memory"); }

// Barriers and TMEM, once per CTA.
template <bool PAIR, int ST>
__device__ __forceinline__ void setup(Sync &sy)
{
    if (threadIdx.x == 0) {
        for (int q = 0; q < ST; ++q) {
            mbar_init(&sy.full[q], 1);
            mbar_init(&sy.empty[q], 1);
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(&sy.done[q], 1);
            mbar_init(&sy.free_[q], (PAIR ? 2 : 1) * EPI);
        }
        mbar_init(&sy.fin, 1);
        sy.abort = sy.issued = sy.consumed = sy.last = 0;
        fence_mbar_init();
    }
    if ((threadIdx.x >> 5) == 1) {
        if (PAIR)
            tmem_alloc_pair(&sy.tmem, Tile<PAIR>::COLS);
        else
            tmem_alloc(&sy.tmem, Tile<PAIR>::COLS);
    }
    tc_fence_before();
    __syncthreads();
    group_sync<PAIR>();  // both CTAs' barriers exist before any cross-CTA signal
    tc_fence_after();
}
template <bool PAIR, int ST>
__device__ __forceinline__ void teardown(Sync &sy, Ctl *ctl, bool even)
{
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int g = sy.consumed; even && g < sy.consumed + ST && g < sy.issued; ++g)  // not consumed (abort only)
            wait_bounded(&sy.full[g % ST], (uint32_t)(g / ST) & 1u, &sy.abort, ctl, true);
        wait_bounded(&sy.fin, 0, &sy.abort, ctl, true);  // no MMA is left in flight
    }
    __syncthreads();
    group_sync<PAIR>();
    if ((threadIdx.x >> 5) == 1) {
        tc_fence_after();
        if (PAIR)
            tmem_dealloc_pair(sy.tmem, Tile<PAIR>::COLS);
        else
            tmem_dealloc(sy.tmem, Tile<PAIR>::COLS);
    }
}

// The TMA producer: for every stage of every item, issue(item, stage, k, buffer, barrier).
template <bool PAIR, int ST, class Load>
__device__ __forceinline__ void producer(Sync &sy, uint8_t *stages, const Item *items, int first, int last,
                                         uint32_t rank, Ctl *ctl, Load load)
{
    constexpr uint32_t STAGE = Tile<PAIR>::STAGE;
    int g = 0;
    for (int n = first; n < last; ++n) {
        const Item it = items[n];
        for (int s = it.s0; s < it.s1; ++s, ++g) {
            const int st = g % ST;
            if (!wait_bounded(&sy.empty[st], ((uint32_t)(g / ST) & 1u) ^ 1u, &sy.abort, ctl)) {
                sy.issued = g;
                return;
            }
            if (!PAIR || rank == 0)
                mbar_arrive_expect_tx(&sy.full[st], (PAIR ? 2 : 1) * STAGE);
            load(it, s, stages + (size_t)st * STAGE, &sy.full[st]);
        }
    }
    sy.issued = g;
}

// The MMA issuer (a whole warp): every stage into a fresh accumulator, buffer g & 1.  mn(item,
// stage) gives which operands are MN-major (bit 0: B, bit 1: A).
template <bool PAIR, int ST, class Mn>
__device__ __forceinline__ void issuer(Sync &sy, uint8_t *stages, const Item *items, int first, int last, Ctl *ctl,
                                       Mn mn)
{
    constexpr uint32_t idesc = idesc_bf16_f32(Tile<PAIR>::M, Tile<PAIR>::N), STAGE = Tile<PAIR>::STAGE;
    const uint32_t leader = elect_one();
    const uint32_t tmem = __shfl_sync(0xffffffffu, sy.tmem, 0);
    int g = 0, st = 0;
    uint32_t ph = 0;  // stage st and its phase
    bool ok = true;
    for (int n = first; n < last && ok; ++n) {
        const Item it = items[n];
        const int s0 = __shfl_sync(0xffffffffu, (int)it.s0, 0), s1 = __shfl_sync(0xffffffffu, (int)it.s1, 0);
        for (int s = s0; s < s1; ++s, ++g) {
            const int buf = g & 1;
            ok = wait_bounded(&sy.free_[buf], ((uint32_t)(g >> 1) & 1u) ^ 1u, &sy.abort, ctl) &&
                 wait_bounded(&sy.full[st], ph, &sy.abort, ctl);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok)
                break;
            tc_fence_after();
            const uint32_t base = smem_u32(stages + (size_t)st * STAGE);
            const uint32_t dacc = tmem + (uint32_t)buf * (Tile<PAIR>::NACC * Tile<PAIR>::N);
            const int m = __shfl_sync(0xffffffffu, mn(it, s), 0);
            const uint32_t id = idesc | ((m & 1) ? IDESC_B_MN : 0u) | ((m & 2) ? IDESC_A_MN : 0u);
            // descriptors of part 0 at K slice 0; a part adds its bytes, a slice 32 B (K-major) or 2 KB (MN-major)
            const uint64_t a0 = (m & 2) ? sdesc_mn_sw128(base, A_BYTES / 2) : sdesc_k_sw128(base);
            const uint64_t b0 = (m & 1) ? sdesc_mn_sw128(base + 3 * A_BYTES, A_BYTES / 2)
                                        : sdesc_k_sw128(base + 3 * A_BYTES);
            const uint32_t a_lo = (uint32_t)a0, a_hi = (uint32_t)(a0 >> 32), b_lo = (uint32_t)b0, b_hi = (uint32_t)(b0 >> 32);
            const uint32_t as = (m & 2) ? 2048 >> 4 : 32 >> 4, bs = (m & 1) ? 2048 >> 4 : 32 >> 4;
            constexpr uint32_t APART = A_BYTES >> 4, BPART = Tile<PAIR>::B_PART >> 4;
            // smallest products first: m.m, h.l, l.h, then h.m, m.h, then h.h
            constexpr int pa[6] = {1, 0, 2, 0, 1, 0}, pb[6] = {1, 2, 0, 1, 0, 0};
#pragma unroll
            for (int t = 0; t < 6; ++t)
#pragma unroll
                for (int kk = 0; kk < BK / 16; ++kk)
                    mma_bf16_warp<PAIR>(leader, dacc + (kk % Tile<PAIR>::NACC) * Tile<PAIR>::N,
                                        a_lo + pa[t] * APART + kk * as, a_hi, b_lo + pb[t] * BPART + kk * bs, b_hi, id,
                                        !(t == 0 && kk < Tile<PAIR>::NACC));
            mma_commit_warp<PAIR>(leader, &sy.empty[st]);
            mma_commit_warp<PAIR>(leader, &sy.done[buf]);
            if (++st == ST) {
                st = 0;
                ph ^= 1u;
            }
        }
    }
    sy.consumed = g;
    // an mbarrier that both CTAs of a pair are told of; only the even one waits on it
    mma_commit_warp<PAIR>(leader, &sy.fin);
}

// ---- the epilogue's side of the main loop ---------------------------------------------
// Tile sums in registers: acc[c][q] is register q of the fragment (see
// tmem_ld_frag16_nowait) of this warp's 16-column chunk c.
template <int NCH>
__device__ __forceinline__ void drain(uint32_t taddr, float (&acc)[NCH][16])
{
    uint32_t v[2][2][16];  // two chunks in flight while the two before are added
    tmem_ld_frag16_nowait(taddr, v[0][0]);
    tmem_ld_frag16_nowait(taddr + 16, v[0][1]);
#pragma unroll
    for (int c = 0; c < NCH; c += 2) {
        const int b = (c >> 1) & 1;
        tmem_wait16(v[b][0]);
        tmem_wait16(v[b][1]);
        if (c + 2 < NCH) {
            tmem_ld_frag16_nowait(taddr + (c + 2) * 16, v[b ^ 1][0]);
            tmem_ld_frag16_nowait(taddr + (c + 3) * 16, v[b ^ 1][1]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 16; ++q)
                acc[c + h][q] += __uint_as_float(v[b][h][q]);
    }
}
template <int NCH>
__device__ __forceinline__ void clear(float (&acc)[NCH][16])
{
#pragma unroll
    for (int c = 0; c < NCH; ++c)
#pragma unroll
        for (int q = 0; q < 16; ++q)
            acc[c][q] = 0.0f;
}
// to and from a slot: thread tt's register quads at [(4 c + q)][tt] (coalesced, 16 bytes each)
template <int NCH>
__device__ __forceinline__ void put_slot(float *slot, int tt, const float (&acc)[NCH][16])
{
#pragma unroll
    for (int c = 0; c < NCH; ++c)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            __stcg(reinterpret_cast<float4 *>(slot) + (4 * c + q) * (32 * EPI) + tt,
                   make_float4(acc[c][4 * q], acc[c][4 * q + 1], acc[c][4 * q + 2], acc[c][4 * q + 3]));
}
template <int NCH>
__device__ __forceinline__ void add_slot(const float *slot, int tt, float (&acc)[NCH][16])
{
#pragma unroll
    for (int c = 0; c < NCH; ++c)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 v = __ldcg(reinterpret_cast<const float4 *>(slot) + (4 * c + q) * (32 * EPI) + tt);
            acc[c][4 * q] += v.x;
            acc[c][4 * q + 1] += v.y;
            acc[c][4 * q + 2] += v.z;
            acc[c][4 * q + 3] += v.w;
        }
}
__device__ __forceinline__ void get_slot16(const float *slot, int c, int tt, uint32_t (&r)[16])
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(slot) + (4 * c + q) * (32 * EPI) + tt);
        r[4 * q] = v.x;
        r[4 * q + 1] = v.y;
        r[4 * q + 2] = v.z;
        r[4 * q + 3] = v.w;
    }
}
// registers back into TMEM, for the epilogue's loop over chunks
template <int NCH>
__device__ __forceinline__ void put_tmem(uint32_t taddr, const float (&acc)[NCH][16])
{
#pragma unroll
    for (int c = 0; c < NCH; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            asm volatile("tcgen05.st.sync.aligned.16x256b.x2.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(
                             taddr + c * 16 + ((uint32_t)(16 * h) << 16)),
                         "r"(__float_as_uint(acc[c][8 * h])), "r"(__float_as_uint(acc[c][8 * h + 1])),
                         "r"(__float_as_uint(acc[c][8 * h + 2])), "r"(__float_as_uint(acc[c][8 * h + 3])),
                         "r"(__float_as_uint(acc[c][8 * h + 4])), "r"(__float_as_uint(acc[c][8 * h + 5])),
                         "r"(__float_as_uint(acc[c][8 * h + 6])), "r"(__float_as_uint(acc[c][8 * h + 7]))
                         : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Whether this CTA is the last of a cut tile's parts to arrive (its own sums
// are in their slot): then every part's sums are visible to all its epilogue
// threads.  The counter goes back to zero for the next launch.
__device__ __forceinline__ bool arrive_last(Sync &sy, int *counter, int nparts, int tt)
{
    __threadfence();
    epi_bar();
    if (tt == 0) {
        const int k = atomicAdd(counter, 1);
        sy.last = k == nparts - 1;
        if (k == nparts - 1)
            *counter = 0;
        __threadfence();
    }
    epi_bar();
    return *(volatile int *)&sy.last != 0;
}

// One item's stages: sums the drained stages into acc and releases each TMEM
// buffer, the last one only if `keep` is false.  at_r(): called between the
// last R-num stage and the first A-num stage (s == nR).
template <bool PAIR, class AtR>
__device__ __forceinline__ bool sum_stages(Sync &sy, const Item &it, int nR, int &g, uint32_t tq, uint32_t free_even,
                                           bool keep, Ctl *ctl, float (&acc)[Tile<PAIR>::NCH][16], AtR at_r)
{
    const int lane = threadIdx.x & 31;
    bool live = true;
    for (int s = it.s0; s < it.s1; ++s, ++g) {
        const int buf = g & 1;
        if (s == nR && s > it.s0)
            at_r();
        live = live && wait_bounded(&sy.done[buf], (uint32_t)(g >> 1) & 1u, &sy.abort, ctl) &&
               !*(volatile int *)&sy.abort;
        live = __all_sync(0xffffffffu, live);
        if (!live)
            continue;
        tc_fence_after();
#pragma unroll
        for (int q = 0; q < Tile<PAIR>::NACC; ++q)
            drain<Tile<PAIR>::NCH>(tq + (uint32_t)(buf * Tile<PAIR>::NACC + q) * Tile<PAIR>::N, acc);
        if (!(keep && s + 1 == it.s1)) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (PAIR)
                    mbar_arrive_cluster(free_even + buf * (uint32_t)sizeof(uint64_t));
                else
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&sy.free_[buf])) : "memory");
            }
        }
    }
    return live;
}

// ---------------------------------------------------------------------------
// Phase 1
// ---------------------------------------------------------------------------
template <bool PAIR>
__global__ void __cluster_dims__(PAIR ? 2 : 1, 1, 1) __launch_bounds__(NTHREADS, 1)
    k_f32_phase1(const __grid_constant__ F32Maps maps, const __grid_constant__ Dev d, int cur,
                 const int *__restrict__ off, const Item *__restrict__ items)
{
    constexpr int N = Tile<PAIR>::N, NCH = Tile<PAIR>::NCH, SLOT = Tile<PAIR>::SLOT, ST = stages_of<PAIR, false>();
    constexpr uint32_t STAGE = Tile<PAIR>::STAGE, B_PART = Tile<PAIR>::B_PART;
    Ctl *ctl = d.ctl;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *stages = align1024(smem_raw);
    Sync &sy = *reinterpret_cast<Sync *>(stages + ST * STAGE);
    float *colvec = reinterpret_cast<float *>(stages + ST * STAGE + ((sizeof(Sync) + 15) & ~size_t(15)));
    float *colred = colvec + 3 * N;    // [quarter][column] sums of W'^2
    float *rowred = colred + 4 * N;    // [half][row]
    double *hred = reinterpret_cast<double *>(rowred + 2 * 128);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = PAIR ? cluster_ctarank() : 0;
    const int worker = PAIR ? blockIdx.x >> 1 : blockIdx.x;
    const int nR = ceil_div(d.Tp, BK);
    setup<PAIR, ST>(sy);
    const bool active = ctl->active;  // every CTA sees the same value
    const int first = off[worker], last = active ? off[worker + 1] : first;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        if (warp == 0 && lane == 0) {
            producer<PAIR, ST>(sy, stages, items, first, last, rank, ctl,
                           [&](const Item &it, int s, uint8_t *b, uint64_t *bar) {
                               const int m0 = (int)(it.a & 0xffffu) * Tile<PAIR>::M + 128 * (int)rank;
                               const int n0 = (int)(it.a >> 16) * N, nb0 = n0 + 128 * (int)rank;
                               if (s < nR) {  // P_off rows x W columns, K over TFs
                                   const int k = s * BK;
                                   for (int p = 0; p < 3; ++p) {
                                       load_box<PAIR>(b + p * A_BYTES, &maps.P[p], bar, k, m0);
                                       for (int h = 0; h < Tile<PAIR>::BROWS / 64; ++h)
                                           load_box<PAIR>(b + 3 * A_BYTES + p * B_PART + h * (A_BYTES / 2),
                                                          &maps.Wm[cur][p], bar, nb0 + 64 * h, k);
                                   }
                                   return;
                               }
                               const int k = (s - nR) * BK;
                               for (int p = 0; p < 3; ++p) {
                                   load_box<PAIR>(b + p * A_BYTES, &maps.W[cur][p], bar, k, m0);
                                   uint8_t *bb = b + 3 * A_BYTES + p * B_PART;
                                   if (k >= n0) {  // C_off[j][k] at or past the tile's diagonal block: stored rows
                                       load_box<PAIR>(bb, PAIR ? &maps.C[p] : &maps.Cm[p], bar, k, nb0);
                                   } else {        // C_off[k][j], rows k of the upper triangle
                                       for (int h = 0; h < Tile<PAIR>::BROWS / 64; ++h)
                                           load_box<PAIR>(bb + h * (A_BYTES / 2), &maps.Cm[p], bar, nb0 + 64 * h, k);
                                   }
                               }
                           });
        } else if (warp == 1 && rank == 0) {
            issuer<PAIR, ST>(sy, stages, items, first, last, ctl, [&](const Item &it, int s) {
                return (s < nR || (s - nR) * BK < (int)(it.a >> 16) * N) ? 1 : 0;
            });
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        const int e = warp - 4, wq = warp & 3, half = e >> 2, tt = threadIdx.x - 128;
        const int er = lane >> 2, ec = 8 * (lane & 1) + 2 * (lane & 2);
        const uint32_t free_even = PAIR ? mapa_shared(smem_u32(&sy.free_[0]), 0) : 0;
        const uint32_t tq = sy.tmem + ((uint32_t)(wq * 32) << 16) + half * (N / 2);  // this warp's lanes and columns
        const int nx = cur ^ 1;
        const float *W = d.W[cur];
        float *Wn = d.W[nx];
        __nv_bfloat16 *Ws[3] = {d.Wh[nx], d.Wm[nx], d.Wl[nx]};
        int g = 0;
        for (int n = first; n < last; ++n) {
            const Item it = items[n];
            const bool cut = it.nparts > 1;
            const int nt = (int)(it.a >> 16), m0 = (int)(it.a & 0xffffu) * Tile<PAIR>::M + 128 * (int)rank;
            const int n0 = nt * N;
            // slots: this CTA's own for an uncut tile's R-num; a cut tile's R-num and parts
            float *rslot = d.p1_acc + (size_t)blockIdx.x * SLOT;
            float *fix = d.p1_fix + (size_t)((PAIR ? 2 : 1) * it.slot) * SLOT + (size_t)rank * SLOT;
            constexpr size_t FS = (size_t)(PAIR ? 2 : 1) * SLOT;
            if (cut)
                rslot = fix;
            // what the epilogue needs besides the sums comes in while the stages run (a pair's registers
            // are taken by the sums: only the columns' vectors); read after them, its latency and a
            // barrier were 1.5 us of a 34 us iteration at 125 x 125, 1 of 68 at 250 x 2100
            for (int j = tt; j < N; j += 32 * EPI) {
                const int gj = n0 + j;
                const bool cj = gj < d.G;
                colvec[j] = cj ? d.cdf[gj] : 0.0f;
                colvec[N + j] = cj ? d.csqW[gj] : 0.0f;
                colvec[2 * N + j] = cj ? d.csqC[gj] : 0.0f;
            }
            const int k0 = m0 + wq * 32;
            const bool rows_in = m0 < d.Tp;
            float pdi[4], rsp[4], rsw[4], rowsq[4];
            auto fetch_rows = [&]() {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = k0 + er + 8 * i;
                    const bool ri = r < d.T;
                    pdi[i] = ri ? d.pdf[r] : 0.0f;
                    rsp[i] = ri ? d.rsqP[r] : 0.0f;
                    rsw[i] = ri ? d.rsqW[r] : 0.0f;
                    rowsq[i] = 0.0f;
                }
            };
            const size_t wo = (size_t)(k0 + er) * d.Gp + n0 + half * (N / 2) + ec;
            uint4 wq0[4];
            auto fetch_w = [&](int c) {
                if (c < NCH && rows_in && n0 + half * (N / 2) + c * 16 < d.Gp) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        wq0[i] = *reinterpret_cast<const uint4 *>(W + wo + (size_t)(8 * i) * d.Gp + c * 16);
                }
            };
            if (!PAIR) {
                fetch_rows();
                fetch_w(0);
            }
            float acc[NCH][16];
            clear<NCH>(acc);
            bool live = sum_stages<PAIR>(sy, it, nR, g, tq, free_even, PAIR && !cut, ctl, acc, [&]() {
                put_slot<NCH>(rslot, tt, acc);
                clear<NCH>(acc);
            });
            const int lastbuf = (g - 1) & 1;
            bool mine = true;
            if (cut) {
                if (it.s1 <= nR) {  // all of R-num and nothing else
                    put_slot<NCH>(rslot, tt, acc);
                    clear<NCH>(acc);
                }
                put_slot<NCH>(fix + (1 + it.part) * FS, tt, acc);
                mine = arrive_last(sy, d.p1_flag + (PAIR ? 2 : 1) * it.fix + rank, it.nparts, tt);
                if (mine && live) {
                    clear<NCH>(acc);
                    for (int p = 0; p < it.nparts; ++p)
                        add_slot<NCH>(fix + (1 + p) * FS, tt, acc);
                }
            }
            if (!mine)
                continue;
            // the sums in TMEM: the last stage's buffer of an uncut tile on a pair (kept until the
            // epilogue is done), else columns that no stage uses (one CTA), else wait-free reuse of the
            // slot of part 0 (a pair's cut tile)
            const uint32_t tsum = PAIR ? tq + (uint32_t)lastbuf * N : tq + 4 * N;
            const bool in_tmem = !(PAIR && cut);
            float *aslot = fix + FS;
            if (live) {
                if (in_tmem)
                    put_tmem<NCH>(tsum, acc);
                else
                    put_slot<NCH>(aslot, tt, acc);
            }
            if (PAIR) {
                fetch_rows();
                fetch_w(0);
            }
            const Damp damp(ctl->alpha, 2.0f);
            // a row's squares and |W' - W| are added four columns at a time, these over the chunks: no chain
            // of additions is longer than 8 (32 and 128 in one left 15% to 20% more error than FFMA's
            // slots of 128 columns)
            float hsum = 0.0f;
            epi_bar();  // colvec is complete; colred and rowred of the item before are no longer read
            // W, R-num and the sums one chunk ahead
            uint32_t rq0[16], ar[16];
            auto fetch_r = [&](int c) {
                if (c < NCH && live && rows_in && n0 + half * (N / 2) + c * 16 < d.Gp)
                    get_slot16(rslot, c, tt, rq0);
            };
            auto fetch_sums = [&](int c) {
                if (in_tmem)
                    tmem_ld_frag16_nowait(tsum + c * 16, ar);
                else
                    get_slot16(aslot, c, tt, ar);
            };
            fetch_r(0);
            if (live)
                fetch_sums(0);
#pragma unroll 1
            for (int c = 0; c < NCH && live; ++c) {
                const int cc = half * (N / 2) + c * 16, j0 = n0 + cc;
                float cs[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                float x[4][4], y[4][4], w[4][4];
                if (in_tmem)
                    tmem_wait16(ar);
                frag_to_rows(ar, y);
                if (c + 1 < NCH)
                    fetch_sums(c + 1);
                frag_to_rows(rq0, x);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    w[i][0] = __uint_as_float(wq0[i].x);
                    w[i][1] = __uint_as_float(wq0[i].y);
                    w[i][2] = __uint_as_float(wq0[i].z);
                    w[i][3] = __uint_as_float(wq0[i].w);
                }
                fetch_w(c + 1);
                fetch_r(c + 1);
                if (rows_in && j0 < d.Gp) {
                    const float4 c4 = *reinterpret_cast<const float4 *>(colvec + cc + ec);
                    const float4 w4 = *reinterpret_cast<const float4 *>(colvec + N + cc + ec);
                    const float4 q4 = *reinterpret_cast<const float4 *>(colvec + 2 * N + cc + ec);
                    const float cd[4] = {c4.x, c4.y, c4.z, c4.w}, nw[4] = {w4.x, w4.y, w4.z, w4.w},
                                nc[4] = {q4.x, q4.y, q4.z, q4.w};
                    float hc = 0.0f;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const bool ri = k0 + er + 8 * i < d.T;
                        float wn[4], r4 = 0.0f, h4 = 0.0f;
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float rnum = x[i][u] + pdi[i] * w[i][u];   // P_i. . W_.j
                            const float anum = y[i][u] + w[i][u] * cd[u];    // W_i. . C_.j
                            const float R = tanimoto_newton(rnum, rsp[i], nw[u]);
                            const float A = tanimoto_newton(anum, rsw[i], nc[u]);
                            const float v = damp(w[i][u], A + R);
                            wn[u] = ri && j0 + ec + u < d.G ? v : 0.0f;
                            h4 += fabsf(wn[u] - w[i][u]);  // (padding holds zeros)
                            r4 = fmaf(wn[u], wn[u], r4);
                            cs[u] = fmaf(wn[u], wn[u], cs[u]);
                        }
                        hc += h4;
                        rowsq[i] += r4;
                        const size_t o = wo + (size_t)(8 * i) * d.Gp + c * 16;
                        *reinterpret_cast<float4 *>(Wn + o) = make_float4(wn[0], wn[1], wn[2], wn[3]);
                        uint32_t p0[3], p1[3];
                        split3(wn[0], wn[1], p0);
                        split3(wn[2], wn[3], p1);
#pragma unroll
                        for (int p = 0; p < 3; ++p)
                            *reinterpret_cast<uint2 *>(Ws[p] + o) = make_uint2(p0[p], p1[p]);
                    }
                    hsum += hc;
                }
                const float t = lanes8_reduce_scatter4(cs);
                if (!(lane & 4))
                    colred[wq * N + cc + ec + (lane >> 3 & 1) + 2 * (lane >> 4)] = t;
            }
            if (in_tmem && PAIR && live) {  // the buffer that held the sums
                tc_fence_before();
                __syncwarp();
                if (lane == 0)
                    mbar_arrive_cluster(free_even + lastbuf * (uint32_t)sizeof(uint64_t));
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                rowsq[i] += __shfl_xor_sync(0xffffffffu, rowsq[i], 1);
                rowsq[i] += __shfl_xor_sync(0xffffffffu, rowsq[i], 2);
                if ((lane & 3) == 0)
                    rowred[half * 128 + wq * 32 + er + 8 * i] = rowsq[i];
            }
            double hv = (double)hsum;
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1)
                hv += __shfl_xor_sync(0xffffffffu, hv, o);
            if (lane == 0)
                hred[e] = hv;
            epi_bar();
            if (live && rows_in) {
                const int slot = m0 / 128;  // this CTA's 128-row block
                for (int j = tt; j < N; j += 32 * EPI)
                    if (n0 + j < d.Gp)
                        d.wcol_part[(size_t)slot * d.Gp + n0 + j] =
                            ((colred[j] + colred[N + j]) + colred[2 * N + j]) + colred[3 * N + j];
                if (tt < 128)
                    d.wrow_part[(size_t)nt * d.Tp + m0 + tt] = rowred[tt] + rowred[128 + tt];
                if (tt == 0) {
                    double hs = 0.0;
                    for (int q = 0; q < EPI; ++q)
                        hs += hred[q];
                    d.hpart[(size_t)nt * d.nbT + slot] = hs;
                }
            }
        }
    }
    teardown<PAIR, ST>(sy, ctl, !PAIR || rank == 0);
}

// ---------------------------------------------------------------------------
// Phase 2
// ---------------------------------------------------------------------------
template <bool PAIR, bool SIM>
__global__ void __cluster_dims__(PAIR ? 2 : 1, 1, 1) __launch_bounds__(NTHREADS, 1)
    k_f32_phase2(const __grid_constant__ F32Maps maps, const __grid_constant__ Dev d, int cur,
                 const int *__restrict__ off, const Item *__restrict__ items)
{
    constexpr int N = Tile<PAIR>::N, NCH = Tile<PAIR>::NCH, SLOT = Tile<PAIR>::SLOT, NS = SIM ? 3 : 2;
    constexpr int ST = stages_of<PAIR, SIM>(), MR = mirror_rows<PAIR, SIM>();
    constexpr uint32_t STAGE = Tile<PAIR>::STAGE, B_PART = Tile<PAIR>::B_PART;
    Ctl *ctl = d.ctl;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *stages = align1024(smem_raw);
    Sync &sy = *reinterpret_cast<Sync *>(stages + ST * STAGE);
    float *colnrm = reinterpret_cast<float *>(stages + ST * STAGE + ((sizeof(Sync) + 15) & ~size_t(15)));
    float *colred = colnrm + N;             // [quarter][sum][column]
    float *rowred = colred + 4 * NS * N;    // [half][sum][row]
    float *blocks = rowred + 2 * NS * 128;  // per epilogue warp: MR x 16 staging block, rows of 17
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = PAIR ? cluster_ctarank() : 0;
    const int worker = PAIR ? blockIdx.x >> 1 : blockIdx.x;
    setup<PAIR, ST>(sy);
    const bool active = ctl->active;
    const int first = off[worker], last = active ? off[worker + 1] : first;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        if (warp == 0 && lane == 0) {
            producer<PAIR, ST>(sy, stages, items, first, last, rank, ctl,
                           [&](const Item &it, int s, uint8_t *b, uint64_t *bar) {
                               const int m0 = (int)(it.a & 0x7fffu) * Tile<PAIR>::M + 128 * (int)rank;
                               const int n0 = (int)(it.a >> 15 & 0x7fffu) * N + 128 * (int)rank, k = s * BK;
                               for (int p = 0; p < 3; ++p) {
                                   uint8_t *bb = b + 3 * A_BYTES + p * B_PART;
                                   if (it.a >> 31) {  // P: rows of W', K over genes
                                       load_box<PAIR>(b + p * A_BYTES, &maps.W[cur][p], bar, k, m0);
                                       load_box<PAIR>(bb, PAIR ? &maps.W[cur][p] : &maps.Wm[cur][p], bar, k, n0);
                                       continue;
                                   }
                                   // C: columns of W', K over TFs, MN-major
                                   for (int h = 0; h < 2; ++h)
                                       load_box<PAIR>(b + p * A_BYTES + h * (A_BYTES / 2), &maps.Wm[cur][p], bar,
                                                      m0 + 64 * h, k);
                                   for (int h = 0; h < Tile<PAIR>::BROWS / 64; ++h)
                                       load_box<PAIR>(bb + h * (A_BYTES / 2), &maps.Wm[cur][p], bar, n0 + 64 * h, k);
                               }
                           });
        } else if (warp == 1 && rank == 0) {
            issuer<PAIR, ST>(sy, stages, items, first, last, ctl,
                         [](const Item &it, int) { return it.a >> 31 ? 0 : 3; });
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        const int e = warp - 4, wq = warp & 3, half = e >> 2, tt = threadIdx.x - 128;
        const int er = lane >> 2, ec = 8 * (lane & 1) + 2 * (lane & 2);
        const uint32_t free_even = PAIR ? mapa_shared(smem_u32(&sy.free_[0]), 0) : 0;
        const uint32_t tq = sy.tmem + ((uint32_t)(wq * 32) << 16) + half * (N / 2);
        float *blk = blocks + (size_t)e * (MR * 17);
        int g = 0;
        for (int n = first; n < last; ++n) {
            const Item it = items[n];
            const bool cut = it.nparts > 1, isP = it.a >> 31;
            const int bm = (int)(it.a & 0x7fffu), bn = (int)(it.a >> 15 & 0x7fffu);
            constexpr size_t FS = (size_t)(PAIR ? 2 : 1) * SLOT;
            float *fix = d.p1_fix + (size_t)((PAIR ? 2 : 1) * it.slot) * SLOT + (size_t)rank * SLOT;
            const int nn = isP ? d.T : d.G, ld = isP ? d.Tp : d.Gp;
            const int m0 = bm * Tile<PAIR>::M + 128 * (int)rank, n0 = bn * N;
            const float *nrm = isP ? d.rsqW : d.csqW;
            float *X = isP ? d.Poff : d.Coff;
            const bool rows_in = m0 < ld;
            const int k0 = m0 + wq * 32;
            // what the epilogue needs besides the sums comes in while the stages run (as in phase 1)
            for (int j = tt; j < N; j += 32 * EPI)
                colnrm[j] = n0 + j < nn ? nrm[n0 + j] : 0.0f;
            float nrow[4], r1[4], r2[4], rv[4];
            auto fetch_rows = [&]() {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    nrow[i] = k0 + er + 8 * i < nn ? nrm[k0 + er + 8 * i] : 0.0f;
                    r1[i] = r2[i] = rv[i] = 0.0f;
                }
            };
            const size_t xo = (size_t)(k0 + er) * ld + n0 + half * (N / 2) + ec;
            // old values (and the sums below) one chunk ahead (three ahead measured the same)
            uint4 o0[4];
            auto fetch = [&](int c) {
                if (c < NCH && rows_in && n0 + half * (N / 2) + c * 16 < ld) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        o0[i] = *reinterpret_cast<const uint4 *>(X + xo + (size_t)(8 * i) * ld + c * 16);
                }
            };
            if (!PAIR) {
                fetch_rows();
                fetch(0);
            }
            float acc[NCH][16];
            clear<NCH>(acc);
            const bool live = sum_stages<PAIR>(sy, it, -1, g, tq, free_even, PAIR && !cut, ctl, acc, []() {});
            const int lastbuf = (g - 1) & 1;
            bool mine = true;
            if (cut) {
                put_slot<NCH>(fix + it.part * FS, tt, acc);
                mine = arrive_last(sy, d.p1_flag + (PAIR ? 2 : 1) * it.fix + rank, it.nparts, tt);
                if (mine && live) {
                    clear<NCH>(acc);
                    for (int p = 0; p < it.nparts; ++p)
                        add_slot<NCH>(fix + p * FS, tt, acc);
                }
            }
            if (!mine)
                continue;
            const uint32_t tsum = PAIR ? tq + (uint32_t)lastbuf * N : tq + 4 * N;
            const bool in_tmem = !(PAIR && cut);
            if (live) {
                if (in_tmem)
                    put_tmem<NCH>(tsum, acc);
                else
                    put_slot<NCH>(fix, tt, acc);
            }
            __nv_bfloat16 *Xs[3] = {isP ? d.Ph : d.Ch, isP ? d.Pm : d.Cm, isP ? d.Pl : d.Cl};
            // split copies of the lower triangle: all of P, of C only inside diagonal tiles
            const bool mirror = isP || (PAIR ? bm == bn : bm == bn >> 1);
            const Damp damp(ctl->alpha, 1.0f);
            if (PAIR) {
                fetch_rows();
                fetch(0);
            }
            epi_bar();  // colnrm is complete; colred and rowred of the item before are no longer read
            uint32_t ar[16];
            auto fetch_sums = [&](int c) {
                if (in_tmem)
                    tmem_ld_frag16_nowait(tsum + c * 16, ar);
                else
                    get_slot16(fix, c, tt, ar);
            };
            if (live)
                fetch_sums(0);
#pragma unroll 1
            for (int c = 0; c < NCH && live; ++c) {
                const int cc = half * (N / 2) + c * 16, j0 = n0 + cc;
                float cs[8], cv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    cs[u] = cs[4 + u] = cv[u] = 0.0f;
                float x[4][4], v[4][4];
                if (in_tmem)
                    tmem_wait16(ar);
                frag_to_rows(ar, x);
                if (c + 1 < NCH)
                    fetch_sums(c + 1);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    v[i][0] = __uint_as_float(o0[i].x);
                    v[i][1] = __uint_as_float(o0[i].y);
                    v[i][2] = __uint_as_float(o0[i].z);
                    v[i][3] = __uint_as_float(o0[i].w);
                }
                fetch(c + 1);
                // a block with no entry above the diagonal or inside the network has nothing to do
                if (rows_in && j0 < ld && k0 < j0 + 15) {
                    const float4 n4 = *reinterpret_cast<const float4 *>(colnrm + cc + ec);
                    const float nj[4] = {n4.x, n4.y, n4.z, n4.w};
                    const bool inner = k0 + 31 < j0 && j0 + 15 < nn;
                    float l1 = 0.0f, l2 = 0.0f, lv = 0.0f;
                    auto update = [&](int i, int u, bool valid) {
                        const float s = tanimoto_newton(x[i][u], nrow[i], nj[u]);
                        const float w = valid ? damp(v[i][u], s) : 0.0f;
                        const float y = SIM ? (valid ? s : 0.0f) : w;
                        // a row's four columns first, then the chunks (as in phase 1)
                        l1 = u ? l1 + y : y;
                        l2 = u ? fmaf(y, y, l2) : y * y;
                        cs[u] += y;
                        cs[4 + u] = fmaf(y, y, cs[4 + u]);
                        if (SIM) {
                            lv = u ? fmaf(w, w, lv) : w * w;
                            cv[u] = fmaf(w, w, cv[u]);
                        }
                        if (u == 3) {
                            r1[i] += l1;
                            r2[i] += l2;
                            if (SIM)
                                rv[i] += lv;
                        }
                        v[i][u] = w;
                    };
                    if (inner) {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                update(i, u, true);
                        const size_t ro = xo + c * 16, r8 = (size_t)8 * ld;
                        uint32_t p0[4][3], p1[4][3];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            split3(v[i][0], v[i][1], p0[i]);
                            split3(v[i][2], v[i][3], p1[i]);
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            *reinterpret_cast<float4 *>(X + ro + i * r8) =
                                make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
#pragma unroll
                        for (int p = 0; p < 3; ++p)
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                *reinterpret_cast<uint2 *>(Xs[p] + ro + i * r8) = make_uint2(p0[i][p], p1[i][p]);
                    } else {
                        uint32_t vm = 0;  // bit 4 i + u: entry (row i, column u) counts
#pragma unroll
                        for (int i = 0; i < 4; ++i)
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const bool valid = k0 + er + 8 * i < j0 + ec + u && j0 + ec + u < nn;
                                vm |= valid ? 1u << (4 * i + u) : 0u;
                                update(i, u, valid);
                            }
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const size_t ro = xo + (size_t)(8 * i) * ld + c * 16;
                            const uint32_t m = vm >> (4 * i) & 15u;
                            uint32_t p0[3], p1[3];
                            split3(v[i][0], v[i][1], p0);
                            split3(v[i][2], v[i][3], p1);
                            if (m == 15u) {
                                *reinterpret_cast<float4 *>(X + ro) = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
#pragma unroll
                                for (int p = 0; p < 3; ++p)
                                    *reinterpret_cast<uint2 *>(Xs[p] + ro) = make_uint2(p0[p], p1[p]);
                            } else if (m) {
#pragma unroll
                                for (int u = 0; u < 4; ++u)
                                    if (m >> u & 1u) {
                                        X[ro + u] = v[i][u];
#pragma unroll
                                        for (int p = 0; p < 3; ++p)
                                            reinterpret_cast<uint16_t *>(Xs[p])[ro + u] =
                                                (uint16_t)((u < 2 ? p0[p] : p1[p]) >> (16 * (u & 1)));
                                    }
                            }
                        }
                    }
                    // mirrored entries (j, k) through this warp's staging block, MR rows at a time: lane l
                    // takes column (l & 15), rows (MR / 2) (l >> 4) + 0 .. MR / 2 - 1
                    if (mirror) {
                        constexpr int H = MR / 2;
                        const int col = lane & 15, jm = j0 + col;
#pragma unroll 1
                        for (int r0 = 0; r0 < 32; r0 += MR) {
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                if (8 * i >= r0 && 8 * i < r0 + MR)
#pragma unroll
                                    for (int u = 0; u < 4; ++u)
                                        blk[(er + 8 * i - r0) * 17 + ec + u] = v[i][u];
                            __syncwarp();
                            const int km = k0 + r0 + H * (lane >> 4);
                            constexpr uint32_t all = (1u << H) - 1u;
                            const uint32_t mm =
                                jm >= nn ? 0u : (km + H - 1 < jm ? all : (km >= jm ? 0u : ((1u << (jm - km)) - 1u)));
                            if (mm) {
                                uint32_t q3[3][H / 2];
#pragma unroll
                                for (int q = 0; q < H / 2; ++q) {
                                    const float *b = blk + (H * (lane >> 4) + 2 * q) * 17 + col;
                                    uint32_t p[3];
                                    split3(b[0], b[17], p);
                                    q3[0][q] = p[0];
                                    q3[1][q] = p[1];
                                    q3[2][q] = p[2];
                                }
                                const size_t mo = (size_t)jm * ld + km;
#pragma unroll
                                for (int p = 0; p < 3; ++p) {
                                    if (mm == all) {
                                        if (H == 8)
                                            *reinterpret_cast<uint4 *>(Xs[p] + mo) =
                                                make_uint4(q3[p][0], q3[p][1], q3[p][H / 2 - 2], q3[p][H / 2 - 1]);
                                        else
                                            *reinterpret_cast<uint2 *>(Xs[p] + mo) = make_uint2(q3[p][0], q3[p][1]);
                                    } else {
#pragma unroll
                                        for (int q = 0; q < H; ++q)
                                            if (mm >> q & 1u)
                                                reinterpret_cast<uint16_t *>(Xs[p])[mo + q] =
                                                    (uint16_t)(q3[p][q >> 1] >> (16 * (q & 1)));
                                    }
                                }
                            }
                            __syncwarp();  // the block is rewritten
                        }
                    }
                }
                const float t = lanes8_reduce_scatter8(cs);
                colred[(wq * NS + (lane >> 4)) * N + cc + ec + (lane >> 2 & 1) + 2 * (lane >> 3 & 1)] = t;
                if (SIM) {
                    const float tv = lanes8_reduce_scatter4(cv);
                    if (!(lane & 4))
                        colred[(wq * NS + 2) * N + cc + ec + (lane >> 3 & 1) + 2 * (lane >> 4)] = tv;
                }
            }
            if (in_tmem && PAIR && live) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0)
                    mbar_arrive_cluster(free_even + lastbuf * (uint32_t)sizeof(uint64_t));
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float q1 = r1[i], q2 = r2[i], qv = rv[i];
#pragma unroll
                for (int o = 1; o <= 2; o <<= 1) {
                    q1 += __shfl_xor_sync(0xffffffffu, q1, o);
                    q2 += __shfl_xor_sync(0xffffffffu, q2, o);
                    if (SIM)
                        qv += __shfl_xor_sync(0xffffffffu, qv, o);
                }
                if ((lane & 3) == 0) {
                    const int row = wq * 32 + er + 8 * i;
                    rowred[(half * NS + 0) * 128 + row] = q1;
                    rowred[(half * NS + 1) * 128 + row] = q2;
                    if (SIM)
                        rowred[(half * NS + 2) * 128 + row] = qv;
                }
            }
            epi_bar();
            if (live && rows_in) {
                const int nb = ceil_div(ld, N);
#pragma unroll
                for (int w = 0; w < 3; ++w) {
                    float *S = w == 0 ? (isP ? d.ps_sum : d.cs_sum) : w == 1 ? (isP ? d.ps_sq : d.cs_sq)
                                                                            : (isP ? d.ps_vsq : d.cs_vsq);
                    const int wc = (!SIM && w == 2) ? 1 : w;  // sum of v^2 = sum of x^2 unless D2
                    auto colsum = [&](int j) {
                        return ((colred[(0 * NS + wc) * N + j] + colred[(1 * NS + wc) * N + j]) +
                                colred[(2 * NS + wc) * N + j]) + colred[(3 * NS + wc) * N + j];
                    };
                    auto rowsum = [&](int r) { return rowred[wc * 128 + r] + rowred[(NS + wc) * 128 + r]; };
                    if (PAIR) {  // row role in slot bn, column role of this CTA's rows in slot nb + 2 bm + rank
                        for (int j = tt; j < N; j += 32 * EPI)
                            if (n0 + j < ld)
                                S[(size_t)(nb + 2 * bm + (int)rank) * ld + n0 + j] = colsum(j);
                        if (tt < 128)
                            S[(size_t)bn * ld + m0 + tt] = rowsum(tt);
                    } else {  // row role in slot bn, column role in slot nb + bm
                        if (tt < N)
                            S[(size_t)(nb + bm) * ld + n0 + tt] = colsum(tt);
                        if (tt < 128)
                            S[(size_t)bn * ld + m0 + tt] = rowsum(tt);
                    }
                }
            }
        }
    }
    teardown<PAIR, ST>(sy, ctl, !PAIR || rank == 0);
}

// h, m, l of a whole array (padding stays zero): four values per thread
__global__ void k_split3(const float *__restrict__ X, size_t n4, __nv_bfloat16 *__restrict__ H,
                         __nv_bfloat16 *__restrict__ M, __nv_bfloat16 *__restrict__ L)
{
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < n4; q += (size_t)gridDim.x * blockDim.x) {
        const float4 v = reinterpret_cast<const float4 *>(X)[q];
        uint32_t p0[3], p1[3];
        split3(v.x, v.y, p0);
        split3(v.z, v.w, p1);
        reinterpret_cast<uint2 *>(H)[q] = make_uint2(p0[0], p1[0]);
        reinterpret_cast<uint2 *>(M)[q] = make_uint2(p0[1], p1[1]);
        reinterpret_cast<uint2 *>(L)[q] = make_uint2(p0[2], p1[2]);
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct Phase {
    std::vector<int> off;      // per worker, its range of items (once finished)
    std::vector<Item> items;
    std::vector<int> who, order;  // while it is made: each item's worker; the order they are given out in
    int fixes = 0, slots = 0;  // cut tiles; slots per CTA rank that they meet in
    double cost = 0;           // of the busiest worker, in stages
};

// The items from `from` on, whose costs are given: longest first (equals in the order they stand
// in) to the least loaded worker (the first of equals); the largest load.  There are few different
// costs, so the order takes one pass.
double assign(Phase &ph, int from, const std::vector<double> &cost, int workers)
{
    std::vector<double> kinds;
    std::vector<uint16_t> kind(cost.size());
    size_t k = 0;
    for (size_t q = 0; q < cost.size(); ++q) {
        if (k >= kinds.size() || kinds[k] != cost[q])
            k = std::find(kinds.begin(), kinds.end(), cost[q]) - kinds.begin();
        if (k == kinds.size())
            kinds.push_back(cost[q]);
        kind[q] = (uint16_t)k;
    }
    std::vector<int> rank(kinds.size());
    for (size_t q = 0; q < rank.size(); ++q)
        rank[q] = (int)q;
    std::sort(rank.begin(), rank.end(), [&kinds](int x, int y) { return kinds[x] > kinds[y]; });
    std::vector<int> at(kinds.size());  // where each kind's items go in the order
    for (uint16_t q : kind)
        ++at[q];
    int n = from;
    for (int r : rank) {
        const int c = at[r];
        at[r] = n;
        n += c;
    }
    ph.order.resize(ph.items.size());
    for (int q = 0; q < from; ++q)
        ph.order[q] = q;
    for (size_t q = 0; q < kind.size(); ++q)
        ph.order[at[kind[q]]++] = from + (int)q;
    // a heap of (load, worker), the least at the root
    std::vector<std::pair<double, int>> heap(workers);
    for (int w = 0; w < workers; ++w)
        heap[w] = {0.0, w};
    double most = 0.0;
    ph.who.resize(ph.items.size());
    for (size_t q = from; q < ph.items.size(); ++q) {
        std::pair<double, int> x = heap[0];
        ph.who[ph.order[q]] = x.second;
        x.first += cost[ph.order[q] - from];
        most = std::max(most, x.first);
        int h = 0;
        for (int c = 1; c < workers; c = 2 * h + 1) {
            c += c + 1 < workers && heap[c + 1] < heap[c];
            if (!(heap[c] < x))
                break;
            heap[h] = heap[c];
            h = c;
        }
        heap[h] = x;
    }
    return most;
}
// The lists, worker by worker, each in the order in which its items were given out
void finish(Phase &ph, int workers)
{
    ph.off.assign(workers + 1, 0);
    for (int w : ph.who)
        ++ph.off[w + 1];
    for (int w = 0; w < workers; ++w)
        ph.off[w + 1] += ph.off[w];
    std::vector<int> next(ph.off.begin(), ph.off.end() - 1);
    std::vector<Item> lists(ph.items.size());
    for (size_t q = 0; q < lists.size(); ++q) {
        const int n = ph.order.empty() ? (int)q : ph.order[q];
        lists[next[ph.who[n]]++] = ph.items[n];
    }
    ph.items = std::move(lists);
    ph.who = ph.order = std::vector<int>();
}

// Costs in stages of K = 64 (measured: 1.9 us on a pair, 0.8 us on one CTA): a
// finished tile's epilogue, and what a cut costs each part (its sums to L2, the
// counter, a pipeline that starts empty) and the part that finishes.
constexpr double EPILOGUE[2] = {6.0, 10.0}, CUT[2] = {4.0, 3.0}, CUT_LAST[2] = {4.0, 3.0};  // [one CTA], [pair]
constexpr double STAGE_US[2] = {0.8, 1.9};
constexpr int MIN_PART = 4;
constexpr int tile_m(bool pair) { return pair ? Tile<true>::M : Tile<false>::M; }
constexpr int tile_n(bool pair) { return pair ? Tile<true>::N : Tile<false>::N; }

// Phase 1 with the tiles from `whole` on cut in one of two ways, the ones
// before whole, in rounds: np > 0, every tile in np equal parts (the first
// holds all of R-num), longest first to the least loaded worker; np = 0, the
// tiles' work as one line dealt out in equal shares, tiles cut where a share
// ends (never inside R-num, and no part under MIN_PART stages).
Phase plan_phase1_cut(const Dev &d, int workers, bool pair, int whole, int np)
{
    const int nmt = ceil_div(d.Tp, tile_m(pair)), ntile = nmt * ceil_div(d.Gp, tile_n(pair));
    const int nR = ceil_div(d.Tp, BK), K = nR + ceil_div(d.Gp, BK), rest = ntile - whole;
    const double E = EPILOGUE[pair];
    Phase ph;
    std::vector<double> load(workers, 0.0), parts;  // of the workers; costs of the parts to give out
    ph.items.reserve(whole + 2 * (size_t)std::max(rest, np * rest));
    ph.who.reserve(ph.items.capacity());
    auto give = [&ph](const Item &it, int w) {
        ph.items.push_back(it);
        ph.who.push_back(w);
    };
    for (int t = 0; t < whole; ++t) {
        Item it{};
        it.a = (uint32_t)(t % nmt) | (uint32_t)(t / nmt) << 16;
        it.s1 = (uint16_t)K;
        it.nparts = 1;
        give(it, t % workers);
        load[t % workers] += K + E;
    }
    const double share = rest > 0 ? rest * (K + E) / workers : 1.0;
    std::vector<int> order, cut;
    if (np == 0) {  // equal shares go TF-block-major, so that the workers on one gene block's TF blocks
        for (int m = 0; m < nmt; ++m)  // run side by side
            for (int t = whole + ((m - whole) % nmt + nmt) % nmt; t < ntile; t += nmt)
                order.push_back(t);
    }
    for (int q = 0; q < rest; ++q) {
        const int t = np == 0 ? order[q] : whole + q;
        cut.assign(1, 0);  // part p: stages [cut[p], cut[p + 1])
        const double x0 = q * (K + E);
        if (np > 0) {
            const int e0 = std::max(K / np, nR);
            for (int p = 0; p < np; ++p)
                cut.push_back(e0 + (np > 1 ? (K - e0) * p / (np - 1) : K - e0));
        } else {
            for (int w = (int)(x0 / share) + 1; w * share < x0 + K + E; ++w) {
                int c = (int)(w * share - x0 + 0.5);
                if (c < nR)
                    c = c < nR / 2 ? 0 : nR;
                if (c - cut.back() >= MIN_PART && K - c >= MIN_PART)
                    cut.push_back(c);
            }
            cut.push_back(K);
        }
        const int n = (int)cut.size() - 1;
        for (int p = 0; p < n; ++p) {
            Item it{};
            it.a = (uint32_t)(t % nmt) | (uint32_t)(t / nmt) << 16;
            it.s0 = (uint16_t)cut[p]; it.s1 = (uint16_t)cut[p + 1];
            it.part = (uint16_t)p; it.nparts = (uint16_t)n;
            if (n > 1) {
                it.fix = (uint16_t)ph.fixes;
                it.slot = (uint16_t)ph.slots;
            }
            const double c = it.s1 - it.s0 + (n > 1 ? CUT[pair] : 0.0) +
                             (p == n - 1 ? E + (n > 1 ? CUT_LAST[pair] : 0.0) : 0.0);
            if (np > 0) {
                ph.items.push_back(it);
                parts.push_back(c);
            } else {
                const int w = std::min(workers - 1, (int)((x0 + 0.5 * (cut[p] + cut[p + 1])) / share));
                give(it, w);
                load[w] += c;
            }
        }
        if (n > 1) {
            ph.fixes += 1;
            ph.slots += 1 + n;  // R-num and every part's A-num
        }
    }
    if (np > 0)
        ph.cost = ceil_div(whole, workers) * (K + E) + assign(ph, whole, parts, workers);
    else
        ph.cost = *std::max_element(load.begin(), load.end());
    return ph;
}

// Phase 1's lists, tiles in the gene-block-major order (the TF blocks of a gene
// block side by side share C's rows in L2): all whole; or, when that leaves
// the last round more than 5% short, the tiles of the last two rounds cut,
// whichever way leaves the busiest worker the least.
Phase plan_phase1(const Dev &d, int workers, bool pair)
{
    const int ntile = ceil_div(d.Tp, tile_m(pair)) * ceil_div(d.Gp, tile_n(pair));
    const int nR = ceil_div(d.Tp, BK), K = nR + ceil_div(d.Gp, BK);
    Phase best = plan_phase1_cut(d, workers, pair, ntile, 1);
    if ((double)ceil_div(ntile, workers) * workers <= 1.05 * ntile) {
        finish(best, workers);
        return best;
    }
    const int whole = std::max(0, ntile / workers - 1) * workers;
    for (int np : {0, 2, 3, 4, 6, 8, 12}) {
        if (np > 0 && ((ntile - whole) * np > 4 * workers || K - std::max(K / np, nR) < (np - 1) * MIN_PART))
            continue;
        Phase ph = plan_phase1_cut(d, workers, pair, whole, np);
        if (ph.cost < best.cost)
            best = std::move(ph);
    }
    finish(best, workers);
    return best;
}

// Phase 2: every upper-triangle tile in equal parts of at most `cap` stages,
// longest first to the least loaded worker.
Phase plan_phase2_cap(const Dev &d, int workers, bool pair, int cap)
{
    const int M = tile_m(pair), N = tile_n(pair);
    const double E = EPILOGUE[pair];
    Phase ph;
    std::vector<double> cost;
    for (int isP = 1; isP >= 0; --isP) {
        const int ld = isP ? d.Tp : d.Gp, nbm = ceil_div(ld, M), nbn = ceil_div(ld, N), K = ceil_div(isP ? d.Gp : d.Tp, BK);
        const int np = std::min(ceil_div(K, cap), 64);
        const size_t most = ph.items.size() + (size_t)nbm * (nbn + M / N) / 2 * np;
        ph.items.reserve(most);
        cost.reserve(most);
        for (int bm = 0; bm < nbm; ++bm)
            for (int bn = bm * (M / N); bn < nbn; ++bn) {
                for (int p = 0; p < np; ++p) {
                    Item it{};
                    it.a = (uint32_t)bm | (uint32_t)bn << 15 | (isP ? 0x80000000u : 0u);
                    it.s0 = (uint16_t)(K * p / np); it.s1 = (uint16_t)(K * (p + 1) / np);
                    it.part = (uint16_t)p; it.nparts = (uint16_t)np;
                    if (np > 1) {
                        it.fix = (uint16_t)ph.fixes;
                        it.slot = (uint16_t)ph.slots;
                    }
                    // (a mirrored tile's epilogue takes almost twice as long)
                    const double e = isP || bn < (bm + 1) * (M / N) ? 1.8 * E : E;
                    ph.items.push_back(it);
                    cost.push_back(it.s1 - it.s0 + (np > 1 ? CUT[pair] : 0.0) +
                                   (p == np - 1 ? e + (np > 1 ? CUT_LAST[pair] : 0.0) : 0.0));
                }
                if (np > 1) {
                    ph.fixes += 1;
                    ph.slots += np;
                }
            }
    }
    ph.cost = assign(ph, 0, cost, workers);
    return ph;
}

Phase plan_phase2(const Dev &d, int workers, bool pair)
{
    auto tiles = [&](int ld) { return (long long)ceil_div(ld, tile_m(pair)) * (ceil_div(ld, tile_n(pair)) + 2) / 2; };
    Phase best;
    for (int cap : {1 << 20, 256, 64, 32, 16, 8, 5}) {
        const long long parts = tiles(d.Tp) * ceil_div(ceil_div(d.Gp, BK), cap) +
                                tiles(d.Gp) * ceil_div(ceil_div(d.Tp, BK), cap);
        if (cap < (1 << 20) && parts > 8LL * workers)  // enough items to balance without cutting more
            break;
        Phase ph = plan_phase2_cap(d, workers, pair, cap);
        if (best.items.empty() || ph.cost < best.cost)
            best = std::move(ph);
    }
    finish(best, workers);
    return best;
}

struct F32Plan {
    bool pair;
    Phase p1, p2;
};

// What both phases' busiest workers cost at least: every tile whole, all workers equally busy
double least_cost(const Dev &d, int workers, bool pair)
{
    const int M = tile_m(pair), N = tile_n(pair), kT = ceil_div(d.Tp, BK), kG = ceil_div(d.Gp, BK);
    const double E = EPILOGUE[pair];
    double c = (double)ceil_div(d.Tp, M) * ceil_div(d.Gp, N) * (kT + kG + E);
    for (int isP = 0; isP < 2; ++isP) {
        const int ld = isP ? d.Tp : d.Gp, nbm = ceil_div(ld, M), nbn = ceil_div(ld, N);
        for (int bm = 0; bm < nbm; ++bm)
            c += (nbn - bm * (M / N)) * ((isP ? kG : kT) + E);
    }
    return c / workers;
}

// The tile shape whose busiest worker is done first by the stage times; one
// CTA per tile only where pairs would have few tiles each (it reads three times
// the operand bytes per flop).
F32Plan f32_plan_for(const Dev &d, int nsm)
{
    F32Plan best{};
    double t_best = 0.0;
    for (int pair = 1; pair >= 0; --pair) {
        if (!pair && (long long)ceil_div(d.Gp, 256) * ceil_div(d.Tp, 256) > 2LL * nsm)
            continue;
        const int workers = pair ? nsm / 2 : nsm;
        if (!best.p1.off.empty() && STAGE_US[pair] * least_cost(d, workers, pair != 0) > t_best * (1.0 + 1e-9))
            continue;  // not even with its work spread evenly
        F32Plan p{pair != 0, plan_phase1(d, workers, pair != 0), plan_phase2(d, workers, pair != 0)};
        const double t = STAGE_US[pair] * (p.p1.cost + p.p2.cost);
        if (best.p1.off.empty() || t < t_best) {
            best = std::move(p);
            t_best = t;
        }
    }
    return best;
}

// CTAs of a phase: the workers up to the last that has an item.  A CTA takes an SM to itself (217 KB
// of shared memory, all of TMEM), so one that finds nothing to do keeps another network of a set
// waiting: with 152 CTAs whatever the work, 64 networks of 125 x 125 took 286 us an iteration (81
// now), 64 of 60 x 300 382 (154), 16 of 250 x 600 184 (144).
int grid_of(const F32Plan &p, int phase)
{
    const Phase &ph = phase ? p.p2 : p.p1;
    int n = (int)ph.off.size() - 1;
    while (n > 1 && ph.off[n - 1] == ph.off[n])
        --n;
    return (p.pair ? 2 : 1) * n;
}

struct F32Host {
    F32Maps maps;
    F32Plan plan;  // its lists are on the device once `ready`
    bool ready = false;
    int grid[2] = {0, 0};  // CTAs of the two phases
    int *off[2] = {nullptr, nullptr};
    Item *items[2] = {nullptr, nullptr};
};

template <bool PAIR, class K1, class K2, class K3>
cudaError_t smem_limits(K1 p1, K2 p2, K3 p2s)
{
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(p1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p1_smem<PAIR>())) ||
        (e = cudaFuncSetAttribute(p2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p2_smem<PAIR, false>())))
        return e;
    return cudaFuncSetAttribute(p2s, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p2_smem<PAIR, true>());
}

cudaError_t all_smem_limits()
{
    cudaError_t e = smem_limits<true>(k_f32_phase1<true>, k_f32_phase2<true, false>, k_f32_phase2<true, true>);
    return e ? e : smem_limits<false>(k_f32_phase1<false>, k_f32_phase2<false, false>, k_f32_phase2<false, true>);
}

cudaError_t make_maps(const Dev &d, F32Maps &m)
{
    std::memset(&m, 0, sizeof m);
    __nv_bfloat16 *P[3] = {d.Ph, d.Pm, d.Pl}, *C[3] = {d.Ch, d.Cm, d.Cl};
    cudaError_t e;
    for (int p = 0; p < 3; ++p) {
        if ((e = tc_make_map(&m.P[p], P[p], d.Tp, d.Tp, 128)) || (e = tc_make_map(&m.C[p], C[p], d.Gp, d.Gp, 128)) ||
            (e = tc_make_map(&m.Cm[p], C[p], d.Gp, d.Gp, 64)))
            return e;
        for (int b = 0; b < 2; ++b) {
            __nv_bfloat16 *W[3] = {d.Wh[b], d.Wm[b], d.Wl[b]};
            if ((e = tc_make_map(&m.W[b][p], W[p], d.Tp, d.Gp, 128)) ||
                (e = tc_make_map(&m.Wm[b][p], W[p], d.Tp, d.Gp, 64)))
                return e;
        }
    }
    return cudaSuccess;
}

// panda_step_static's work lists and control block, by value in one launch
struct StaticArgs {
    Item items[2][F32_STATIC_ITEMS];
    int n[2];
    float alpha;
    double e2;
};
constexpr size_t STATIC_LIST = F32_STATIC_LIST_BYTES / 2;  // one phase: its offsets (256 bytes), then its items
static_assert((F32_STATIC_ITEMS + 1) * sizeof(int) <= 256, "the offsets fit");

__global__ void k_f32_static_lists(const __grid_constant__ StaticArgs a, uint8_t *lists, Ctl *ctl, double *e2tab, int *flags)
{
    const int t = threadIdx.x;
    for (int ph = 0; ph < 2; ++ph) {
        int *off = reinterpret_cast<int *>(lists + ph * STATIC_LIST);
        Item *it = reinterpret_cast<Item *>(lists + ph * STATIC_LIST + 256);
        if (t <= a.n[ph])
            off[t] = t;  // CTA t: item t
        if (t < a.n[ph])
            it[t] = a.items[ph][t];
    }
    if (t < 4)
        flags[t] = 0;
    if (t == 0) {
        Ctl c{};
        c.active = 1;
        c.stop_at = 1;
        c.alpha = a.alpha;
        c.tol = -1.0;
        *ctl = c;
        e2tab[0] = 1.0;
        e2tab[1] = a.e2;
    }
}

// On the stream of the kernels that read it, which does not wait for the default stream: a plain
// cudaMemcpy from pageable memory may return with its last bytes still on the way.  v lives until the
// caller has waited for s.
template <class T>
cudaError_t to_device(T **dst, const std::vector<T> &v, cudaStream_t s)
{
    cudaError_t e = cudaMalloc(dst, std::max<size_t>(1, v.size()) * sizeof(T));
    if (!e && !v.empty())
        e = cudaMemcpyAsync(*dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, s);
    return e;
}

template <bool PAIR>
cudaError_t launch_phase(const F32Host &h, const Dev &d, int cur, cudaStream_t s, int phase)
{
    const int grid = h.grid[phase - 1];
    if (phase == 1)
        return launch(k_f32_phase1<PAIR>, grid, NTHREADS, p1_smem<PAIR>(), s, h.maps, d, cur, h.off[0], h.items[0]);
    if (d.diag == 2)
        return launch(k_f32_phase2<PAIR, true>, grid, NTHREADS, p2_smem<PAIR, true>(), s, h.maps, d, cur, h.off[1],
                            h.items[1]);
    return launch(k_f32_phase2<PAIR, false>, grid, NTHREADS, p2_smem<PAIR, false>(), s, h.maps, d, cur, h.off[1],
                        h.items[1]);
}

}  // namespace

const char *const F32_KERNEL_NAMES[F32_KERNELS] = {"k_f32_phase1", "k_reduce_wnorms", "k_f32_phase2", "k_fin"};

void f32_plan(Dev &d, int nsm, size_t *slot_floats, size_t *fix_floats, int *fixes, bool *pair)
{
    F32Host *h = static_cast<F32Host *>(d.f32_host);
    if (!h) {
        d.f32_host = h = new F32Host;
        h->plan = f32_plan_for(d, nsm);
        for (int q = 0; q < 2; ++q)
            h->grid[q] = grid_of(h->plan, q);
    }
    const F32Plan &p = h->plan;
    const size_t slot = p.pair ? Tile<true>::SLOT : Tile<false>::SLOT, ranks = p.pair ? 2 : 1;
    *slot_floats = slot * (size_t)h->grid[0];  // (phase 1's alone)
    *fix_floats = slot * ranks * (size_t)std::max(p.p1.slots, p.p2.slots);
    *fixes = std::max(p.p1.fixes, p.p2.fixes);
    *pair = p.pair;
}

void f32_plan_info(const Dev &d, int nsm, bool *pair, int *ctas, int *items, int *cuts)
{
    const F32Plan p = f32_plan_for(d, nsm);
    *pair = p.pair;
    for (int q = 0; q < 2; ++q) {
        const Phase &ph = q ? p.p2 : p.p1;
        ctas[q] = grid_of(p, q);
        items[q] = (int)ph.items.size();
        cuts[q] = ph.fixes;
    }
}

int f32_diag_block(const Dev &d) { return static_cast<const F32Host *>(d.f32_host)->plan.pair ? 256 : 64; }

cudaError_t f32_prepare(Dev &d, int cur, cudaStream_t s, bool restored)
{
    auto split = [&](const float *X, size_t n, __nv_bfloat16 *h, __nv_bfloat16 *m, __nv_bfloat16 *l) {
        k_split3<<<(int)std::min<size_t>(2432, (n / 4 + 255) / 256), 256, 0, s>>>(X, n / 4, h, m, l);
    };
    if (restored) {
        split(d.W[cur], (size_t)d.Tp * d.Gp, d.Wh[cur], d.Wm[cur], d.Wl[cur]);
        split(d.Poff, (size_t)d.Tp * d.Tp, d.Ph, d.Pm, d.Pl);
        split(d.Coff, (size_t)d.Gp * d.Gp, d.Ch, d.Cm, d.Cl);
    }
    cudaError_t e = cudaGetLastError();
    F32Host *h = static_cast<F32Host *>(d.f32_host);
    if (e || h->ready)
        return e;
    if ((e = make_maps(d, h->maps)) || (e = all_smem_limits()))
        return e;
    const F32Plan &p = h->plan;
    if ((e = to_device(&h->off[0], p.p1.off, s)) || (e = to_device(&h->items[0], p.p1.items, s)) ||
        (e = to_device(&h->off[1], p.p2.off, s)) || (e = to_device(&h->items[1], p.p2.items, s)))
        return e;
    h->ready = true;
    return cudaSuccess;
}

void f32_release(Dev &d)
{
    F32Host *h = static_cast<F32Host *>(d.f32_host);
    if (h) {
        for (int q = 0; q < 2; ++q) {
            cudaFree(h->off[q]);
            cudaFree(h->items[q]);
        }
        delete h;
    }
    d.f32_host = nullptr;
}

cudaError_t launch_iteration_f32(const Dev &d, int cur, cudaStream_t s, KernelEvents &ke)
{
    const F32Host &h = *static_cast<const F32Host *>(d.f32_host);
    cudaError_t e;
    ke.mark(s);
    if ((e = h.plan.pair ? launch_phase<true>(h, d, cur, s, 1) : launch_phase<false>(h, d, cur, s, 1)))
        return e;
    ke.mark(s);
    if ((e = launch_reduce_wnorms(d, s)))
        return e;
    ke.mark(s);
    if ((e = h.plan.pair ? launch_phase<true>(h, d, cur ^ 1, s, 2) : launch_phase<false>(h, d, cur ^ 1, s, 2)))
        return e;
    ke.mark(s);
    return launch_fin(d, s, ke);
}

cudaError_t f32_static_host(const Dev &d, void *lists, void **host)
{
    F32Host *h = new F32Host;
    cudaError_t e;
    if ((e = make_maps(d, h->maps)) || (e = all_smem_limits())) {
        delete h;
        return e;
    }
    h->plan.pair = false;
    h->ready = true;
    for (int ph = 0; ph < 2; ++ph) {
        h->off[ph] = reinterpret_cast<int *>(static_cast<uint8_t *>(lists) + ph * STATIC_LIST);
        h->items[ph] = reinterpret_cast<Item *>(static_cast<uint8_t *>(lists) + ph * STATIC_LIST + 256);
    }
    const int nt = d.Gp / 64, mt = d.Tp / 128;
    h->grid[0] = nt * mt;
    for (int ld : {d.Tp, d.Gp})
        for (int bm = 0; bm < ld / 128; ++bm)
            h->grid[1] += ld / 64 - 2 * bm;
    *host = h;
    return cudaSuccess;
}

cudaError_t f32_static_lists(const Dev &d, float alpha, double e2, void *lists, int *flags, cudaStream_t s)
{
    StaticArgs a{};
    a.alpha = alpha;
    a.e2 = e2;
    auto add = [&](int ph, uint32_t code, int stages) {
        Item it{};
        it.a = code;
        it.s1 = (uint16_t)stages;
        it.nparts = 1;
        a.items[ph][a.n[ph]++] = it;
    };
    const int nR = d.Tp / BK, nA = d.Gp / BK;
    for (int nt = 0; nt < d.Gp / 64; ++nt)
        for (int mt = 0; mt < d.Tp / 128; ++mt)
            add(0, (uint32_t)mt | (uint32_t)nt << 16, nR + nA);
    for (int isP = 1; isP >= 0; --isP) {
        const int ld = isP ? d.Tp : d.Gp;
        for (int bm = 0; bm < ld / 128; ++bm)
            for (int bn = 2 * bm; bn < ld / 64; ++bn)
                add(1, (uint32_t)bm | (uint32_t)bn << 15 | (isP ? 0x80000000u : 0u), isP ? nA : nR);
    }
    k_f32_static_lists<<<1, 64, 0, s>>>(a, static_cast<uint8_t *>(lists), d.ctl, d.e2tab, flags);
    return cudaGetLastError();
}

}  // namespace panda
