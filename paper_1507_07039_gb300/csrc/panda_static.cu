// panda_step_static: one message-passing iteration on caller-owned device
// networks that allocates no device memory at all.
//
// Some callers cannot call cudaMalloc: code that must run within a fixed
// device-memory budget handed out by a host framework's own allocator or
// pool, plug-ins loaded into a process that forbids allocation once it is
// running, or latency-critical loops where a cudaMalloc (an implicit device
// synchronisation) is not acceptable.  For them this entry point takes its
// working memory from one file-scope device array of fixed size instead.
//
// The array is `g_scratch` below: STATIC_BYTES bytes (about 11.5 MB), sized
// for networks of at most PANDA_STATIC_MAX_NODES TFs and genes.  Every GPU
// that loads the library's device code holds it until the process exits (with
// CUDA's lazy module loading that happens at the first call on the device, so
// a caller with a fixed budget makes that call at start-up).  In host code its
// name only stands for the device array; the device address is looked up once
// per device with cudaGetSymbolAddress, with that device current, on the
// first call made on it.  All calls share the array, so two calls that overlap
// on the GPU (for example on two streams) race with each other.
//
// The iteration itself is the FP32 path of panda_step (the same kernels, whole
// tiles), run on a copy of the caller's networks laid out in the array.
//
// One call is bound by its launches and its wait for the device.  Everything is
// queued at once and waited for once: the kernels that read the networks check
// them and zero the padding on the way, the iteration runs whatever the checks
// find, and the kernels that write the results back look at the findings
// themselves.  At 64 x 256 a call took 282 us with the array cleared, the
// networks copied, checked, waited for and stripped in passes of their own
// and FFMA products.
#include "panda.h"
#include "panda_internal.cuh"

#include <cmath>
#include <mutex>
#include <string>

namespace panda {

// Sets the message panda_last_error(NULL) returns (defined in panda_api.cu).
void set_global_error(const std::string &msg);

namespace {

constexpr int SMAX = PANDA_STATIC_MAX_NODES;  // a multiple of TILE
constexpr int SNB = SMAX / TILE;
constexpr size_t al256(size_t b) { return (b + 255) & ~size_t(255); }
constexpr size_t SQ = al256(sizeof(float) * SMAX * SMAX);  // one padded square matrix
constexpr size_t VF = al256(sizeof(float) * SMAX);
constexpr size_t VD = al256(sizeof(double) * SMAX);
constexpr size_t PART = al256(sizeof(float) * 3 * SNB * SMAX);  // partial-sum slots
constexpr size_t BF = al256(sizeof(__nv_bfloat16) * SMAX * SMAX);  // one part of a padded square matrix
static_assert(2 * BF >= SQ, "two neighbouring parts hold a dense matrix");
constexpr size_t STATIC_BYTES = 4 * SQ                  // W[2], Poff, Coff
                                + 12 * BF               // three parts of W[2], P, C
                                + 2 * VD + 6 * VF       // pd, cd; pdf, cdf, rsqP, csqC, rsqW, csqW
                                + 8 * PART              // wrow, wcol, ps_sum/sq/vsq, cs_sum/sq/vsq
                                + al256(sizeof(double) * 2 * SNB * SNB)  // hpart
                                + al256(sizeof(Ctl) + 4 * sizeof(int)) + 2 * al256(2 * sizeof(double))  // ctl, hist, e2tab
                                + al256(F32_STATIC_SLOT_BYTES) + al256(F32_STATIC_LIST_BYTES);

__device__ __align__(256) unsigned char g_scratch[STATIC_BYTES];

constexpr int MAX_DEVICES = 64;
std::mutex g_mu;
unsigned char *g_addr[MAX_DEVICES] = {};
void *g_host[MAX_DEVICES][SNB][SNB] = {};  // tensor maps over the array, per padded shape

// Device address of g_scratch on the current device (looked up once).
cudaError_t scratch_address(int dev, unsigned char **out)
{
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_addr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
        if (e != cudaSuccess)
            return e;
        g_addr[dev] = static_cast<unsigned char *>(p);
    }
    *out = g_addr[dev];
    return cudaSuccess;
}

int fail(int code, const std::string &msg)
{
    set_global_error(msg);
    return code;
}

}  // namespace
}  // namespace panda

using namespace panda;

#define SCU(call)                                                                           \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess)                                                              \
            return fail(PANDA_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_));   \
    } while (0)

extern "C" int panda_step_static(int T, int G, float *dW, float *dP, float *dC, float alpha, int t,
                                 int diag, double *h_out, void *stream)
{
    if (T < 1 || G < 1 || T > SMAX || G > SMAX)
        return fail(PANDA_EINVAL, "panda_step_static: T and G must be in [1, " +
                                      std::to_string(SMAX) + "] (the size of its static scratch)");
    if (!dW || !dP || !dC)
        return fail(PANDA_EINVAL, "panda_step_static: W, P and C must not be NULL");
    if (!(alpha >= 0.0f && alpha <= 1.0f) || t < 1 || diag < 0 || diag > 2)
        return fail(PANDA_EINVAL, "panda_step_static: need alpha in [0, 1], t >= 1, diag in 0..2");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int dev = 0;
    SCU(cudaGetDevice(&dev));
    if (dev < 0 || dev >= MAX_DEVICES)
        return fail(PANDA_EUNSUPPORTED, "panda_step_static: device index out of range");
    if (!tc_supported())
        return fail(PANDA_EUNSUPPORTED, "panda_step_static: needs an sm_103 device");
    unsigned char *base = nullptr;
    SCU(scratch_address(dev, &base));

    // carve the array (every region sized for the maximum network)
    Dev d{};
    d.T = T; d.G = G;
    d.Tp = round_up(T, TILE); d.Gp = round_up(G, TILE);
    d.nbT = d.Tp / TILE; d.nbG = d.Gp / TILE;
    d.nwr = 2 * d.nbG;
    d.narrow = 1;
    d.diag = diag;
    d.inv_n1P = T > 1 ? 1.0 / (T - 1) : 0.0;
    d.inv_n1C = G > 1 ? 1.0 / (G - 1) : 0.0;
    unsigned char *p = base;
    auto take = [&p](size_t bytes) { unsigned char *q = p; p += bytes; return q; };
    auto part = [&take]() { return (__nv_bfloat16 *)take(BF); };
    for (int b = 0; b < 2; ++b) {
        d.W[b] = (float *)take(SQ);
        d.Wh[b] = part(); d.Wm[b] = part(); d.Wl[b] = part();
    }
    d.Poff = (float *)take(SQ);
    d.Coff = (float *)take(SQ);
    d.Ph = part(); d.Pm = part(); d.Pl = part();
    d.Ch = part(); d.Cm = part(); d.Cl = part();
    d.pd = (double *)take(VD);
    d.cd = (double *)take(VD);
    d.pdf = (float *)take(VF);
    d.cdf = (float *)take(VF);
    d.rsqP = (float *)take(VF);
    d.csqC = (float *)take(VF);
    d.rsqW = (float *)take(VF);
    d.csqW = (float *)take(VF);
    d.wrow_part = (float *)take(PART);
    d.wcol_part = (float *)take(PART);
    d.ps_sum = (float *)take(PART);
    d.ps_sq = (float *)take(PART);
    d.ps_vsq = (float *)take(PART);
    d.cs_sum = (float *)take(PART);
    d.cs_sq = (float *)take(PART);
    d.cs_vsq = (float *)take(PART);
    d.hpart = (double *)take(al256(sizeof(double) * 2 * SNB * SNB));
    d.ctl = (Ctl *)take(al256(sizeof(Ctl) + 4 * sizeof(int)));
    d.hist = (double *)take(al256(2 * sizeof(double)));
    d.e2tab = (double *)take(al256(2 * sizeof(double)));
    int *flags = (int *)(d.ctl + 1);  // read back with the control block

    d.p1_acc = (float *)take(al256(F32_STATIC_SLOT_BYTES));
    void *lists = take(al256(F32_STATIC_LIST_BYTES));
    {
        std::lock_guard<std::mutex> lock(g_mu);
        void *&host = g_host[dev][d.nbT - 1][d.nbG - 1];
        if (!host)
            SCU(f32_static_host(d, lists, &host));
        d.f32_host = host;
    }

    // one iteration at index t: counter 0, growth factor e^{2 alpha t} in slot 1
    SCU(f32_static_lists(d, alpha, std::exp(2.0 * (double)alpha * (double)t), lists, flags, s));
    // the state, exactly as a context builds it; a network that is not on this device is copied to
    // where its matrix lives, and back from the room that its old values or its parts took
    const bool hW = where_is(dW, dev) == Where::HERE, hP = where_is(dP, dev) == Where::HERE,
               hC = where_is(dC, dev) == Where::HERE;
    SymOut po{d.Poff, !hP, Parts{d.Ph, d.Pm, d.Pl}, 1, 64, d.Tp, d.pd, d.pdf};
    SymOut xo{d.Coff, !hC, Parts{d.Ch, d.Cm, d.Cl}, 0, 64, d.Gp, d.cd, d.cdf};
    StateIn in{hW ? dW : d.W[0], hP ? dP : d.Poff, hC ? dC : d.Coff, T, G, hW ? G : d.Gp, hP ? T : d.Tp, hC ? G : d.Gp,
               nullptr, nullptr, nullptr};
    struct Moved { bool here; float *user, *in; int rows, cols, ld; float *out; };
    const Moved moved[3] = {{hW, dW, d.W[0], T, G, d.Gp, d.W[0]},
                            {hP, dP, d.Poff, T, T, d.Tp, reinterpret_cast<float *>(d.Ph)},   // Ph and Pm: 4 bytes an entry
                            {hC, dC, d.Coff, G, G, d.Gp, reinterpret_cast<float *>(d.Ch)}};  // Ch and Cm
    for (const Moved &m : moved)
        if (!m.here)
            SCU(cudaMemcpy2DAsync(m.in, (size_t)m.ld * 4, m.user, (size_t)m.cols * 4, (size_t)m.cols * 4, m.rows,
                                  cudaMemcpyDefault, s));
    SCU(launch_load(in, d.W[0], Parts{d.Wh[0], d.Wm[0], d.Wl[0]}, d.Tp, d.Gp, po, xo, flags, s));
    in.W = d.W[0];
    in.ldw = d.Gp;
    SCU(launch_norms(StateNorms{in, d.pd, d.cd, d.rsqW, d.csqW, d.rsqP, d.csqC}, s));
    KernelEvents ke{nullptr, 0, false};
    SCU(launch_iteration_f32(d, 0, s, ke));
    // results back into the caller's buffers, diagonals from the FP64 vectors; a failed call leaves
    // the caller's networks as they were
    SCU(launch_store(StateOut{T, G, d.Tp, d.Gp, d.W[1], d.Poff, d.Coff, nullptr, nullptr, d.pd, d.cd,
                              hW ? dW : moved[0].out, hP ? dP : moved[1].out, hC ? dC : moved[2].out, flags, d.ctl},
                     s));
    struct { Ctl ctl; int flags[4]; } back{};
    SCU(cudaMemcpyAsync(&back, d.ctl, sizeof(Ctl) + 4 * sizeof(int), cudaMemcpyDeviceToHost, s));
    SCU(cudaStreamSynchronize(s));
    const Ctl &hc = back.ctl;
    const int *hflags = back.flags;
    if (hflags[0])
        return fail(PANDA_ENONFINITE, "panda_step_static: a network has a non-finite entry");
    if (hflags[1])
        return fail(PANDA_EASYM, "panda_step_static: P or C is not exactly symmetric");
    if (hc.status & ST_TIMEOUT)
        return fail(PANDA_ETIMEOUT, "panda_step_static: a bounded device wait expired");
    if (hc.status & ST_NONFINITE)
        return fail(PANDA_ENONFINITE, "panda_step_static: the networks became non-finite (left unchanged)");
    for (const Moved &m : moved)
        if (!m.here)
            SCU(cudaMemcpyAsync(m.user, m.out, (size_t)m.rows * m.cols * 4, cudaMemcpyDefault, s));
    if (!hW || !hP || !hC)
        SCU(cudaStreamSynchronize(s));
    if (h_out)
        *h_out = hc.h_last;
    return PANDA_OK;
}
