// host.h -- host-side helpers shared by the C-ABI drivers (workspace,
// timing, CUDA-graph capture of a sweep, parameter checks) and the FP64
// two-sided sweep runner used by the plain and the mixed-precision drivers.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <utility>
#include <vector>

#include "internal.h"

namespace jac {

constexpr double U64 = 1.1102230246251565e-16;  // 2^-53

// Stream-ordered workspace that is released when the call returns.  The
// environment variable JACOBI_WORKSPACE_LIMIT=<bytes> caps what one
// Workspace may hold (host-side fault injection: the call then returns
// JACOBI_ERR_ALLOC before it launches anything, as on a real allocation
// failure).
struct Workspace {
    cudaStream_t s;
    std::vector<void*> ptrs;
    bool failed = false;
    size_t used = 0, limit = (size_t)-1;
    explicit Workspace(cudaStream_t st) : s(st)
    {
        if (const char* e = getenv("JACOBI_WORKSPACE_LIMIT")) limit = (size_t)strtoull(e, nullptr, 10);
    }
    template <class T>
    T* get(size_t count)
    {
        T* p = try_get<T>(count);
        if (!p) failed = true;
        return p;
    }
    // For what a call can do without: null where it does not fit (asked for
    // after everything the call needs).
    template <class T>
    T* try_get(size_t count)
    {
        const size_t bytes = (count == 0 ? 1 : count) * sizeof(T);
        if (failed || bytes > limit - used) return nullptr;
        void* p = nullptr;
        if (workspace_alloc(&p, bytes, s) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        used += bytes;
        ptrs.push_back(p);
        return (T*)p;
    }
    ~Workspace()
    {
        for (void* p : ptrs) cudaFreeAsync(p, s);
        cudaStreamSynchronize(s);
    }
};

struct Timer {
    cudaEvent_t a = nullptr, b = nullptr;
    cudaStream_t s;
    explicit Timer(cudaStream_t st) : s(st)
    {
        cudaEventCreate(&a);
        cudaEventCreate(&b);
        cudaEventRecord(a, s);
    }
    double stop()
    {
        float ms = 0.f;
        cudaEventRecord(b, s);
        cudaEventSynchronize(b);
        cudaEventElapsedTime(&ms, a, b);
        return ms;
    }
    ~Timer()
    {
        cudaEventDestroy(a);
        cudaEventDestroy(b);
    }
};

inline float elapsed_ms(cudaEvent_t a, cudaEvent_t b)
{
    float t = 0.f;
    if (cudaEventElapsedTime(&t, a, b) != cudaSuccess) {
        cudaGetLastError();
        return 0.f;
    }
    return t;
}

// Events recorded between the kernels of a sweep (inside the captured graph),
// read after the sweep to split the device time into pivot and update phases.
struct PhaseEvents {
    std::vector<cudaEvent_t> ev;
    explicit PhaseEvents(size_t n) : ev(n, nullptr)
    {
        for (auto& e : ev) cudaEventCreate(&e);
    }
    ~PhaseEvents()
    {
        for (auto& e : ev)
            if (e) cudaEventDestroy(e);
    }
    float ms(size_t a, size_t b) const { return elapsed_ms(ev[a], ev[b]); }
    float at(size_t i) const { return i ? ms(0, i) : 0.f; }   // from the first
};

// Spans of device time, in ms from a sweep's first event, and the time that any of
// them covers (update kernels of two streams can run at the same time).
using Spans = std::vector<std::pair<float, float>>;
inline double covered_ms(Spans& v)
{
    std::sort(v.begin(), v.end());
    double t = 0.0;
    float end = 0.f;
    for (const auto& x : v) {
        t += std::max(0.f, x.second - std::max(x.first, end));
        end = std::max(end, x.second);
    }
    return t;
}

// The spans of a side stream's update kernels, by number; those that a sweep did
// not open are left out.
struct SideTimes {
    PhaseEvents pe;
    std::vector<char> on;
    explicit SideTimes(size_t n) : pe(2 * n), on(n, 0) {}
    cudaError_t open(size_t i, cudaStream_t s)
    {
        on[i] = 1;
        return cudaEventRecordWithFlags(pe.ev[2 * i], s, cudaEventRecordExternal);
    }
    cudaError_t close(size_t i, cudaStream_t s) { return cudaEventRecordWithFlags(pe.ev[2 * i + 1], s, cudaEventRecordExternal); }
    void add(Spans& v, cudaEvent_t base) const
    {
        for (size_t i = 0; i < on.size(); ++i)
            if (on[i]) v.emplace_back(elapsed_ms(base, pe.ev[2 * i]), elapsed_ms(base, pe.ev[2 * i + 1]));
    }
};

// A low-priority stream beside the caller's, with the events that fork from it
// and join it again.  Destroyed only after its work is done.
struct SideStream {
    cudaStream_t s = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr, done[2] = {nullptr, nullptr};   // done: Q's update, by step parity
    bool open()
    {
        int lo = 0, hi = 0;
        bool ok = cudaDeviceGetStreamPriorityRange(&lo, &hi) == cudaSuccess &&
                  cudaStreamCreateWithPriority(&s, cudaStreamNonBlocking, lo) == cudaSuccess;
        for (cudaEvent_t* e : {&fork, &join, &done[0], &done[1]})
            ok = ok && cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess;
        if (!ok) cudaGetLastError();
        return ok;
    }
    ~SideStream()
    {
        if (s) {
            cudaStreamSynchronize(s);
            cudaStreamDestroy(s);
        }
        for (cudaEvent_t e : {fork, join, done[0], done[1]})
            if (e) cudaEventDestroy(e);
    }
};

// A captured sweep, replayed on the caller's stream.
struct SweepGraph {
    cudaGraphExec_t exec = nullptr;
    ~SweepGraph()
    {
        if (exec) cudaGraphExecDestroy(exec);
    }
};

// Capture `body` (a function issuing launches on stream cs) into g; returns
// false when capture is not possible, in which case the caller launches
// directly.
template <class F>
inline bool capture(SweepGraph& g, F body)
{
    // the highest priority: a sweep's own kernels go before those of a SideStream
    cudaStream_t cs;
    int lo = 0, hi = 0;
    if (cudaDeviceGetStreamPriorityRange(&lo, &hi) != cudaSuccess ||
        cudaStreamCreateWithPriority(&cs, cudaStreamNonBlocking, hi) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    bool ok = false;
    if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeRelaxed) == cudaSuccess) {
        bool launched = body(cs);
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamEndCapture(cs, &graph);
        if (launched && e == cudaSuccess && graph) {
            ok = cudaGraphInstantiate(&g.exec, graph, 0) == cudaSuccess;
        }
        if (graph) cudaGraphDestroy(graph);
    }
    cudaGetLastError();
    cudaStreamDestroy(cs);
    return ok;
}

// The emulated FP64 products slice an operand once into an image (V once
// per step in the update; both operands once per refinement product) by
// default; JACOBI_EMU_IMAGE=0 makes every tile slice its operands itself
// (the same slices, so the same results bit for bit).
inline bool emu_image_wanted()
{
    const char* e = getenv("JACOBI_EMU_IMAGE");
    return !(e && e[0] == '0');
}

// Cluster size for the pivot solves of a step with npairs pairs of order k:
// automatic unless JACOBI_PIVOT_CLUSTER is set ("1" = one CTA per pair,
// up to "16" = that size when it fits).
inline int choose_pivot_cluster(int k, int npairs)
{
    int dev = 0, smem = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (const char* env = getenv("JACOBI_PIVOT_CLUSTER")) {
        const int want = atoi(env);
        if (want == 1) return 1;
        if (want > 1 && pivot_pos_fits(k, want, (size_t)smem)) return want;
    }
    return pivot_cluster_size(k, npairs, (size_t)smem);
}

// Whether the pivot solves leave SMs for a side stream's kernels, and those are
// worth the events (n = 256: 12.64 ms without, 12.8 with them; n = 500: 31.0 and
// 29.1).
inline bool sms_left(int np, int npairs, int pcl)
{
    int dev = 0, sms = 0;
    return np >= 384 && cudaGetDevice(&dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
           npairs * pcl < sms;
}

inline int check_params(const jacobi_params& p)
{
    if (p.b < 1) return -7;
    if (p.b > 128) return JACOBI_ERR_UNSUPPORTED;
    if (p.ordering != JACOBI_ORDER_ROUND_ROBIN && p.ordering != JACOBI_ORDER_ANTI_DIAGONAL) return -7;
    if (p.max_sweeps < 0 || p.max_sweeps > 1000 || p.inner_max_sweeps < 0) return -7;
    if (!(p.tol >= 0.0) || !(p.inner_tol >= 0.0)) return -7;
    if (p.conv != JACOBI_CONV_OFF_ABS && p.conv != JACOBI_CONV_REL) return -7;
    if (p.pivot_order < 0 || p.pivot_order > 2) return -7;
    if (p.precision < JACOBI_PREC_FP64 || p.precision > JACOBI_PREC_FP64_EMU) return -7;
    if (p.fp64_products != 0 && p.fp64_products != 1) return -7;
    if (p.svd_qr != 0 && p.svd_qr != 1) return -7;
    return 0;
}

inline void fill_counters(jacobi_stats* st, const DevCounters& c)
{
    st->rotations = (long long)c.rotations;
    st->inner_sweeps = (long long)c.inner_sweeps;
    st->pair_solves = (long long)c.pair_solves;
    st->flops_fp64 = (double)c.flops_fp64;
    st->flops_update = (double)c.flops_update;
    st->flops_fp32 = (double)c.flops_fp32;
    st->flops_lowp = (double)c.flops_lowp;
}


// Plain FP64 two-sided driver on an already loaded, padded working pair
// (Aw[cur], Qw[cur]).  Runs until the stop test passes; on return *cur
// indexes the buffers holding the result.  Used by jacobi_syev and by the
// closing sweeps of the mixed form.
struct EvdState {
    int np, b, k;
    int n_real;   // rows/columns >= n_real are zero padding
    int pcl = 1;  // pivot cluster size (1: one CTA per pair)
    Ordering ord;
    int2* dpairs;
    double* Aw[2];
    double* Qw[2];
    double* Vb[2];   // by the step's parity (cur): Q's update reads one while the next pivots write the other
    int* rot[2];
    double* gscratch;
    double* partial;
    unsigned* ticket;
    double* result;
    DevCounters* cnt;
    // FP64 products on the tensor cores (JACOBI_PREC_FP64_EMU): the stage-1
    // products and the timeout word
    double* T64 = nullptr;
    int* err = nullptr;
    // the step's V sliced once (bf16 digit images) and its column scales
    unsigned char* vimg[2] = {nullptr, nullptr};
    int* vexp[2] = {nullptr, nullptr};
    // and the step's stage-1 operands (A's pair-blocks, Q's column pairs)
    unsigned char* aimg = nullptr;
    int* atab = nullptr;
    unsigned char* qimg = nullptr;
    int* qexp = nullptr;
    SideStream* side = nullptr;   // what runs beside the pivot solves: those images, Q's update
    bool pending = false;         // Q's update of the last step is still to be launched there
    EmuUpdArgs pending_q{};
    int pending_cur = 0;
    SideTimes* times = nullptr;   // two intervals a step (the images of A's operands; Q's) and the last step's Q

    // The odd steps' transforms: buffers of their own where a side stream may
    // read the even steps' meanwhile and they fit, else the even steps'.
    void parity_buffers(Workspace& ws)
    {
        Vb[1] = Vb[0];
        rot[1] = rot[0];
        vimg[1] = vimg[0];
        vexp[1] = vexp[0];
        if (ws.failed || !(aimg || Qw[0]) || !sms_left(np, ord.dev_per_step, pcl)) return;
        double* v = ws.try_get<double>((size_t)ord.max_pairs * 2 * k * k);
        int* r = v ? ws.try_get<int>(ord.max_pairs) : nullptr;
        unsigned char* vi = r && vimg[0] ? ws.try_get<unsigned char>(emu_update_vimg_bytes(ord.dev_per_step, k)) : nullptr;
        int* ve = vi ? ws.try_get<int>(emu_update_vexp_ints(ord.dev_per_step, k)) : nullptr;
        if (!r || (vimg[0] && !ve)) return;
        Vb[1] = v;
        rot[1] = r;
        vimg[1] = vi;
        vexp[1] = ve;
    }
    // pivot_order == 2: the per-pair QRCP scratch of the pivoting step
    double* qrws = nullptr;
    // emulated products: balance by the diagonal (relative stop criterion)
    int balance = 0;
};

// Result of a run of sweeps: code 0 converged, 1 max_sweeps ran out, <0 error.
struct SweepResult {
    int code;
    int sweeps;
};

SweepResult run_evd_sweeps(EvdState& E, const jacobi_params& p, int& cur, double target,
                           int sweep0, jacobi_stats* st, cudaStream_t s, bool use_rel);

// Mixed-precision two-sided driver (low-precision sweeps on the tensor
// cores, refinement against A0 in FP64, FP64 closing sweeps).
int syev_mixed(int n, double* A, int lda, double* w, double* Q, int ldq, const jacobi_params& p,
               jacobi_stats* st, cudaStream_t s);

}  // namespace jac
