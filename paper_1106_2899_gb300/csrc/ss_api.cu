// ss_api.cu -- host runtime behind the C ABI of include/slipspring.h.
//
// A context holds one or more elements (ensembles of equal-length chains).
// Each element owns its device state and observables; ss_run enqueues, per
// chunk of chunk_steps steps, one launch of the chain kernel per element.
// Parameters are validated here, on the host; kernels assume valid input.
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#include <mutex>
#include <string>
#include <vector>

#include "slipspring.h"
#include "ss_kernels.cuh"
#include "ss_adjoint.cuh"
#include "ss_corr.cuh"
#include "ss_launch.h"
#include "ss_state.cuh"

namespace {

constexpr int kThreads = ssk::kChunkThreads;
constexpr int kWarpsPerCta = kThreads / 32;

struct Elem {
    int M = 0, N = 0, W = 16, B = 2, NP = 32, zmax = 0;
    uint32_t chain_base = 0;
    int slices = 0, groups = 0;
    int parts = 1;            // correlator CTAs per slice
    void* R = nullptr;
    void* A = nullptr;
    int32_t* S = nullptr;
    int32_t* Z = nullptr;
    void* hist = nullptr;    // [M][L][6][16] T: newest 16 samples per correlator level and series row
    double* acc64 = nullptr;  // [slices * parts][L][96] FP64 sums
    double* acc64tt = nullptr;  // [slices * parts][L][48] FP64 sums of channel TT (optional)
    void* ser = nullptr;     // [ser_cap][M][6] T: stress series of one launch
    void* lev = nullptr;     // [2][ser_cap / 4 + 1][M][6] T: correlator level samples (ping-pong)
    int ser_cap = 0;
    double* logs = nullptr;  // in the context's block
    double* kap_d = nullptr;
    long long* kfrom_d = nullptr;
    int n_kap_d = 0;
    std::vector<long long> kfrom{0};
    std::vector<double> kap = std::vector<double>(9, 0.0);
    bool flow_dirty = true;
};

// one layout class of the batched launch: its items and graph node
struct BatchedClass {
    int k = 0;
    int2* items = nullptr;
    int n_items = 0, smem = 0;
    cudaGraphNode_t node = nullptr;
};

}  // namespace

struct ss_ctx {
    cudaStream_t stream = nullptr;
    int prec = SS_FP32;
    int dev = 0, sms = 1;  // the device and its SMs
    uint64_t seed = 0;
    std::vector<Elem> el;
    ss_params P{};
    bool have_params = false;
    bool initialized = false;
    double k_b = 0, k_s = 0;
    int levels = 0;
    long long step = 0;
    long long nsamp = 0;
    long long log_m0 = 0;
    unsigned long long* counters = nullptr;  // [kCounterCopies][8]
    int32_t* status = nullptr;
    // stress logs of all elements, one block [element][max_logs][groups][14]
    double* logs = nullptr;
    size_t logs_n = 0;
    std::vector<double> logs_host;  // what the last read copied back
    bool logs_read = false;         // logs_host holds the whole block as it is now
    bool logs_captured = false;     // a graph that writes the logs was captured: its replays are not seen here
    void* stage = nullptr;  // device staging for state uploads and correlator readout
    size_t stage_bytes = 0;
    long long launches = 0;
    bool timing = false;
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> events;  // chain-kernel launches while timing
    // batched mode: one graph launch per chunk over all elements
    bool batched = false;
    bool tuned = false;
    bool graph_dirty = true;
    int batch_logs = 0;  // log steps of a launch at most
    ssk::ChunkArgs* d_elems = nullptr;
    int2* d_items = nullptr;
    std::vector<BatchedClass> bclasses;
    cudaGraphExec_t gexec = nullptr;
    cudaGraph_t graph = nullptr;
    // differentiation window
    struct Window {
        long long n = 0, t_start = 0;
        int ce = 0, nseg = 0;
        bool have_tape = false, forward_done = false;
        bool complete = false;  // every buffer below is allocated
        uint8_t* tape = nullptr;
        void* series = nullptr;
        void* ckR = nullptr;  // [nseg+1] states
        void* ckA = nullptr;
        int32_t* ckS = nullptr;
        int32_t* ckZ = nullptr;
        void* snR = nullptr;  // [ce+1] states
        void* snA = nullptr;
        int32_t* snS = nullptr;
        int32_t* snZ = nullptr;
        void* xbar = nullptr;
        void* ybar = nullptr;
        double* scratch = nullptr;
        void* Rb = nullptr;
        void* Ab = nullptr;
        double* grad = nullptr;
        double* wgt = nullptr;
    } win;
    // options of the next chain-kernel launches (set by the window calls)
    int opt_tape_mode = 0;
    bool opt_snap = false, opt_series = false, opt_corr_off = false;
    long long opt_snap_t0 = 0;
    cudaEvent_t xev = nullptr;  // orders the context's stream against a caller's stream
    std::vector<cudaStream_t> side;  // streams beside the context's, for several elements (made on first use)
    std::vector<cudaEvent_t> side_ev;
    std::string err;
};

namespace {

int fail(ss_ctx* c, int code, const std::string& msg) {
    if (c) c->err = msg;
    return code;
}

#define SS_CUDA(ctx, call)                                                                  \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess) {                                                            \
            cudaGetLastError(); /* reported here: not to be found again by a later call */  \
            return fail((ctx), e_ == cudaErrorMemoryAllocation ? SS_ENOMEM : SS_ECUDA,      \
                        std::string(#call) + ": " + cudaGetErrorString(e_));                 \
        }                                                                                   \
    } while (0)

size_t tsize(const ss_ctx* c) { return c->prec == SS_FP64 ? sizeof(double) : sizeof(float); }

// NVTX range for profilers (a no-op unless a tool is attached)
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

// device staging of at least `bytes`, grown on demand and kept for the context
int stage_at_least(ss_ctx* c, size_t bytes) {
    if (c->stage_bytes >= bytes) return SS_OK;
    if (c->stage) {
        SS_CUDA(c, cudaStreamSynchronize(c->stream));
        cudaFree(c->stage);
        c->stage = nullptr;
        c->stage_bytes = 0;
    }
    SS_CUDA(c, cudaMalloc(&c->stage, bytes));
    c->stage_bytes = bytes;
    return SS_OK;
}

void free_elem(Elem& e) {
    void* ptrs[] = {e.R, e.A, e.S, e.Z, e.hist, e.acc64, e.acc64tt, e.ser, e.lev, e.kap_d, e.kfrom_d};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    e.R = e.A = e.hist = e.ser = e.lev = nullptr;
    e.ser_cap = 0;
    e.S = e.Z = nullptr;
    e.acc64 = e.acc64tt = e.logs = e.kap_d = nullptr;
    e.kfrom_d = nullptr;
    e.n_kap_d = 0;
}

void free_logs(ss_ctx* c) {
    if (c->logs) cudaFree(c->logs);
    c->logs = nullptr;
    c->logs_n = 0;
    c->logs_read = c->logs_captured = false;
    for (Elem& e : c->el) e.logs = nullptr;
}

// Work that changes the logs is about to be enqueued: what was read of them is out of
// date, and stays so from read to read once the stream is captured into a graph.
int logs_change(ss_ctx* c) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (c->logs) SS_CUDA(c, cudaStreamIsCapturing(c->stream, &st));
    if (st != cudaStreamCaptureStatusNone) c->logs_captured = true;
    c->logs_read = false;
    return SS_OK;
}

// The first n stress logs of an element on the host.  The logs of several elements
// are usually read one after another, so a block of up to kLogBlockBytes comes over
// in one copy and stays until the next run or reset (512 elements: 512 copies and
// synchronisations took 7 ms), but for a context whose runs were captured into a graph.
constexpr size_t kLogBlockBytes = 4 << 20;
int read_logs(ss_ctx* c, const Elem& e, int n, const double** out) {
    const bool all = c->el.size() > 1 && !c->logs_captured && c->logs_n * sizeof(double) <= kLogBlockBytes;
    const size_t first = (size_t)(e.logs - c->logs), count = (size_t)n * e.groups * 14;
    if (!all || !c->logs_read) {
        c->logs_host.resize(all ? c->logs_n : count);
        SS_CUDA(c, cudaMemcpyAsync(c->logs_host.data(), all ? c->logs : e.logs, c->logs_host.size() * sizeof(double),
                                   cudaMemcpyDeviceToHost, c->stream));
        SS_CUDA(c, cudaStreamSynchronize(c->stream));
        c->logs_read = all;
    }
    *out = c->logs_host.data() + (all ? first : 0);
    return SS_OK;
}

// Chain layout for N beads: W lanes per chain, B beads per lane (W*B >= N).  Every
// layout of the chain kernel rounds each sum over beads alike, so the choice is
// free.  Eight lanes per chain leave fewer lanes idle at N <= 8 and 17..24 and share
// the slot work and the reductions of a warp among four chains, but run half as
// many warps: they win once the chip is full (us per step, 8 against 16 lanes:
// N = 24: 1.70 / 1.46 at 4096 chains, 2.39 / 2.50 at 8192, 14.6 / 16.5 at 65536;
// N = 16: 3.10 / 2.89 at 16384, 10.0 / 10.4 at 65536).  FP64 work is bound by the
// FP64 pipe of the SM partitions a launch reaches, and takes the wider layouts.
void layout_for(int M, int N, int prec, int integrator, int* W, int* B) {
    const bool narrow = prec == SS_FP32 && integrator == SS_EULER;
    if (N <= 8) {
        *W = 8, *B = 1;
    } else if (N <= 16) {
        if (narrow && M >= 40000)
            *W = 8, *B = 2;
        else
            *W = 16, *B = 1;
    } else if (N <= 24 && narrow && M >= 8192) {
        *W = 8, *B = 3;
    } else if (N <= 32) {
        *W = 16, *B = 2;
    } else if (N <= 48) {
        *W = 16, *B = 3;
    } else if (N <= 64) {
        *W = 16, *B = 4;
    } else if (N <= 96) {
        *W = 32, *B = 3;
    } else {
        *W = 32, *B = 4;
    }
}

int chains_per_cta(int W) { return kWarpsPerCta * (32 / W); }

// the chain kernel of this precision (windows refuse a velocity gradient)
template <typename T>
const void* chunk_fn(int W, int B, int win, bool flow, bool heun, bool corr, bool alt) {
    if (sizeof(T) == 8)
        return flow ? ssk::chunk_fn_f64_flow(W, B, win, heun, corr, alt) : ssk::chunk_fn_f64(W, B, win, heun, corr, alt);
    return flow ? ssk::chunk_fn_f32_flow(W, B, win, heun, corr, alt) : ssk::chunk_fn_f32(W, B, win, heun, corr, alt);
}
// Lets a kernel be launched with more than the default 48 KiB of dynamic shared memory
// (fixed: its static shared memory).  The limit belongs to the function on the current
// device, not to a context: it is always set to all that an SM offers a CTA, so that no
// context or thread lowers what another one's launches or graphs need.
cudaError_t allow_smem(const void* fn, int bytes, int fixed = 0) {
    if (bytes <= 48 * 1024 - fixed) return cudaSuccess;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024 - fixed);
}
// its shared memory with nlog log steps; series: a stress series may be written
template <typename T>
int chunk_smem(int W, int B, int nlog, bool flow, bool heun, bool series, bool alt) {
    return ssk::smem_plan<T>(kWarpsPerCta, W, B, nlog, series ? ssk::red_steps<T>(W, B, heun, flow, alt) : 0).total;
}
// and its warps per SM
template <typename T>
int chunk_resident(int W, int B, int nlog, bool flow, bool heun, bool series, bool alt) {
    return std::min(ssk::chunk_warps_per_sm<T>(W, B, heun, flow, alt),
                    ssk::ctas_by_smem(chunk_smem<T>(W, B, nlog, flow, heun, series, alt)));
}
// Whether M chains of a layout run the second form of the chain kernel: by the waves of
// warps that each form takes.  More warps per SM do the same work per time, or a little
// less, but may save a wave (first / second form, N = 49..64, us of 400 steps: 4000 x 60,
// 13.2 warps per SM, Euler-Maruyama 1516 / 1335, with shear 1592 / 1355, Heun 2104 / 1740;
// 9000 x 62, 29.6 per SM: 2578 / 2640, 2718 / 2680, 3852 / 3490; 2500 x 52: 951 / 1079, 1001 /
// 1145, 1376 / 1420; 300 steps with shear: 6000 x 48, 19.7 per SM, 1147 / 948; 10200 x 24
// 1034 / 892; Heun 6000 x 32 985 / 884, 4400 x 48 1642 / 1319).  At N = 49..64 Heun with flow
// has more warps in the first form, which does more per time (30000 x 60: 15.1 / 17.4 ms;
// 3000 x 60: 1.87 / 2.53); the second is faster in one wave of its own and in two where the
// first, of whose warps 12 fit an SM, takes two as well (2300 x 60: 1.67 / 1.59; 3500 x 60:
// 1.97 / 2.69; 4000 x 60: 2.98 / 2.77).  (Heun figures before its records by slot, which took
// 4-9% off both forms.)
template <typename T>
bool second_form(int M, int W, int B, int sms, int nlog, bool flow, bool heun, bool series) {
    if (sizeof(T) == 8 || !ssk::has_second_form(W, B, heun, flow)) return false;
    const long long warps = ((long long)M * W + 31) / 32;
    const int a = sms * chunk_resident<T>(W, B, nlog, flow, heun, series, false);
    const int b = sms * chunk_resident<T>(W, B, nlog, flow, heun, series, true);
    if (B == 4 && heun && flow) return warps <= b || (warps > 12 * sms && warps <= 2 * b);
    const auto cost = [&](int slots) { return (warps + slots - 1) / slots * slots; };
    return cost(b) * 23 < cost(a) * 20;
}

// z_max by default: one slot per bead (Sec. 3.2), at most SS_MAX_SLOTS
int default_zmax(int N) { return std::min(N, SS_MAX_SLOTS); }

// Inverse standard normal CDF by bisection on erfc: the destruction
// threshold on a standard normal draw (host constant).
double norm_ppf(double p) {
    if (p >= 1.0) return std::numeric_limits<double>::infinity();
    if (p <= 0.0) return -std::numeric_limits<double>::infinity();
    double lo = -40.0, hi = 40.0;
    for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (mid == lo || mid == hi) break;
        if (0.5 * std::erfc(-mid / std::sqrt(2.0)) < p)
            lo = mid;
        else
            hi = mid;
    }
    return 0.5 * (lo + hi);
}

template <typename T>
ssk::StepConst<T> step_const(const ss_ctx* c, int N) {
    const ss_params& p = c->P;
    ssk::StepConst<T> s{};
    s.k_b = T(c->k_b);
    s.k_s = T(c->k_s);
    s.mob = T(p.dt / p.zeta);
    s.amp = T(std::sqrt(2.0 * p.kT * p.dt / p.zeta));
    s.dt = T(p.dt);
    s.pref = T(p.dt * p.kT / p.zeta_s);
    s.chop = T(c->k_s / (4.0 * p.kT));
    s.sa = T(std::sqrt(p.kT / c->k_s));
    const double pd = p.dt * p.kT / p.zeta_s;
    s.cd = T(norm_ppf(pd < 1.0 ? pd : 1.0));
    s.NkT = T((double)N * p.kT);
    s.kT = T(p.kT);
    s.pc[0] = T(0);
    for (int K = 1; K <= ssk::kMaxSlots; ++K) {
        double pc = p.dt * p.kT / (p.zeta_s * p.N0 * (double)K);
        if (pc > 0.5) pc = 0.5;
        s.pc[K] = T(pc);
    }
    s.two_pref = T(2.0 * p.dt * p.kT / p.zeta_s);
    s.c2 = T(2.0 * (c->k_s / (4.0 * p.kT)) * 1.4426950408889634);
    s.c2_f = (float)(2.0 * (c->k_s / (4.0 * p.kT)) * 1.4426950408889634);
    s.two_pref_f = (float)(2.0 * p.dt * p.kT / p.zeta_s);
    s.hmob = T(0.5 * (p.dt / p.zeta));
    s.hdt = T(0.5 * p.dt);
    uint32_t k0 = (uint32_t)c->seed, k1 = (uint32_t)(c->seed >> 32);
    for (int r = 0; r < 10; ++r) {
        s.rk0[r] = k0;
        s.rk1[r] = k1;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return s;
}

// The correlator kernel of one launch: all levels over the launch's series of the
// chains m0 (a multiple of kSliceChains) .. m1 - 1
// (ns rows of [M][6]); each CTA folds its chains' sums into acc64.  n0:
// samples before the launch; lev: two level-sample buffers of lev_half
// elements.  Returns the number of kernels launched, or -1.
// chains: those of one FP64 sum (a part of a slice, or a whole one).
template <typename T, bool TT>
int corr_launches_t(const T* ser, int m0, int m1, int chains, int ns, int M, int L, long long n0, T* hist,
                    double* acc64, double* acc64tt, T* lev, size_t lev_half, cudaStream_t st) {
    // one sum per slice: the FP32 kernel takes whole slices, the FP64 one (more
    // registers) half of every slice at a time
    constexpr bool whole = sizeof(T) == 4 && !TT;
    int launched = 0;
    const int part = std::min(chains, whole ? ssk::kSliceChains : ssk::kCorrPartChains);
    const int b0 = m0 / chains;
    const dim3 grid((m1 - m0 + chains - 1) / chains), block(ssk::corr_threads(part));
    for (int first = 0; first < chains && m0 + first < m1; first += part) {
        if (ns == 1 && part <= ssk::kCorrPartChains) {
            ssk::corr_step_kernel<T, TT>
                <<<grid, block, 0, st>>>(ser, b0, part, first, chains, n0, M, L, hist, acc64, acc64tt);
        } else if (whole && part > ssk::kCorrPartChains) {
            if constexpr (whole)
                ssk::corr_kernel<T, TT, ssk::kSliceChains>
                    <<<grid, block, 0, st>>>(ser, b0, part, first, chains, ns, n0, M, L, hist, lev, lev_half, acc64, acc64tt);
        } else {
            ssk::corr_kernel<T, TT, ssk::kCorrPartChains>
                <<<grid, block, 0, st>>>(ser, b0, part, first, chains, ns, n0, M, L, hist, lev, lev_half, acc64, acc64tt);
        }
        if (cudaGetLastError() != cudaSuccess) return -1;
        ++launched;
    }
    return launched;
}

// acc64tt null: channel TT off
template <typename T>
int corr_launches(const T* ser, int m0, int m1, int chains, int ns, int M, int L, long long n0, T* hist, double* acc64,
                  double* acc64tt, T* lev, size_t lev_half, cudaStream_t st) {
    return acc64tt ? corr_launches_t<T, true>(ser, m0, m1, chains, ns, M, L, n0, hist, acc64, acc64tt, lev, lev_half, st)
                   : corr_launches_t<T, false>(ser, m0, m1, chains, ns, M, L, n0, hist, acc64, nullptr, lev, lev_half, st);
}

// Whether element e has a nonzero velocity gradient at any step of t0 ..
// t0 + nsteps - 1 (the schedule entry active at t0 and every entry that starts
// inside the window, as the chain kernel walks them).
bool flow_in_window(const Elem& e, long long t0, int nsteps) {
    const int n = (int)e.kfrom.size();
    int ki = 0;
    while (ki + 1 < n && t0 >= e.kfrom[ki + 1]) ++ki;
    for (int k = ki; k < n; ++k) {
        if (k > ki && e.kfrom[k] >= t0 + nsteps) break;
        for (int d = 0; d < 9; ++d)
            if (e.kap[9 * (size_t)k + d] != 0.0) return true;
    }
    return false;
}

// Stress-log steps of one launch of the chain kernel at most.  Every CTA keeps 112 bytes
// per log step of its launch in shared memory, and CTAs are single warps: a launch with
// many log steps would leave room for few of them on an SM (N = 32: 20 without logs, 17
// with 16, 10 with 103, one with 1024).  Where a context's warps do not fit the chip at
// once, a chunk is split into launches of 16 log steps (us per step of 65536 x 32 under
// shear, log_every 10 / 1: 27.2 / 685 unsplit, 19.3 / 86.1 at 16 log steps, 20.5 / 86.3 at
// 32).  A smaller context takes as many as leave room for its warps: it is bound by
// latency, and a launch costs it some steps' time (256 x 16, log_every 1: 3.25 us per
// step with 16 log steps per launch, 2.85 with 1024; 4096 x 40: 49.6 unsplit, 6.8 with 16
// log steps, 6.4 with the 62 that fit).  The sums of every warp enter device
// memory by FP64 atomics, which bound a log at every step of a large ensemble.
constexpr int kLaunchLogs = 16;
// bytes0: shared memory of a CTA without logs
int launch_logs(const ss_ctx* c, int bytes0) {
    long long warps = 0;
    for (const Elem& e : c->el) warps += ((long long)e.M * e.W + 31) / 32;
    const long long per_sm = std::max(1ll, (warps + c->sms - 1) / c->sms);
    const long long room = 228 * 1024 / per_sm / 128 * 128 - 1024 - bytes0;
    return (int)std::max<long long>(kLaunchLogs, room / 112);
}
// steps from t on, n at most, with no more than `logs` log steps
int log_bounded_steps(const ss_params& p, long long t, int n, int logs) {
    if (p.log_every <= 0) return n;
    return (int)std::min<long long>(n, (t / p.log_every + logs + 1) * p.log_every - 1 - t);
}
// log steps of the longest launch over an element
template <typename T>
int logs_per_launch(const ss_ctx* c, const Elem& e, bool flow, bool heun, bool series) {
    if (c->P.log_every <= 0) return 0;
    return std::min(launch_logs(c, chunk_smem<T>(e.W, e.B, 0, flow, heun, series, false)),
                    c->P.chunk_steps / c->P.log_every + 1);
}

template <typename T>
int launch_chunk(ss_ctx* c, Elem& e, int m0, int m1, long long t0, int nsteps, cudaStream_t st) {
    NvtxRange range("chain kernel + correlator launch");
    const ss_params& p = c->P;
    ssk::ChunkArgs a{};
    a.R = e.R;
    a.A = e.A;
    a.S = e.S;
    a.Z = e.Z;
    a.logs = e.logs;
    a.counters = c->counters;
    a.cnt_mask = ssk::kCounterCopies - 1;
    a.status = c->status;
    a.kap = e.kap_d;
    a.kap_from = e.kfrom_d;
    a.n_kap = e.n_kap_d;
    a.M = e.M;
    a.N = e.N;
    a.zmax = e.zmax;
    a.create_mode = p.create_mode;
    a.destroy_new = p.destroy_new;
    a.log_every = p.log_every;
    a.recenter_every = p.recenter_every;
    a.log_m0 = c->log_m0;
    a.max_logs = p.max_logs;
    a.groups = e.groups;
    a.slices = e.slices;
    a.key0 = (uint32_t)c->seed;
    a.key1 = (uint32_t)(c->seed >> 32);
    a.chain_base = e.chain_base;
    // the correlator's input: this launch's stress series (a window keeps the
    // series of the whole window for its adjoint)
    const bool corr = c->levels > 0 && !c->opt_corr_off;
    if (corr && nsteps > ssk::kCorrMaxSteps) return fail(c, SS_EINVAL, "launch longer than the correlator accepts");
    if (corr) {
        if (c->opt_series) {
            a.series = c->win.series;
            a.series_row0 = t0 - c->win.t_start;
        } else {
            a.series = e.ser;
            a.series_row0 = 0;
        }
    }
    if (c->opt_corr_off) a.log_every = 0;  // recomputation: no observables at all
    if (c->opt_tape_mode) {
        a.tape = c->win.tape;
        a.tape_mode = c->opt_tape_mode;
        a.tape_t0 = c->win.t_start;
        a.tape_rows = c->win.n;
    }
    if (c->opt_snap) {
        a.snapR = c->win.snR;
        a.snapA = c->win.snA;
        a.snapS = c->win.snS;
        a.snapZ = c->win.snZ;
        a.snap_t0 = c->opt_snap_t0;
        a.snap_steps = c->win.ce;
    }
    // differentiation windows run the instantiations with the window hooks (they
    // refuse a velocity gradient), a launch without a velocity gradient the one
    // without the flow terms
    const int win = c->opt_tape_mode == 1 ? ssk::kWinRecord : (c->opt_tape_mode == 2 ? ssk::kWinReplay : ssk::kWinOff);
    // (the window kernels have the series compiled in, also for a replay without it)
    const bool flow = flow_in_window(e, t0, nsteps), heun = c->P.integrator == SS_HEUN;
    const bool series = corr || win != ssk::kWinOff;
    const int max_logs = logs_per_launch<T>(c, e, flow, heun, series);
    // (elements beside one another fill each other's waves: the first form)
    const bool alt = win == ssk::kWinOff && c->el.size() == 1 &&
                     second_form<T>(e.M, e.W, e.B, c->sms, max_logs, flow, heun, series);
    const void* kern = chunk_fn<T>(e.W, e.B, win, flow, heun, corr, alt);
    if (!kern) return fail(c, SS_EINVAL, "no chain kernel for this layout");
    ssk::StepConst<T> sc = step_const<T>(c, e.N);
    const int cpc = chains_per_cta(e.W), ctas = (m1 - m0 + cpc - 1) / cpc;
    a.cta0 = m0 / cpc;
    void* args[] = {(void*)&a, (void*)&sc};
    const long long row0 = a.series_row0;
    for (int done = 0; done < nsteps; done += a.nsteps) {
        a.t0 = t0 + done;
        a.nsteps = a.log_every > 0 ? log_bounded_steps(p, a.t0, nsteps - done, max_logs) : nsteps - done;
        a.series_row0 = row0 + done;
        a.nlog_chunk = a.log_every > 0 ? (int)((a.t0 + a.nsteps) / a.log_every - a.t0 / a.log_every) : 0;
        const int smem = chunk_smem<T>(e.W, e.B, a.nlog_chunk, flow, heun, series, alt);
        SS_CUDA(c, allow_smem(kern, smem));
        cudaEvent_t ev0 = nullptr, ev1 = nullptr;
        if (c->timing) {
            SS_CUDA(c, cudaEventCreate(&ev0));
            SS_CUDA(c, cudaEventCreate(&ev1));
            SS_CUDA(c, cudaEventRecord(ev0, st));
        }
        SS_CUDA(c, cudaLaunchKernel(kern, dim3(ctas), dim3(kThreads), args, smem, st));
        if (c->timing) {
            SS_CUDA(c, cudaEventRecord(ev1, st));
            c->events.emplace_back(ev0, ev1);
        }
        c->launches++;
    }
    if (corr) {
        const T* ser = static_cast<const T*>(a.series) + (size_t)row0 * e.M * 6;
        const int nl = corr_launches<T>(ser, m0, m1, ssk::corr_chains(e.M), nsteps, e.M, c->levels, c->nsamp, static_cast<T*>(e.hist), e.acc64,
                                        e.acc64tt, static_cast<T*>(e.lev), (size_t)(e.ser_cap / 4 + 1) * e.M * 6,
                                        st);
        if (nl < 0) return fail(c, SS_ECUDA, "correlator kernel launch failed");
        c->launches += nl;
    }
    return SS_OK;
}

template <typename T>
int launch_init(ss_ctx* c, Elem& e) {
    const ss_params& p = c->P;
    const double lam = (double)e.N / p.N0;
    const double sb = std::sqrt(p.kT / c->k_b), sa = std::sqrt(p.kT / c->k_s);
    const int blocks = (e.M + 127) / 128;
    const uint32_t k0 = (uint32_t)c->seed, k1 = (uint32_t)(c->seed >> 32);
    switch (e.NP) {
        case 16:
            ssk::init_kernel<T, 16><<<blocks, 128, 0, c->stream>>>((T*)e.R, (T*)e.A, e.S, e.Z, e.M, e.N, e.zmax, sb,
                                                                   sa, lam, k0, k1, e.chain_base);
            break;
        case 32:
            ssk::init_kernel<T, 32><<<blocks, 128, 0, c->stream>>>((T*)e.R, (T*)e.A, e.S, e.Z, e.M, e.N, e.zmax, sb,
                                                                   sa, lam, k0, k1, e.chain_base);
            break;
        case 48:
            ssk::init_kernel<T, 48><<<blocks, 128, 0, c->stream>>>((T*)e.R, (T*)e.A, e.S, e.Z, e.M, e.N, e.zmax, sb,
                                                                   sa, lam, k0, k1, e.chain_base);
            break;
        case 64:
            ssk::init_kernel<T, 64><<<blocks, 128, 0, c->stream>>>((T*)e.R, (T*)e.A, e.S, e.Z, e.M, e.N, e.zmax, sb,
                                                                   sa, lam, k0, k1, e.chain_base);
            break;
        default:
            ssk::init_kernel<T, 128><<<blocks, 128, 0, c->stream>>>((T*)e.R, (T*)e.A, e.S, e.Z, e.M, e.N, e.zmax,
                                                                    sb, sa, lam, k0, k1, e.chain_base);
    }
    SS_CUDA(c, cudaGetLastError());
    c->launches++;
    return SS_OK;
}

int upload_flow(ss_ctx* c, Elem& e) {
    if (!e.flow_dirty) return SS_OK;
    if (e.kap_d) cudaFree(e.kap_d);
    if (e.kfrom_d) cudaFree(e.kfrom_d);
    e.kap_d = nullptr;
    e.kfrom_d = nullptr;
    const int n = (int)e.kfrom.size();
    SS_CUDA(c, cudaMalloc(&e.kap_d, sizeof(double) * 9 * n));
    SS_CUDA(c, cudaMalloc(&e.kfrom_d, sizeof(long long) * n));
    SS_CUDA(c, cudaMemcpyAsync(e.kap_d, e.kap.data(), sizeof(double) * 9 * n, cudaMemcpyHostToDevice,
                               c->stream));
    SS_CUDA(c, cudaMemcpyAsync(e.kfrom_d, e.kfrom.data(), sizeof(long long) * n, cudaMemcpyHostToDevice,
                               c->stream));
    SS_CUDA(c, cudaStreamSynchronize(c->stream));
    e.n_kap_d = n;
    e.flow_dirty = false;
    c->graph_dirty = true;
    return SS_OK;
}

int zero_observables(ss_ctx* c) {
    const size_t ts = tsize(c);
    for (Elem& e : c->el) {
        if (e.hist) SS_CUDA(c, cudaMemsetAsync(e.hist, 0, (size_t)e.M * c->levels * 96 * ts, c->stream));
        if (e.acc64)
            SS_CUDA(c, cudaMemsetAsync(e.acc64, 0, (size_t)e.slices * e.parts * c->levels * 96 * sizeof(double),
                                       c->stream));
        if (e.acc64tt)
            SS_CUDA(c, cudaMemsetAsync(e.acc64tt, 0, (size_t)e.slices * e.parts * c->levels * 48 * sizeof(double),
                                       c->stream));
    }
    if (const int rl = logs_change(c)) return rl;
    if (c->logs) SS_CUDA(c, cudaMemsetAsync(c->logs, 0, c->logs_n * sizeof(double), c->stream));
    c->nsamp = 0;
    c->log_m0 = c->P.log_every > 0 ? c->step / c->P.log_every : 0;
    return SS_OK;
}

bool finite_pos(double x) { return std::isfinite(x) && x > 0; }

Elem* elem_at(ss_ctx* c, int e) {
    if (!c || e < 0 || e >= (int)c->el.size()) return nullptr;
    return &c->el[e];
}

template <typename T>
int get_state_t(ss_ctx* c, Elem& e, double* R, int32_t* Z, int32_t* S, double* A) {
    const int W = e.NP, N = e.N, zm = e.zmax;
    std::vector<T> Rd((size_t)e.M * 3 * W), Ad((size_t)e.M * 3 * W);
    std::vector<int32_t> Sd((size_t)e.M * W), Zd(e.M);
    SS_CUDA(c, cudaMemcpyAsync(Rd.data(), e.R, Rd.size() * sizeof(T), cudaMemcpyDeviceToHost, c->stream));
    SS_CUDA(c, cudaMemcpyAsync(Ad.data(), e.A, Ad.size() * sizeof(T), cudaMemcpyDeviceToHost, c->stream));
    SS_CUDA(c, cudaMemcpyAsync(Sd.data(), e.S, Sd.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
    SS_CUDA(c, cudaMemcpyAsync(Zd.data(), e.Z, Zd.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
    SS_CUDA(c, cudaStreamSynchronize(c->stream));
    for (int m = 0; m < e.M; ++m) {
        if (R)
            for (int i = 0; i < N; ++i)
                for (int d = 0; d < 3; ++d) R[((size_t)m * N + i) * 3 + d] = (double)Rd[((size_t)m * 3 + d) * W + i];
        if (Z) Z[m] = Zd[m];
        for (int j = 0; j < zm; ++j) {
            const bool occ = j < Zd[m];
            if (S) S[(size_t)m * zm + j] = occ ? Sd[(size_t)m * W + j] : -1;
            if (A)
                for (int d = 0; d < 3; ++d)
                    A[((size_t)m * zm + j) * 3 + d] = occ ? (double)Ad[((size_t)m * 3 + d) * W + j] : 0.0;
        }
    }
    return SS_OK;
}

template <typename T>
int check_convert_state(ss_ctx* c, Elem& e, const double* dR, const double* dA, const int32_t* dS, const int32_t* dZ,
                        int* dF);

template <typename T>
int set_state_t(ss_ctx* c, Elem& e, const double* R, const int32_t* Z, const int32_t* S, const double* A) {
    // the caller's arrays go to the device as they are; checked and converted there
    const size_t M = e.M, N = e.N, zm = e.zmax;
    const size_t bR = M * N * 3 * sizeof(double), bA = M * zm * 3 * sizeof(double);
    const size_t bS = M * zm * sizeof(int32_t), bZ = M * sizeof(int32_t);
    const size_t oA = (bR + 255) & ~(size_t)255, oS = (oA + bA + 255) & ~(size_t)255;
    const size_t oZ = (oS + bS + 255) & ~(size_t)255, oF = (oZ + bZ + 255) & ~(size_t)255;
    int rc = stage_at_least(c, oF + sizeof(int));
    if (rc != SS_OK) return rc;
    char* st = static_cast<char*>(c->stage);
    const double* dR = reinterpret_cast<const double*>(st);
    const double* dA = reinterpret_cast<const double*>(st + oA);
    const int32_t* dS = reinterpret_cast<const int32_t*>(st + oS);
    const int32_t* dZ = reinterpret_cast<const int32_t*>(st + oZ);
    int* dF = reinterpret_cast<int*>(st + oF);
    SS_CUDA(c, cudaMemcpyAsync(st, R, bR, cudaMemcpyHostToDevice, c->stream));
    SS_CUDA(c, cudaMemcpyAsync(st + oA, A, bA, cudaMemcpyHostToDevice, c->stream));
    SS_CUDA(c, cudaMemcpyAsync(st + oS, S, bS, cudaMemcpyHostToDevice, c->stream));
    SS_CUDA(c, cudaMemcpyAsync(st + oZ, Z, bZ, cudaMemcpyHostToDevice, c->stream));
    return check_convert_state<T>(c, e, dR, dA, dS, dZ, dF);
}

// Check a state in the caller's layout held in device memory (dR [M][N][3],
// dA [M][zm][3] double, dS [M][zm], dZ [M] int32) and, if it is valid, convert
// it into the element's device layout.  dF: a device int used as the check
// flag.  Synchronises the context's stream to read the flag.
template <typename T>
int check_convert_state(ss_ctx* c, Elem& e, const double* dR, const double* dA, const int32_t* dS, const int32_t* dZ,
                        int* dF) {
    SS_CUDA(c, cudaMemsetAsync(dF, 0, sizeof(int), c->stream));
    const int width = std::max(e.N, e.zmax);
    const long long nchk = (long long)e.M * width, ncv = (long long)e.M * e.NP;
    ssk::state_check_kernel<<<(unsigned)((nchk + 255) / 256), 256, 0, c->stream>>>(dR, dA, dS, dZ, e.M, e.N, e.zmax,
                                                                                  width, dF);
    SS_CUDA(c, cudaGetLastError());
    int bad = 0;
    SS_CUDA(c, cudaMemcpyAsync(&bad, dF, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    SS_CUDA(c, cudaStreamSynchronize(c->stream));
    if (bad & 1) return fail(c, SS_EINVAL, "Z out of range");
    if (bad & 2) return fail(c, SS_EINVAL, "S out of range");
    if (bad & 4) return fail(c, SS_EINVAL, "non-finite A");
    if (bad & 8) return fail(c, SS_EINVAL, "non-finite R");
    ssk::state_convert_kernel<T><<<(unsigned)((ncv + 255) / 256), 256, 0, c->stream>>>(
        dR, dA, dS, dZ, e.M, e.N, e.zmax, e.NP, static_cast<T*>(e.R), static_cast<T*>(e.A), e.S, e.Z);
    SS_CUDA(c, cudaGetLastError());
    c->launches += 2;
    return SS_OK;
}

// group sums [G][L][16][2][3] (W = 96) or, of channel TT, [G][L][16][3] (W = 48)
// from the device sums of the parts, summed on the device
template <int W>
int group_corr(ss_ctx* c, Elem& e, const double* acc, std::vector<double>& out) {
    const int L = c->levels;
    const size_t n = (size_t)e.groups * L * W;
    int rc = stage_at_least(c, n * sizeof(double));
    if (rc != SS_OK) return rc;
    double* d = static_cast<double*>(c->stage);
    ssk::corr_group_kernel<W><<<(unsigned)((n + 127) / 128), 128, 0, c->stream>>>(acc, e.slices, e.parts, e.groups, L, d);
    SS_CUDA(c, cudaGetLastError());
    out.resize(n);
    SS_CUDA(c, cudaMemcpyAsync(out.data(), d, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    SS_CUDA(c, cudaStreamSynchronize(c->stream));
    return SS_OK;
}

// chains of each group (slices are dealt to groups in contiguous runs), one pass over the slices
std::vector<int> group_sizes(const Elem& e) {
    const int sc = ssk::kSliceChains;
    std::vector<int> n(e.groups, 0);
    for (int s = 0; s < e.slices; ++s) n[(int)(((long long)s * e.groups) / e.slices)] += std::min(sc, e.M - s * sc);
    return n;
}

// ------------------------------------------------------------ batched ----
// Lane layouts the batched path can use; one kernel per layout.
constexpr int kBatchedLayouts = 10;
constexpr int kLayoutW[kBatchedLayouts] = {16, 16, 16, 16, 8, 8, 8, 32, 32, 32};
constexpr int kLayoutB[kBatchedLayouts] = {1, 2, 3, 4, 1, 2, 3, 1, 3, 4};

int layout_class(int W, int B) {
    for (int k = 0; k < kBatchedLayouts; ++k)
        if (kLayoutW[k] == W && kLayoutB[k] == B) return k;
    return -1;
}

void free_batched(ss_ctx* c) {
    if (c->gexec) cudaGraphExecDestroy(c->gexec);
    if (c->graph) cudaGraphDestroy(c->graph);
    if (c->d_elems) cudaFree(c->d_elems);
    if (c->d_items) cudaFree(c->d_items);
    c->gexec = nullptr;
    c->graph = nullptr;
    c->d_elems = nullptr;
    c->d_items = nullptr;
    c->bclasses.clear();
    c->graph_dirty = true;
}

// one element's kernel arguments in batched mode (no correlator)
ssk::ChunkArgs make_desc(const ss_ctx* c, const Elem& e) {
    const ss_params& p = c->P;
    ssk::ChunkArgs a{};
    a.R = e.R;
    a.A = e.A;
    a.S = e.S;
    a.Z = e.Z;
    a.logs = e.logs;
    a.counters = c->counters;
    a.cnt_mask = ssk::kCounterCopies - 1;
    a.status = c->status;
    a.kap = e.kap_d;
    a.kap_from = e.kfrom_d;
    a.n_kap = e.n_kap_d;
    a.M = e.M;
    a.N = e.N;
    a.zmax = e.zmax;
    a.create_mode = p.create_mode;
    a.destroy_new = p.destroy_new;
    a.log_every = p.log_every;
    a.recenter_every = p.recenter_every;
    a.max_logs = p.max_logs;
    a.groups = e.groups;
    a.slices = e.slices;
    a.key0 = (uint32_t)c->seed;
    a.key1 = (uint32_t)(c->seed >> 32);
    a.chain_base = e.chain_base;
    a.W = e.W;
    a.B = e.B;
    return a;
}

// Work items (element, first chain of a CTA tile) of one layout class,
// longest chains and largest elements first.
std::vector<int2> make_items(const std::vector<Elem>& el, int W, int B) {
    std::vector<int> order;
    for (size_t i = 0; i < el.size(); ++i)
        if (el[i].W == W && el[i].B == B) order.push_back((int)i);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        return el[a].N != el[b].N ? el[a].N > el[b].N : el[a].M > el[b].M;
    });
    std::vector<int2> items;
    for (int e : order) {
        const int cpc = chains_per_cta(W);
        for (int m = 0; m < el[e].M; m += cpc) items.push_back(make_int2(e, m));
    }
    return items;
}

template <typename T>
const void* batched_fn_of(int k) {
    return sizeof(T) == 8 ? ssk::batched_fn_f64(kLayoutW[k], kLayoutB[k]) : ssk::batched_fn_f32(kLayoutW[k], kLayoutB[k]);
}

// shared memory of a class beside the kernel's own copy of an element's arguments
template <typename T>
int batched_smem_bytes(int k, int nlog) {
    return ssk::smem_plan<T>(kWarpsPerCta, kLayoutW[k], kLayoutB[k], nlog, 0).total;
}

template <typename T>
int batched_launch_direct(ss_ctx* c, int k, const ssk::ChunkArgs* d_elems, const int2* d_items, int n_items,
                          long long t0, int ns, int smem) {
    ssk::RunInfo info{t0, ns, c->log_m0};
    ssk::StepConst<T> sc = step_const<T>(c, 32);
    void* args[] = {(void*)&d_elems, (void*)&d_items, (void*)&info, (void*)&sc};
    SS_CUDA(c, cudaLaunchKernel(batched_fn_of<T>(k), dim3(n_items), dim3(kThreads), args, smem, c->stream));
    return SS_OK;
}

// Candidate lane layouts of the batched kernel for `total` chains of length N, the
// default first: by the waves of warps they take (24 warps per SM at one bead per
// lane, 20 at two).  N = 9..16: 16 x 1 while it fits one wave (7296 chains on 152
// SMs), 8 x 2 while that does (12160), 16 x 1 for its two and a half waves (19000),
// then 8 x 2, which does less per chain (us per step at 4096 / 16384 / 65536 chains:
// 16 x 1 0.99 / 2.89 / 10.4, 8 x 2 1.35 / 3.10 / 10.0).  N = 17..32: 32 x 1 for
// ensembles of one wave (1024 chains: 1.27 us per step, 16 x 2 1.5), then 16 x 2, or
// 8 x 3 as in layout_for.  FP64 takes the same lines (us per step: N = 24, 16 x 2 / 8 x 3,
// 1000 chains 8.4 / 13.0, 9000 57.0 / 53.9, 20000 121 / 98.8; N = 32, 32 x 1 / 16 x 2, 1000
// 7.05 / 8.9, 20000 126 / 121; N = 16, 16 x 1 / 8 x 2, 1000 4.85 / 9.1, 9000 33.7 / 35.6, 30000
// 100.9 / 98.0).
std::vector<std::pair<int, int>> layout_candidates(int N, long long total, long long sms) {
    using L = std::vector<std::pair<int, int>>;
    if (N <= 8) return {{8, 1}};
    if (N <= 16) {
        const bool wide = total <= 48 * sms || (total > 80 * sms && total <= 125 * sms);
        return wide ? L{{16, 1}, {8, 2}} : L{{8, 2}, {16, 1}};
    }
    if (N <= 32) {
        const std::pair<int, int> two = N <= 24 && total >= 8192 ? std::pair<int, int>{8, 3} : std::pair<int, int>{16, 2};
        return total <= 24 * sms ? L{{32, 1}, two} : L{two, {32, 1}};
    }
    if (N <= 48) return {{16, 3}};
    if (N <= 64) return {{16, 4}};
    if (N <= 96) return {{32, 3}};
    return {{32, 4}};
}

// Project-written autotuner: for each chain length, time every candidate layout
// on a trial ensemble (equilibrium start, no flow, no logs, up to 65536 chains)
// with the batched kernel of that layout, twice each, and keep the fastest
// (the default layout unless another is at least a quarter faster).  Results are
// cached for the process by what they depend on: the device, the length, the
// precision and the default, which follows the number of chains.  (Cached by length
// and precision alone, a context of 65536 chains of N = 32 after one of 1000 ran
// 32 x 1, the layout for one wave.)
template <typename T>
int autotune(ss_ctx* c) {
    static std::mutex mu;
    struct Tuned {
        int dev, N, prec;
        std::pair<int, int> first, best;  // layouts (W, B): the default and the one kept
    };
    static std::vector<Tuned> cache;
    std::vector<int> lengths;
    for (const Elem& e : c->el)
        if (std::find(lengths.begin(), lengths.end(), e.N) == lengths.end()) lengths.push_back(e.N);
    for (int N : lengths) {
        int bestW = -1, bestB = -1;
        long long total = 0;
        for (const Elem& e : c->el)
            if (e.N == N) total += e.M;
        const auto cand = layout_candidates(N, total, c->sms);
        {
            std::lock_guard<std::mutex> lk(mu);
            for (const Tuned& r : cache)
                if (r.dev == c->dev && r.N == N && r.prec == c->prec && r.first == cand[0])
                    bestW = r.best.first, bestB = r.best.second;
        }
        if (bestW < 0) {
            bestW = cand[0].first, bestB = cand[0].second;
            if (cand.size() > 1) {
                Elem t;
                // as many chains as the workload has, up to enough for many waves:
                // the comparison is then one of steady throughput
                t.M = (int)std::max<long long>(256, std::min<long long>(65536, total));
                t.N = N;
                t.W = bestW;
                t.B = bestB;
                t.NP = ssk::row_stride(N);
                t.zmax = c->P.z_max > 0 ? std::min(c->P.z_max, N) : default_zmax(N);
                t.slices = (t.M + ssk::kSliceChains - 1) / ssk::kSliceChains;
                t.groups = 1;
                const size_t ts = sizeof(T);
                int rc = SS_OK;
                if (cudaMalloc(&t.R, (size_t)t.M * 3 * t.NP * ts) != cudaSuccess ||
                    cudaMalloc(&t.A, (size_t)t.M * 3 * t.NP * ts) != cudaSuccess ||
                    cudaMalloc(&t.S, (size_t)t.M * t.NP * sizeof(int32_t)) != cudaSuccess ||
                    cudaMalloc(&t.Z, (size_t)t.M * sizeof(int32_t)) != cudaSuccess)
                    rc = fail(c, SS_ENOMEM, "autotune: allocation failed");
                if (rc == SS_OK) rc = launch_init<T>(c, t);
                if (rc == SS_OK) rc = upload_flow(c, t);
                ssk::ChunkArgs* dd = nullptr;
                int2* di = nullptr;
                unsigned long long* dcnt = nullptr;  // the trials count into scratch, not the context
                if (rc == SS_OK && (cudaMalloc(&dd, sizeof(ssk::ChunkArgs)) != cudaSuccess ||
                                    cudaMalloc(&di, sizeof(int2) * t.M) != cudaSuccess ||
                                    cudaMalloc(&dcnt, (ssk::kCounterCopies + 1) * 8 * sizeof(unsigned long long)) != cudaSuccess))
                    rc = fail(c, SS_ENOMEM, "autotune: allocation failed");
                const long long saved_m0 = c->log_m0;
                const int saved_log = c->P.log_every;
                c->log_m0 = 0;
                c->P.log_every = 0;
                // each candidate timed twice, in alternating order, keeping its
                // faster trial
                std::vector<float> cand_ms(cand.size(), 1e30f);
                for (int trial = 0; trial < 2 * (int)cand.size(); ++trial) {
                    if (rc != SS_OK) break;
                    const size_t ci = (size_t)trial % cand.size();
                    const auto& lb = cand[ci];
                    t.W = lb.first;
                    t.B = lb.second;
                    const int k = layout_class(t.W, t.B);
                    std::vector<Elem> one = {t};
                    std::vector<int2> items = make_items(one, t.W, t.B);
                    ssk::ChunkArgs desc = make_desc(c, t);
                    desc.counters = dcnt;
                    desc.status = reinterpret_cast<int32_t*>(dcnt + 8 * ssk::kCounterCopies);
                    const int smem = batched_smem_bytes<T>(k, 0);
                    SS_CUDA(c, allow_smem(batched_fn_of<T>(k), smem, sizeof(ssk::ChunkArgs)));
                    SS_CUDA(c, cudaMemcpy(dd, &desc, sizeof(desc), cudaMemcpyHostToDevice));
                    SS_CUDA(c, cudaMemcpy(di, items.data(), sizeof(int2) * items.size(), cudaMemcpyHostToDevice));
                    cudaEvent_t e0, e1;
                    SS_CUDA(c, cudaEventCreate(&e0));
                    SS_CUDA(c, cudaEventCreate(&e1));
                    rc = batched_launch_direct<T>(c, k, dd, di, (int)items.size(), 0, 32, smem);
                    cudaEventRecord(e0, c->stream);
                    if (rc == SS_OK)
                        rc = batched_launch_direct<T>(c, k, dd, di, (int)items.size(), 32, 256, smem);
                    cudaEventRecord(e1, c->stream);
                    cudaEventSynchronize(e1);
                    float ms = 0.f;
                    cudaEventElapsedTime(&ms, e0, e1);
                    cudaEventDestroy(e0);
                    cudaEventDestroy(e1);
                    if (rc == SS_OK) cand_ms[ci] = std::min(cand_ms[ci], ms);
                }
                // the default layout (the first candidate) gives way only to one
                // at least a quarter faster: the candidates are within a few percent
                // of one another near the lines of the default, and a choice by
                // timing noise would differ from one process to the next
                size_t pick = 0;
                for (size_t ci = 1; ci < cand.size(); ++ci)
                    if (cand_ms[ci] < 0.75f * cand_ms[0] && cand_ms[ci] < cand_ms[pick]) pick = ci;
                bestW = cand[pick].first;
                bestB = cand[pick].second;
                c->log_m0 = saved_m0;
                c->P.log_every = saved_log;
                if (dd) cudaFree(dd);
                if (di) cudaFree(di);
                if (dcnt) cudaFree(dcnt);
                free_elem(t);
                if (rc != SS_OK) return rc;
                std::lock_guard<std::mutex> lk(mu);
                cache.push_back({c->dev, N, c->prec, cand[0], cand[pick]});
            }
        }
        for (Elem& e : c->el)
            if (e.N == N) e.W = bestW, e.B = bestB;
    }
    c->tuned = true;
    c->graph_dirty = true;
    return SS_OK;
}

// Descriptors, work items and the graph of one batched launch: a kernel per
// layout class, on independent branches so that they share the GPU.
template <typename T>
int batched_prepare(ss_ctx* c) {
    free_batched(c);
    std::vector<ssk::ChunkArgs> descs;
    for (const Elem& e : c->el) descs.push_back(make_desc(c, e));
    std::vector<std::vector<int2>> cls(kBatchedLayouts);
    size_t total = 0;
    for (int k = 0; k < kBatchedLayouts; ++k) {
        cls[k] = make_items(c->el, kLayoutW[k], kLayoutB[k]);
        total += cls[k].size();
    }
    SS_CUDA(c, cudaMalloc(&c->d_elems, sizeof(ssk::ChunkArgs) * descs.size()));
    SS_CUDA(c, cudaMalloc(&c->d_items, sizeof(int2) * std::max<size_t>(1, total)));
    SS_CUDA(c, cudaMemcpy(c->d_elems, descs.data(), sizeof(ssk::ChunkArgs) * descs.size(), cudaMemcpyHostToDevice));
    SS_CUDA(c, cudaGraphCreate(&c->graph, 0));
    c->batch_logs = 0;
    if (c->P.log_every > 0) {
        c->batch_logs = c->P.chunk_steps / c->P.log_every + 1;
        for (int k = 0; k < kBatchedLayouts; ++k)
            if (!cls[k].empty())
                c->batch_logs = std::min(
                    c->batch_logs, launch_logs(c, batched_smem_bytes<T>(k, 0) + (int)sizeof(ssk::ChunkArgs)));
    }
    size_t off = 0;
    for (int k = 0; k < kBatchedLayouts; ++k) {
        if (cls[k].empty()) continue;
        SS_CUDA(c, cudaMemcpy(c->d_items + off, cls[k].data(), sizeof(int2) * cls[k].size(), cudaMemcpyHostToDevice));
        BatchedClass bc;
        bc.k = k;
        bc.items = c->d_items + off;
        bc.n_items = (int)cls[k].size();
        bc.smem = batched_smem_bytes<T>(k, c->batch_logs);
        SS_CUDA(c, allow_smem(batched_fn_of<T>(k), bc.smem, sizeof(ssk::ChunkArgs)));
        ssk::RunInfo info{0, 1, 0};
        ssk::StepConst<T> sc = step_const<T>(c, 32);
        const ssk::ChunkArgs* pe = c->d_elems;
        void* args[] = {(void*)&pe, (void*)&bc.items, (void*)&info, (void*)&sc};
        cudaKernelNodeParams kp{};
        kp.func = (void*)batched_fn_of<T>(k);
        kp.gridDim = dim3(bc.n_items);
        kp.blockDim = dim3(kThreads);
        kp.sharedMemBytes = bc.smem;
        kp.kernelParams = args;
        SS_CUDA(c, cudaGraphAddKernelNode(&bc.node, c->graph, nullptr, 0, &kp));
        c->bclasses.push_back(bc);
        off += cls[k].size();
    }
    SS_CUDA(c, cudaGraphInstantiate(&c->gexec, c->graph, 0));
    c->graph_dirty = false;
    return SS_OK;
}

// One graph launch per chunk; the chunk's first step enters through the kernel
// nodes' parameters.
template <typename T>
int batched_chunk(ss_ctx* c, long long t0, int ns) {
    ssk::RunInfo info{t0, ns, c->log_m0};
    ssk::StepConst<T> sc = step_const<T>(c, 32);
    const ssk::ChunkArgs* pe = c->d_elems;
    for (BatchedClass& bc : c->bclasses) {
        void* args[] = {(void*)&pe, (void*)&bc.items, (void*)&info, (void*)&sc};
        cudaKernelNodeParams kp{};
        kp.func = (void*)batched_fn_of<T>(bc.k);
        kp.gridDim = dim3(bc.n_items);
        kp.blockDim = dim3(kThreads);
        kp.sharedMemBytes = bc.smem;
        kp.kernelParams = args;
        SS_CUDA(c, cudaGraphExecKernelNodeSetParams(c->gexec, bc.node, &kp));
    }
    SS_CUDA(c, cudaGraphLaunch(c->gexec, c->stream));
    c->launches += (long long)c->bclasses.size();
    return SS_OK;
}

template <typename T>
int batched_run(ss_ctx* c, long long n_steps) {
    if (!c->tuned) {
        int rc = autotune<T>(c);
        if (rc != SS_OK) return rc;
    }
    if (c->graph_dirty) {
        int rc = batched_prepare<T>(c);
        if (rc != SS_OK) return rc;
    }
    long long left = n_steps;
    while (left > 0) {
        const int ns =
            log_bounded_steps(c->P, c->step, (int)std::min<long long>(left, c->P.chunk_steps), c->batch_logs);
        int rc = batched_chunk<T>(c, c->step, ns);
        if (rc != SS_OK) return rc;
        c->step += ns;
        left -= ns;
    }
    return SS_OK;
}

// ------------------------------------------------------------- window ----
void free_window(ss_ctx* c) {
    auto& w = c->win;
    void* ptrs[] = {w.tape, w.series, w.ckR, w.ckA, w.ckS, w.ckZ, w.snR, w.snA, w.snS, w.snZ,
                    w.xbar, w.ybar, w.scratch, w.Rb, w.Ab, w.grad, w.wgt};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    w = ss_ctx::Window();
}

int copy_state(ss_ctx* c, const Elem& e, void* dR, void* dA, int32_t* dS, int32_t* dZ, const void* sR,
               const void* sA, const int32_t* sS, const int32_t* sZ) {
    const size_t ts = tsize(c);
    SS_CUDA(c, cudaMemcpyAsync(dR, sR, (size_t)e.M * 3 * e.NP * ts, cudaMemcpyDeviceToDevice, c->stream));
    SS_CUDA(c, cudaMemcpyAsync(dA, sA, (size_t)e.M * 3 * e.NP * ts, cudaMemcpyDeviceToDevice, c->stream));
    SS_CUDA(c, cudaMemcpyAsync(dS, sS, (size_t)e.M * e.NP * sizeof(int32_t), cudaMemcpyDeviceToDevice, c->stream));
    SS_CUDA(c, cudaMemcpyAsync(dZ, sZ, (size_t)e.M * sizeof(int32_t), cudaMemcpyDeviceToDevice, c->stream));
    return SS_OK;
}

// steps of checkpoint segment seg (the last one may be shorter)
int seg_len(const ss_ctx* c, int seg) {
    const long long left = c->win.n - (long long)seg * c->win.ce;
    return (int)std::min<long long>(c->win.ce, left);
}

template <typename T>
int launch_adjoint(ss_ctx* c, Elem& e, int seg) {
    auto& w = c->win;
    const size_t ts = sizeof(T);
    ssk::AdjArgs a{};
    a.snapR = w.snR;
    a.snapA = w.snA;
    a.snapS = w.snS;
    a.snapZ = w.snZ;
    a.tape = w.tape + (size_t)seg * w.ce * e.M * e.NP;
    a.xbar = static_cast<char*>(w.xbar) + (size_t)seg * w.ce * e.M * 3 * ts;
    a.ybar = static_cast<char*>(w.ybar) + (size_t)seg * w.ce * e.M * 3 * ts;
    a.Rb = w.Rb;
    a.Ab = w.Ab;
    a.grad = w.grad;
    a.M = e.M;
    a.N = e.N;
    a.ns = seg_len(c, seg);
    a.t0 = w.t_start + (long long)seg * w.ce;
    a.key0 = (uint32_t)c->seed;
    a.key1 = (uint32_t)(c->seed >> 32);
    a.chain_base = e.chain_base;
    a.destroy_new = c->P.destroy_new;
    a.create_mode = c->P.create_mode;
    a.zmax = e.zmax;
    // (snapshots and tape have the same columns in every layout; 8 x 2 would round
    // the sums of a gradient otherwise than 16 x 1)
    const bool two = e.W == 8 && e.B == 2;
    const int W = two ? 16 : e.W, B = two ? 1 : e.B;
    const int smem = kWarpsPerCta * 32 * B * (int)(2 * sizeof(ssk::Pos<T>) + sizeof(ssk::SlotRec<T>) + 8);
    const void* kern = sizeof(T) == 8 ? ssk::adjoint_fn_f64(W, B) : ssk::adjoint_fn_f32(W, B);
    if (!kern) return fail(c, SS_EINVAL, "no adjoint kernel for this layout");
    SS_CUDA(c, allow_smem(kern, smem));
    const int ctas = (e.M + chains_per_cta(W) - 1) / chains_per_cta(W);
    ssk::StepConst<T> sc = step_const<T>(c, e.N);
    void* args[] = {(void*)&a, (void*)&sc};
    SS_CUDA(c, cudaLaunchKernel(kern, dim3(ctas), dim3(kThreads), args, smem, c->stream));
    c->launches++;
    return SS_OK;
}

template <typename T>
int window_backward_t(ss_ctx* c, const double* dL_dG, double grad[3]) {
    auto& w = c->win;
    Elem& e = c->el[0];
    const int L = c->levels;
    const double kT = c->P.kT;
    // weights of the later x origin products of each (level, lag) slot, TOTAL channel
    std::vector<T> wg((size_t)L * 16, T(0));
    for (int l = 0; l < L; ++l)
        for (int k = (l == 0 ? 0 : 8); k < 16; ++k) {
            const long long cnt = std::max(0ll, (w.n >> l) - k);
            if (cnt > 0 && dL_dG[l * 16 + k] != 0.0)
                wg[(size_t)l * 16 + k] = T(dL_dG[l * 16 + k] / (3.0 * e.M * e.N * kT * kT * (double)cnt));
        }
    SS_CUDA(c, cudaMemcpyAsync(w.wgt, wg.data(), sizeof(T) * wg.size(), cudaMemcpyHostToDevice, c->stream));
    {
        // correlator adjoint: block means per level, per-block lag sums, per-sample sums
        const long long P = 3ll * e.M, n = w.n, cap = 2 * (n + 1) * P;
        T* X = reinterpret_cast<T*>(w.scratch);
        T* Y = X + cap;
        T* CX = Y + cap;
        T* CY = CX + cap;
        const T* wt = reinterpret_cast<const T*>(w.wgt);
        const int thr = 256;
        auto blocks = [&](long long items) { return (unsigned)((items + thr - 1) / thr); };
        ssk::adj_level0_kernel<T><<<blocks(n * P), thr, 0, c->stream>>>(static_cast<const T*>(w.series), n, e.M, X, Y);
        SS_CUDA(c, cudaGetLastError());
        c->launches++;
        long long off = 0;
        for (int l = 0; l < L && (n >> l) > 0; ++l) {
            const long long nl = n >> l;
            if (l > 0) {
                ssk::adj_level_mean_kernel<T><<<blocks(nl * P), thr, 0, c->stream>>>(X, Y, off - (n >> (l - 1)), off,
                                                                                   nl, P);
                SS_CUDA(c, cudaGetLastError());
                c->launches++;
            }
            const unsigned grid = blocks(P) * (unsigned)((nl + ssk::kAdjBlock - 1) / ssk::kAdjBlock);
            if (l == 0)
                ssk::adj_block_sums_kernel<T, 0><<<grid, thr, 0, c->stream>>>(X + off * P, Y + off * P, CX + off * P,
                                                                              CY + off * P, nl, P, T(1), wt);
            else
                ssk::adj_block_sums_kernel<T, ssk::kP / 2><<<grid, thr, 0, c->stream>>>(
                    X + off * P, Y + off * P, CX + off * P, CY + off * P, nl, P, T(1.0 / (double)(1ll << l)),
                    wt + l * 16);
            SS_CUDA(c, cudaGetLastError());
            c->launches++;
            off += nl;
        }
        ssk::adj_sample_sums_kernel<T><<<blocks(P) * (unsigned)((n + ssk::kAdjBlock - 1) / ssk::kAdjBlock), thr, 0,
                                         c->stream>>>(CX, CY, n, P, L,
                                                                             static_cast<T*>(w.xbar),
                                                                             static_cast<T*>(w.ybar));
        SS_CUDA(c, cudaGetLastError());
        c->launches++;
    }
    const size_t ts = sizeof(T);
    SS_CUDA(c, cudaMemsetAsync(w.Rb, 0, (size_t)e.M * 3 * e.NP * ts, c->stream));
    SS_CUDA(c, cudaMemsetAsync(w.Ab, 0, (size_t)e.M * 3 * e.NP * ts, c->stream));
    SS_CUDA(c, cudaMemsetAsync(w.grad, 0, (size_t)e.M * 3 * sizeof(double), c->stream));
    const size_t stR = (size_t)e.M * 3 * e.NP * ts, stS = (size_t)e.M * e.NP * sizeof(int32_t);
    for (int seg = w.nseg - 1; seg >= 0; --seg) {
        // recompute the segment from its checkpoint with the recorded decisions,
        // keeping the state before every step
        int rc = copy_state(c, e, e.R, e.A, e.S, e.Z, static_cast<char*>(w.ckR) + seg * stR,
                            static_cast<char*>(w.ckA) + seg * stR,
                            reinterpret_cast<int32_t*>(reinterpret_cast<char*>(w.ckS) + seg * stS),
                            w.ckZ + (size_t)seg * e.M);
        if (rc != SS_OK) return rc;
        c->opt_tape_mode = 2;
        c->opt_snap = true;
        c->opt_corr_off = true;
        c->opt_snap_t0 = w.t_start + (long long)seg * w.ce;
        rc = launch_chunk<T>(c, e, 0, e.M, c->opt_snap_t0, seg_len(c, seg), c->stream);
        c->opt_tape_mode = 0;
        c->opt_snap = false;
        c->opt_corr_off = false;
        if (rc != SS_OK) return rc;
        rc = launch_adjoint<T>(c, e, seg);
        if (rc != SS_OK) return rc;
    }
    // the live state is the window's final state again
    int rc = copy_state(c, e, e.R, e.A, e.S, e.Z, static_cast<char*>(w.ckR) + w.nseg * stR,
                        static_cast<char*>(w.ckA) + w.nseg * stR,
                        reinterpret_cast<int32_t*>(reinterpret_cast<char*>(w.ckS) + w.nseg * stS),
                        w.ckZ + (size_t)w.nseg * e.M);
    if (rc != SS_OK) return rc;
    std::vector<double> g((size_t)e.M * 3);
    SS_CUDA(c, cudaMemcpyAsync(g.data(), w.grad, sizeof(double) * g.size(), cudaMemcpyDeviceToHost, c->stream));
    SS_CUDA(c, cudaStreamSynchronize(c->stream));
    grad[0] = grad[1] = grad[2] = 0.0;
    for (int m = 0; m < e.M; ++m)
        for (int k = 0; k < 3; ++k) grad[k] += g[(size_t)m * 3 + k];
    return SS_OK;
}

}  // namespace

// ================================================================== C ABI ====
namespace {
// Work enqueued on `later` from now on runs after what is enqueued on `first`.
int order_streams(ss_ctx* c, cudaStream_t first, cudaStream_t later) {
    if (first == later) return SS_OK;
    if (!c->xev) SS_CUDA(c, cudaEventCreateWithFlags(&c->xev, cudaEventDisableTiming));
    SS_CUDA(c, cudaEventRecord(c->xev, first));
    SS_CUDA(c, cudaStreamWaitEvent(later, c->xev, 0));
    return SS_OK;
}

// warps per SM of the chain kernel's launches over an element
template <typename T>
int resident_warps(const ss_ctx* c, const Elem& e, bool flow) {
    const bool heun = c->P.integrator == SS_HEUN, series = c->levels > 0;
    const int nlog = logs_per_launch<T>(c, e, flow, heun, series);
    const bool alt = second_form<T>(e.M, e.W, e.B, c->sms, nlog, flow, heun, series);
    return chunk_resident<T>(e.W, e.B, nlog, flow, heun, series, alt);
}

constexpr int kSideStreams = 7;    // beside the context's own
// Parts of one element's chains that run side by side: for runs long enough to pay
// for the launches (256 steps), of more warps than the chip holds at once.  Four
// parts fill the last wave best (16384 x 8: 4.49 -> 4.02 ms, two parts 4.20; 4096 x
// 80: 7.41 -> 6.74, 6.72); from eight waves on the tail is small and two parts let
// the correlator overlap (65536 x 32: 34.7 -> 34.4 ms, four parts 34.6).
int run_parts(const ss_ctx* c, const Elem& e, long long n_steps) {
    const bool flow = flow_in_window(e, c->step, (int)std::min<long long>(n_steps, 1 << 30));
    const int per_sm = c->prec == SS_FP64 ? resident_warps<double>(c, e, flow) : resident_warps<float>(c, e, flow);
    const long long warps = ((long long)e.M * e.W + 31) / 32, slots = (long long)per_sm * c->sms;
    if (n_steps < 256 || warps <= slots) return 1;
    return std::min(e.slices, warps < 8 * slots ? 4 : 2);
}

constexpr int kSideMinSteps = 32;  // steps of a call from which several elements run side by side

// Work enqueued on the first lanes - 1 side streams from now on runs after what is
// enqueued on the context's stream.
int fork_streams(ss_ctx* c, int lanes) {
    if (lanes <= 1) return SS_OK;
    while ((int)c->side.size() < lanes - 1) {
        cudaStream_t s = nullptr;
        cudaEvent_t ev = nullptr;
        SS_CUDA(c, cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        c->side_ev.push_back(ev);
        SS_CUDA(c, cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
        c->side.push_back(s);
    }
    if (!c->xev) SS_CUDA(c, cudaEventCreateWithFlags(&c->xev, cudaEventDisableTiming));
    SS_CUDA(c, cudaEventRecord(c->xev, c->stream));
    for (int k = 0; k < lanes - 1; ++k) SS_CUDA(c, cudaStreamWaitEvent(c->side[k], c->xev, 0));
    return SS_OK;
}
// And the context's stream goes on after what is enqueued on them.
int join_streams(ss_ctx* c, int lanes) {
    for (int k = 0; k < lanes - 1 && k < (int)c->side.size(); ++k) {
        SS_CUDA(c, cudaEventRecord(c->side_ev[k], c->side[k]));
        SS_CUDA(c, cudaStreamWaitEvent(c->stream, c->side_ev[k], 0));
    }
    return SS_OK;
}
}  // namespace

extern "C" {

int ss_create(ss_ctx** out, const ss_element* elems, int n_elems, int precision, uint64_t seed,
              void* cuda_stream) {
    if (!out) return SS_EINVAL;
    *out = nullptr;
    if (!elems || n_elems <= 0) return SS_EINVAL;
    if (precision != SS_FP32 && precision != SS_FP64) return SS_EINVAL;
    long long total = 0;
    for (int i = 0; i < n_elems; ++i) {
        if (elems[i].n_chains <= 0 || elems[i].n_beads < 2 || elems[i].n_beads > SS_MAX_BEADS) return SS_EINVAL;
        total += elems[i].n_chains;
    }
    if (total > 0xFFFFFFFFll) return SS_EINVAL;
    ss_ctx* c = new (std::nothrow) ss_ctx();
    if (!c) return SS_ENOMEM;
    c->stream = static_cast<cudaStream_t>(cuda_stream);
    c->prec = precision;
    c->seed = seed;
    uint32_t base = 0;
    for (int i = 0; i < n_elems; ++i) {
        Elem e;
        e.M = elems[i].n_chains;
        e.N = elems[i].n_beads;
        layout_for(e.M, e.N, precision, SS_EULER, &e.W, &e.B);
        e.NP = ssk::row_stride(e.N);
        e.chain_base = base;
        base += (uint32_t)e.M;
        c->el.push_back(e);
    }
    if (cudaMalloc(&c->counters, ssk::kCounterCopies * 8 * sizeof(unsigned long long)) != cudaSuccess ||
        cudaMalloc(&c->status, sizeof(int32_t)) != cudaSuccess) {
        ss_destroy(c);
        return SS_ECUDA;
    }
    if (cudaGetDevice(&c->dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, c->dev) != cudaSuccess) {
        ss_destroy(c);
        return SS_ECUDA;
    }
    cudaMemset(c->counters, 0, ssk::kCounterCopies * 8 * sizeof(unsigned long long));
    cudaMemset(c->status, 0, sizeof(int32_t));
    *out = c;
    return SS_OK;
}

int ss_set_params(ss_ctx* c, const ss_params* pin) {
    if (!c || !pin) return SS_EINVAL;
    ss_params p = *pin;
    if (p.N0 == 0) p.N0 = 4.0;
    if (p.Ns == 0) p.Ns = 0.5;
    if (p.zeta_s == 0) p.zeta_s = 0.1;
    if (p.dt == 0) p.dt = 0.01;
    if (p.b == 0) p.b = 1.0;
    if (p.kT == 0) p.kT = 1.0;
    if (p.zeta == 0) p.zeta = 1.0;
    if (p.recenter_every == 0) p.recenter_every = 100;
    if (p.corr_levels == 0) p.corr_levels = 24;
    if (p.groups == 0) p.groups = 32;
    if (p.chunk_steps == 0) p.chunk_steps = 1024;
    if (!(p.N0 > 0) || std::isnan(p.N0)) return fail(c, SS_EINVAL, "N0 must be > 0 (inf allowed)");
    if (!finite_pos(p.Ns) || !finite_pos(p.zeta_s) || !finite_pos(p.dt) || !finite_pos(p.b) ||
        !finite_pos(p.kT) || !finite_pos(p.zeta))
        return fail(c, SS_EINVAL, "Ns, zeta_s, dt, b, kT, zeta must be finite and > 0");
    const double kb = p.k_b > 0 ? p.k_b : 3.0 * p.kT / (p.b * p.b);
    const double ks = p.k_s > 0 ? p.k_s : 3.0 * p.kT / (p.Ns * p.b * p.b);
    if (!finite_pos(kb) || !finite_pos(ks)) return fail(c, SS_EINVAL, "k_b, k_s must be finite and > 0");
    if (!(p.dt * (4.0 * kb + ks) / p.zeta < 2.0))
        return fail(c, SS_EINVAL, "Euler step unstable: dt (4 k_b + k_s) / zeta must be < 2");
    if (p.create_mode != 0 && p.create_mode != 1) return fail(c, SS_EINVAL, "create_mode must be 0 or 1");
    if (p.corr_tt != 0 && p.corr_tt != 1) return fail(c, SS_EINVAL, "corr_tt must be 0 or 1");
    if (p.integrator != SS_EULER && p.integrator != SS_HEUN)
        return fail(c, SS_EINVAL, "integrator must be SS_EULER or SS_HEUN");
    if (p.destroy_new != 0 && p.destroy_new != 1) return fail(c, SS_EINVAL, "destroy_new must be 0 or 1");
    if (p.corr_levels > SS_MAX_LEVELS) return fail(c, SS_EINVAL, "corr_levels must be <= 32");
    if (p.groups < 1 || p.chunk_steps < 1 || p.log_every < 0 || p.max_logs < 0)
        return fail(c, SS_EINVAL, "groups, chunk_steps must be >= 1; log_every, max_logs >= 0");
    if (p.log_every > 0 && p.max_logs <= 0) return fail(c, SS_EINVAL, "log_every > 0 needs max_logs > 0");
    for (const Elem& e : c->el) {
        const int zm = p.z_max > 0 ? p.z_max : default_zmax(e.N);
        if (zm < 1 || zm > std::min(e.N, SS_MAX_SLOTS)) return fail(c, SS_EINVAL, "z_max must be in 1..min(N, 64)");
    }
    if (c->counters) cudaStreamSynchronize(c->stream);
    for (Elem& e : c->el) free_elem(e);
    free_logs(c);
    free_batched(c);
    free_window(c);
    c->P = p;
    c->k_b = kb;
    c->k_s = ks;
    c->levels = p.corr_levels > 0 ? p.corr_levels : 0;
    c->tuned = false;
    c->step = 0;
    c->initialized = false;
    // with the correlator on, a launch covers at most kCorrMaxSteps steps
    if (c->levels > 0) c->P.chunk_steps = std::min(c->P.chunk_steps, ssk::kCorrMaxSteps);
    const size_t ts = tsize(c);
    for (Elem& e : c->el) {
        e.zmax = p.z_max > 0 ? p.z_max : default_zmax(e.N);
        layout_for(e.M, e.N, c->prec, p.integrator, &e.W, &e.B);
        e.slices = (e.M + ssk::kSliceChains - 1) / ssk::kSliceChains;
        e.groups = std::min(p.groups, e.slices);
        e.parts = ssk::corr_parts(e.M);
        SS_CUDA(c, cudaMalloc(&e.R, (size_t)e.M * 3 * e.NP * ts));
        SS_CUDA(c, cudaMalloc(&e.A, (size_t)e.M * 3 * e.NP * ts));
        SS_CUDA(c, cudaMalloc(&e.S, (size_t)e.M * e.NP * sizeof(int32_t)));
        SS_CUDA(c, cudaMalloc(&e.Z, (size_t)e.M * sizeof(int32_t)));
        SS_CUDA(c, cudaMemsetAsync(e.Z, 0, (size_t)e.M * sizeof(int32_t), c->stream));
        if (c->levels > 0) {
            SS_CUDA(c, cudaMalloc(&e.hist, (size_t)e.M * c->levels * 96 * ts));
            e.ser_cap = c->P.chunk_steps;
            SS_CUDA(c, cudaMalloc(&e.ser, (size_t)e.M * 6 * e.ser_cap * ts));
            SS_CUDA(c, cudaMalloc(&e.lev, (size_t)2 * (e.ser_cap / 4 + 1) * e.M * 6 * ts));
            SS_CUDA(c, cudaMalloc(&e.acc64, (size_t)e.slices * e.parts * c->levels * 96 * sizeof(double)));
            if (p.corr_tt)
                SS_CUDA(c, cudaMalloc(&e.acc64tt, (size_t)e.slices * e.parts * c->levels * 48 * sizeof(double)));
        }
        e.flow_dirty = true;
    }
    if (p.max_logs > 0) {
        for (const Elem& e : c->el) c->logs_n += (size_t)p.max_logs * e.groups * 14;
        SS_CUDA(c, cudaMalloc(&c->logs, c->logs_n * sizeof(double)));
        size_t off = 0;
        for (Elem& e : c->el) {
            e.logs = c->logs + off;
            off += (size_t)p.max_logs * e.groups * 14;
        }
    }
    SS_CUDA(c, cudaMemsetAsync(c->counters, 0, ssk::kCounterCopies * 8 * sizeof(unsigned long long), c->stream));
    SS_CUDA(c, cudaMemsetAsync(c->status, 0, sizeof(int32_t), c->stream));
    c->launches = 0;
    int rc = zero_observables(c);
    if (rc != SS_OK) return rc;
    c->have_params = true;
    return SS_OK;
}

int ss_set_flow(ss_ctx* c, int elem, int64_t from_step, const double kappa[9]) {
    if (!c || !kappa || from_step < 0) return SS_EINVAL;
    for (int i = 0; i < 9; ++i)
        if (!std::isfinite(kappa[i])) return fail(c, SS_EINVAL, "kappa must be finite");
    if (elem < -1 || elem >= (int)c->el.size()) return fail(c, SS_EINVAL, "bad element index");
    for (int i = 0; i < (int)c->el.size(); ++i) {
        if (elem >= 0 && i != elem) continue;
        Elem& e = c->el[i];
        size_t n = 0;
        while (n < e.kfrom.size() && e.kfrom[n] < from_step) ++n;
        e.kfrom.resize(n + 1);
        e.kap.resize(9 * (n + 1));
        e.kfrom[n] = from_step;
        for (int k = 0; k < 9; ++k) e.kap[9 * n + k] = kappa[k];
        e.flow_dirty = true;
    }
    c->graph_dirty = true;
    return SS_OK;
}

int ss_set_flow_table(ss_ctx* c, int n, const int32_t* elem, const int64_t* from_step, const double* kappa) {
    if (!c || n < 0 || (n > 0 && (!elem || !from_step || !kappa))) return SS_EINVAL;
    for (int i = 0; i < n; ++i) {
        if (elem[i] < 0 || elem[i] >= (int)c->el.size()) return fail(c, SS_EINVAL, "bad element index");
        if (i > 0 && elem[i] == elem[i - 1] && from_step[i] <= from_step[i - 1])
            return fail(c, SS_EINVAL, "flow table: steps must increase within an element");
    }
    for (int i = 0; i < n; ++i) {
        const int rc = ss_set_flow(c, elem[i], from_step[i], kappa + 9 * (size_t)i);
        if (rc != SS_OK) return rc;
    }
    return SS_OK;
}

int ss_set_batched(ss_ctx* c, int enable) {
    if (!c) return SS_EINVAL;
    c->batched = enable != 0;
    c->graph_dirty = true;
    if (!c->batched) {  // back to the per-element kernels' layouts (same padded stride)
        for (Elem& e : c->el) layout_for(e.M, e.N, c->prec, c->P.integrator, &e.W, &e.B);
        c->tuned = false;
    }
    return SS_OK;
}

int ss_run(ss_ctx* c, int64_t n_steps) {
    if (!c) return SS_EINVAL;
    NvtxRange range("ss_run");
    if (!c->have_params) return fail(c, SS_ESTATE, "ss_set_params must precede ss_run");
    if (n_steps < 0) return fail(c, SS_EINVAL, "n_steps must be >= 0");
    if (c->step + n_steps > 0xFFFFFFFFll) return fail(c, SS_EOVERFLOW, "step counter would pass 2^32");
    const ss_params& p = c->P;
    if (p.log_every > 0) {
        const long long nlog = (c->step + n_steps) / p.log_every - c->log_m0;
        if (nlog > p.max_logs) return fail(c, SS_EINVAL, "stress log capacity (max_logs) exceeded");
    }
    if (const int rl = logs_change(c)) return rl;
    for (Elem& e : c->el) {
        int rc = upload_flow(c, e);
        if (rc != SS_OK) return rc;
    }
    if (!c->initialized) {
        for (Elem& e : c->el) {
            int rc = c->prec == SS_FP64 ? launch_init<double>(c, e) : launch_init<float>(c, e);
            if (rc != SS_OK) return rc;
        }
        c->initialized = true;
    }
    if (c->batched) {
        if (c->levels > 0) return fail(c, SS_EINVAL, "batched mode keeps stress logs only: set corr_levels < 0");
        if (p.integrator != SS_EULER) return fail(c, SS_EINVAL, "batched mode runs the Euler-Maruyama integrator");
        return c->prec == SS_FP64 ? batched_run<double>(c, n_steps) : batched_run<float>(c, n_steps);
    }
    // Several elements run side by side, and so do parts of a large one: one after
    // another, launches leave the SMs idle behind their last wave of CTAs (six
    // ensembles of 4096 x 40 fill 0.84 of a wave each, 16384 x 8 1.12), and the
    // correlator, bound by memory, would run alone instead of beside the chain
    // kernel.  A unit of work stays on one stream, so its launches keep their order.
    // Calls of a few steps are launch-bound and stay on one stream, as do runs whose
    // launches are timed.
    struct Unit {
        Elem* e;
        int m0, m1;
    };
    std::vector<Unit> units;
    const bool side = n_steps >= kSideMinSteps && !c->timing;
    for (Elem& e : c->el) {
        const int parts = side && c->el.size() == 1 ? run_parts(c, e, n_steps) : 1;
        const int sc = ssk::kSliceChains;
        for (int k = 0; k < parts; ++k) {
            const int s0 = (int)((long long)e.slices * k / parts), s1 = (int)((long long)e.slices * (k + 1) / parts);
            units.push_back({&e, s0 * sc, std::min(e.M, s1 * sc)});
        }
    }
    const int n_units = (int)units.size();
    const int lanes = side ? std::min(n_units, kSideStreams + 1) : 1;
    int rc = fork_streams(c, lanes);
    long long left = n_steps;
    while (rc == SS_OK && left > 0) {
        const int ns = (int)std::min<long long>(left, p.chunk_steps);
        for (int i = 0; rc == SS_OK && i < n_units; ++i) {
            const Unit& u = units[i];
            const cudaStream_t st = i % lanes == 0 ? c->stream : c->side[i % lanes - 1];
            rc = c->prec == SS_FP64 ? launch_chunk<double>(c, *u.e, u.m0, u.m1, c->step, ns, st)
                                    : launch_chunk<float>(c, *u.e, u.m0, u.m1, c->step, ns, st);
        }
        if (rc != SS_OK) break;
        c->step += ns;
        if (c->levels > 0) c->nsamp += ns;
        left -= ns;
    }
    const int rj = join_streams(c, lanes);
    return rc != SS_OK ? rc : rj;
}

int ss_stress(ss_ctx* c, int elem, double* t, double* mean, double* sem, int cap, int* n_out) {
    Elem* e = elem_at(c, elem);
    if (!e || cap < 0) return fail(c, SS_EINVAL, "bad element or capacity");
    if (!c->have_params) return fail(c, SS_ESTATE, "no parameters");
    const ss_params& p = c->P;
    const int n = p.log_every > 0 ? (int)std::min<long long>(c->step / p.log_every - c->log_m0, p.max_logs) : 0;
    if (n_out) *n_out = n;
    if (n == 0 || cap == 0) return SS_OK;
    const std::vector<int> gsz = group_sizes(*e);
    const double* L = nullptr;
    const int rc = read_logs(c, *e, n, &L);
    if (rc != SS_OK) return rc;
    for (int i = 0; i < std::min(n, cap); ++i) {
        if (t) t[i] = (double)((c->log_m0 + 1 + i) * p.log_every) * p.dt;
        for (int k = 0; k < 6; ++k) {
            double tot = 0.0, gm = 0.0, gm2 = 0.0;
            for (int g = 0; g < e->groups; ++g) {
                const double sg = L[((size_t)i * e->groups + g) * 14 + k];
                tot += sg;
                const double mg = sg / gsz[g];
                gm += mg;
                gm2 += mg * mg;
            }
            if (mean) mean[i * 6 + k] = tot / e->M;
            if (sem) {
                const int G = e->groups;
                const double mu = gm / G;
                sem[i * 6 + k] = G > 1 ? std::sqrt(std::max(0.0, (gm2 - G * mu * mu) / (G - 1)) / G) : 0.0;
            }
        }
    }
    return SS_OK;
}

int ss_correlator(ss_ctx* c, int elem, int channel, double* t, double* G, double* sem, int cap, int* n_out) {
    Elem* e = elem_at(c, elem);
    if (!e || cap < 0) return fail(c, SS_EINVAL, "bad element or capacity");
    if (channel < SS_CH_AUTO || channel > SS_CH_VIRTUAL) return fail(c, SS_EINVAL, "bad channel");
    if (!c->have_params || c->levels <= 0) return fail(c, SS_ESTATE, "correlator not enabled");
    const bool tt = channel == SS_CH_TT || channel == SS_CH_VIRTUAL;
    if (tt && !e->acc64tt) return fail(c, SS_ESTATE, "channel TT needs corr_tt = 1");
    const int L = c->levels, NG = e->groups;
    int n_slots = 0;  // lags with at least one product: level 0 lags 0..15, level l >= 1 lags 8..15
    for (int l = 0; l < L; ++l)
        for (int k = (l == 0 ? 0 : 8); k < 16; ++k) n_slots += (c->nsamp >> l) - k > 0;
    if (n_out) *n_out = n_slots;
    if (cap == 0 || (!t && !G && !sem)) return SS_OK;  // a size query reads nothing from the device
    std::vector<double> acc, acc_tt;
    int rc = group_corr<96>(c, *e, e->acc64, acc);
    if (rc != SS_OK) return rc;
    if (tt) {
        rc = group_corr<48>(c, *e, e->acc64tt, acc_tt);
        if (rc != SS_OK) return rc;
    }
    const std::vector<int> gsz = group_sizes(*e);
    const double norm = (double)e->N * c->P.kT * c->P.kT;
    int n = 0;
    for (int l = 0; l < L; ++l)
        for (int k = (l == 0 ? 0 : 8); k < 16; ++k) {
            const long long cnt = std::max(0ll, (c->nsamp >> l) - k);
            if (cnt <= 0) continue;
            double tot = 0.0, gm = 0.0, gm2 = 0.0;
            for (int g = 0; g < NG; ++g) {
                double v = 0.0;
                for (int d = 0; d < 3; ++d) {
                    const double* base = &acc[((((size_t)g * L + l) * 16 + k) * 2) * 3];
                    const double auto_ = base[d], total = base[3 + d];
                    const double ttv = tt ? acc_tt[(((size_t)g * L + l) * 16 + k) * 3 + d] : 0.0;
                    switch (channel) {
                        case SS_CH_AUTO: v += auto_; break;
                        case SS_CH_CROSS: v += total - auto_; break;
                        case SS_CH_TOTAL: v += total; break;
                        case SS_CH_TT: v += ttv; break;
                        default: v += ttv - total; break;  // SS_CH_VIRTUAL
                    }
                }
                v /= 3.0;
                tot += v;
                const double mg = v / ((double)cnt * gsz[g] * norm);
                gm += mg;
                gm2 += mg * mg;
            }
            if (n < cap) {
                if (t) t[n] = (double)((long long)k << l) * c->P.dt;
                if (G) G[n] = tot / ((double)cnt * e->M * norm);
                if (sem) {
                    const double mu = gm / NG;
                    sem[n] = NG > 1 ? std::sqrt(std::max(0.0, (gm2 - NG * mu * mu) / (NG - 1)) / NG) : 0.0;
                }
            }
            ++n;
        }
    if (n_out) *n_out = n;
    return SS_OK;
}

int ss_destroy(ss_ctx* c) {
    if (!c) return SS_OK;
    if (c->stream || c->counters) cudaStreamSynchronize(c->stream);
    for (auto& pr : c->events) {
        cudaEventDestroy(pr.first);
        cudaEventDestroy(pr.second);
    }
    for (Elem& e : c->el) free_elem(e);
    free_logs(c);
    free_batched(c);
    free_window(c);
    if (c->counters) cudaFree(c->counters);
    if (c->status) cudaFree(c->status);
    if (c->stage) cudaFree(c->stage);
    if (c->xev) cudaEventDestroy(c->xev);
    for (cudaStream_t s : c->side) cudaStreamDestroy(s);
    for (cudaEvent_t ev : c->side_ev) cudaEventDestroy(ev);
    delete c;
    return SS_OK;
}

const char* ss_last_error(const ss_ctx* c) {
    if (!c) return "no context";
    return c->err.c_str();
}

int ss_get_state(ss_ctx* c, int elem, double* R, int32_t* Z, int32_t* S, double* A) {
    Elem* e = elem_at(c, elem);
    if (!e) return fail(c, SS_EINVAL, "bad element");
    if (!c->have_params) return fail(c, SS_ESTATE, "no parameters");
    return c->prec == SS_FP64 ? get_state_t<double>(c, *e, R, Z, S, A) : get_state_t<float>(c, *e, R, Z, S, A);
}

int ss_set_state(ss_ctx* c, int elem, const double* R, const int32_t* Z, const int32_t* S, const double* A) {
    Elem* e = elem_at(c, elem);
    if (!e || !R || !Z || !S || !A) return fail(c, SS_EINVAL, "bad element or NULL array");
    if (!c->have_params) return fail(c, SS_ESTATE, "ss_set_params must precede ss_set_state");
    int rc = c->prec == SS_FP64 ? set_state_t<double>(c, *e, R, Z, S, A) : set_state_t<float>(c, *e, R, Z, S, A);
    if (rc != SS_OK) return rc;
    // every element must hold a state before stepping: sample the others once
    if (!c->initialized) {
        for (int i = 0; i < (int)c->el.size(); ++i) {
            if (i == elem) continue;
            rc = c->prec == SS_FP64 ? launch_init<double>(c, c->el[i]) : launch_init<float>(c, c->el[i]);
            if (rc != SS_OK) return rc;
        }
        c->initialized = true;
    }
    return SS_OK;
}

// ---- the state through caller-owned device memory, the Z histogram
int ss_get_state_dev(ss_ctx* c, int elem, double* R, int32_t* Z, int32_t* S, double* A, void* cuda_stream) {
    Elem* e = elem_at(c, elem);
    if (!e) return fail(c, SS_EINVAL, "bad element");
    if (!c->have_params) return fail(c, SS_ESTATE, "no parameters");
    if (!R && !Z && !S && !A) return SS_OK;
    const int width = std::max(e->N, e->zmax);
    const unsigned blocks = (unsigned)(((long long)e->M * width + 255) / 256);
    if (c->prec == SS_FP64)
        ssk::state_export_kernel<double><<<blocks, 256, 0, c->stream>>>(
            static_cast<const double*>(e->R), static_cast<const double*>(e->A), e->S, e->Z, e->M, e->N, e->zmax,
            e->NP, R, A, S, Z);
    else
        ssk::state_export_kernel<float><<<blocks, 256, 0, c->stream>>>(
            static_cast<const float*>(e->R), static_cast<const float*>(e->A), e->S, e->Z, e->M, e->N, e->zmax,
            e->NP, R, A, S, Z);
    SS_CUDA(c, cudaGetLastError());
    c->launches++;
    const cudaStream_t user = cuda_stream ? static_cast<cudaStream_t>(cuda_stream) : c->stream;
    return order_streams(c, c->stream, user);
}

int ss_set_state_dev(ss_ctx* c, int elem, const double* R, const int32_t* Z, const int32_t* S, const double* A,
                     void* cuda_stream) {
    Elem* e = elem_at(c, elem);
    if (!e || !R || !Z || !S || !A) return fail(c, SS_EINVAL, "bad element or NULL array");
    if (!c->have_params) return fail(c, SS_ESTATE, "ss_set_params must precede ss_set_state_dev");
    const cudaStream_t user = cuda_stream ? static_cast<cudaStream_t>(cuda_stream) : c->stream;
    int rc = order_streams(c, user, c->stream);
    if (rc != SS_OK) return rc;
    rc = stage_at_least(c, sizeof(int));
    if (rc != SS_OK) return rc;
    int* dF = static_cast<int*>(c->stage);
    rc = c->prec == SS_FP64 ? check_convert_state<double>(c, *e, R, A, S, Z, dF)
                            : check_convert_state<float>(c, *e, R, A, S, Z, dF);
    if (rc != SS_OK) return rc;
    if (!c->initialized) {
        for (int i = 0; i < (int)c->el.size(); ++i) {
            if (i == elem) continue;
            rc = c->prec == SS_FP64 ? launch_init<double>(c, c->el[i]) : launch_init<float>(c, c->el[i]);
            if (rc != SS_OK) return rc;
        }
        c->initialized = true;
    }
    return SS_OK;
}

int ss_zhist(ss_ctx* c, int elem, int64_t* hist, int cap, int* n_out) {
    Elem* e = elem_at(c, elem);
    if (!e || !n_out || cap < 0) return fail(c, SS_EINVAL, "bad element, NULL n_out or negative cap");
    if (!c->have_params) return fail(c, SS_ESTATE, "no parameters");
    const int nb = e->zmax + 1;
    *n_out = nb;
    if (!hist || cap == 0) return SS_OK;
    if (!c->initialized) return fail(c, SS_ESTATE, "no state yet: ss_run or ss_set_state first");
    int rc = stage_at_least(c, (size_t)(nb + 1) * sizeof(unsigned long long));
    if (rc != SS_OK) return rc;
    unsigned long long* dh = static_cast<unsigned long long*>(c->stage);
    SS_CUDA(c, cudaMemsetAsync(dh, 0, (size_t)(nb + 1) * sizeof(unsigned long long), c->stream));
    const int blocks = std::max(1, std::min((e->M + 255) / 256, 1024));
    ssk::zhist_kernel<<<blocks, 256, 0, c->stream>>>(e->Z, e->M, nb, dh);
    SS_CUDA(c, cudaGetLastError());
    c->launches++;
    std::vector<unsigned long long> h(nb + 1);
    SS_CUDA(c, cudaMemcpyAsync(h.data(), dh, h.size() * sizeof(unsigned long long), cudaMemcpyDeviceToHost,
                               c->stream));
    SS_CUDA(c, cudaStreamSynchronize(c->stream));
    for (int z = 0; z < std::min(cap, nb); ++z) hist[z] = (int64_t)h[z];
    if (h[nb] != 0) return fail(c, SS_EOVERFLOW, "a chain's Z is outside 0..z_max (see ss_status)");
    return SS_OK;
}

int ss_set_chain_offset(ss_ctx* c, uint32_t offset) {
    if (!c) return SS_EINVAL;
    long long base = offset;
    for (const Elem& e : c->el) base += e.M;
    if (base > 0xFFFFFFFFll) return fail(c, SS_EINVAL, "chain ids would pass 2^32");
    uint32_t b = offset;
    for (Elem& e : c->el) {
        e.chain_base = b;
        b += (uint32_t)e.M;
    }
    return SS_OK;
}

int ss_step_count(ss_ctx* c, int64_t* steps) {
    if (!c || !steps) return SS_EINVAL;
    *steps = c->step;
    return SS_OK;
}

int ss_set_step_count(ss_ctx* c, int64_t step) {
    if (!c) return SS_EINVAL;
    if (!c->have_params) return fail(c, SS_ESTATE, "no parameters");
    if (step < 0 || step > 0xFFFFFFFFll) return fail(c, SS_EINVAL, "step must be in 0..2^32");
    if (c->win.forward_done && !c->win.have_tape) return fail(c, SS_ESTATE, "window state inconsistent");
    c->step = step;
    return zero_observables(c);
}

int ss_reset_observables(ss_ctx* c) {
    if (!c) return SS_EINVAL;
    if (!c->have_params) return fail(c, SS_ESTATE, "no parameters");
    return zero_observables(c);
}

int ss_corr_sums(ss_ctx* c, int elem, double* acc, int* n_groups, int64_t* n_samples) {
    Elem* e = elem_at(c, elem);
    if (!e) return fail(c, SS_EINVAL, "bad element");
    if (!c->have_params || c->levels <= 0) return fail(c, SS_ESTATE, "correlator not enabled");
    std::vector<double> g;
    int rc = group_corr<96>(c, *e, e->acc64, g);
    if (rc != SS_OK) return rc;
    if (acc) std::memcpy(acc, g.data(), g.size() * sizeof(double));
    if (n_groups) *n_groups = e->groups;
    if (n_samples) *n_samples = c->nsamp;
    return SS_OK;
}

int ss_corr_sums_tt(ss_ctx* c, int elem, double* acc_tt, int* n_groups, int64_t* n_samples) {
    Elem* e = elem_at(c, elem);
    if (!e) return fail(c, SS_EINVAL, "bad element");
    if (!c->have_params || c->levels <= 0 || !e->acc64tt) return fail(c, SS_ESTATE, "channel TT not enabled");
    std::vector<double> g;
    int rc = group_corr<48>(c, *e, e->acc64tt, g);
    if (rc != SS_OK) return rc;
    if (acc_tt) std::memcpy(acc_tt, g.data(), g.size() * sizeof(double));
    if (n_groups) *n_groups = e->groups;
    if (n_samples) *n_samples = c->nsamp;
    return SS_OK;
}

int ss_log_sums(ss_ctx* c, int elem, int64_t* log_step, double* sums, int cap, int* n_out, int* n_groups) {
    Elem* e = elem_at(c, elem);
    if (!e || cap < 0) return fail(c, SS_EINVAL, "bad element or capacity");
    if (!c->have_params) return fail(c, SS_ESTATE, "no parameters");
    const ss_params& p = c->P;
    const int n = p.log_every > 0 ? (int)std::min<long long>(c->step / p.log_every - c->log_m0, p.max_logs) : 0;
    if (n_out) *n_out = n;
    if (n_groups) *n_groups = e->groups;
    const int k = std::min(n, cap);
    if (k > 0 && sums) {
        const double* L = nullptr;
        const int rc = read_logs(c, *e, k, &L);
        if (rc != SS_OK) return rc;
        std::memcpy(sums, L, (size_t)k * e->groups * 14 * sizeof(double));
    }
    if (log_step)
        for (int i = 0; i < k; ++i) log_step[i] = (c->log_m0 + 1 + i) * p.log_every;
    return SS_OK;
}

int ss_counters(ss_ctx* c, int64_t out[8]) {
    if (!c || !out) return SS_EINVAL;
    unsigned long long all[ssk::kCounterCopies][8], h[8] = {0};
    SS_CUDA(c, cudaMemcpyAsync(all, c->counters, sizeof(all), cudaMemcpyDeviceToHost, c->stream));
    SS_CUDA(c, cudaStreamSynchronize(c->stream));
    for (const auto& copy : all)
        for (int i = 0; i < 8; ++i) h[i] += copy[i];
    for (int i = 0; i < 5; ++i) out[i] = (int64_t)h[i];
    out[5] = c->launches;
    out[6] = (int64_t)h[6];
    out[7] = (int64_t)h[7];
    return SS_OK;
}

int ss_status(ss_ctx* c, int32_t* status) {
    if (!c || !status) return SS_EINVAL;
    SS_CUDA(c, cudaMemcpyAsync(status, c->status, sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
    SS_CUDA(c, cudaStreamSynchronize(c->stream));
    return SS_OK;
}

int ss_synchronize(ss_ctx* c) {
    if (!c) return SS_EINVAL;
    SS_CUDA(c, cudaStreamSynchronize(c->stream));
    return SS_OK;
}

int ss_kernel_timing(ss_ctx* c, int enable) {
    if (!c) return SS_EINVAL;
    c->timing = enable != 0;
    return SS_OK;
}

int ss_kernel_time(ss_ctx* c, double* chain_kernel_ms, int64_t* chain_launches) {
    if (!c) return SS_EINVAL;
    SS_CUDA(c, cudaStreamSynchronize(c->stream));
    double total = 0.0;
    for (auto& pr : c->events) {
        float ms = 0.0f;
        SS_CUDA(c, cudaEventElapsedTime(&ms, pr.first, pr.second));
        total += ms;
    }
    if (chain_kernel_ms) *chain_kernel_ms = total;
    if (chain_launches) *chain_launches = (int64_t)c->events.size();
    for (auto& pr : c->events) {
        cudaEventDestroy(pr.first);
        cudaEventDestroy(pr.second);
    }
    c->events.clear();
    return SS_OK;
}


int ss_window_forward(ss_ctx* c, int64_t n_steps, int checkpoint_every, int replay) {
    if (!c) return SS_EINVAL;
    NvtxRange range("ss_window_forward");
    if (!c->have_params) return fail(c, SS_ESTATE, "ss_set_params must precede a window");
    if (c->el.size() != 1) return fail(c, SS_EINVAL, "a differentiation window needs exactly one element");
    if (c->levels <= 0) return fail(c, SS_EINVAL, "a differentiation window needs the correlator (corr_levels > 0)");
    if (c->batched) return fail(c, SS_EINVAL, "a differentiation window runs on the per-element path");
    if (c->P.integrator != SS_EULER)
        return fail(c, SS_EINVAL, "differentiation windows differentiate the Euler-Maruyama step");
    if (checkpoint_every < 1 || n_steps < 1) return fail(c, SS_EINVAL, "n_steps, checkpoint_every must be >= 1");
    if (checkpoint_every > c->P.chunk_steps) return fail(c, SS_EINVAL, "checkpoint_every must be <= chunk_steps");
    Elem& e = c->el[0];
    for (double k : e.kap)
        if (k != 0.0) return fail(c, SS_EINVAL, "differentiation windows run without flow");
    if (c->step + n_steps > 0xFFFFFFFFll) return fail(c, SS_EOVERFLOW, "step counter would pass 2^32");
    auto& w = c->win;
    if (replay && !(w.have_tape && w.n == n_steps && w.ce == checkpoint_every))
        return fail(c, SS_ESTATE, "replay needs a recorded window of the same length");
    if (c->P.log_every > 0) {
        const long long ts = replay ? w.t_start : c->step;
        if ((ts + n_steps) / c->P.log_every - ts / c->P.log_every > c->P.max_logs)
            return fail(c, SS_EINVAL, "stress log capacity (max_logs) exceeded");
    }
    int rc = upload_flow(c, e);
    if (rc != SS_OK) return rc;
    if (!c->initialized) {
        rc = c->prec == SS_FP64 ? launch_init<double>(c, e) : launch_init<float>(c, e);
        if (rc != SS_OK) return rc;
        c->initialized = true;
    }
    const size_t ts = tsize(c);
    const size_t stR = (size_t)e.M * 3 * e.NP * ts, stS = (size_t)e.M * e.NP * sizeof(int32_t);
    // the buffers of a window of the same shape are kept (a fit evaluates one window
    // again and again; allocating them took 5 ms of a 2048-step window of 8192 chains)
    if (!replay && w.complete && w.n == n_steps && w.ce == checkpoint_every) {
        w.have_tape = w.forward_done = false;
    } else if (!replay) {
        free_window(c);
        w.n = n_steps;
        w.ce = checkpoint_every;
        w.nseg = (int)((n_steps + checkpoint_every - 1) / checkpoint_every);
        SS_CUDA(c, cudaMalloc(&w.tape, (size_t)n_steps * e.M * e.NP));
        SS_CUDA(c, cudaMalloc(&w.series, (size_t)n_steps * e.M * 6 * ts));
        SS_CUDA(c, cudaMalloc(&w.ckR, (w.nseg + 1) * stR));
        SS_CUDA(c, cudaMalloc(&w.ckA, (w.nseg + 1) * stR));
        SS_CUDA(c, cudaMalloc(&w.ckS, (w.nseg + 1) * stS));
        SS_CUDA(c, cudaMalloc(&w.ckZ, (size_t)(w.nseg + 1) * e.M * sizeof(int32_t)));
        SS_CUDA(c, cudaMalloc(&w.snR, (size_t)(w.ce + 1) * stR));
        SS_CUDA(c, cudaMalloc(&w.snA, (size_t)(w.ce + 1) * stR));
        SS_CUDA(c, cudaMalloc(&w.snS, (size_t)(w.ce + 1) * stS));
        SS_CUDA(c, cudaMalloc(&w.snZ, (size_t)(w.ce + 1) * e.M * sizeof(int32_t)));
        SS_CUDA(c, cudaMalloc(&w.xbar, (size_t)n_steps * e.M * 3 * ts));
        SS_CUDA(c, cudaMalloc(&w.ybar, (size_t)n_steps * e.M * 3 * ts));
        SS_CUDA(c, cudaMalloc(&w.scratch, (size_t)8 * (n_steps + 1) * e.M * 3 * ts));  // 4 level arrays of 2(n+1) rows
        SS_CUDA(c, cudaMalloc(&w.Rb, stR));
        SS_CUDA(c, cudaMalloc(&w.Ab, stR));
        SS_CUDA(c, cudaMalloc(&w.grad, (size_t)e.M * 3 * sizeof(double)));
        SS_CUDA(c, cudaMalloc(&w.wgt, (size_t)c->levels * 16 * sizeof(double)));
        w.complete = true;
    }
    c->logs_read = false;
    // a replayed window draws the noise of the recorded one: same step indices
    if (replay) c->step = w.t_start;
    rc = zero_observables(c);
    if (rc != SS_OK) return rc;
    w.t_start = c->step;
    for (int seg = 0; seg <= w.nseg; ++seg) {
        rc = copy_state(c, e, static_cast<char*>(w.ckR) + seg * stR, static_cast<char*>(w.ckA) + seg * stR,
                        reinterpret_cast<int32_t*>(reinterpret_cast<char*>(w.ckS) + seg * stS),
                        w.ckZ + (size_t)seg * e.M, e.R, e.A, e.S, e.Z);
        if (rc != SS_OK) return rc;
        if (seg == w.nseg) break;
        c->opt_tape_mode = replay ? 2 : 1;
        c->opt_series = true;
        const int len = seg_len(c, seg);
        rc = c->prec == SS_FP64 ? launch_chunk<double>(c, e, 0, e.M, c->step, len, c->stream)
                                : launch_chunk<float>(c, e, 0, e.M, c->step, len, c->stream);
        c->opt_tape_mode = 0;
        c->opt_series = false;
        if (rc != SS_OK) return rc;
        c->step += len;
        c->nsamp += len;
    }
    w.have_tape = true;
    w.forward_done = true;
    return SS_OK;
}

int ss_set_coefficients(ss_ctx* c, double k_b, double k_s, double zeta) {
    if (!c) return SS_EINVAL;
    if (!c->have_params) return fail(c, SS_ESTATE, "ss_set_params must precede ss_set_coefficients");
    if (!finite_pos(k_b) || !finite_pos(k_s) || !finite_pos(zeta))
        return fail(c, SS_EINVAL, "k_b, k_s, zeta must be finite and > 0");
    if (!(c->P.dt * (4.0 * k_b + k_s) / zeta < 2.0))
        return fail(c, SS_EINVAL, "Euler step unstable: dt (4 k_b + k_s) / zeta must be < 2");
    c->k_b = k_b;
    c->k_s = k_s;
    c->P.zeta = zeta;
    c->P.k_b = k_b;
    c->P.k_s = k_s;
    return SS_OK;
}

int ss_window_backward(ss_ctx* c, const double* dL_dG, double grad[3]) {
    if (!c || !dL_dG || !grad) return SS_EINVAL;
    if (!c->win.forward_done) return fail(c, SS_ESTATE, "ss_window_forward must precede ss_window_backward");
    NvtxRange range("ss_window_backward");
    return c->prec == SS_FP64 ? window_backward_t<double>(c, dL_dG, grad) : window_backward_t<float>(c, dL_dG, grad);
}
}  // extern "C"

// ====================================================== allocation-free run ===
// Working memory of ss_run_noalloc: one array per GPU for the life of the
// process.  In host code g_noalloc_scratch names a host-side stand-in, not a
// device address; the device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_noalloc_scratch[SS_NOALLOC_SCRATCH_BYTES];

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
unsigned char* g_noalloc_ptr[kMaxDevices] = {nullptr};

// Device address of the scratch array on the current device (looked up once).
int noalloc_scratch(unsigned char** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SS_ECUDA;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return SS_ECUDA;
        g_noalloc_ptr[dev] = static_cast<unsigned char*>(p);
    }
    *out = g_noalloc_ptr[dev];
    return SS_OK;
}

// Slice sums [slices][L][3][32] -> one output [L][16][2][3], slices added in order.
__global__ void noalloc_reduce_kernel(const double* acc64, int slices, int L, double* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L * 96) return;
    const int l = i / 96, r = i % 96, d = r / 32, cell = r % 32;
    double sum = 0.0;
    for (int sl = 0; sl < slices; ++sl) sum += acc64[((size_t)sl * L + l) * 96 + r];
    out[((l * 16 + (cell & 15)) * 2 + (cell >> 4)) * 3 + d] = sum;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

template <typename T>
int noalloc_launches(ss_ctx* c, int W, int B, const ss_params& p, int M, int N, int zmax, uint32_t chain_base, int64_t t0,
                     int64_t n_steps, void* R, void* A, int32_t* S, int32_t* Z, unsigned char* scr,
                     size_t off_hist, size_t off_ser, size_t off_lev, int ser_cap, size_t off_acc64, size_t off_cnt,
                     int32_t* status, const double* kappa, cudaStream_t st) {
    ssk::ChunkArgs a{};
    a.R = R;
    a.A = A;
    a.S = S;
    a.Z = Z;
    a.logs = nullptr;
    a.counters = reinterpret_cast<unsigned long long*>(scr + off_cnt);
    a.status = status;
    // the velocity gradient goes by value, in the kernel's arguments
    if (kappa) std::memcpy(a.kap0, kappa, sizeof(a.kap0));
    const bool flow = std::any_of(a.kap0, a.kap0 + 9, [](double k) { return k != 0.0; });
    a.M = M;
    a.N = N;
    a.zmax = zmax;
    a.create_mode = p.create_mode;
    a.destroy_new = p.destroy_new;
    a.log_every = 0;
    a.recenter_every = p.recenter_every;
    a.log_m0 = 0;
    a.max_logs = 0;
    a.groups = 1;
    a.slices = (M + ssk::kSliceChains - 1) / ssk::kSliceChains;
    a.key0 = (uint32_t)c->seed;
    a.key1 = (uint32_t)(c->seed >> 32);
    a.chain_base = chain_base;
    a.nlog_chunk = 0;
    if (c->levels > 0) {
        a.series = scr + off_ser;
        a.series_row0 = 0;
    }
    bool alt = false;
    if (sizeof(T) == 4 && ssk::has_second_form(W, B, false, flow)) {
        int dev = 0, sms = 1;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return SS_ECUDA;
        alt = second_form<T>(M, W, B, sms, 0, flow, false, c->levels > 0);
    }
    const void* kern = chunk_fn<T>(W, B, ssk::kWinOff, flow, false, c->levels > 0, alt);
    if (!kern) return SS_EINVAL;
    const int cpc = chains_per_cta(W);
    const int smem = chunk_smem<T>(W, B, 0, flow, false, c->levels > 0, alt);
    if (allow_smem(kern, smem) != cudaSuccess) return SS_ECUDA;
    ssk::StepConst<T> sc = step_const<T>(c, N);
    void* args[] = {(void*)&a, (void*)&sc};
    int64_t done = 0;
    while (done < n_steps) {
        const int ns = (int)std::min<int64_t>(n_steps - done, c->levels > 0 ? ser_cap : p.chunk_steps);
        a.t0 = t0 + done;
        a.nsteps = ns;
        if (cudaLaunchKernel(kern, dim3((M + cpc - 1) / cpc), dim3(kThreads), args, smem, st) != cudaSuccess)
            return SS_ECUDA;
        if (c->levels > 0 &&
            corr_launches<T>(static_cast<const T*>(a.series), 0, M, ssk::kSliceChains, ns, M, c->levels, done,
                             reinterpret_cast<T*>(scr + off_hist), reinterpret_cast<double*>(scr + off_acc64), nullptr,
                             reinterpret_cast<T*>(scr + off_lev), (size_t)(ser_cap / 2 + 1) * M * 6, st) < 0)
            return SS_ECUDA;
        done += ns;
    }
    return SS_OK;
}

}  // namespace

extern "C" int ss_run_noalloc(const ss_params* params, int precision, uint64_t seed, int32_t n_chains,
                              int32_t n_beads, uint32_t chain_base, int64_t t0, int64_t n_steps,
                              const double* kappa, void* R, void* A, int32_t* S, int32_t* Z, double* corr_out,
                              int32_t* status_out, void* cuda_stream) {
    if (!params || !R || !A || !S || !Z) return SS_EINVAL;
    if (precision != SS_FP32 && precision != SS_FP64) return SS_EINVAL;
    if (n_chains <= 0 || n_beads < 2 || n_beads > SS_MAX_BEADS || t0 < 0 || n_steps < 0) return SS_EINVAL;
    if ((long long)chain_base + n_chains > 0xFFFFFFFFll) return SS_EINVAL;
    if (t0 + n_steps > 0xFFFFFFFFll) return SS_EOVERFLOW;
    if (params->log_every != 0 || params->integrator != SS_EULER) return SS_EINVAL;
    if (kappa)
        for (int i = 0; i < 9; ++i)
            if (!std::isfinite(kappa[i])) return SS_EINVAL;
    // Parameter validation and defaults through a context that owns no device
    // memory (ss_set_params with no elements allocates nothing).
    ss_ctx c;
    c.prec = precision;
    c.seed = seed;
    Elem e;
    e.M = n_chains;
    e.N = n_beads;
    layout_for(n_chains, n_beads, precision, SS_EULER, &e.W, &e.B);
    e.NP = ssk::row_stride(e.N);
    c.el.push_back(e);
    {
        ss_params q = *params;
        // the validation of ss_set_params without its allocations
        if (q.N0 == 0) q.N0 = 4.0;
        if (q.Ns == 0) q.Ns = 0.5;
        if (q.zeta_s == 0) q.zeta_s = 0.1;
        if (q.dt == 0) q.dt = 0.01;
        if (q.b == 0) q.b = 1.0;
        if (q.kT == 0) q.kT = 1.0;
        if (q.zeta == 0) q.zeta = 1.0;
        if (q.recenter_every == 0) q.recenter_every = 100;
        if (q.corr_levels == 0) q.corr_levels = 24;
        if (q.chunk_steps == 0) q.chunk_steps = 1024;
        if (!(q.N0 > 0) || std::isnan(q.N0)) return SS_EINVAL;
        if (!finite_pos(q.Ns) || !finite_pos(q.zeta_s) || !finite_pos(q.dt) || !finite_pos(q.b) ||
            !finite_pos(q.kT) || !finite_pos(q.zeta))
            return SS_EINVAL;
        const double kb = q.k_b > 0 ? q.k_b : 3.0 * q.kT / (q.b * q.b);
        const double ks = q.k_s > 0 ? q.k_s : 3.0 * q.kT / (q.Ns * q.b * q.b);
        if (!finite_pos(kb) || !finite_pos(ks) || !(q.dt * (4.0 * kb + ks) / q.zeta < 2.0)) return SS_EINVAL;
        if ((q.create_mode != 0 && q.create_mode != 1) || (q.destroy_new != 0 && q.destroy_new != 1))
            return SS_EINVAL;
        if (q.corr_levels > SS_MAX_LEVELS || q.chunk_steps < 1) return SS_EINVAL;
        const int zm = q.z_max > 0 ? q.z_max : default_zmax(n_beads);
        if (zm < 1 || zm > std::min(n_beads, SS_MAX_SLOTS)) return SS_EINVAL;
        c.P = q;
        c.k_b = kb;
        c.k_s = ks;
        c.levels = q.corr_levels > 0 ? q.corr_levels : 0;
        if (c.levels > 0) c.P.chunk_steps = std::min(c.P.chunk_steps, ssk::kCorrMaxSteps);
        c.el[0].zmax = zm;
    }
    // scratch layout
    const size_t ts = tsize(&c);
    const int slices = (n_chains + ssk::kSliceChains - 1) / ssk::kSliceChains;
    const bool corr = c.levels > 0;
    size_t off = 0;
    const size_t off_hist = off;
    off = align256(off + (corr ? (size_t)n_chains * c.levels * 96 * ts : 0));
    const size_t off_acc64 = off;
    off = align256(off + (corr ? (size_t)slices * c.levels * 96 * sizeof(double) : 0));
    const size_t off_zero = off;  // history and sums start at zero
    off = align256(off + 9 * sizeof(double)) + 256;
    const size_t off_cnt = off;
    off = align256(off + 8 * sizeof(unsigned long long));
    const size_t off_status = off;
    off = align256(off + sizeof(int32_t));
    if (off > (size_t)SS_NOALLOC_SCRATCH_BYTES) return SS_ETOOBIG;
    // the stress series of one launch and the correlator's level samples take
    // the rest: (cap + 2 (cap / 2 + 1)) rows of [M][6], cap <= chunk_steps
    const size_t off_ser = off;
    int ser_cap = 0;
    size_t off_lev = off;
    if (corr) {
        const size_t row = (size_t)n_chains * 6 * ts;
        const size_t rows = ((size_t)SS_NOALLOC_SCRATCH_BYTES - off) / row;  // >= 2 cap + 2 needed
        ser_cap = (int)std::min<size_t>(c.P.chunk_steps, rows >= 2 ? (rows - 2) / 2 : 0);
        if (ser_cap < 1) return SS_ETOOBIG;
        off_lev = align256(off_ser + (size_t)ser_cap * row);
        if (off_lev + (size_t)2 * (ser_cap / 2 + 1) * row > (size_t)SS_NOALLOC_SCRATCH_BYTES) {
            ser_cap -= 1;  // the alignment pad
            off_lev = align256(off_ser + (size_t)ser_cap * row);
            if (ser_cap < 1) return SS_ETOOBIG;
        }
    }

    unsigned char* scr = nullptr;
    int rc = noalloc_scratch(&scr);
    if (rc != SS_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    // what must start at zero: history and sums of the correlator, the status word
    // (the event counters are not read)
    if (corr && cudaMemsetAsync(scr, 0, off_zero, st) != cudaSuccess) return SS_ECUDA;
    if (status_out && cudaMemsetAsync(status_out, 0, sizeof(int32_t), st) != cudaSuccess) return SS_ECUDA;
    int32_t* status = status_out ? status_out : reinterpret_cast<int32_t*>(scr + off_status);
    const int zm = c.el[0].zmax;
#define SS_NOALLOC_ARGS                                                                                          \
    &c, e.W, e.B, c.P, n_chains, n_beads, zm, chain_base, t0, n_steps, R, A, S, Z, scr, off_hist, off_ser, off_lev,       \
        ser_cap, off_acc64, off_cnt, status, kappa, st
    rc = precision == SS_FP64 ? noalloc_launches<double>(SS_NOALLOC_ARGS) : noalloc_launches<float>(SS_NOALLOC_ARGS);
#undef SS_NOALLOC_ARGS
    if (rc != SS_OK) return rc;
    if (corr_out && corr) {
        const int n = c.levels * 96;
        noalloc_reduce_kernel<<<(n + 127) / 128, 128, 0, st>>>(reinterpret_cast<const double*>(scr + off_acc64),
                                                                slices, c.levels, corr_out);
        if (cudaGetLastError() != cudaSuccess) return SS_ECUDA;
    }
    return SS_OK;
}
