// ss_kernels.cuh -- sm_103a kernels of the single-chain slip-spring time step
// (T. Uneyama, arXiv:1106.2899, Sec. 3.1), with a per-step stress series
// for the multiple-tau correlator (a separate kernel) and ensemble stress logs.
//
// Layout: one chain per W-lane segment of a warp (W = 32: one chain per warp,
// W = 16: two, W = 8: four), B beads per lane: lane l of a segment owns beads and
// slip-spring slots l, l + W, ..., so N <= W*B and z_max <= N (the paper's
// one-slot-per-bead bound, Sec. 3.2); slots above 64 stay empty (z_max <= 64,
// so a 64-bit mask covers a bead's springs).  A launch advances each chain `nsteps`
// steps with its whole state in registers; neighbouring beads are read from a
// per-warp shared-memory position table, stress parts wait in shared memory for a
// few steps and are summed there (FP32) or reduced with shuffles (FP64, log steps).
//
// Random numbers: Philox4x32-10 (Salmon et al., SC'11), counter = (index,
// step, purpose, chain id), key = seed.  Per step, slot/bead index l draws
// one block: two Box-Muller pairs give the bead noise (x, y, z) and a fourth
// normal n3; the low bytes of the first three words give a 24-bit uniform u.
// Slot l uses u for its hop (occupied) or its creation attempt (empty) and n3
// for its destruction test n3 < Phi^{-1}(p_destroy).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "ss_math64.cuh"

namespace ssk {

constexpr int kP = 16;      // multiple-tau points per level
constexpr int kCells = 32;  // (channel, lag) cells per level and component: channel*16 + lag
constexpr uint32_t kPurposeStep = 1, kPurposeCreate = 2, kPurposeInitBond = 3,
                   kPurposeInitZ = 4, kPurposeInitS = 5, kPurposeInitA = 6;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxBeads = 128;  // beads per chain
constexpr int kMaxSlots = 64;   // slip-spring slots per chain (z_max <= min(N, kMaxSlots))
constexpr int kSliceChains = 64;  // chains per FP64 correlator/log slice
constexpr int kMaxCorrLevels = 32;  // correlator levels the library accepts

// ---------------------------------------------------------------- Philox ----
// Ten rounds of the Philox4x32 bijection: words 0 and 2 are multiplied by
// the two round multipliers (high and low halves kept), the high halves are
// xored with words 1 and 3 and the round key, and the key advances by the
// two Weyl increments after every round.
__device__ __forceinline__ uint4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                               uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const unsigned long long p0 = (unsigned long long)0xD2511F53u * c0;
        const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * c2;
        c0 = (uint32_t)(p1 >> 32) ^ c1 ^ k0;
        c2 = (uint32_t)(p0 >> 32) ^ c3 ^ k1;
        c1 = (uint32_t)p1;
        c3 = (uint32_t)p0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return make_uint4(c0, c1, c2, c3);
}

// The same bijection with the ten round keys precomputed (kernel parameters).
__device__ __forceinline__ uint4 philox4x32_10_rk(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                  const uint32_t (&rk0)[10], const uint32_t (&rk1)[10]) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const unsigned long long p0 = (unsigned long long)0xD2511F53u * c0;
        const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * c2;
        c0 = (uint32_t)(p1 >> 32) ^ c1 ^ rk0[r];
        c2 = (uint32_t)(p0 >> 32) ^ c3 ^ rk1[r];
        c1 = (uint32_t)p1;
        c3 = (uint32_t)p0;
    }
    return make_uint4(c0, c1, c2, c3);
}

// The same generator for the step draws of a fixed (index, purpose, chain):
// counter (idx, t, P, cid).  Round 0 and most of round 1 do not depend on the
// step t, so their results are computed once per slot (pre) and per step
// (shared by all slots of a lane); philox_step finishes rounds 1..9 and
// returns the same words as philox4x32_10_rk(idx, t, P, cid).
struct PhiloxPre {
    uint32_t c3_1;  // lo(M0 idx) after round 0
    uint32_t c0_2;  // hi(M1 c2_1) ^ lo(M1 P) ^ rk0[1]
    uint32_t c1_2;  // lo(M1 c2_1)
};
__device__ __forceinline__ PhiloxPre philox_pre(uint32_t idx, uint32_t P, uint32_t cid, const uint32_t (&rk0)[10],
                                                const uint32_t (&rk1)[10]) {
    const unsigned long long p0 = (unsigned long long)0xD2511F53u * idx;
    const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * P;
    const uint32_t c2_1 = (uint32_t)(p0 >> 32) ^ cid ^ rk1[0];
    const uint32_t c1_1 = (uint32_t)p1;
    const unsigned long long q1 = (unsigned long long)0xCD9E8D57u * c2_1;
    PhiloxPre r;
    r.c3_1 = (uint32_t)p0;
    r.c0_2 = (uint32_t)(q1 >> 32) ^ c1_1 ^ rk0[1];
    r.c1_2 = (uint32_t)q1;
    return r;
}
// step part shared by the slots: c0 after round 0 is hi(M1 P) ^ t ^ rk0[0]
__device__ __forceinline__ unsigned long long philox_step_shared(uint32_t t, uint32_t P, const uint32_t (&rk0)[10]) {
    const uint32_t c0_1 = (uint32_t)(((unsigned long long)0xCD9E8D57u * P) >> 32) ^ t ^ rk0[0];
    return (unsigned long long)0xD2511F53u * c0_1;
}
__device__ __forceinline__ uint4 philox_step(const PhiloxPre& pre, unsigned long long p0_1, const uint32_t (&rk0)[10],
                                             const uint32_t (&rk1)[10]) {
    uint32_t c0 = pre.c0_2, c1 = pre.c1_2;
    uint32_t c2 = (uint32_t)(p0_1 >> 32) ^ pre.c3_1 ^ rk1[1];
    uint32_t c3 = (uint32_t)p0_1;
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        const unsigned long long p0 = (unsigned long long)0xD2511F53u * c0;
        const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * c2;
        c0 = (uint32_t)(p1 >> 32) ^ c1 ^ rk0[r];
        c2 = (uint32_t)(p0 >> 32) ^ c3 ^ rk1[r];
        c1 = (uint32_t)p1;
        c3 = (uint32_t)p0;
    }
    return make_uint4(c0, c1, c2, c3);
}

// ------------------------------------------------------------ math traits ---
template <typename T>
struct Mth;

template <>
struct Mth<float> {
    // log2 of a normal x > 0 by the hardware approximation, without the scaling of
    // subnormal arguments that __log2f carries (every argument here is >= 2^-24)
    static __device__ __forceinline__ float log2(float x) {
        float r;
        asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
        return r;
    }
    static __device__ __forceinline__ float neg2log(float x) { return log2(x) * -1.3862943611198906f; }
    // sqrt of x >= 0 by the hardware approximation (sqrt.approx); x = 0 gives 0
    static __device__ __forceinline__ float sqrt(float x) {
        float r;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
        return r;
    }
    static __device__ __forceinline__ void sincos(float x, float* s, float* c) { __sincosf(x, s, c); }
    static __device__ __forceinline__ float exp(float x) { return __expf(x); }
    static __device__ __forceinline__ float div(float a, float b) { return __fdividef(a, b); }
    static __device__ __forceinline__ bool finite(float x) { return isfinite(x); }
    static __device__ __forceinline__ float inf() { return __int_as_float(0x7f800000); }
};

template <>
struct Mth<double> {
    static __device__ __forceinline__ double neg2log(double x) { return -2.0 * ::log(x); }
    static __device__ __forceinline__ double sqrt(double x) { return ::sqrt(x); }
    static __device__ __forceinline__ void sincos(double x, double* s, double* c) { ::sincos(x, s, c); }
    static __device__ __forceinline__ double exp(double x) { return ::exp(x); }
    static __device__ __forceinline__ double div(double a, double b) { return a / b; }
    static __device__ __forceinline__ bool finite(double x) { return isfinite(x); }
    static __device__ __forceinline__ double inf() { return __longlong_as_double(0x7ff0000000000000ll); }
};

// pi / 2^23 in both precisions (a power-of-two scaling of pi)
template <typename T>
__device__ __forceinline__ T pi_over_2p23();
template <>
__device__ __forceinline__ float pi_over_2p23<float>() { return 3.14159265358979323846f / 8388608.0f; }
template <>
__device__ __forceinline__ double pi_over_2p23<double>() { return 3.14159265358979323846 / 8388608.0; }

// Box-Muller pair from two words: radius sqrt(-2 ln v), v = (hi24(wa)+1)/2^24
// in (0,1]; angle pi (2 hi24(wb)/2^24 - 1) in [-pi, pi).
template <typename T>
__device__ __forceinline__ void box_muller(uint32_t wa, uint32_t wb, T& n_cos, T& n_sin) {
    const T v = T((wa >> 8) + 1u) * T(1.0 / 16777216.0);
    const T r = Mth<T>::sqrt(Mth<T>::neg2log(v));
    const T th = T(int(wb >> 8) - (1 << 23)) * pi_over_2p23<T>();
    T s, c;
    Mth<T>::sincos(th, &s, &c);
    n_cos = r * c;
    n_sin = r * s;
}

// The pair of the step and creation draws: in FP64 by the tables of ss_math64.cuh.
template <typename T>
__device__ __forceinline__ void draw_pair(uint32_t wa, uint32_t wb, T& n_cos, T& n_sin) {
    if constexpr (sizeof(T) == 8)
        box_muller_lattice(wa, wb, n_cos, n_sin);
    else
        box_muller<T>(wa, wb, n_cos, n_sin);
}

// 24-bit uniform in [0, 1) from the low bytes of words x, y, z
__device__ __forceinline__ uint32_t lo24_bits(uint4 w) {
    return (w.x & 0xFFu) | ((w.y & 0xFFu) << 8) | ((w.z & 0xFFu) << 16);
}
template <typename T>
__device__ __forceinline__ T uniform_lo24(uint4 w) {
    return T(lo24_bits(w)) * T(1.0 / 16777216.0);
}

// ---- packed FP32x2 arithmetic (sm_100 and later: one instruction per pair).
// Where a lane carries an even number of FP32 beads, the identical scalar
// operations of two beads (sub-slots 2p and 2p+1) are issued as one packed
// instruction; each half is rounded exactly as the scalar operation, so the
// results are bit-identical to the scalar forms.
__device__ __forceinline__ float2 pk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 pk(float a) { return make_float2(a, a); }

// Box-Muller pairs of two beads (words a_k, b_k of bead k), the operations of
// box_muller<float> on each.
__device__ __forceinline__ void box_muller_x2(uint32_t a0, uint32_t b0, uint32_t a1, uint32_t b1, float& c0,
                                              float& s0, float& c1, float& s1) {
    const float2 v = __fmul2_rn(pk(float((a0 >> 8) + 1u), float((a1 >> 8) + 1u)), pk(1.0f / 16777216.0f));
    const float2 m = __fmul2_rn(pk(Mth<float>::log2(v.x), Mth<float>::log2(v.y)), pk(-1.3862943611198906f));
    const float2 r = pk(Mth<float>::sqrt(m.x), Mth<float>::sqrt(m.y));
    const float2 th = __fmul2_rn(pk(float(int(b0 >> 8) - (1 << 23)), float(int(b1 >> 8) - (1 << 23))),
                                 pk(3.14159265358979323846f / 8388608.0f));
    float sa, ca, sb, cb;
    __sincosf(th.x, &sa, &ca);
    __sincosf(th.y, &sb, &cb);
    const float2 cc = __fmul2_rn(r, pk(ca, cb));
    const float2 ss = __fmul2_rn(r, pk(sa, sb));
    c0 = cc.x;
    c1 = cc.y;
    s0 = ss.x;
    s1 = ss.y;
}

template <typename T>
__device__ __forceinline__ T shfl(T v, int src, int width) {
    return __shfl_sync(kFull, v, src, width);
}

// ------------------------------------------------------------- arguments ----
template <typename T>
struct StepConst {
    T k_b, k_s;   // bond and slip-spring stiffness
    T mob;        // dt / zeta
    T amp;        // sqrt(2 kT dt / zeta)
    T dt;
    T pref;       // dt kT / zeta_s: hop and destruction prefactor
    T chop;       // k_s / (4 kT): Glauber exponent per change of squared length
    T sa;         // sqrt(kT / k_s): anchor spread of a new spring
    T cd;         // Phi^{-1}(min(dt kT/zeta_s, 1)) (+inf when that is 1)
    T NkT, kT;
    T pc[kMaxSlots + 1];  // creation probability per end and attempt, by K
    T two_pref;           // 2 dt kT / zeta_s
    T c2;                 // 2 chop log2(e): base-2 exponent per change of squared length
    T hmob, hdt;          // mob / 2, dt / 2: the stochastic Heun corrector
    float c2_f, two_pref_f;  // c2, two_pref in FP32: the hop filter of FP64 runs
    uint32_t rk0[10], rk1[10];  // Philox round keys (key + r * Weyl increment)
};

struct ChunkArgs {
    void* R;            // [M][3][W] T
    void* A;            // [M][3][W] T
    int32_t* S;         // [M][W]
    int32_t* Z;         // [M]
    double* logs;       // [max_logs][groups][14]
    // [cnt_mask + 1][8]: events 0..4, 6 non-finite states, 7 broken invariants.  A CTA
    // adds to copy blockIdx.x & cnt_mask: one copy for all would serialise the
    // additions of a launch of few steps.
    unsigned long long* counters;
    int cnt_mask;
    int32_t* status;
    const double* kap;          // [n_kap][9]
    const long long* kap_from;  // [n_kap]
    int n_kap;                  // 0: the constant gradient kap0
    double kap0[9];
    int M, N, zmax, create_mode, destroy_new;
    int cta0;                   // first CTA tile of this launch
    int log_every, recenter_every;
    long long log_m0;           // logs are taken at steps m*log_every with m > log_m0
    int max_logs, groups, slices;  // slices of kSliceChains chains
    long long t0;               // first step index of this launch
    int nsteps;
    uint32_t key0, key1, chain_base;
    int nlog_chunk;             // log slots reserved in shared memory
    int W, B;                   // lane layout (read by the batched kernel)
    // differentiation windows (all optional, null when unused):
    uint8_t* tape;              // [steps][M][NP] decisions per slot and step
    int tape_mode;              // 0 off, 1 record, 2 replay (decisions frozen)
    long long tape_t0;          // step of tape row 0
    long long tape_rows;        // rows of the tape (steps outside are neither read nor written)
    void* snapR;                // [steps+1][M][3][NP] T: state before each step
    void* snapA;
    int32_t* snapS;             // [steps+1][M][NP]
    int32_t* snapZ;             // [steps+1][M]
    long long snap_t0;
    int snap_steps;
    // stress series for the correlator (null: not written): element
    // [((series_row0 + s) * M + m) * 6 + q] is, after step s of this launch,
    // sigma_off (q = 0..2: xy, xz, yz) or (sigma + sigma^(v))_off (q = 3..5)
    void* series;
    long long series_row0;
};

// decision byte of one slot in one step (tape): hop, creation, destruction
constexpr uint8_t kTapeUp = 1, kTapeDown = 2, kTapeNew0 = 4, kTapeNewN = 8, kTapeKillOld = 16, kTapeKillNew = 32;

// One slip-spring record in shared memory: a vector and an integer (the bead
// index in the re-indexing, a flag in the spring tables), 16 bytes in FP32.
template <typename T>
struct __align__(16) SlotRec {
    T x, y, z;
    int s;
};

// One bead position in the per-warp shared position table.
template <typename T>
struct __align__(16) Pos {
    T x, y, z, w;
};

// Threads per CTA of the chain kernels: one warp, so that a small ensemble spreads
// over the SMs and the last CTAs of a large one leave no warps waiting for their
// CTA (against CTAs of four warps: 1.04-1.24x at N = 128 x 4096 chains and
// N = 60 x 16384, 1.005x at N = 32 x 65536).
constexpr int kChunkThreads = 32;
constexpr int kCounterCopies = 64;  // power of two
// Resident warps per SM the kernels are compiled for.  Two beads per lane fit 96
// registers; three or more need 128 (N = 40, 65536 chains: 26.4 us per step at 16
// warps, 28.8 at 20 with the spills of 96 registers).  FP64 work is bound by the
// FP64 pipe long before twelve warps.
//
// A kernel of fewer warps with more registers does as much per time or more, but takes a
// second wave for what more warps take in one.  Some layouts therefore have two forms
// (ALT the second), which give the same bits, and the host takes the better one by the
// waves of an ensemble (second_form):
//   16 x 4 (N = 49..64), Euler-Maruyama: 168 registers without spills, 12 warps, or 128
//     with 130-190 bytes of spills, 16 warps (N = 62, 9000 chains, 400 steps: 2.97 -> 2.67
//     ms at 12; N = 56, 16000 chains: 4.62 -> 4.20)
//   16 x 4, Heun: 128 registers, 13 warps by shared memory with reduction batches of five
//     steps, 16 with two; with 168 registers the compiler contracts its sums in another
//     order and the results differ in the last bits
//   16 x 4, Heun with flow: 10 warps (168 registers, of which 12 fit), or 8 without spills
//   16 x 3 and 8 x 3 with flow: 16 or 20 warps; with Heun 12 or 16
//   16 x 2, Heun with flow: 16 or 20 warps
constexpr bool has_second_form(int W, int B, bool heun, bool flow) {
    return (W == 16 && B == 4) || (W <= 16 && B == 3 && flow) || (W == 16 && B == 2 && heun && flow);
}
template <typename T>
constexpr int chunk_warps_per_sm(int W, int B, bool heun = false, bool flow = false, bool alt = false) {
    if (sizeof(T) == 8) return heun && flow ? 8 : 12;
    if (W == 16 && B == 4) return heun && flow ? (alt ? 8 : 10) : (heun || alt ? 16 : 12);
    const int more = alt ? 4 : 0;
    if (heun && flow) return B == 1 ? 20 : (B == 2 ? 16 : 12) + more;  // both states live at once
    return B == 1 ? 24 : (B == 2 ? 20 : 16) + more;
}

// Columns of a chain's row in device memory (R, A [3][NP], S, tape [NP]): a
// property of the chain length alone, so layouts of fewer lanes x beads than
// that (8 x 1, 8 x 3, 32 x 3) read and write the same arrays.
__host__ __device__ constexpr int row_stride(int n) {
    return n <= 64 ? (n + 15) / 16 * 16 : kMaxBeads;
}
// Slot sub-slots of a lane: slots above kMaxSlots never hold a spring.
__host__ __device__ constexpr int slot_sub(int W, int B) { return W * B <= kMaxSlots ? B : kMaxSlots / W; }

// shared memory carve-up (bytes), identical on host and device
struct SmemPlan {
    int off_rec, off_pos, off_bq, off_msk, off_red, off_kap, off_log, total;
};

// Stress samples are reduced in batches of kRedSteps steps (FP32): the six
// per-lane parts of each step wait in shared memory, and then each lane adds up
// whole rows (one value of one chain and step), five steps filling 60 of 64, 30
// of 32 or 120 of 128 row slots of a warp.  (A shuffle reduction of every step,
// with its selects and its five dependent rounds, took 12 instructions per
// warp-step more.)
constexpr int kRedSteps = 5;
// of a chain kernel whose stress series may be written (0: FP64, no batches)
template <typename T>
constexpr int red_steps(int W, int B, bool heun, bool flow, bool alt) {
    if (sizeof(T) == 8) return 0;
    // a second form of more warps: as many as leave room for them
    if (alt && heun && flow) return B == 3 ? 4 : kRedSteps;
    return alt ? 2 : kRedSteps;
}
// Rows of W + 4 words, so that eight lanes reading 16 bytes of eight rows each
// cover every bank once; the chains of a warp lie W words (mod 32) apart, so that
// the 32 lanes writing one value of each do, too.
__host__ __device__ constexpr int red_row(int W) { return W + 4; }
__host__ __device__ constexpr int red_chain(int W, int steps) {
    const int n = steps * 6 * red_row(W), pad = (W - n % 32 + 32) % 32;
    return n + (W == 32 ? 0 : pad);
}

// red: steps of a reduction batch, 0 without a stress series.  Nothing touches the
// reduction buffer then, a third of the shared memory of a CTA: left out, the batched kernel and the
// chain kernel without the correlator run the warps their registers are planned for
// (16 x 2 with 11 log steps: 17 and 18 warps/SM -> 20; 512 elements, 1000 steps: 57.4 ->
// 52.3 ms, six ensembles of 4096 x 40 under shear: 11.1 -> 10.7 ms).
template <typename T>
__host__ __device__ inline SmemPlan smem_plan(int warps, int W, int B, int nlog_chunk, int red) {
    SmemPlan p;
    const int chains = warps * (32 / W), NL = W * B;
    p.off_rec = 0;
    // per chain 3 NL spring records: the first spring of each bead, the second, and by slot
    int sz = chains * 3 * NL * (int)sizeof(SlotRec<T>);
    p.off_pos = (sz + 15) & ~15;
    // per chain NL positions between two guard entries
    sz = p.off_pos + chains * (NL + 2) * (int)sizeof(Pos<T>);
    p.off_bq = (sz + 15) & ~15;
    // per chain NL + 1 bond vectors: entry i + 1 holds bead i's, entry 0 zeros
    sz = p.off_bq + chains * (NL + 1) * (int)sizeof(Pos<T>);
    p.off_msk = (sz + 15) & ~15;
    sz = p.off_msk + chains * NL * (int)(NL <= 32 ? sizeof(unsigned) : sizeof(unsigned long long));
    p.off_red = (sz + 15) & ~15;
    sz = p.off_red + (red > 0 ? chains * red_chain(W, red) * (int)sizeof(T) : 0);
    p.off_kap = (sz + 15) & ~15;
    sz = p.off_kap + warps * 3 * (int)sizeof(Pos<T>);
    p.off_log = (sz + 15) & ~15;
    sz = p.off_log + nlog_chunk * 14 * (int)sizeof(double);
    p.total = (sz + 15) & ~15;
    return p;
}

// CTAs that `bytes` of shared memory each leave room for on an SM: 228 KB, 1 KB per CTA
// for the system, granules of 128 bytes
constexpr int ctas_by_smem(int bytes) { return 228 * 1024 / ((bytes + 1024 + 127) / 128 * 128); }

// -------------------------------------------------------------- helpers -----
// 1 + index of the lowest set bit (0 for none) of a 32- or 64-bit slot mask
__device__ __forceinline__ int mask_ffs(unsigned m) { return __ffs((int)m); }
__device__ __forceinline__ int mask_ffs(unsigned long long m) { return __ffsll((long long)m); }
// number of set bits of a slot mask
__device__ __forceinline__ int mask_popc(unsigned m) { return __popc(m); }
__device__ __forceinline__ int mask_popc(unsigned long long m) { return __popcll(m); }

// Sum over the W lanes of a segment; every lane of the segment gets the sum.
template <typename T, int W>
__device__ __forceinline__ T seg_sum(T v) {
#pragma unroll
    for (int off = W / 2; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off, W);
    return v;
}

// Sums over the W lanes of a segment of six per-lane values v[0..5]
// (sigma_xy, sigma_xz, sigma_yz and the same components of sigma + sigma^(v))
// by a transpose reduction: the first round splits the two tensors between
// the lane halves, the second the xy/xz pair (yz summed on both sides), the
// third xy-or-xz against yz; butterflies finish.  On return lane ll holds
// the total of value seg6_value(ll).
template <int W>
__device__ __forceinline__ int seg6_value(int ll) {
    const int comp = (ll & (W / 8)) ? 2 : ((ll & (W / 4)) ? 1 : 0);
    return ((ll & (W / 2)) ? 3 : 0) + comp;
}
template <typename T, int W>
__device__ __forceinline__ T seg_reduce6(const T (&v)[6], int ll) {
    T w[3];
    {
        const bool hi = (ll & (W / 2)) != 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const T send = hi ? v[k] : v[k + 3];
            const T keep = hi ? v[k + 3] : v[k];
            w[k] = keep + __shfl_xor_sync(kFull, send, W / 2, W);
        }
    }
    T x, y;
    {
        const bool hi = (ll & (W / 4)) != 0;
        const T send = hi ? w[0] : w[1];
        const T keep = hi ? w[1] : w[0];
        x = keep + __shfl_xor_sync(kFull, send, W / 4, W);
        y = w[2] + __shfl_xor_sync(kFull, w[2], W / 4, W);
    }
    T r;
    {
        const bool hi = (ll & (W / 8)) != 0;
        const T send = hi ? x : y;
        const T keep = hi ? y : x;
        r = keep + __shfl_xor_sync(kFull, send, W / 8, W);
    }
#pragma unroll
    for (int off = W / 16; off > 0; off >>= 1) r += __shfl_xor_sync(kFull, r, off, W);
    return r;
}

// Glauber hop probability of Sec. 3.1 item 2, min{pref (1 - tanh y), 1/2},
// y = chop (d_new - d_old), with 1 - tanh y written 2 / (1 + e^{2y}) and y
// clamped to [-40, 40].
template <typename T>
__device__ __forceinline__ T hop_prob(const StepConst<T>& c, T d_new, T d_old) {
    T y = c.chop * (d_new - d_old);
    y = y > T(40) ? T(40) : (y < T(-40) ? T(-40) : y);
    const T w = c.pref * Mth<T>::div(T(2), T(1) + Mth<T>::exp(T(2) * y));
    return w < T(0.5) ? w : T(0.5);
}

// FP32 form of the same probability for the two moves from one slot (new squared
// lengths dnew.x, dnew.y): e^{2y} = 2^t with t = c2 (d_new - d_old) (c2 = 2 chop
// log2 e) by ex2.approx, 2/(1+e^{2y}) by rcp.approx, the additions and
// multiplications packed.  t is capped at 80 log2 e (y <= 40), where the
// probability is still a normal float; below y = -40 the expression already
// equals its limit 2 pref.
__device__ __forceinline__ float2 hop_prob_x2(const StepConst<float>& c, float2 dnew, float d_old) {
    const float2 t = __fmul2_rn(pk(c.c2), __fadd2_rn(dnew, pk(-d_old)));
    float ea, eb, ra, rb;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ea) : "f"(fminf(t.x, 115.41560327111707f)));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(eb) : "f"(fminf(t.y, 115.41560327111707f)));
    const float2 den = __fadd2_rn(pk(1.0f), pk(ea, eb));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(ra) : "f"(den.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rb) : "f"(den.y));
    const float2 w = __fmul2_rn(pk(c.two_pref), pk(ra, rb));
    return make_float2(fminf(w.x, 0.5f), fminf(w.y, 0.5f));
}

// An FP64 number in FP32, truncated, by integer operations; `odd` is set if it is
// not a normal number there (zero among them).
__device__ __forceinline__ float trunc_f32(double x, bool& odd) {
    const unsigned hi = (unsigned)__double2hiint(x), fs = __funnelshift_l((unsigned)__double2loint(x), hi, 3);
    odd |= (hi & 0x7fffffffu) - (897u << 20) >= (253u << 20);
    return __uint_as_float(((fs ^ 0x40000000u) & 0x7fffffffu) | (hi & 0x80000000u));
}
// Hop decision of an FP64 slot in FP32 where that is certain: spring vectors to
// the bead, the one above and the one below, the 24-bit uniform k.  With vectors
// truncated to 23 bits a squared length is off by less than 4.2e-7 of itself, the
// exponent by less than 6e-7 c2 (sum of two squared lengths), a probability by
// less than 1.1e-7 two_pref times that plus 6e-7 two_pref; the margin is nine
// times as wide in the first part and six times in the second.  Returns false if the uniform lies within it (about 1e-5 of all hops):
// the FP64 probabilities then decide.  These are 70 FP64 instructions (two
// exponentials, two divisions) of 64 cycles each.
__device__ __forceinline__ bool hop_filter(const StepConst<double>& c, const double (&r0)[3], const double (&rp)[3],
                                           const double (&rm)[3], bool has_up, bool has_dn, uint32_t k, bool& up,
                                           bool& dn) {
    bool odd = false;
    float d[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float x0 = trunc_f32(r0[i], odd), xp = trunc_f32(rp[i], odd), xm = trunc_f32(rm[i], odd);
        d[0] = fmaf(x0, x0, d[0]);
        d[1] = fmaf(xp, xp, d[1]);
        d[2] = fmaf(xm, xm, d[2]);
    }
    float p[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        float e, r;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(fminf(c.c2_f * (d[1 + i] - d[0]), 115.41560327111707f)));
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.0f + e));
        p[i] = fminf(c.two_pref_f * r, 0.5f);
    }
    const float margin = c.two_pref_f * fmaf(c.c2_f * 1e-6f, d[0] + d[1] + d[2], 4e-6f);
    const float u = (float)k * (1.0f / 16777216.0f), pp = has_up ? p[0] : 0.0f, ps = pp + (has_dn ? p[1] : 0.0f);
    up = u < pp;
    dn = !up && u < ps;
    return !odd && fabsf(u - pp) > margin && fabsf(u - ps) > 2.0f * margin;
}

// ---------------------------------------------------------- chunk kernel ----
// W lanes per chain, B beads per lane: bead i and slot i of a chain live on
// lane i % W as its sub-slot i / W (NL = W*B >= N beads; slots only up to
// kMaxSlots, SB sub-slots of a lane).  NP is the row stride in device memory.
//
// The spring forces of a step read, per bead, the vectors of up to two springs
// from two tables that the slot lanes keep up to date (rec).  A third spring on
// one bead is rare and handled in a branch.  (A gather by bit scans of the
// masks spends 24 instructions on every bead, most of which carry no spring.)
constexpr int kWinOff = 0, kWinRecord = 1, kWinReplay = 2;  // differentiation-window hooks

// State of one chain before a step, for the recompute of a differentiation window.
template <typename T, int W, int B, int SB, typename Args>
__device__ __forceinline__ void snapshot_store(const Args& a, long long row, int mm, int ll, const T (&R)[B][3],
                                               const T (&A)[SB][3], const int (&S)[SB], int Z) {
    constexpr int NP = row_stride(W * B);
    T* sR = static_cast<T*>(a.snapR) + ((size_t)row * a.M + mm) * 3 * NP;
    T* sA = static_cast<T*>(a.snapA) + ((size_t)row * a.M + mm) * 3 * NP;
    int32_t* sS = a.snapS + ((size_t)row * a.M + mm) * NP;
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const int i = ll + b * W;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            sR[d * NP + i] = R[b][d];
            sA[d * NP + i] = b < SB && i < Z ? A[b < SB ? b : 0][d] : T(0);
        }
        sS[i] = b < SB && i < Z ? S[b < SB ? b : 0] : -1;
    }
    if (ll == 0) a.snapZ[(size_t)row * a.M + mm] = Z;
}

constexpr int kNever = 0x7fffffff;
// absolute step as an offset from t0 (kNever: beyond any launch)
__device__ __forceinline__ int rel_step(long long t_abs, long long t0) {
    const long long r = t_abs - t0;
    return r > (long long)kNever ? kNever : (int)r;
}

// Place in the velocity-gradient schedule: entry, offset of the next entry in
// this launch, whether the entry is non-zero.
struct KappaState {
    int ki, next_from;
    bool nz;
};
// The entry of the schedule for step t0 + s (from entry ki on), its matrix in
// the rows kap.  All lanes of the warp call this together.  The loads are __ldg:
// through pointers that come from memory, plain ones might read shared memory for
// all the compiler knows, and cost the batched kernel 27 us per step instead of 18
// (N = 32, 65536 chains).
template <typename T, typename Args>
__device__ __forceinline__ KappaState kappa_at(Args& a, int ki, long long t0, int s, Pos<T>* kap) {
    const int lane = threadIdx.x & 31;
    const int n = a.n_kap;
    const double* const k = a.kap;
    const long long* const from = a.kap_from;
    while (ki + 1 < n && t0 + s >= __ldg(from + ki + 1)) ++ki;
    T v = T(0);
    if (lane < 9) v = n > 0 ? T(__ldg(k + ki * 9 + lane)) : T(a.kap0[lane]);
    if (lane < 9) reinterpret_cast<T*>(kap + lane / 3)[lane % 3] = v;
    KappaState r;
    r.ki = ki;
    r.next_from = ki + 1 < n ? rel_step(__ldg(from + ki + 1), t0) : kNever;
    r.nz = __any_sync(kFull, v != T(0));
    __syncwarp();
    return r;
}
// The chains of one CTA: chains cta_first .. cta_first + chains per CTA - 1 of
// the element described by `a` (all warps of the CTA call this together).
// FLOW: the velocity-gradient terms are compiled in (without them the launch
// must have kappa = 0 throughout; recentring is then never needed).  CORR: the
// stress series is compiled in, its samples reduced RED steps at a time.  VL = 2: eight lanes do the work of sixteen.
// Sub-slots of even and of odd b are the beads of lanes l and l + 8 of a 16-lane
// segment; summing them apart and adding the two is the first round of that
// segment's reduction, so every sum over beads is rounded as there.
// PAIR (one bead per lane): the stress of a log step is summed as with two beads per
// lane, those of lanes l and l + W/2 in one fused sum.
template <typename T, int W, int B, int WIN, bool FLOW, bool HEUN, bool CORR, int VL, int RED, bool PAIR, typename Args>
__device__ __forceinline__ void run_chains(Args& a, const StepConst<T>& c, const int cta_first,
                                           const T NkT, const long long t0_, const int nsteps_,
                                           const long long log_m0_, const int nlog_) {
    constexpr int SEGS = 32 / W;
    constexpr int NL = W * B;               // beads of a chain's lanes
    constexpr int NP = row_stride(NL);      // columns of a chain's rows in device memory
    constexpr int SB = slot_sub(W, B);      // slot sub-slots
    constexpr int G8 = W / 8;               // lanes per value group after seg_reduce6
    constexpr int BP = std::is_same<T, float>::value ? B / 2 * 2 : 0;  // beads in packed FP32x2 pairs
    // the uniform of a slot: itself in FP32, its 24 bits in FP64 (compared as integers)
    constexpr bool INT_U = sizeof(T) == 8;
    using U = typename std::conditional<INT_U, uint32_t, T>::type;
    auto u_value = [](U u) -> T {
        if constexpr (INT_U)
            return T(u) * T(1.0 / 16777216.0);
        else
            return u;
    };
    // per-bead slot masks: 32 bits cover every slot when NL <= 32
    using Mask = typename std::conditional<(NL <= 32), unsigned, unsigned long long>::type;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    const int seg = lane / W;
    const int ll = lane % W;
    const int cslot = warp * SEGS + seg;
    const int m = cta_first + cslot;
    const bool live = m < a.M;
    const int mm = live ? m : 0;
    const uint32_t chain_id = a.chain_base + (uint32_t)mm;
    const int N = a.N;
    const unsigned segmask = (W == 32) ? kFull : (((1u << W) - 1u) << (seg * W));
    const unsigned lt = ((1u << lane) - 1u) & segmask;  // lanes of this segment below this one

    extern __shared__ __align__(16) unsigned char smem[];
    const SmemPlan plan = smem_plan<T>(nwarps, W, B, nlog_, RED);
    // spring records of this chain: [0, NL) the first spring of each bead, [NL, 2 NL)
    // the second (zeros where there is none), [2 NL, 3 NL) by slot: springs beyond
    // the second of a bead, and scratch of the re-indexing
    SlotRec<T>* rec = reinterpret_cast<SlotRec<T>*>(smem + plan.off_rec) + cslot * 3 * NL;
    SlotRec<T>* tab = rec + 2 * NL;
    // positions, with a guard entry on either side (read for a hop beyond an end,
    // whose probability is then replaced by 0)
    Pos<T>* pos = reinterpret_cast<Pos<T>*>(smem + plan.off_pos) + cslot * (NL + 2) + 1;
    // bond vectors Q_i = R_{i+1} - R_i of the current state times k_b, one entry up:
    // bq[i + 1] = k_b Q_i, bq[0] = 0 (bead 0 has no left bond); with HEUN Q_i itself,
    // whose corrector rounds the bond force from it
    Pos<T>* bq = reinterpret_cast<Pos<T>*>(smem + plan.off_bq) + cslot * (NL + 1);
    Mask* msk = reinterpret_cast<Mask*>(smem + plan.off_msk) + cslot * NL;
    [[maybe_unused]] T* const red = reinterpret_cast<T*>(smem + plan.off_red) + warp * SEGS * red_chain(W, RED);
    double* slog = reinterpret_cast<double*>(smem + plan.off_log);

    for (int i = threadIdx.x; i < nlog_ * 14; i += blockDim.x) slog[i] = 0.0;

    // ---- flow schedule, as step offsets in this launch
    const int never = kNever;
    // The velocity gradient waits in shared memory, row by row (three 16-byte
    // broadcast loads a step): nine registers for the whole launch would spill.
    KappaState ks{0, never, false};
    [[maybe_unused]] Pos<T>* const kap = reinterpret_cast<Pos<T>*>(smem + plan.off_kap) + warp * 3;
    auto kx = [&](int d) { return kap[d].x; };
    auto ky = [&](int d) { return kap[d].y; };
    auto kz = [&](int d) { return kap[d].z; };
    auto load_kappa = [&](int s) {
        ks = kappa_at<T>(a, ks.ki, t0_, s, kap);
    };
    if constexpr (FLOW) load_kappa(0);

    // ---- load state
    const T* Rg = static_cast<const T*>(a.R);
    const T* Ag = static_cast<const T*>(a.A);
    T R[B][3], A[SB][3];
    int S[SB];
    int Z = live ? a.Z[mm] : 0;
    SlotRec<T> zrec;
    zrec.x = zrec.y = zrec.z = T(0);
    zrec.s = 0;
    Pos<T> zpos;
    zpos.x = zpos.y = zpos.z = zpos.w = T(0);
    auto store_pos = [&](const T (&X)[B][3]) {
#pragma unroll
        for (int b = 0; b < B; ++b) {
            Pos<T> p;
            p.x = X[b][0];
            p.y = X[b][1];
            p.z = X[b][2];
            p.w = T(0);
            pos[ll + b * W] = p;
        }
    };
#pragma unroll
    for (int b = 0; b < SB; ++b) {
        const int i = ll + b * W;
        S[b] = (live && i < Z) ? a.S[(size_t)mm * NP + i] : 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) A[b][d] = (live && i < Z) ? Ag[((size_t)mm * 3 + d) * NP + i] : T(0);
    }
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const int i = ll + b * W;
#pragma unroll
        for (int d = 0; d < 3; ++d) R[b][d] = (live && i < N) ? Rg[((size_t)mm * 3 + d) * NP + i] : T(0);
        rec[i] = zrec;
        rec[NL + i] = zrec;
        msk[i] = Mask(0);
    }
    store_pos(R);
    if (ll == 0) {
        pos[-1] = zpos;
        pos[NL] = zpos;
        bq[0] = zpos;
    }

    // Values that change only with Z, kept from one change to the next: per
    // sub-slot the bound on u below which it creates a spring (2 p_c on the
    // creation attempts of substep 3a, slots Z .. c_last - 1; 0 elsewhere) and the
    // bound on n3 below which a spring at an end is destroyed (cd on occupied
    // slots, -inf elsewhere) and its stiffness in the stress (0 on empty slots); an
    // attempt dropped at the cap, counted on lane 0; and
    // the largest Z of this warp's chains (sub-slots at or above it hold no spring).
    U thr_c[SB];
    int z_w = 0;
    bool c_drop = false;
    auto attempts_end = [&]() { return Z < a.zmax ? ((a.create_mode == 0) ? a.zmax : Z + 1) : Z; };
    auto set_create = [&]() {
        c_drop = Z >= a.zmax && a.create_mode == 1 && ll == 0 && live;
        z_w = (int)__reduce_max_sync(kFull, (unsigned)Z);
        const int c_last = attempts_end();
        const T pc2 = T(2) * c.pc[c_last - Z];
        U thr;  // u < 2 p_c as a bound on U
        if constexpr (INT_U)
            thr = (U)__double2uint_ru(pc2 * 16777216.0);
        else
            thr = pc2;
#pragma unroll
        for (int b = 0; b < SB; ++b) {
            const int i = ll + b * W;
            thr_c[b] = (i >= Z && i < c_last) ? thr : U(0);
        }
    };
    set_create();

    // stress series of this launch (the correlator reads it afterwards)
    T* const ser = static_cast<T*>(a.series);
    const bool corr_on = CORR && ser != nullptr;
    const int gq = seg6_value<W>(ll);  // value this lane holds after seg_reduce6
    // one writer per value: the lowest lane of its group (yz is held twice over)
    [[maybe_unused]] T* const ser_m = (corr_on && live && (ll % G8) == 0 && !((gq % 3) == 2 && (ll & (W / 4))))
                         ? ser + ((size_t)a.series_row0 * a.M + mm) * 6 + gq
                         : nullptr;
    const size_t ser_step = (size_t)a.M * 6;
    // Batched reduction (FP32): value q of step n of a batch is row 6 n + q of its
    // chain, W lane parts summed in pairs as the butterflies of seg_reduce6 pair
    // the lanes.
    [[maybe_unused]] int red_n = 0;  // steps waiting
    [[maybe_unused]] T* red_w = red + seg * red_chain(W, RED) + ll;
    [[maybe_unused]] auto red_put = [&](const T (&v)[6]) {
#pragma unroll
        for (int q = 0; q < 6; ++q) red_w[q * red_row(W)] = v[q];
        red_w += 6 * red_row(W);
    };
    [[maybe_unused]] auto red_flush = [&](int s_end) {
        const int rows = 6 * red_n;  // of each chain
        for (int r = lane; r < rows * SEGS; r += 32) {
            const int ch = SEGS == 1 ? 0 : r / rows, rr = r - ch * rows;
            const float4* row = reinterpret_cast<const float4*>(red + ch * red_chain(W, RED) + rr * red_row(W));
            float4 x[W / 4];
#pragma unroll
            for (int k = 0; k < W / 4; ++k) x[k] = row[k];
#pragma unroll
            for (int h = W / 8; h > 0; h >>= 1) {
#pragma unroll
                for (int k = 0; k < h; ++k) {
                    x[k].x += x[k + h].x;
                    x[k].y += x[k + h].y;
                    x[k].z += x[k + h].z;
                    x[k].w += x[k + h].w;
                }
            }
            const float sum = (x[0].x + x[0].z) + (x[0].y + x[0].w);
            const int st = rr / 6, q = rr - 6 * st, m = cta_first + warp * SEGS + ch;
            if (m < a.M) ser[((size_t)(a.series_row0 + s_end - red_n + st) * a.M + m) * 6 + q] = sum;
        }
        red_n = 0;
        red_w = red + seg * red_chain(W, RED) + ll;
    };
    if (nlog_ > 0)
        __syncthreads();  // the CTA's stress-log buffer is zeroed
    else
        __syncwarp();

    // ---- periodic events, as step offsets in this launch
    int next_log = a.log_every > 0 ? rel_step((t0_ / a.log_every + 1) * a.log_every - 1, t0_) : never;
    int next_rc = a.recenter_every > 0 ? rel_step((t0_ / a.recenter_every + 1) * a.recenter_every - 1, t0_) : never;
    int log_slot = 0;
    const uint32_t t0lo = (uint32_t)t0_;

    unsigned cnt_up = 0, cnt_dn = 0, cnt_cr = 0, cnt_de = 0, cnt_drop = 0;

    __syncwarp();  // positions, zeroed records and masks of this warp's chains are in place

    // Spring vectors d_j = R_{S_j} - A_j into the tables the forces of the next
    // step read: the first slot to enter its bit in the bead's mask takes the
    // bead's first record, the next one the second (their sum is the same either
    // way), any other its own slot's record; the record names its slot, so that a
    // bead of three or more can add them in slot order.  The masks and the records
    // of beads 0 .. NL - 1 are zero before: each slot clears what it wrote before
    // it moves.  loc: this slot's record; more3: some bead of the warp has three.
    // With BY_SLOT (Heun at three and four beads per lane) every record is written by
    // slot as well while some bead has three, so that the sums in slot order read them
    // without a search: that kernel gathers twice a step with a flow and is short of
    // registers (us of 200 steps, before / with: 16000 x 60 3122 / 2927, with shear 4185 /
    // 3997, 16000 x 48 with shear 2810 / 2517, 16000 x 128 4764 / 4369; in the Euler-Maruyama
    // step, which gathers once, it cost 2.4% at N = 32).
    // The slots of an idle lane (no spring) do the same work without a branch: a
    // stale S is a valid bead, and their record is their own slot's, which nothing
    // reads.  Sub-slots at or above every Z of the warp are skipped (the first
    // never is).
    int loc[SB];
    bool more3 = false;
    constexpr bool BY_SLOT = HEUN && B >= 3;
    auto skip = [&](int b, int z) { return b > 0 && b * W >= z; };
    auto register_springs = [&](const T (&d)[SB][3]) {
        bool third = false;
#pragma unroll
        for (int b = 0; b < SB; ++b) {
            const int i = ll + b * W;
            if (!skip(b, z_w)) {
                const bool occ = i < Z;
                Mask old = ~Mask(0);
                if (occ) old = atomicOr(&msk[S[b]], Mask(1) << i);
                const bool late = (old & (old - Mask(1))) != Mask(0);  // two or more before it, or no spring
                third |= occ && late;
                int l = old != Mask(0) ? NL + S[b] : S[b];
                l = late ? 2 * NL + i : l;
                loc[b] = l;
                SlotRec<T> r;
                r.x = d[b][0];
                r.y = d[b][1];
                r.z = d[b][2];
                r.s = i;
                rec[l] = r;
            }
        }
        more3 = __any_sync(kFull, third);
        if constexpr (BY_SLOT) {
            if (more3) {
#pragma unroll
                for (int b = 0; b < SB; ++b) {
                    const int i = ll + b * W;
                    if (!skip(b, z_w)) {
                        SlotRec<T> r;
                        r.x = d[b][0];
                        r.y = d[b][1];
                        r.z = d[b][2];
                        r.s = i;
                        tab[i] = r;
                    }
                }
            }
        }
    };
    auto spring_vectors = [&](T (&d)[SB][3]) {
#pragma unroll
        for (int b = 0; b < SB; ++b) {
            if (!skip(b, z_w)) {
                const Pos<T> ps = pos[S[b]];
                d[b][0] = ps.x - A[b][0];
                d[b][1] = ps.y - A[b][1];
                d[b][2] = ps.z - A[b][2];
            }
        }
    };
    // the vectors again, from shifted or predicted coordinates, in the same records
    auto rewrite_springs = [&]() {
#pragma unroll
        for (int b = 0; b < SB; ++b) {
            if (!skip(b, z_w)) {
                const Pos<T> ps = pos[S[b]];
                SlotRec<T>& r = rec[loc[b]];
                r.x = ps.x - A[b][0];
                r.y = ps.y - A[b][1];
                r.z = ps.z - A[b][2];
                if constexpr (BY_SLOT) {
                    if (more3) tab[ll + b * W] = r;
                }
            }
        }
    };
    {
        T d[SB][3];
        spring_vectors(d);
        register_springs(d);
    }
    PhiloxPre ppre[B];
#pragma unroll
    for (int b = 0; b < B; ++b) ppre[b] = philox_pre((uint32_t)(ll + b * W), kPurposeStep, chain_id, c.rk0, c.rk1);
    // Bond vectors of the current positions (the position table holds them):
    // the stress of a step and the bond forces of the next step both use
    // them.  The last bead and padding beads read themselves: Q = 0.
    T Q[B][3];
    auto bond_vectors = [&]() {
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int i = ll + b * W;
            const Pos<T> p1 = pos[i < N - 1 ? i + 1 : i];
            Q[b][0] = p1.x - R[b][0];
            Q[b][1] = p1.y - R[b][1];
            Q[b][2] = p1.z - R[b][2];
            Pos<T> qq;
            const T f = HEUN ? T(1) : c.k_b;
            qq.x = f * Q[b][0];
            qq.y = f * Q[b][1];
            qq.z = f * Q[b][2];
            qq.w = T(0);
            bq[i + 1] = qq;
        }
    };
    bond_vectors();
    // the first step's forces read records, masks and bond vectors that other lanes
    // of the chain have written (the later steps' lie behind the barrier that ends a
    // step)
    __syncwarp();

    // Random numbers of step tt: block (i, tt, STEP, chain) per bead/slot i.
    // They do not depend on the state: a step draws its own at its top, where their
    // integer work interleaves with the forces.
    auto draw = [&](const uint32_t tt, T (&nrm)[B][4], U (&u)[B]) {
        const unsigned long long p_shared = philox_step_shared(tt, kPurposeStep, c.rk0);
#pragma unroll
        for (int b = 0; b < BP; b += 2) {
            const uint4 w0 = philox_step(ppre[b], p_shared, c.rk0, c.rk1);
            const uint4 w1 = philox_step(ppre[b + 1], p_shared, c.rk0, c.rk1);
            if constexpr (std::is_same<T, float>::value) {
                box_muller_x2(w0.x, w0.y, w1.x, w1.y, nrm[b][0], nrm[b][1], nrm[b + 1][0], nrm[b + 1][1]);
                box_muller_x2(w0.z, w0.w, w1.z, w1.w, nrm[b][2], nrm[b][3], nrm[b + 1][2], nrm[b + 1][3]);
                const float2 uu = __fmul2_rn(pk(float(lo24_bits(w0)), float(lo24_bits(w1))), pk(1.0f / 16777216.0f));
                u[b] = uu.x;
                u[b + 1] = uu.y;
            }
        }
#pragma unroll
        for (int b = BP; b < B; ++b) {
            const uint4 w = philox_step(ppre[b], p_shared, c.rk0, c.rk1);
            if constexpr (std::is_same<T, float>::value) {  // the bead's two Box-Muller pairs packed
                box_muller_x2(w.x, w.y, w.z, w.w, nrm[b][0], nrm[b][1], nrm[b][2], nrm[b][3]);
            } else {
                draw_pair<T>(w.x, w.y, nrm[b][0], nrm[b][1]);
                draw_pair<T>(w.z, w.w, nrm[b][2], nrm[b][3]);
            }
            if constexpr (INT_U)
                u[b] = lo24_bits(w);
            else
                u[b] = uniform_lo24<T>(w);
        }
    };
    // decisions of a replayed step, loaded one step ahead
    auto tape_at = [&](int s, int b) -> uint8_t {
        const long long row = (long long)t0_ + s - a.tape_t0;
        return (live && s < nsteps_ && row >= 0 && row < a.tape_rows)
                   ? a.tape[((size_t)row * a.M + mm) * NP + ll + b * W]
                   : (uint8_t)0;
    };
    [[maybe_unused]] uint8_t tape_next[SB];
    if constexpr (WIN == kWinReplay) {
#pragma unroll
        for (int b = 0; b < SB; ++b) tape_next[b] = tape_at(0, b);
    }
    int s = 0;
    for (;;) {  // stretches of one velocity gradient
    const int s_end = FLOW ? min(nsteps_, ks.next_from) : nsteps_;
    for (; s < s_end; ++s) {
        const uint32_t t = t0lo + (uint32_t)s;
        if (WIN == kWinReplay && a.snapR != nullptr && live) {
            const long long sr = (long long)t0_ + s - a.snap_t0;
            if (sr >= 0 && sr <= a.snap_steps) snapshot_store<T, W, B, SB>(a, sr, mm, ll, R, A, S, Z);
        }
        [[maybe_unused]] uint8_t tb[SB];
        if constexpr (WIN != kWinOff) {
#pragma unroll
            for (int b = 0; b < SB; ++b) {
                tb[b] = WIN == kWinReplay ? tape_next[b] : (uint8_t)0;
                if (WIN == kWinReplay) tape_next[b] = tape_at(s + 1, b);
            }
        }

        T nrm[B][4];
        U u[B];
        draw(t, nrm, u);
        // ---- substep 1: forces at time t, Euler-Maruyama, anchor advection.
        // Forces on positions Ro (this lane's beads; the other beads from the
        // position table) with the spring vectors of the tables: bonds
        // k_b (R_{i-1} + R_{i+1} - 2 R_i), springs -k_s sum_{j: S_j = i} d_j.
        // With bonds_from_q the bond forces come from the bond vectors of the
        // state (this lane's Q and the left neighbour's from the table):
        // k_b (Q_i - Q_{i-1}), the same terms as from positions.
        auto forces = [&](T (&Fo)[B][3], const T (&Ro)[B][3], const bool bonds_from_q) {
            if (bonds_from_q) {
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    const Pos<T> qm = bq[ll + b * W];  // k_b Q_{i-1} (0 for bead 0; HEUN: Q_{i-1})
                    const T Qm[3] = {qm.x, qm.y, qm.z};
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        if constexpr (HEUN)
                            Fo[b][d] = c.k_b * Q[b][d] - c.k_b * Qm[d];
                        else
                            Fo[b][d] = fma(c.k_b, Q[b][d], -Qm[d]);
                    }
                }
            } else {
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    const int i = ll + b * W;
                    const Pos<T> pl = pos[i > 0 ? i - 1 : 0];
                    const Pos<T> pr = pos[i < N - 1 ? i + 1 : i];
                    const T Rl[3] = {pl.x, pl.y, pl.z}, Rr[3] = {pr.x, pr.y, pr.z};
                    // an end bead reads itself for its missing neighbour: that term is 0
#pragma unroll
                    for (int d = 0; d < 3; ++d) Fo[b][d] = c.k_b * (Rl[d] - Ro[b][d]) + c.k_b * (Rr[d] - Ro[b][d]);
                }
            }
            // springs on this bead: -k_s sum_j d_j, slots in ascending order
            // (zero records where there is none)
            T sp[B][3];
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const SlotRec<T> r0 = rec[ll + b * W], r1 = rec[NL + ll + b * W];
                sp[b][0] = r0.x + r1.x;
                sp[b][1] = r0.y + r1.y;
                sp[b][2] = r0.z + r1.z;
            }
            if (more3) {  // a third spring on one bead of the warp: rare
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    Mask mb = msk[ll + b * W];
                    if (mask_popc(mb) > 2) {
                        // the springs of the mask in slot order: the first two, then the rest
                        const int j0 = BY_SLOT ? 0 : rec[ll + b * W].s, j1 = BY_SLOT ? 0 : rec[NL + ll + b * W].s;
                        auto take = [&]() {
                            const int j = mask_ffs(mb) - 1;
                            mb &= mb - Mask(1);
                            if constexpr (BY_SLOT) return tab[j];
                            else return rec[j == j0 ? ll + b * W : (j == j1 ? NL + ll + b * W : 2 * NL + j)];
                        };
                        const SlotRec<T> q0 = take(), q1 = take();
                        Fo[b][0] -= c.k_s * (q0.x + q1.x);
                        Fo[b][1] -= c.k_s * (q0.y + q1.y);
                        Fo[b][2] -= c.k_s * (q0.z + q1.z);
                        sp[b][0] = sp[b][1] = sp[b][2] = T(0);
                        while (mb) {
                            const SlotRec<T> q = take();
                            sp[b][0] += q.x;
                            sp[b][1] += q.y;
                            sp[b][2] += q.z;
                        }
                    }
                }
            }
#pragma unroll
            for (int b = 0; b < B; ++b)
#pragma unroll
                for (int d = 0; d < 3; ++d) Fo[b][d] -= c.k_s * sp[b][d];
        };
        T F[B][3];
        forces(F, R, true);
        // Padding beads (i >= N) are stepped like the others: their bond
        // vectors are zero, they exert no force, carry no spring, enter no
        // stress and are never stored.
        T Rn[B][3];
        [[maybe_unused]] T A0[SB][3];
        if constexpr (HEUN) {
#pragma unroll
            for (int b = 0; b < SB; ++b)
#pragma unroll
                for (int d = 0; d < 3; ++d) A0[b][d] = A[b][d];
        }
#pragma unroll
        for (int b = 0; b < B; ++b) {
            if (ks.nz) {
                if constexpr (std::is_same<T, float>::value) {
                    if (b < BP) {
                        // beads b and b + 1 together; the same operations as the scalar form below
                        if ((b & 1) == 0) {
                            const int b1 = b + 1 < B ? b + 1 : b;
                            const float2 r0 = pk(R[b][0], R[b1][0]), r1 = pk(R[b][1], R[b1][1]),
                                         r2 = pk(R[b][2], R[b1][2]);
#pragma unroll
                            for (int d = 0; d < 3; ++d) {
                                const float2 flow = __ffma2_rn(pk(kz(d)), r2,
                                                               __ffma2_rn(pk(ky(d)), r1,
                                                                          __fmul2_rn(pk(kx(d)), r0)));
                                const float2 e = __ffma2_rn(
                                    pk(c.amp), pk(nrm[b][d], nrm[b1][d]),
                                    __ffma2_rn(pk(c.dt), flow,
                                               __ffma2_rn(pk(c.mob), pk(F[b][d], F[b1][d]), pk(R[b][d], R[b1][d]))));
                                Rn[b][d] = e.x;
                                Rn[b1][d] = e.y;
                            }
                        }
                    } else {
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            const float flow = __fmaf_rn(
                                kz(d), R[b][2],
                                __fmaf_rn(ky(d), R[b][1], __fmul_rn(kx(d), R[b][0])));
                            Rn[b][d] =
                                __fmaf_rn(c.amp, nrm[b][d], __fmaf_rn(c.dt, flow, __fmaf_rn(c.mob, F[b][d], R[b][d])));
                        }
                    }
                } else {
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const T flow = kx(d) * R[b][0] + ky(d) * R[b][1] + kz(d) * R[b][2];
                        Rn[b][d] = R[b][d] + c.mob * F[b][d] + c.dt * flow + c.amp * nrm[b][d];
                    }
                }
            } else if (b < BP) {
                if constexpr (std::is_same<T, float>::value) {
                    if ((b & 1) == 0) {  // beads b and b + 1 together
                        const int b1 = b + 1 < B ? b + 1 : b;
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            const float2 e = __ffma2_rn(pk(c.amp), pk(nrm[b][d], nrm[b1][d]),
                                                        __ffma2_rn(pk(c.mob), pk(F[b][d], F[b1][d]),
                                                                   pk(R[b][d], R[b1][d])));
                            Rn[b][d] = e.x;
                            Rn[b1][d] = e.y;
                        }
                    }
                }
            } else {
#pragma unroll
                for (int d = 0; d < 3; ++d) Rn[b][d] = R[b][d] + c.mob * F[b][d] + c.amp * nrm[b][d];
            }
        }
        if (ks.nz) {
#pragma unroll
            for (int b = 0; b < SB; ++b) {
                if (ll + b * W < Z) {
                    T An[3];
#pragma unroll
                    for (int d = 0; d < 3; ++d)
                        An[d] = A[b][d] +
                                c.dt * (kx(d) * A[b][0] + ky(d) * A[b][1] + kz(d) * A[b][2]);
#pragma unroll
                    for (int d = 0; d < 3; ++d) A[b][d] = An[d];
                }
            }
        }
        if constexpr (HEUN && !FLOW) {
            // Stochastic Heun corrector without a velocity gradient: the
            // anchors stay where they are, so the springs' force at the
            // predicted positions is the step's spring force less
            // k_s n_i (Rn_i - R_i), n_i the number of springs on bead i (the
            // same sum, reordered); only the bond forces are recomputed.
            store_pos(Rn);
            __syncwarp();
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int i = ll + b * W;
                const Pos<T> pl = pos[i > 0 ? i - 1 : 0];
                const Pos<T> pr = pos[i < N - 1 ? i + 1 : i];
                const Pos<T> qm = bq[i];  // Q_{i-1} of the step's start
                const T nsp = T(mask_popc(msk[i]));
                const T Rl[3] = {pl.x, pl.y, pl.z}, Rr[3] = {pr.x, pr.y, pr.z}, Qm[3] = {qm.x, qm.y, qm.z};
                T F2[3];
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const T fb1 = c.k_b * Q[b][d] - c.k_b * Qm[d];  // the bond part of F
                    F2[d] = c.k_b * (Rl[d] - Rn[b][d]) + c.k_b * (Rr[d] - Rn[b][d]) + (F[b][d] - fb1) -
                            c.k_s * nsp * (Rn[b][d] - R[b][d]);
                }
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    Rn[b][d] = R[b][d] + c.hmob * (F[b][d] + F2[d]) + c.amp * nrm[b][d];
            }
        } else if constexpr (HEUN) {
            // Stochastic Heun corrector (the second-order stochastic Runge-Kutta
            // step for additive noise): the Euler state above is the predictor;
            // the drift is averaged between the start and the predicted state
            // (predicted anchors A under a flow), with the springs and the
            // noise of this step.
            __syncwarp();
            store_pos(Rn);
            __syncwarp();
            rewrite_springs();
            __syncwarp();
            T F2[B][3];
            forces(F2, Rn, false);
#pragma unroll
            for (int b = 0; b < B; ++b) {
                T fl[3] = {T(0), T(0), T(0)};
                if (ks.nz) {
#pragma unroll
                    for (int d = 0; d < 3; ++d)
                        fl[d] = (kx(d) * R[b][0] + ky(d) * R[b][1] + kz(d) * R[b][2]) +
                                (kx(d) * Rn[b][0] + ky(d) * Rn[b][1] + kz(d) * Rn[b][2]);
                }
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    Rn[b][d] = R[b][d] + c.hmob * (F[b][d] + F2[b][d]) + c.hdt * fl[d] + c.amp * nrm[b][d];
            }
#pragma unroll
            for (int b = 0; b < SB; ++b) {
                if (ks.nz && ll + b * W < Z) {
                    T An[3];
#pragma unroll
                    for (int d = 0; d < 3; ++d)
                        An[d] = A0[b][d] + c.hdt * ((kx(d) * A0[b][0] + ky(d) * A0[b][1] +
                                                     kz(d) * A0[b][2]) +
                                                    (kx(d) * A[b][0] + ky(d) * A[b][1] +
                                                     kz(d) * A[b][2]));
#pragma unroll
                    for (int d = 0; d < 3; ++d) A[b][d] = An[d];
                }
            }
        }
        // the Heun corrector above read other lanes' positions, so they are
        // overwritten only after a barrier; in the Euler step the last reads
        // of the position table lie behind the barrier that ended the last step
        // (or the setup of the launch) already
        if constexpr (HEUN) __syncwarp();
        store_pos(Rn);
        __syncwarp();

        // ---- substep 2: hops on the new positions, one uniform per spring;
        // sub-slots above every chain's Z in this warp are skipped.  Each slot
        // clears its record and its bead's mask (the forces have read them) and
        // keeps the spring vector dd after the move.
        const int zw = z_w;
        T dd[SB][3];
        bool cand = false;
#pragma unroll
        for (int b = 0; b < SB; ++b) {
            if (!skip(b, zw)) {
                const int i = ll + b * W;
                const bool occ = i < Z;
                const int si = S[b];  // a valid bead index in every slot, occupied or not
                rec[loc[b]] = zrec;
                msk[si] = Mask(0);
                bool up, dn;
                if constexpr (WIN == kWinReplay) {
                    // (a tape recorded from another state must not move a spring off the chain)
                    up = occ && (tb[b] & kTapeUp) && si < N - 1;
                    dn = occ && (tb[b] & kTapeDown) && si > 0;
                    S[b] = up ? si + 1 : (dn ? si - 1 : si);
                    const Pos<T> ps = pos[S[b]];
                    dd[b][0] = ps.x - A[b][0];
                    dd[b][1] = ps.y - A[b][1];
                    dd[b][2] = ps.z - A[b][2];
                } else {
                    const Pos<T> q0 = pos[si], qp = pos[si + 1], qm = pos[si - 1];
                    const T r0[3] = {q0.x - A[b][0], q0.y - A[b][1], q0.z - A[b][2]};
                    const T rp[3] = {qp.x - A[b][0], qp.y - A[b][1], qp.z - A[b][2]};
                    const T rm[3] = {qm.x - A[b][0], qm.y - A[b][1], qm.z - A[b][2]};
                    if constexpr (sizeof(T) == 8) {
                        const bool sure = hop_filter(c, r0, rp, rm, si < N - 1, si > 0, u[b], up, dn);
                        if (__any_sync(kFull, occ && !sure)) {
                            const T d0 = r0[0] * r0[0] + r0[1] * r0[1] + r0[2] * r0[2];
                            const T dp = rp[0] * rp[0] + rp[1] * rp[1] + rp[2] * rp[2];
                            const T dm = rm[0] * rm[0] + rm[1] * rm[1] + rm[2] * rm[2];
                            const T pp = (si < N - 1) ? hop_prob<T>(c, dp, d0) : T(0);
                            const T pm = (si > 0) ? hop_prob<T>(c, dm, d0) : T(0);
                            up = u_value(u[b]) < pp;
                            dn = !up && u_value(u[b]) < pp + pm;
                        }
                        up = occ && up;
                        dn = occ && dn;
                    } else {
                        const T d0 = r0[0] * r0[0] + r0[1] * r0[1] + r0[2] * r0[2];
                        const T dp = fma(rp[2], rp[2], fma(rp[1], rp[1], rp[0] * rp[0]));
                        const T dm = fma(rm[2], rm[2], fma(rm[1], rm[1], rm[0] * rm[0]));
                        const float2 ppm = hop_prob_x2(c, make_float2(dp, dm), d0);
                        const T pp = (si < N - 1) ? ppm.x : T(0);
                        const T pm = (si > 0) ? ppm.y : T(0);
                        up = occ && (u[b] < pp);
                        dn = occ && !up && (u[b] < pp + pm);
                    }
                    if constexpr (WIN == kWinRecord) tb[b] = (up ? kTapeUp : 0) | (dn ? kTapeDown : 0);
                    S[b] = up ? si + 1 : (dn ? si - 1 : si);
#pragma unroll
                    for (int d = 0; d < 3; ++d) dd[b][d] = up ? rp[d] : (dn ? rm[d] : r0[d]);
                }
                cnt_up += up ? 1u : 0u;
                cnt_dn += dn ? 1u : 0u;
                if constexpr (WIN != kWinReplay)
                    cand |= occ && (nrm[b][3] < c.cd) && ((unsigned)(S[b] - 1) >= (unsigned)(N - 2));
            }
        }

        // ---- substep 3a: creation, K attempts at both ends
        if (c_drop) ++cnt_drop;
        // a slot can change only if it may create (u < 2 p_c on an attempt) or
        // sits at an end with a destruction hit: the detailed work below runs
        // only when some slot of the warp can
#pragma unroll
        for (int b = 0; b < SB; ++b) {
            if constexpr (WIN == kWinReplay)
                cand |= (tb[b] & (kTapeNew0 | kTapeNewN | kTapeKillOld | kTapeKillNew)) != 0;
            else  // S = 0 or S = N - 1: S - 1 >= N - 2 as unsigned numbers
                cand |= u[b] < thr_c[b];
        }
        if (__any_sync(kFull, cand)) {
            // ---- substeps 3a and 3b in detail, then the re-indexing: survivors in
            // slot order (sub-slot major, then lane), new springs at bead 1 in
            // attempt order, new springs at bead N
            const int Zc = Z, last = attempts_end();
            const T pc = c.pc[last - Zc], pc2 = T(2) * pc;
            int end_new[SB];  // the end a spring is created at by this slot's attempt, -1 none
            bool gone[SB];    // an old spring destroyed
            bool any_new = false, any_gone = false;
#pragma unroll
            for (int b = 0; b < SB; ++b) {
                const int i = ll + b * W;
                const bool hit = nrm[b][3] < c.cd;
                const bool att = i >= Zc && i < last;
                if constexpr (WIN == kWinReplay) {
                    end_new[b] = !att ? -1 : ((tb[b] & kTapeNew0) ? 0 : ((tb[b] & kTapeNewN) ? N - 1 : -1));
                    gone[b] = i < Zc && (tb[b] & kTapeKillOld);
                } else {
                    end_new[b] = !att ? -1 : (u_value(u[b]) < pc ? 0 : (u_value(u[b]) < pc2 ? N - 1 : -1));
                    gone[b] = i < Zc && hit && (S[b] == 0 || S[b] == N - 1);
                }
                const bool made = end_new[b] >= 0;
                const bool undone =  // created and destroyed within the step
                    made && (WIN == kWinReplay ? (tb[b] & kTapeKillNew) != 0 : a.destroy_new && hit);
                if constexpr (WIN == kWinRecord)
                    tb[b] |= (made ? (end_new[b] == 0 ? kTapeNew0 : kTapeNewN) : 0) | (gone[b] ? kTapeKillOld : 0) |
                             (undone ? kTapeKillNew : 0);
                cnt_cr += made ? 1u : 0u;
                cnt_de += (gone[b] ? 1u : 0u) + (undone ? 1u : 0u);
                if (undone) end_new[b] = -1;
                any_new |= end_new[b] >= 0;
                any_gone |= gone[b];
            }
            int base = Zc;  // springs placed so far
            if (__any_sync(kFull, any_gone)) {
                int dest[SB];
                base = 0;
#pragma unroll
                for (int b = 0; b < SB; ++b) {
                    const bool stays = ll + b * W < Zc && !gone[b];
                    const unsigned kb = __ballot_sync(kFull, stays) & segmask;
                    dest[b] = stays ? base + __popc(kb & lt) : -1;
                    base += __popc(kb);
                }
                __syncwarp();
#pragma unroll
                for (int b = 0; b < SB; ++b) {
                    if (dest[b] >= 0) {
                        SlotRec<T> r;
                        r.x = A[b][0];
                        r.y = A[b][1];
                        r.z = A[b][2];
                        r.s = S[b];
                        tab[dest[b]] = r;
                    }
                }
            }
            int Znew = base;
            if (__any_sync(kFull, any_new)) {
                int dest[SB];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
#pragma unroll
                    for (int b = 0; b < SB; ++b) {
                        const bool here = end_new[b] == (e == 0 ? 0 : N - 1);
                        const unsigned nb = __ballot_sync(kFull, here) & segmask;
                        if (here) dest[b] = Znew + __popc(nb & lt);
                        Znew += __popc(nb);
                    }
                }
                __syncwarp();
#pragma unroll
                for (int b = 0; b < SB; ++b) {
                    if (end_new[b] >= 0) {
                        const Pos<T> pe = pos[end_new[b]];
                        const uint4 wc = philox4x32_10_rk((uint32_t)(ll + b * W), t, kPurposeCreate, chain_id, c.rk0,
                                                          c.rk1);
                        T n3[4];
                        draw_pair<T>(wc.x, wc.y, n3[0], n3[1]);
                        draw_pair<T>(wc.z, wc.w, n3[2], n3[3]);
                        SlotRec<T> r;
                        r.x = pe.x + c.sa * n3[0];
                        r.y = pe.y + c.sa * n3[1];
                        r.z = pe.z + c.sa * n3[2];
                        r.s = end_new[b];
                        tab[dest[b]] = r;
                    }
                }
            }
            __syncwarp();
            // slots whose content moved: all of a chain that lost a spring, else the new ones
#pragma unroll
            for (int b = 0; b < SB; ++b) {
                const int i = ll + b * W;
                if (i < Znew && (base != Zc || i >= Zc)) {
                    const SlotRec<T> r = tab[i];
                    S[b] = r.s;
                    A[b][0] = r.x;
                    A[b][1] = r.y;
                    A[b][2] = r.z;
                }
            }
            __syncwarp();
            Z = Znew;
            set_create();
            spring_vectors(dd);
        }
        if constexpr (WIN == kWinRecord) {
            const long long row = (long long)t0_ + s - a.tape_t0;
            if (live && row >= 0 && row < a.tape_rows) {
#pragma unroll
                for (int b = 0; b < SB; ++b) a.tape[((size_t)row * a.M + mm) * NP + ll + b * W] = tb[b];
            }
        }
        // ---- spring vectors of the new state: this step's stress (with a stiffness
        // of 0 in an empty slot), the next step's spring forces
        __syncwarp();  // every slot has cleared its record and mask
        register_springs(dd);
        const int zn = z_w;
        T sv[VL][3];  // this lane's parts of sigma^(v)_xy, xz, yz
#pragma unroll
        for (int v = 0; v < VL; ++v) sv[v][0] = sv[v][1] = sv[v][2] = T(0);
#pragma unroll
        for (int b = 0; b < SB; ++b) {
            T(&x)[3] = sv[b % VL];
            if (!skip(b, zn)) {
                const T ks_b = ll + b * W < Z ? c.k_s : T(0);
                const T kd0 = ks_b * dd[b][0], kd1 = ks_b * dd[b][1];
                x[0] = fma(kd0, dd[b][1], x[0]);
                x[1] = fma(kd0, dd[b][2], x[1]);
                x[2] = fma(kd1, dd[b][2], x[2]);
            }
        }
#pragma unroll
        for (int b = 0; b < B; ++b)
#pragma unroll
            for (int d = 0; d < 3; ++d) R[b][d] = Rn[b][d];

        // ---- bond vectors of the new state: this step's stress, the next
        // step's bond forces
        bond_vectors();

        // ---- stress of the new state (Eq. stress_tensor_single_chain, App. B)
        const bool do_log = (s == next_log);
        if (do_log) next_log += a.log_every;
        const bool do_rc = (s == next_rc) && ks.nz;
        if (s == next_rc) next_rc += a.recenter_every;
        // per-lane parts of the off-diagonal sigma_ab (bonds) and sigma_ab +
        // sigma^(v)_ab (v[0..5]), and with `diag` the bond part of sigma_aa
        auto stress_parts = [&](T (&vs)[6], T (&dgs)[3], const bool diag) {
            T v[VL][3], dgp[VL][3];
#pragma unroll
            for (int p = 0; p < VL; ++p)
#pragma unroll
                for (int k = 0; k < 3; ++k) v[p][k] = dgp[p][k] = T(0);
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const T(&q)[3] = Q[b];  // the last bead's is 0
                T(&x)[3] = v[b % VL];
                T(&dg)[3] = dgp[b % VL];
                const T kq0 = c.k_b * q[0], kq1 = c.k_b * q[1];
                x[0] = fma(kq0, q[1], x[0]);
                x[1] = fma(kq0, q[2], x[1]);
                x[2] = fma(kq1, q[2], x[2]);
                if (diag) {
                    dg[0] += kq0 * q[0];
                    dg[1] += kq1 * q[1];
                    dg[2] += c.k_b * q[2] * q[2];
                }
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                vs[k] = v[0][k];
                vs[3 + k] = sv[0][k] + v[0][k];
                dgs[k] = dgp[0][k];
                if constexpr (VL == 2) {
                    vs[k] += v[VL - 1][k];
                    vs[3 + k] += sv[VL - 1][k] + v[VL - 1][k];
                    dgs[k] += dgp[VL - 1][k];
                }
            }
        };
        if (corr_on) {  // every step: the correlator's input
            T v[6], dgp[3];
            stress_parts(v, dgp, false);
            if constexpr (sizeof(T) == 4) {
                red_put(v);
            } else {
                const T r = seg_reduce6<T, W>(v, ll);
                if (ser_m != nullptr) ser_m[(size_t)s * ser_step] = r;
            }
        }
        if (do_log) {
            // a log step (warp-uniform, every log_every steps): the stress
            // again with its diagonal, kept out of the every-step path
            T v[6], dgp[3];
            stress_parts(v, dgp, true);
            if constexpr (PAIR) {
                static_assert(B == 1 && VL == 1, "lanes of one bead");
                constexpr int H = W / 2;
                const T ks_h = ll + H < Z ? c.k_s : T(0);  // stiffness of the upper lane's slot
                T q[3], d[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    q[k] = __shfl_down_sync(kFull, Q[0][k], H, W);
                    d[k] = __shfl_down_sync(kFull, dd[0][k], H, W);
                }
                const bool low = ll < H;
#pragma unroll
                for (int k = 0; k < 3; ++k) {  // xy, xz, yz
                    const int a0 = k == 2 ? 1 : 0, a1 = k == 0 ? 1 : 2;
                    const T b = fma(c.k_b * q[a0], q[a1], v[k]);
                    v[k] = low ? b : T(0);
                    v[3 + k] = low ? fma(ks_h * d[a0], d[a1], sv[0][k]) + b : T(0);
                    dgp[k] = low ? fma(c.k_b * q[k], q[k], dgp[k]) : T(0);
                }
            }
            const T r6 = seg_reduce6<T, W>(v, ll);
            T sig[3], dg[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                sig[d] = shfl(r6, d == 0 ? 0 : (d == 1 ? W / 4 : W / 8), W);
                dg[d] = seg_sum<T, W>(dgp[d]) - NkT;
            }
            const int slot = log_slot++;
            if (live && ll == 0 && slot < nlog_) {
                double* L = slog + slot * 14;
                const double v6[6] = {(double)dg[0], (double)dg[1], (double)dg[2],
                                      (double)sig[0], (double)sig[1], (double)sig[2]};
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    atomicAdd(L + k, v6[k]);
                    atomicAdd(L + 6 + k, v6[k] * v6[k]);
                }
                atomicAdd(L + 12, (double)Z);
                atomicAdd(L + 13, (double)Z * (double)Z);
            }
        }
        if (do_rc) {
            T csum[VL][3];
#pragma unroll
            for (int p = 0; p < VL; ++p) csum[p][0] = csum[p][1] = csum[p][2] = T(0);
#pragma unroll
            for (int b = 0; b < B; ++b)
#pragma unroll
                for (int d = 0; d < 3; ++d) csum[b % VL][d] += (ll + b * W < N) ? R[b][d] : T(0);
            T com[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if constexpr (VL == 2) csum[0][d] += csum[VL - 1][d];
                com[d] = seg_sum<T, W>(csum[0][d]) / T(N);
            }
            __syncwarp();
#pragma unroll
            for (int b = 0; b < B; ++b)
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    if (ll + b * W < N) R[b][d] -= com[d];
#pragma unroll
            for (int b = 0; b < SB; ++b)
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    if (ll + b * W < Z) A[b][d] -= com[d];
            store_pos(R);
            // the spring and bond vectors from the shifted coordinates, as a
            // launch starting here computes them: results do not depend on
            // where the launches end
            __syncwarp();
            bond_vectors();
            rewrite_springs();
        }
        __syncwarp();
        if constexpr (sizeof(T) == 4) {
            if (corr_on && ++red_n == RED) red_flush(s + 1);
        }
    }
    if (!FLOW || s >= nsteps_) break;
    load_kappa(s);
    }
    if constexpr (sizeof(T) == 4) {
        if (corr_on) red_flush(nsteps_);
    }

    if (WIN == kWinReplay && a.snapR != nullptr && live) {
        const long long sr = (long long)t0_ + nsteps_ - a.snap_t0;
        if (sr >= 0 && sr <= a.snap_steps) snapshot_store<T, W, B, SB>(a, sr, mm, ll, R, A, S, Z);
    }

    // ---- store state
    T* Rw = static_cast<T*>(a.R);
    T* Aw = static_cast<T*>(a.A);
    bool bad = false, broken = false;  // non-finite position; broken invariant 0 <= Z <= z_max, 0 <= S < N
    if (live) {
        if (ll == 0) a.Z[mm] = Z;
        broken = Z < 0 || Z > a.zmax;
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int i = ll + b * W;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if (i < N) {
                    Rw[((size_t)mm * 3 + d) * NP + i] = R[b][d];
                    bad |= !Mth<T>::finite(R[b][d]);
                }
            }
        }
#pragma unroll
        for (int i0 = 0; i0 < NP; i0 += W) {  // every column: slots above this layout's are empty
            const int i = i0 + ll, b = i0 / W;
            const int sj = b < SB ? S[b < SB ? b : 0] : 0;
            const bool occ = b < SB && i < Z;
            a.S[(size_t)mm * NP + i] = occ ? sj : -1;
            broken |= occ && (sj < 0 || sj >= N);
#pragma unroll
            for (int d = 0; d < 3; ++d)
                Aw[((size_t)mm * 3 + d) * NP + i] = occ ? A[b < SB ? b : 0][d] : T(0);
        }
    }
    unsigned long long* const counters = a.counters + (blockIdx.x & a.cnt_mask) * 8;
    if (__any_sync(kFull, bad) && lane == 0) {
        atomicOr(a.status, 1);
        atomicAdd(counters + 6, 1ull);
    }
    if (__any_sync(kFull, broken) && lane == 0) {
        atomicOr(a.status, 2);
        atomicAdd(counters + 7, 1ull);
    }

    // ---- event counters (padding segments beyond the element's chains count nothing)
    {
        unsigned v[5] = {cnt_up, cnt_dn, cnt_cr, cnt_de, cnt_drop};
        if (!live) v[0] = v[1] = v[2] = v[3] = v[4] = 0u;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const unsigned x = __reduce_add_sync(kFull, v[k]);
            if (lane == 0 && x) atomicAdd(counters + k, (unsigned long long)x);
        }
    }

    // ---- stress logs: add this CTA's sums to its group
    if (a.log_every > 0 && nlog_ > 0) {
        __syncthreads();
        const long long first_m = t0_ / a.log_every + 1;  // first log multiple in or after t0+1
        const int slice = cta_first / kSliceChains;
        const int grp = (int)(((long long)slice * a.groups) / a.slices);
        for (int i = threadIdx.x; i < nlog_ * 14; i += blockDim.x) {
            const int slot = i / 14, k = i % 14;
            const long long idx = first_m + slot - log_m0_ - 1;
            const long long step = (first_m + slot) * a.log_every;
            if (step <= t0_ + nsteps_ && idx >= 0 && idx < a.max_logs && slog[i] != 0.0)
                atomicAdd(a.logs + ((size_t)idx * a.groups + grp) * 14 + k, slog[i]);
        }
    }
}

// WIN: the differentiation-window hooks are compiled in (kWinRecord,
// kWinReplay); the plain kernel (kWinOff) carries none of them.  FLOW: the
// velocity-gradient terms are compiled in (launches with kappa = 0 throughout
// may use the instantiation without them).  HEUN: the stochastic Heun
// integrator instead of Euler-Maruyama for substep 1.  CORR: a stress series may
// be written (without one, its registers are free).  ALT: the second form of a layout.
template <typename T, int W, int B, int WIN, bool FLOW, bool HEUN, bool CORR, bool ALT = false>
__global__ void __launch_bounds__(kChunkThreads, chunk_warps_per_sm<T>(W, B, HEUN, FLOW, ALT))
    chunk_kernel(const ChunkArgs a, const StepConst<T> c) {
    run_chains<T, W, B, WIN, FLOW, HEUN, CORR, W == 8 ? 2 : 1, CORR ? red_steps<T>(W, B, HEUN, FLOW, ALT) : 0, false>(
        a, c, (blockIdx.x + a.cta0) * (blockDim.x / W), c.NkT, a.t0, a.nsteps, a.log_m0, a.nlog_chunk);
}

// ------------------------------------------------------ batched kernel ------
// Many elements in one launch per lane layout: CTA k runs work item k (element,
// first chain of a CTA tile) of its layout class for all steps of the launch.  The
// items are ordered longest first and the hardware starts CTAs in order, as slots
// free up.  Each element's arguments (state pointers, sizes, flow schedule, log
// buffers) live in a device array; a CTA reads them from shared memory.
struct RunInfo {
    long long t0;     // first step of this launch
    int nsteps;
    long long log_m0;
};

template <typename T, int W, int B>
__global__ void __launch_bounds__(kChunkThreads, chunk_warps_per_sm<T>(W, B))
    batched_kernel(const ChunkArgs* __restrict__ elems, const int2* __restrict__ items, const RunInfo info,
                   const StepConst<T> c) {
    static_assert(sizeof(ChunkArgs) % 8 == 0, "copied in 8-byte words");
    __shared__ unsigned long long args_s[sizeof(ChunkArgs) / 8];
    // volatile: read where they are used (most of them in rare branches), not kept
    // in registers for the whole launch
    const volatile ChunkArgs& a = *reinterpret_cast<const volatile ChunkArgs*>(args_s);
    const int2 wi = items[blockIdx.x];
    for (int i = threadIdx.x; i < (int)(sizeof(ChunkArgs) / 8); i += blockDim.x)
        args_s[i] = reinterpret_cast<const unsigned long long*>(elems + wi.x)[i];
    __syncthreads();
    const int nlog = a.log_every > 0 ? (int)((info.t0 + info.nsteps) / a.log_every - info.t0 / a.log_every) : 0;
    // 8 x 2 adds the stress of a lane's two beads in one fused sum here and in two in
    // chunk_kernel: the stress logs of the two paths differ by FP32 rounding there.  (The
    // centre of mass, the only sum over beads that enters a state, is the same either
    // way.)  16 x 1 and 32 x 1 sum as 8 x 2 and 16 x 2 do, so that the logs of a length
    // are the same in every layout it may run in.
    constexpr bool PAIR = B == 1 && W > 8;
    constexpr int VL = W == 8 && B != 2 ? 2 : 1;
    run_chains<T, W, B, kWinOff, true, false, false, VL, 0, PAIR>(a, c, wi.y, T((double)a.N) * c.kT, info.t0, info.nsteps,
                                                        info.log_m0, nlog);
}

}  // namespace ssk
