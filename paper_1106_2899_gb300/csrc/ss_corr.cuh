// ss_corr.cuh -- multiple-tau correlator of the chain kernel's stress series.
#pragma once
#include "ss_kernels.cuh"

namespace ssk {

// ----------------------------------------------------- correlator kernels ----
// Multiple-tau lag products of one launch's stress series (Eq.
// relaxation_modulus_tensor_green_kubo_form, App. B).  Level 0 holds the raw
// samples; level l >= 1 the means of two consecutive level-(l-1) samples, i.e.
// of blocks of 2^l raw samples aligned to the absolute sample index.  At level
// l, lag k (0..15 at level 0, 8..15 above) adds x_l(j) y_l(j - k) for every
// sample j completed in this launch, with x = sigma_off (the later value) and
// y = sigma_off (AUTO channel) or (sigma + sigma^(v))_off (TOTAL channel).
//
// One thread per (chain, series row q): q = 0..2 are sigma_off (xy, xz, yz),
// q = 3..5 (sigma + sigma^(v))_off; a warp holds 5 chains x 6 rows, and the later
// value x of row q is row q % 3 of the same chain, taken by a shuffle.  A pass takes two levels: the samples of level l stream by from
// memory (the chain kernel's series for level 0, else what the pass below stored),
// their pair means are the samples of level l + 1 and never leave the registers,
// and the pair means of those are stored as the samples of level l + 2.  So the
// sample traffic is 1.7 times the series and there are half as many passes as
// levels.  (One level per pass moved 3 times the series through memory.)
// hist [M][L][6][16] keeps the newest 16 samples of every level and row (oldest
// first, zero after a reset): the lags reach back into earlier launches through a
// 16-entry register ring.  A CTA covers one part of a slice of kSliceChains chains
// and adds its chains' sums of this launch to the part's FP64 sums acc64
// [parts][L][3][32] (component, channel * 16 + lag).  With TT the rows of
// sigma + sigma^(v) also take their own samples as the later value (channel TT,
// acc64tt [parts][L][3][16]).
constexpr int kCorrMaxSteps = 1024;  // samples per launch (the level-sample buffers hold a quarter)
constexpr int kCorrPartChains = 32;  // chains per CTA at most, but for callers that keep one sum per slice

// Chains per CTA: 32 in seven warps, or, in ensembles too small to fill the chip
// with those, 16 in four warps, over twice the SMs.
__host__ __device__ constexpr int corr_chains(int M) { return M >= 8192 ? 32 : 16; }
__host__ __device__ constexpr int corr_parts(int M) {  // parts of a slice
    return kSliceChains / corr_chains(M);
}
constexpr int kCorrChainsPerWarp = 5;
__host__ __device__ constexpr int corr_threads(int chains) {
    return (chains + kCorrChainsPerWarp - 1) / kCorrChainsPerWarp * 32;
}

// Sums of column i of red over the eight chains from c0 on, in FP64.  FP32 values
// are summed in FP32 while the rounding error of every addition is kept exactly
// (TwoSum, Knuth) and summed beside them.  The result has FP64 accuracy with a
// quarter of the FP64 conversions and additions.
template <typename T>
__device__ __forceinline__ double corr_eight_chains(const T* red, int stride, int c0, int i) {
    if constexpr (sizeof(T) == 4) {
        float s = red[(size_t)c0 * stride + i], e = 0.0f;
#pragma unroll
        for (int c = 1; c < 8; ++c) {
            const float x = red[(size_t)(c0 + c) * stride + i];
            const float t = s + x;
            const float bp = t - s;
            e += (s - (t - bp)) + (x - bp);
            s = t;
        }
        return (double)s + (double)e;
    } else {
        double s = 0.0;
#pragma unroll
        for (int c = 0; c < 8; ++c) s += red[(size_t)(c0 + c) * stride + i];
        return s;
    }
}

// This CTA's sums of one level (each thread's lags k0..15 of its row, column col0
// + lag of W columns), folded into out [W]; mine: this thread owns a row.
template <typename T, int W>
__device__ __forceinline__ void corr_fold(const T (&acc)[16], int k0, bool live, bool mine, int c, int col0, int chains,
                                          double* __restrict__ out, T* red) {
    __syncthreads();  // the last fold has read red
    if (mine) {
        T* row = red + (size_t)c * W + col0;
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (k >= k0) row[k] = live ? acc[k] : T(0);
    }
    __syncthreads();
    const int tasks = W * (chains / 8);  // at most two per thread
    double p[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int i = threadIdx.x + k * blockDim.x;
        p[k] = i < tasks && i % kP >= k0 ? corr_eight_chains(red, W, i / W * 8, i % W) : 0.0;
    }
    __syncthreads();
    double* part = reinterpret_cast<double*>(red);
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if ((int)(threadIdx.x + k * blockDim.x) < tasks) part[threadIdx.x + k * blockDim.x] = p[k];
    __syncthreads();
    for (int i = threadIdx.x; i < W; i += blockDim.x) {
        if (i % kP < k0) continue;
        double s = part[i];
        for (int b = 1; b < chains / 8; ++b) s += part[b * W + i];
        out[i] += s;
    }
}

// Sixteen samples of one row's history.
template <typename T>
__device__ __forceinline__ void corr_hist_load(const T* __restrict__ h, T (&r)[16]) {
    using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    constexpr int n = 16 / (sizeof(V) / sizeof(T));
#pragma unroll
    for (int i = 0; i < n; ++i) reinterpret_cast<V*>(r)[i] = reinterpret_cast<const V*>(h)[i];
}
// The newest 16 samples, oldest first, after n samples in the ring: r rotated left
// by n mod 16 (four conditional rotations), stored.
template <typename T>
__device__ __forceinline__ void corr_hist_store(T* __restrict__ h, T (&r)[16], int n) {
#pragma unroll
    for (int s = 8; s > 0; s >>= 1) {
        if (n & s) {
            T x[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = r[(i + s) & 15];
#pragma unroll
            for (int i = 0; i < 16; ++i) r[i] = x[i];
        }
    }
    using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    constexpr int m = 16 / (sizeof(V) / sizeof(T));
#pragma unroll
    for (int i = 0; i < m; ++i) reinterpret_cast<V*>(h)[i] = reinterpret_cast<const V*>(r)[i];
}

// The two levels of one pass for one thread: rings (ring position of a sample: its
// index in this launch mod 16), sums, the newest sample of each level.
template <typename T>
struct CorrPass {
    alignas(16) T rA[16], rB[16];
    T accA[16], accB[16], ttA[16], ttB[16];
    T py, pz;
};

// Samples on their way: groups of eight are copied to shared memory three groups
// ahead of their use (FP32), each lane its own row, by asynchronous 4-byte copies.
// A warp then has 24 rows in flight instead of the eight its registers can hold:
// the loads' latency bound the kernel.
constexpr int kCorrStage = 32;  // samples of a row in shared memory
__device__ __forceinline__ void corr_copy_group(float* st, const float* yrow, size_t stride, int j, int n) {
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        if (j + v < n) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(st + ((j + v) & (kCorrStage - 1)) * 32);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(yrow + (size_t)(j + v) * stride)
                         : "memory");
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// Up to 32 samples of level l from sample j0 on (all 32 unless TAIL) of n: products
// of lags K0..15, and of lags 8..15 of the pair means.  ODD: the first sample of the
// launch completes a pair with the newest one before it.
template <typename T, int K0, bool ODD, bool TT, bool TAIL, bool STAGE>
__device__ __forceinline__ void corr_block(CorrPass<T>& s, const T* yrow, T* st, int src, size_t stride, int j0, int n,
                                           bool has_b, bool odd_b, T* out, bool emit) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        T yv[8];
        if constexpr (STAGE) {
            if (!TAIL || j0 + h * 8 < n) {
                corr_copy_group(st, yrow, stride, j0 + h * 8 + 24, n);
                asm volatile("cp.async.wait_group 3;" ::: "memory");
            }
#pragma unroll
            for (int v = 0; v < 8; ++v) yv[v] = st[(h * 8 + v) * 32];
        } else {
            asm volatile("" ::: "memory");  // one group of loads at a time: all 32 at once would spill
#pragma unroll
            for (int v = 0; v < 8; ++v)  // independent loads first
                if (!TAIL || j0 + h * 8 + v < n) yv[v] = yrow[(size_t)(j0 + h * 8 + v) * stride];
        }
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            const int u = h * 8 + v;
            if (!TAIL || j0 + u < n) {
                const T y = yv[v], x = __shfl_sync(kFull, y, src);
                s.rA[u & 15] = y;
#pragma unroll
                for (int k = K0; k < 16; ++k) s.accA[k] += x * s.rA[(u - k) & 15];
                if constexpr (TT) {
#pragma unroll
                    for (int k = K0; k < 16; ++k) s.ttA[k] += y * s.rA[(u - k) & 15];
                }
                if (has_b && (u & 1) == (ODD ? 0 : 1)) {
                    const int j = u >> 1;  // sample j0 / 2 + j of level l + 1
                    const T z = T(0.5) * (s.py + y), zx = __shfl_sync(kFull, z, src);
                    s.rB[j & 15] = z;
#pragma unroll
                    for (int k = kP / 2; k < 16; ++k) s.accB[k] += zx * s.rB[(j - k) & 15];
                    if constexpr (TT) {
#pragma unroll
                        for (int k = kP / 2; k < 16; ++k) s.ttB[k] += z * s.rB[(j - k) & 15];
                    }
                    if (emit && (j & 1) == (odd_b ? 0 : 1)) out[(size_t)((j0 / 2 + j) >> 1) * stride] = T(0.5) * (s.pz + z);
                    s.pz = z;
                }
                s.py = y;
            }
        }
    }
}

template <typename T, int K0, bool ODD, bool TT, bool STAGE>
__device__ __forceinline__ void corr_levels(CorrPass<T>& s, const T* yrow, T* st, int src, size_t stride, int n,
                                            bool has_b, bool odd_b, T* out, bool emit) {
    if constexpr (STAGE) {
#pragma unroll
        for (int g = 0; g < 3; ++g) corr_copy_group(st, yrow, stride, 8 * g, n);
    }
    int j = 0;
    for (; j + 32 <= n; j += 32)
        corr_block<T, K0, ODD, TT, false, STAGE>(s, yrow, st, src, stride, j, n, has_b, odd_b, out, emit);
    if (j < n) corr_block<T, K0, ODD, TT, true, STAGE>(s, yrow, st, src, stride, j, n, has_b, odd_b, out, emit);
    if constexpr (STAGE) asm volatile("cp.async.wait_all;" ::: "memory");
}

// All levels of one launch: ns samples after n0 earlier ones.  CTA b + b0
// = B has the `chains` <= CHAINS chains from B * span + first on and the sums of
// part B.  lev: two buffers of lev_half elements for the samples the
// passes store.  A pair may join the newest sample of the previous launch (the last
// entry of the level's history) and the first new one.
template <typename T, bool TT, int CHAINS>
__global__ void __launch_bounds__(corr_threads(CHAINS), sizeof(T) == 4 && !TT && CHAINS == kCorrPartChains ? 2 : 1)
    corr_kernel(const T* __restrict__ ser, int b0, int chains, int first, int span, int ns, long long n0, int M, int L, T* __restrict__ hist,
                T* lev, size_t lev_half, double* __restrict__ acc64, double* __restrict__ acc64tt) {
    constexpr bool STAGE = sizeof(T) == 4 && CHAINS == kCorrPartChains;
    __shared__ alignas(16) T red[CHAINS * 96];
    __shared__ T stage[STAGE ? corr_threads(CHAINS) * kCorrStage : 1];
    const int lane = threadIdx.x & 31, q = lane % 6;
    const int c = (threadIdx.x >> 5) * kCorrChainsPerWarp + lane / 6;  // chain of this CTA
    const bool mine = lane < 30 && c < chains;
    const int block = blockIdx.x + b0;
    const int m = block * span + first + c;
    const bool live = mine && m < M;
    const int src = min(lane / 6 * 6 + q % 3, 31);
    const int mm = live ? m : 0;
    T* const st = stage + (STAGE ? (threadIdx.x >> 5) * kCorrStage * 32 + lane : 0);
    const size_t stride = (size_t)M * 6;
    auto count = [&](int l) { return l < L ? (int)(((n0 + ns) >> l) - (n0 >> l)) : 0; };

    const T* yin = ser;  // samples of level l of this launch
    for (int l = 0; l < L && count(l) > 0; l += 2) {
        const int nA = count(l), nB = count(l + 1);
        const bool odd_a = (n0 >> l) & 1, odd_b = (n0 >> (l + 1)) & 1;
        T* const hA = hist + (((size_t)mm * L + l) * 6 + q) * 16;
        T* const hB = hA + 6 * 16;
        CorrPass<T> s;
#pragma unroll
        for (int i = 0; i < 16; ++i) s.accA[i] = s.accB[i] = s.ttA[i] = s.ttB[i] = s.rB[i] = T(0);
        corr_hist_load(hA, s.rA);
        s.py = s.rA[15];
        if (nB > 0) corr_hist_load(hB, s.rB);
        s.pz = s.rB[15];
        T* const yout = lev + (size_t)((l >> 1) & 1) * lev_half;
        T* const out = yout + (size_t)mm * 6 + q;
        const T* yrow = yin + (size_t)mm * 6 + q;
        const bool emit = live && count(l + 2) > 0;
        if (l == 0) {
            if (odd_a)
                corr_levels<T, 0, true, TT, STAGE>(s, yrow, st, src, stride, nA, nB > 0, odd_b, out, emit);
            else
                corr_levels<T, 0, false, TT, STAGE>(s, yrow, st, src, stride, nA, nB > 0, odd_b, out, emit);
        } else {
            if (odd_a)
                corr_levels<T, kP / 2, true, TT, STAGE>(s, yrow, st, src, stride, nA, nB > 0, odd_b, out, emit);
            else
                corr_levels<T, kP / 2, false, TT, STAGE>(s, yrow, st, src, stride, nA, nB > 0, odd_b, out, emit);
        }
        double* const oA = acc64 + ((size_t)block * L + l) * 96;
        const int col = (q % 3) * kCells + (q / 3) * kP;
        corr_fold<T, 96>(s.accA, l == 0 ? 0 : kP / 2, live, mine, c, col, chains, oA, red);
        if (nB > 0) corr_fold<T, 96>(s.accB, kP / 2, live, mine, c, col, chains, oA + 96, red);
        if constexpr (TT) {
            double* const oT = acc64tt + ((size_t)block * L + l) * 48;
            corr_fold<T, 48>(s.ttA, l == 0 ? 0 : kP / 2, live, mine && q >= 3, c, (q - 3) * kP, chains, oT, red);
            if (nB > 0) corr_fold<T, 48>(s.ttB, kP / 2, live, mine && q >= 3, c, (q - 3) * kP, chains, oT + 48, red);
        }
        if (live) {
            corr_hist_store(hA, s.rA, nA);
            if (nB > 0) corr_hist_store(hB, s.rB, nB);
        }
        yin = yout;  // each thread reads back the samples it stored
    }
}

// The same for a launch of one step (programs that do something of their own
// between steps): sample n0 enters level 0 and, while the level's sample completes
// a pair, the levels above.  No sums live across samples, so 28 warps fit an SM
// instead of 14 and nothing but the histories moves.
template <typename T, bool TT>
__global__ void __launch_bounds__(corr_threads(kCorrPartChains), sizeof(T) == 4 ? 4 : 2)
    corr_step_kernel(const T* __restrict__ ser, int b0, int chains, int first, int span, long long n0, int M, int L,
                     T* __restrict__ hist, double* __restrict__ acc64, double* __restrict__ acc64tt) {
    __shared__ alignas(16) T red[kCorrPartChains * 96];
    const int lane = threadIdx.x & 31, q = lane % 6;
    const int c = (threadIdx.x >> 5) * kCorrChainsPerWarp + lane / 6;  // chain of this CTA
    const bool mine = lane < 30 && c < chains;
    const int block = blockIdx.x + b0;
    const int m = block * span + first + c;
    const bool live = mine && m < M;
    const int src = min(lane / 6 * 6 + q % 3, 31);
    const int mm = live ? m : 0;
    T y = ser[(size_t)mm * 6 + q];
    for (int l = 0; l < L; ++l) {
        const int k0 = l == 0 ? 0 : kP / 2;
        T* const h = hist + (((size_t)mm * L + l) * 6 + q) * 16;
        alignas(16) T r[16];
        corr_hist_load(h, r);
        const T x = __shfl_sync(kFull, y, src);
        const bool up = (n0 >> l) & 1;  // completes a pair
        const T mean = T(0.5) * (r[15] + y);
        T acc[16];
        acc[0] = x * y;
#pragma unroll
        for (int k = 1; k < 16; ++k) acc[k] = x * r[16 - k];
        const size_t part = (size_t)block * L + l;
        corr_fold<T, 96>(acc, k0, live, mine, c, (q % 3) * kCells + (q / 3) * kP, chains, acc64 + part * 96, red);
        if constexpr (TT) {
            acc[0] = y * y;
#pragma unroll
            for (int k = 1; k < 16; ++k) acc[k] = y * r[16 - k];
            corr_fold<T, 48>(acc, k0, live, mine && q >= 3, c, (q - 3) * kP, chains, acc64tt + part * 48, red);
        }
        if (live) {
#pragma unroll
            for (int i = 0; i < 15; ++i) r[i] = r[i + 1];
            r[15] = y;
            corr_hist_store(h, r, 0);
        }
        if (!up) break;
        y = mean;
    }
}

// Correlator group sums from the part sums, in order.  acc64 [slices * parts][L]
// [W]: W = 96 (component * 32 + channel * 16 + lag) or 48 (channel TT: component *
// 16 + lag); out[g][l][lag][channel][component], the layout of ss_corr_sums and
// ss_corr_sums_tt.  Group g has the slices s with floor(s * groups / slices) = g.
// One thread per (g, l, cell).
template <int W>
__global__ void corr_group_kernel(const double* __restrict__ acc64, int slices, int parts, int groups, int L,
                                  double* __restrict__ out) {
    constexpr int CH = W / 48;
    const int id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= groups * L * W) return;
    const int g = id / (L * W), l = (id / W) % L, i = id % W;
    const int d = i / (CH * kP), ch = (i / kP) % CH, lag = i % kP;
    const int s0 = (int)(((long long)g * slices + groups - 1) / groups);
    const int s1 = (int)(((long long)(g + 1) * slices + groups - 1) / groups);
    double sum = 0.0;
    for (int sl = s0 * parts; sl < s1 * parts; ++sl) sum += acc64[((size_t)sl * L + l) * W + i];
    out[((((size_t)g * L + l) * 16 + lag) * CH + ch) * 3 + d] = sum;
}

}  // namespace ssk
