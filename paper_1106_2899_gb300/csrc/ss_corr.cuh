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
// q = 3..5 (sigma + sigma^(v))_off; a warp holds 5 chains x 6 rows, and the
// later value x of row q is row q % 3 of the same chain, taken by a shuffle.
// Samples of a level are [j][M][6] arrays (the chain kernel's series for
// level 0).  hist [M][L][6][16] keeps the newest 16 samples of every level
// and row (oldest first, zero after a reset): the lags reach back into
// earlier launches through a 16-entry register ring; each level's pass
// writes its own history when it ends.  A CTA covers one slice of
// kSliceChains chains and adds its chains' sums of this launch, in chain
// order, to the slice's FP64 sums acc64 [slices][L][3][32] (component,
// channel * 16 + lag).  With TT the rows of sigma + sigma^(v) also take their
// own samples as the later value (channel TT, acc64tt [slices][L][3][16]).
constexpr int kCorrChainsPerWarp = 5;
constexpr int kCorrWarps = (kSliceChains + kCorrChainsPerWarp - 1) / kCorrChainsPerWarp;  // 13
constexpr int kCorrThreads = kCorrWarps * 32;
constexpr int kCorrMaxSteps = 1024;  // samples per launch (the level-sample buffers hold half)

// This slice's FP32 sums of one level (each thread's lags k0..15 of its row),
// folded in chain order into FP64.
// Channel TT of the rows q >= 3, folded the same way into out [3][16].
// Sum of column i over the kSliceChains rows of red (row stride `stride`), in
// chain order, in FP64.  FP32 rows go in blocks of eight: a block is summed in
// FP32 while the rounding error of every addition is kept exactly (TwoSum,
// Knuth) and summed beside it, then the block's sum and error are added in
// FP64.  The result has FP64 accuracy with a quarter of the FP64 conversions
// and additions (the FP64 pipe runs at a small fraction of the FP32 rate).
template <typename T>
__device__ __forceinline__ double slice_column_sum(const T* red, int stride, int i) {
    static_assert(kSliceChains % 8 == 0, "blocks of eight chains");
    double sum = 0.0;
    if constexpr (sizeof(T) == 4) {
        for (int c0 = 0; c0 < kSliceChains; c0 += 8) {
            float s = red[(size_t)c0 * stride + i], e = 0.0f;
#pragma unroll
            for (int c = 1; c < 8; ++c) {
                const float x = red[(size_t)(c0 + c) * stride + i];
                const float t = s + x;
                const float bp = t - s;
                e += (s - (t - bp)) + (x - bp);
                s = t;
            }
            sum += (double)s;
            sum += (double)e;
        }
    } else {
        for (int c = 0; c < kSliceChains; ++c) sum += (double)red[(size_t)c * stride + i];
    }
    return sum;
}

template <typename T>
__device__ __forceinline__ void corr_fold_slice_tt(const T (&acc2)[16], int k0, bool live, int slot, int q,
                                                   double* __restrict__ out, T* red) {
    __syncthreads();  // the first fold has read red
    if (slot < kSliceChains && q >= 3) {
        T* row = red + (size_t)slot * 48 + (q - 3) * kP;
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (k >= k0) row[k] = live ? acc2[k] : T(0);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 48; i += blockDim.x) {
        if (i % kP < k0) continue;
        out[i] += slice_column_sum(red, 48, i);
    }
}

template <typename T>
__device__ __forceinline__ void corr_fold_slice(const T (&acc)[16], int k0, bool live, int slot, int q,
                                                double* __restrict__ out, T* red) {
    // red: [kSliceChains][96] T in shared memory, free once every thread is here
    __syncthreads();
    if (slot < kSliceChains) {
        T* row = red + (size_t)slot * 96 + (q % 3) * kCells + (q / 3) * kP;
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (k >= k0) row[k] = live ? acc[k] : T(0);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 96; i += blockDim.x) {
        const int lag = i % kP;
        if (lag < k0) continue;
        out[i] += slice_column_sum(red, 96, i);
    }
}

// Ring of the newest 16 samples of one row: r[i] holds sample base + i - 16
// when the next sample to enter is sample base (i.e. after a whole number of
// 16-sample blocks).  Products of n new samples, sample j given by get(j) (a
// load), each later value x taken from lane src_lane; emit(j, y) sees every
// sample in order (the pair means of the level above are formed there).  nr
// returns the ring position of the next sample (the number of samples in the
// last partial block).  With TT, acc2 also takes the row's own sample as the
// later value (for the rows of sigma + sigma^(v): channel TT).
template <typename T, int K0, bool TT, typename Get, typename Emit>
__device__ __forceinline__ void corr_ring_products(T (&r)[16], T (&acc)[16], T (&acc2)[16], Get get, Emit emit,
                                                   int n, int src_lane, int& nr) {
    int j = 0;
    for (; j + 16 <= n; j += 16) {
        T yv[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) yv[u] = get(j + u);  // independent loads first
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            emit(j + u, yv[u]);
            const T xv = __shfl_sync(kFull, yv[u], src_lane);
            r[u] = yv[u];
#pragma unroll
            for (int k = K0; k < 16; ++k) acc[k] += xv * r[(u - k) & 15];
            if constexpr (TT) {
#pragma unroll
                for (int k = K0; k < 16; ++k) acc2[k] += yv[u] * r[(u - k) & 15];
            }
        }
    }
    const int rem = n - j;
#pragma unroll
    for (int u = 0; u < 16; ++u) {
        if (u < rem) {
            const T yv = get(j + u);
            emit(j + u, yv);
            const T xv = __shfl_sync(kFull, yv, src_lane);
            r[u] = yv;
#pragma unroll
            for (int k = K0; k < 16; ++k) acc[k] += xv * r[(u - k) & 15];
            if constexpr (TT) {
#pragma unroll
                for (int k = K0; k < 16; ++k) acc2[k] += yv * r[(u - k) & 15];
            }
        }
    }
    nr = rem;
}

// The newest 16 samples in ring order after `nr` samples of a partial block:
// out[i] = r[(nr + i) & 15].
template <typename T>
__device__ __forceinline__ void corr_ring_newest(const T (&r)[16], int nr, T* out) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        T v = r[0];
#pragma unroll
        for (int s2 = 1; s2 < 16; ++s2)
            if (((nr + i) & 15) == s2) v = r[s2];
        out[i] = v;
    }
}

// All levels of one launch in one kernel.  Level l's pass reads the level-l
// samples of this launch (the series rows for level 0, else the samples the
// pass below stored), adds their products, and, as the samples stream by,
// stores the pairwise means that are the level-(l+1) samples into one of the
// ping-pong buffers lev (lev_half elements each).  A mean may pair the newest
// level-l sample of the previous launch (the last entry of the level's
// history) with the first new one.  Every thread reads only rows it wrote
// itself (its chain and series row); the block synchronises only for the
// slice folds.
template <typename T, bool TT>
__global__ void __launch_bounds__(kCorrThreads, (sizeof(T) == 4 && !TT) ? 2 : 1)
    corr_kernel(const T* __restrict__ ser, int ns, long long n0, int M, int L, T* __restrict__ hist,
                T* __restrict__ lev, size_t lev_half, double* __restrict__ acc64, double* __restrict__ acc64tt) {
    __shared__ T red[kSliceChains * 96];
    const int lane = threadIdx.x & 31;
    const int cc = lane / 6, q = lane % 6;
    const int slot = (threadIdx.x >> 5) * kCorrChainsPerWarp + cc;  // chain within the slice
    const int fslot = lane < 30 ? slot : kSliceChains;
    const int m = blockIdx.x * kSliceChains + slot;
    const bool live = lane < 30 && slot < kSliceChains && m < M;
    const int mm = live ? m : 0;
    const int src_lane = min(cc * 6 + q % 3, 31);
    const size_t stride = (size_t)M * 6;
    auto cl_of = [&](int l) { return (int)(((n0 + ns) >> l) - (n0 >> l)); };

    const T* yin = ser;  // level-l samples of this launch
    int cl = ns;
    for (int l = 0; l < L && cl > 0; ++l) {
        const int k0 = l == 0 ? 0 : kP / 2;
        T* h = hist + (((size_t)mm * L + l) * 6 + q) * 16;
        T r[16], acc[16], acc2[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            r[i] = live ? h[i] : T(0);
            acc[i] = T(0);
            acc2[i] = T(0);
        }
        // level-(l+1) sample J is the mean of level-l samples off + 2J and
        // off + 2J + 1 of this launch; sample -1 is the newest before it
        const int cn = l + 1 < L ? cl_of(l + 1) : 0;
        const int off = (int)(2 * (n0 >> (l + 1)) - (n0 >> l));  // -1 or 0
        T* const yout = lev + (size_t)(l & 1) * lev_half;
        T* const orow = yout + (size_t)mm * 6 + q;
        T prev = r[15];
        auto emit = [&](int a, T y) {
            const int J = (a - off - 1) >> 1;
            if (((a - off - 1) & 1) == 0 && J < cn && live) orow[(size_t)J * stride] = T(0.5) * (prev + y);
            prev = y;
        };
        const T* yrow = yin + (size_t)mm * 6 + q;
        int nr = 0;
        if (l == 0)
            corr_ring_products<T, 0, TT>(r, acc, acc2, [&](int j) { return yrow[(size_t)j * stride]; }, emit, cl,
                                         src_lane, nr);
        else
            corr_ring_products<T, kP / 2, TT>(r, acc, acc2, [&](int j) { return yrow[(size_t)j * stride]; }, emit,
                                              cl, src_lane, nr);
        corr_fold_slice(acc, k0, live, fslot, q, acc64 + ((size_t)blockIdx.x * L + l) * 96, red);
        if constexpr (TT) corr_fold_slice_tt(acc2, k0, live, fslot, q, acc64tt + ((size_t)blockIdx.x * L + l) * 48, red);
        if (live) {
            T nh[16];
            corr_ring_newest(r, nr, nh);
#pragma unroll
            for (int i = 0; i < 16; ++i) h[i] = nh[i];
        }
        yin = yout;
        cl = cn;
    }
}

// Correlator group sums from the slice sums: out[g][l][lag][ch][d] (the layout
// of ss_corr_sums) = sum over the slices of group g, in slice order, of
// acc64[s][l][d * 32 + ch * 16 + lag].  One thread per (g, l, cell).
__global__ void corr_group_kernel(const double* __restrict__ acc64, int slices, int groups, int L,
                                  double* __restrict__ out) {
    const int id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= groups * L * 96) return;
    const int g = id / (L * 96), l = (id / 96) % L, i = id % 96;
    const int d = i / 32, ch = (i % 32) / 16, lag = i % 16;
    // slices of group g: s with floor(s * groups / slices) == g
    const int s0 = (int)(((long long)g * slices + groups - 1) / groups);
    const int s1 = (int)(((long long)(g + 1) * slices + groups - 1) / groups);
    double sum = 0.0;
    for (int sl = s0; sl < s1; ++sl) sum += acc64[((size_t)sl * L + l) * 96 + i];
    out[((((size_t)g * L + l) * 16 + lag) * 2 + ch) * 3 + d] = sum;
}

}  // namespace ssk
