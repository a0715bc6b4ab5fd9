// ss_state.cuh -- initial state, state upload and export, spring-number histogram.
#pragma once
#include "ss_kernels.cuh"

namespace ssk {

// ------------------------------------------------------- state upload ------
// A caller's state in the host layout (R [M][N][3], A [M][zm][3] double;
// S [M][zm], Z [M] int32), staged on the device as it is, checked and then
// converted to the device layout.  One thread per (chain, bead or slot i).
// bad: bit 1 Z out of 0..zm, 2 S out of 0..N-1, 4 A not finite, 8 R not finite.
__global__ void state_check_kernel(const double* __restrict__ R, const double* __restrict__ A,
                                   const int32_t* __restrict__ S, const int32_t* __restrict__ Z, int M, int N,
                                   int zm, int width, int* __restrict__ bad) {
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (long long)M * width) return;
    const int m = (int)(id / width), i = (int)(id % width);
    const int z = Z[m];
    int f = 0;
    if (i == 0 && (z < 0 || z > zm)) f |= 1;
    if (i < N)
        for (int d = 0; d < 3; ++d)
            if (!isfinite(R[((size_t)m * N + i) * 3 + d])) f |= 8;
    if (i < zm && i < z) {
        const int sj = S[(size_t)m * zm + i];
        if (sj < 0 || sj >= N) f |= 2;
        for (int d = 0; d < 3; ++d)
            if (!isfinite(A[((size_t)m * zm + i) * 3 + d])) f |= 4;
    }
    if (f) atomicOr(bad, f);
}

template <typename T>
__global__ void state_convert_kernel(const double* __restrict__ Rh, const double* __restrict__ Ah,
                                     const int32_t* __restrict__ Sh, const int32_t* __restrict__ Zh, int M, int N,
                                     int zm, int NP, T* __restrict__ R, T* __restrict__ A, int32_t* __restrict__ S,
                                     int32_t* __restrict__ Z) {
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (long long)M * NP) return;
    const int m = (int)(id / NP), i = (int)(id % NP);
    const int z = Zh[m];
    if (i == 0) Z[m] = z;
    for (int d = 0; d < 3; ++d) {
        R[((size_t)m * 3 + d) * NP + i] = i < N ? T(Rh[((size_t)m * N + i) * 3 + d]) : T(0);
        A[((size_t)m * 3 + d) * NP + i] = i < z ? T(Ah[((size_t)m * zm + i) * 3 + d]) : T(0);
    }
    S[(size_t)m * NP + i] = i < z ? Sh[(size_t)m * zm + i] : -1;
}

// The state in the caller's layout (R [M][N][3], A [M][zm][3] double; S
// [M][zm] int32 with -1 for empty slots, Z [M]) from the device layout, into
// caller-owned device arrays (any may be null).  One thread per (chain, i).
template <typename T>
__global__ void state_export_kernel(const T* __restrict__ R, const T* __restrict__ A, const int32_t* __restrict__ S,
                                    const int32_t* __restrict__ Z, int M, int N, int zm, int NP, double* __restrict__ Ro,
                                    double* __restrict__ Ao, int32_t* __restrict__ So, int32_t* __restrict__ Zo) {
    const int width = N > zm ? N : zm;
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (long long)M * width) return;
    const int m = (int)(id / width), i = (int)(id % width);
    const int z = Z[m];
    if (i == 0 && Zo) Zo[m] = z;
    if (i < N && Ro)
        for (int d = 0; d < 3; ++d) Ro[((size_t)m * N + i) * 3 + d] = (double)R[((size_t)m * 3 + d) * NP + i];
    if (i < zm) {
        const bool occ = i < z;
        if (So) So[(size_t)m * zm + i] = occ ? S[(size_t)m * NP + i] : -1;
        if (Ao)
            for (int d = 0; d < 3; ++d)
                Ao[((size_t)m * zm + i) * 3 + d] = occ ? (double)A[((size_t)m * 3 + d) * NP + i] : 0.0;
    }
}

// Histogram of the slip-spring numbers Z of M chains: hist[z] += number of
// chains with Z = z, z = 0..nb-1 (nb <= kMaxSlots + 1), bins per CTA in shared
// memory.  A Z outside 0..nb-1 (never produced by the step) is counted in bin
// nb, the overflow bin.
__global__ void zhist_kernel(const int32_t* __restrict__ Z, int M, int nb, unsigned long long* __restrict__ hist) {
    __shared__ unsigned int h[kMaxSlots + 2];
    for (int i = threadIdx.x; i <= nb; i += blockDim.x) h[i] = 0u;
    __syncthreads();
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < M; m += gridDim.x * blockDim.x) {
        const int z = Z[m];
        atomicAdd(&h[(z >= 0 && z < nb) ? z : nb], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i <= nb; i += blockDim.x)
        if (h[i]) atomicAdd(hist + i, (unsigned long long)h[i]);
}

// ------------------------------------------------------------ init kernel ----
// Equilibrium initial state (Sec. 3.1 sampling): ideal-chain bonds with
// variance kT/k_b per component, Z ~ Poisson(N/N0) by inverse CDF on a 53-bit
// uniform (capped at z_max), S uniform on the beads, anchors Gaussian around
// their bead with variance kT/k_s.  One thread per chain, FP64 arithmetic.
template <typename T, int NP>
__global__ void init_kernel(T* R, T* A, int32_t* S, int32_t* Z, int M, int N, int zmax, double sb,
                            double sa, double lam, uint32_t key0, uint32_t key1, uint32_t chain_base) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const uint32_t cid = chain_base + (uint32_t)m;
    double r[kMaxBeads][3];
    r[0][0] = r[0][1] = r[0][2] = 0.0;
    for (int i = 0; i + 1 < N; ++i) {
        const uint4 w = philox4x32_10((uint32_t)i, 0u, kPurposeInitBond, cid, key0, key1);
        double n[4];
        box_muller<double>(w.x, w.y, n[0], n[1]);
        box_muller<double>(w.z, w.w, n[2], n[3]);
        for (int d = 0; d < 3; ++d) r[i + 1][d] = r[i][d] + sb * n[d];
    }
    for (int i = 0; i < NP; ++i)
        for (int d = 0; d < 3; ++d) R[((size_t)m * 3 + d) * NP + i] = i < N ? T(r[i][d]) : T(0);
    int z = zmax;
    {
        const uint4 w = philox4x32_10(0u, 0u, kPurposeInitZ, cid, key0, key1);
        const double u53 = ((double)(w.x >> 5) * 67108864.0 + (double)(w.y >> 6)) / 9007199254740992.0;
        double pmf = exp(-lam), cdf = pmf;
        for (int k = 0; k < zmax; ++k) {
            if (u53 < cdf) {
                z = k;
                break;
            }
            pmf *= lam / (double)(k + 1);
            cdf += pmf;
        }
    }
    Z[m] = z;
    for (int j = 0; j < NP; ++j) {
        int sj = -1;
        double an[3] = {0.0, 0.0, 0.0};
        if (j < z) {
            const uint4 ws = philox4x32_10((uint32_t)j, 0u, kPurposeInitS, cid, key0, key1);
            sj = (int)(((unsigned long long)ws.x * (unsigned long long)N) >> 32);
            const uint4 wa = philox4x32_10((uint32_t)j, 0u, kPurposeInitA, cid, key0, key1);
            double n[4];
            box_muller<double>(wa.x, wa.y, n[0], n[1]);
            box_muller<double>(wa.z, wa.w, n[2], n[3]);
            for (int d = 0; d < 3; ++d) an[d] = r[sj][d] + sa * n[d];
        }
        S[(size_t)m * NP + j] = sj;
        for (int d = 0; d < 3; ++d) A[((size_t)m * 3 + d) * NP + j] = T(an[d]);
    }
}

}  // namespace ssk
