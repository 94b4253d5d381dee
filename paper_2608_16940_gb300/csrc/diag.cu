// Diagonal streaming update: the diagonal branch of the axis-shifted lowering
// (Alg. 2: multiply each amplitude by the diagonal entry indexed by the
// target bits; Eq. cost-diag-formal: one streaming pass, no permutation, the
// layout unchanged).
//
// A CTA walks tiles of 1024 pairs of amplitudes (16 bytes, physical indices y and
// y + 1), four per thread in flight; three 256-thread CTAs per SM put 48 KiB in
// flight: the memory's latency takes no more, and more turn its bus around more
// often (N = 26, k = 4: 183 / 166 / 171 / 172 us with 2 / 3 / 4 / 5 CTAs; in the L2 the
// last three are alike, N = 20 9.7..10.1, N = 23 18.8 / 17.9 / 18.2).  The entry
// index c(y) (bit j = bit p_j of y) is the OR of a part per thread, per tile and
// per place in the tile; shared tables over the bits of y, 18 KiB formed by every
// CTA, cost a small state most of its launch (N = 20, k = 4: 20.5 us, 6.1 here;
// N = 27, k = 1 / 8 / 12: 0.344 / 0.366 / 0.446 ms, 0.325 / 0.328 / 0.339 here).
// The 2^k-entry FP32 table itself sits in shared memory.  Loads and stores
// stream (evict-first): 16 B per amplitude.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "qsa_internal.h"

namespace qsa {

namespace {

constexpr int kDiagThreads = 256;
constexpr int kDiagUnroll = 4;
constexpr int kDiagCtas = 3;

struct DiagArgs {
    float4* psi;
    uint64_t npairs;
    const float2* d;
    int k;
    int p[QSA_MAX_DIAG];
};

__device__ __forceinline__ float4 cmul2(float4 v, float2 a, float2 b) {
    float4 w;
    w.x = v.x * a.x - v.y * a.y;
    w.y = v.x * a.y + v.y * a.x;
    w.z = v.z * b.x - v.w * b.y;
    w.w = v.z * b.y + v.w * b.x;
    return w;
}

// Part of the entry index from the bits of y in [from, to).
__device__ __forceinline__ uint32_t entry_part(const DiagArgs& a, uint64_t y, int from, int to) {
    const uint32_t lo = static_cast<uint32_t>(y), hi = static_cast<uint32_t>(y >> 32);
    uint32_t c = 0;
#pragma unroll
    for (int j = 0; j < QSA_MAX_DIAG; ++j) {
        if (j >= a.k) break;
        const int p = a.p[j];
        if (p >= from && p < to) c |= (((p < 32 ? lo : hi) >> (p & 31)) & 1u) << j;
    }
    return c;
}

__global__ void __launch_bounds__(kDiagThreads, kDiagCtas) k_apply_diag(const __grid_constant__ DiagArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    float2* d = reinterpret_cast<float2*>(smem);
    for (int i = threadIdx.x; i < (1 << a.k); i += blockDim.x) d[i] = a.d[i];
    // y = tile << 11 | place << 9 | thread << 1 | odd
    const uint32_t odd = entry_part(a, 1, 0, 1), ct = entry_part(a, 2 * threadIdx.x, 1, 9);
    const uint32_t c1 = entry_part(a, 1 << 9, 9, 11), c2 = entry_part(a, 2 << 9, 9, 11);
    __syncthreads();

    constexpr uint64_t kTile = kDiagThreads * kDiagUnroll;
    for (uint64_t q0 = blockIdx.x * kTile; q0 < a.npairs; q0 += gridDim.x * kTile) {
        const uint64_t q = q0 + threadIdx.x;
        float4 v[kDiagUnroll];
#pragma unroll
        for (int u = 0; u < kDiagUnroll; ++u)
            if (q + u * kDiagThreads < a.npairs) v[u] = __ldcs(a.psi + q + u * kDiagThreads);
        const uint32_t c = ct | entry_part(a, q0 << 1, 11, 64);
#pragma unroll
        for (int u = 0; u < kDiagUnroll; ++u)
            if (q + u * kDiagThreads < a.npairs) {
                const uint32_t cu = c | (u & 1 ? c1 : 0u) | (u & 2 ? c2 : 0u);
                __stcs(a.psi + q + u * kDiagThreads, cmul2(v[u], d[cu], d[cu | odd]));
            }
    }
}

}  // namespace

cudaError_t launch_apply_diag(float2* psi, int n, const int* phys, int k, const float* d_tab, cudaStream_t st,
                              uint64_t* launches) {
    if (k < 1 || k > QSA_MAX_DIAG || k > n || n > QSA_MAX_QUBITS) return cudaErrorInvalidValue;
    DiagArgs a{};
    a.psi = reinterpret_cast<float4*>(psi);
    a.npairs = 1ull << (n - 1);
    a.d = reinterpret_cast<const float2*>(d_tab);
    a.k = k;
    for (int j = 0; j < k; ++j) a.p[j] = phys[j];
    const size_t sm = sizeof(float2) << k;   // at most 32 KiB
    const uint64_t tile = kDiagThreads * kDiagUnroll, need = (a.npairs + tile - 1) / tile;
    const uint64_t grid = std::min<uint64_t>(static_cast<uint64_t>(num_sms()) * kDiagCtas, need);
    k_apply_diag<<<static_cast<unsigned>(grid), kDiagThreads, sm, st>>>(a);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace qsa
