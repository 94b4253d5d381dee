// Reductions and sampling on the complex64 state (sm_103a).
//
//   launch_reduce_z      <Z_mask> and the norm: exact squares accumulated per
//                        thread in double-float (about 48 bits), partials
//                        combined in FP64 (App. B: totals kept in FP64).
//   launch_probs_logical p_x = fl64(re^2) + fl64(im^2) for every logical x,
//                        decoded through the layout map (Theorem 1).
//   launch_sample        hierarchical CDF sampler (§IV-E "Sampling": 2^10-entry
//                        blocks, strict upper bound) with integer weights
//                        P_y = floor(re^2 2^60) + floor(im^2 2^60) so that the
//                        CDF is exact and independent of summation order, one
//                        Philox4x64-10 draw per shot, decode through L (§IV-D),
//                        then sort + run-length encode into (outcome, count).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <utility>

#include "qsa_device.cuh"
#include "qsa_internal.h"

namespace qsa {

namespace {

using namespace dev;

constexpr int kRedThreads = 256;
constexpr int kRedBlocksPerSM = 8;

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Per-thread accumulation as an unevaluated float pair s + c: every square is
// split exactly into h + l (FMA two-product, h = fl(v^2), l = v^2 - h) and h
// is added with Knuth's two-sum, whose rounding error goes to c with l.  The
// pair carries about 48 significant bits, so the FP64 value (double)s +
// (double)c of each thread's partial sum matches FP64 accumulation of the
// exact squares, while costing FP32 instructions only (GB300's FP64 rate is a
// small fraction of its FP32 rate).
__device__ __forceinline__ void acc_square(float& s, float& c, float v, bool neg) {
    float h = __fmul_rn(v, v);
    float l = __fmaf_rn(v, v, -h);
    if (neg) {
        h = -h;
        l = -l;
    }
    const float t = __fadd_rn(s, h);
    const float bp = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(h, bp));
    s = t;
    c = __fadd_rn(c, __fadd_rn(e, l));
}

__global__ void __launch_bounds__(kRedThreads) k_reduce_z(const float4* __restrict__ psi2, uint64_t npairs,
                                                           uint64_t physmask, double* __restrict__ partials) {
    float s = 0.f, c = 0.f;
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
    for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < npairs; i += stride) {
        const float4 a = __ldcs(psi2 + i);
        const uint64_t y0 = i << 1;
        const bool n0 = __popcll(y0 & physmask) & 1;
        const bool n1 = __popcll((y0 | 1ull) & physmask) & 1;
        acc_square(s, c, a.x, n0);
        acc_square(s, c, a.y, n0);
        acc_square(s, c, a.z, n1);
        acc_square(s, c, a.w, n1);
    }
    double acc = static_cast<double>(s) + static_cast<double>(c);
    __shared__ double ws[kRedThreads / 32];
    acc = warp_sum_d(acc);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (kRedThreads / 32) ? ws[threadIdx.x] : 0.0;
        v = warp_sum_d(v);
        if (threadIdx.x == 0) partials[blockIdx.x] = v;
    }
}

// Several sign masks in one pass: the squares are formed once per amplitude
// and accumulated per mask exactly as k_reduce_z does (so each result equals
// the single-mask one bit for bit).  Partials of mask m at m * gridDim.x.
__global__ void __launch_bounds__(kRedThreads) k_reduce_z_multi(const float4* __restrict__ psi2, uint64_t npairs,
                                                                ZMasks masks, double* __restrict__ partials) {
    float s[kMaxZMasks] = {}, c[kMaxZMasks] = {};
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
    for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < npairs; i += stride) {
        const float4 a = __ldcs(psi2 + i);
        const uint64_t y0 = i << 1;
#pragma unroll
        for (int m = 0; m < kMaxZMasks; ++m) {
            if (m >= masks.n) break;
            const bool n0 = __popcll(y0 & masks.m[m]) & 1;
            const bool n1 = __popcll((y0 | 1ull) & masks.m[m]) & 1;
            acc_square(s[m], c[m], a.x, n0);
            acc_square(s[m], c[m], a.y, n0);
            acc_square(s[m], c[m], a.z, n1);
            acc_square(s[m], c[m], a.w, n1);
        }
    }
    __shared__ double ws[kRedThreads / 32];
    for (int m = 0; m < masks.n; ++m) {
        double acc = static_cast<double>(s[m]) + static_cast<double>(c[m]);
        acc = warp_sum_d(acc);
        if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x < 32) {
            double v = threadIdx.x < (kRedThreads / 32) ? ws[threadIdx.x] : 0.0;
            v = warp_sum_d(v);
            if (threadIdx.x == 0) partials[static_cast<uint64_t>(m) * gridDim.x + blockIdx.x] = v;
        }
        __syncthreads();
    }
}

// Fixed-order sum of n partials (deterministic for a given grid) by one CTA of
// kRedThreads into *out: its time is a serial chain, so each thread has four
// loads in flight and two rounds of shuffles do the rest.
__device__ __forceinline__ void sum_partials(const double* partials, int n, double* out) {
    __shared__ double ws[kRedThreads / 32];
    double v = 0.0;
    for (int i = threadIdx.x; i < n; i += 4 * kRedThreads) {
        double a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = i + k * kRedThreads < n ? __ldcg(partials + i + k * kRedThreads) : 0.0;
        v += (a[0] + a[1]) + (a[2] + a[3]);
    }
    v = warp_sum_d(v);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        v = warp_sum_d(threadIdx.x < kRedThreads / 32 ? ws[threadIdx.x] : 0.0);
        if (threadIdx.x == 0) *out = v;
    }
    __syncthreads();
}

// As a launch of its own (3.4 us for 304 partials and the gap before it), for
// passes whose CTAs outnumber the SMs many times: CTA m sums partials[m n ..).
__global__ void __launch_bounds__(kRedThreads) k_finalize_sum(const double* __restrict__ partials, int n,
                                                              double* __restrict__ out) {
    sum_partials(partials + static_cast<size_t>(blockIdx.x) * n, n, out + blockIdx.x);
}

// In the pass itself: the CTA that finishes last sums every mask's partials
// (thread 0 of each CTA has written its own).  The count wraps to zero for the
// next pass on the stream.  A launch less: probabilities and norm at N = 12 37.2
// -> 35.3 us a call, two <Z> sums 43.0 -> 40.8, 500 samples with them 106 -> 104.
__device__ __forceinline__ void sum_by_last_cta(const double* partials, int nm, double* out, unsigned* count) {
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicInc(count, gridDim.x - 1) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int m = 0; m < nm; ++m) sum_partials(partials + static_cast<size_t>(m) * gridDim.x, static_cast<int>(gridDim.x), out + m);
}


// States below one tile (N < 12) and outputs off a 16-byte boundary: a gather
// per logical index.
__global__ void k_probs_logical(const float2* __restrict__ psi, Layout lay, double* __restrict__ out) {
    const uint64_t dim = 1ull << lay.n;
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
    for (uint64_t x = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; x < dim; x += stride) {
        const float2 a = psi[encode_logical(x, lay)];
        out[x] = __dadd_rn(__dmul_rn(a.x, a.x), __dmul_rn(a.y, a.y));
    }
}

// v^2 as a double, exactly: the product of the 24-bit mantissas (46..48 bits)
// shifted to 53 bits under the exponent 2 e, in integer instructions.  GB300
// issues two FP64 operations per clock and SM, so forming both squares in FP64
// (two conversions and two products per amplitude) bounds the pass at several
// times its memory traffic; the sum below is the only one left.
__device__ __forceinline__ double square_normal(float v) {
    const uint32_t b = __float_as_uint(v) & 0x7fffffffu;
    const uint32_t M = (b & 0x7fffffu) | 0x800000u;
    const uint64_t P = static_cast<uint64_t>(M) * M;   // in [2^46, 2^48)
    const uint32_t top = static_cast<uint32_t>(P >> 47);
    // value P 2^(2 e - 300): biased exponent 2 e + 769 + top; the leading bit adds one to it
    return __longlong_as_double(static_cast<long long>(
        (P << (6u - top)) + (static_cast<uint64_t>(((b >> 23) << 21) + ((768u + top) << 20)) << 32)));
}
__device__ __forceinline__ double square_exact(float v) {
    const uint32_t b = __float_as_uint(v) & 0x7fffffffu, e = b >> 23;
    if (e == 0u || e == 255u) {   // zero, subnormal, infinite or NaN
        if (b == 0u) return 0.0;
        return static_cast<double>(v) * static_cast<double>(v);
    }
    return square_normal(v);
}
// A zero part leaves the other's square as it is (states with real amplitudes).
__device__ __forceinline__ double probability_exact(float x, float y) {
    if (y == 0.f) return square_exact(x);
    return __dadd_rn(square_exact(x), square_exact(y));
}
// The two probabilities of a 16-byte unit.  One test tells whether its four
// components are normal numbers (a sum that is not finite, if only by overflow,
// takes the other way too), so that the usual unit runs without a branch per
// component (2^27 amplitudes: 0.457 ms with one, 0.411 here; states with real
// amplitudes, which take the other way, 0.421 and 0.404).
__device__ __forceinline__ double2 probabilities(const float4& v) {
    const float least = fminf(fminf(fabsf(v.x), fabsf(v.y)), fminf(fabsf(v.z), fabsf(v.w)));
    const float sum = __fadd_rn(__fadd_rn(fabsf(v.x), fabsf(v.y)), __fadd_rn(fabsf(v.z), fabsf(v.w)));
    if (!(least >= 0x1p-126f && sum <= 0x1.fffffep127f))
        return make_double2(probability_exact(v.x, v.y), probability_exact(v.z, v.w));
    return make_double2(__dadd_rn(square_normal(v.x), square_normal(v.y)), __dadd_rn(square_normal(v.z), square_normal(v.w)));
}

// Probabilities in logical order through tiles of 2^12 amplitudes: the tile's
// bits hold the 64 lowest physical and the 64 lowest logical indices (filled up
// with the next lowest positions), so both the reads (runs of 512 bytes) and
// the writes (runs of 512 bytes) are whole lines; a gather per logical index
// reads a 32-byte sector per amplitude when the layout is permuted.  The tile
// is turned in shared memory, whose 16-byte units are placed by an XOR over
// the tile bits that the writing lanes vary (formed on the host).  With
// partials the norm is taken in the same read (double-float per thread, as
// k_reduce_z).  N = 27, random layout, probabilities and norm:
// 2.01 ms by gather and a second pass, 0.411 ms here (0.317 ms at the copy rate;
// before the test per unit, 0.457 with the three CTAs per SM, 0.524 with two and
// 0.493 with four).
constexpr int kProbT = 12, kProbCtas = 3;

struct ProbArgs {
    const float2* psi;
    double* out;
    double* partials;          // nullable
    double* norm;              // with partials
    unsigned* count;
    uint64_t ntiles;
    int nouter;                // n - 12
    uint8_t opos[24], oq[24];  // outer bit i: its physical position and its logical qubit
    uint64_t poff[kProbT];     // global offset of tile bit b (ascending physical positions)
    uint64_t loff[kProbT];     // logical offset of the tile's i-th lowest logical qubit
    uint16_t pslot[kProbT];    // slot of tile bit b
    uint16_t lslot[kProbT];    // slot of the tile bit that holds the i-th logical qubit
};

__global__ void __launch_bounds__(kRedThreads, kProbCtas) k_probs_tile(const __grid_constant__ ProbArgs a) {
    __shared__ __align__(16) double st[1 << kProbT];
    const int tid = threadIdx.x, lane = tid & 31;
    uint64_t gl = 0, gs = 0;
    uint32_t sl = 0, ss = 0;
#pragma unroll
    for (int b = 0; b < 8; ++b)
        if ((tid >> b) & 1) {
            gl |= a.poff[b + 1];
            sl ^= a.pslot[b + 1];
            gs |= a.loff[b + 1];
            ss ^= a.lslot[b + 1];
        }
    const int op = lane < a.nouter ? a.opos[lane] : 0, oq = lane < a.nouter ? a.oq[lane] : 0;
    float zs = 0.f, zc = 0.f;
    // the tile's base in both orders: lane i places outer bit i
    auto place = [&](uint64_t t, int at) {
        const uint64_t b = lane < a.nouter ? ((t >> lane) & 1ull) << at : 0ull;
        return (static_cast<uint64_t>(__reduce_or_sync(0xffffffffu, static_cast<uint32_t>(b >> 32))) << 32) |
               __reduce_or_sync(0xffffffffu, static_cast<uint32_t>(b));
    };
    float4 v[8];
    auto load = [&](uint64_t t) {
        const uint64_t base = place(t, op) | gl;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            v[k] = __ldcs(reinterpret_cast<const float4*>(a.psi + (base | (k & 1 ? a.poff[9] : 0ull) |
                                                                   (k & 2 ? a.poff[10] : 0ull) | (k & 4 ? a.poff[11] : 0ull))));
    };
    if (blockIdx.x < a.ntiles) load(blockIdx.x);
    for (uint64_t t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        __syncthreads();   // the tile before has been read
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t s = sl ^ (k & 1 ? a.pslot[9] : 0u) ^ (k & 2 ? a.pslot[10] : 0u) ^ (k & 4 ? a.pslot[11] : 0u);
            *reinterpret_cast<double2*>(st + s) =
                probabilities(v[k]);
            if (a.partials) {
                acc_square(zs, zc, v[k].x, false);
                acc_square(zs, zc, v[k].y, false);
                acc_square(zs, zc, v[k].z, false);
                acc_square(zs, zc, v[k].w, false);
            }
        }
        if (t + gridDim.x < a.ntiles) load(t + gridDim.x);   // in flight while this tile is written
        __syncthreads();
        const uint64_t lbase = place(t, oq) | gs;
        const uint32_t s0 = a.lslot[0];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t s = ss ^ (k & 1 ? a.lslot[9] : 0u) ^ (k & 2 ? a.lslot[10] : 0u) ^ (k & 4 ? a.lslot[11] : 0u);
            const uint64_t g = lbase | (k & 1 ? a.loff[9] : 0ull) | (k & 2 ? a.loff[10] : 0ull) |
                               (k & 4 ? a.loff[11] : 0ull);
            __stcs(reinterpret_cast<double2*>(a.out + g), make_double2(st[s], st[s ^ s0]));
        }
    }
    if (a.partials) {
        __shared__ double ws[kRedThreads / 32];
        double acc = warp_sum_d(static_cast<double>(zs) + static_cast<double>(zc));
        if (lane == 0) ws[tid >> 5] = acc;
        __syncthreads();
        if (tid < 32) {
            double x = tid < (kRedThreads / 32) ? ws[tid] : 0.0;
            x = warp_sum_d(x);
            if (tid == 0) a.partials[blockIdx.x] = x;
        }
        sum_by_last_cta(a.partials, 1, a.norm, a.count);
    }
}

// ---------------------------------------------------------------------------
// Sampler
// ---------------------------------------------------------------------------


// One warp per block of `bsz` amplitudes: total integer weight.
__global__ void k_block_weights(const float2* __restrict__ psi, uint64_t nblocks, int bsz,
                                uint64_t* __restrict__ cum) {
    const uint64_t w = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= nblocks) return;
    const float2* p = psi + w * bsz;
    uint64_t s = 0;
    for (int j = lane; j < bsz; j += 32) s += weight(p[j]);
    s = warp_sum_u64(s);
    if (lane == 0) cum[w] = s;
}

// The block weights and, in the same read of the state, <Z_mask> sums for up to
// kMaxZMasks masks: persistent warps walk the 2^bsz-amplitude blocks; each
// thread accumulates its amplitudes' squares per mask as k_reduce_z does
// (double-float); per-CTA partials of mask m at m * gridDim.x.
__global__ void __launch_bounds__(kRedThreads) k_block_weights_z(const float2* __restrict__ psi, uint64_t nblocks,
                                                                 int bsz, uint64_t* __restrict__ cum, ZMasks masks,
                                                                 double* __restrict__ partials) {
    const int lane = threadIdx.x & 31;
    const uint64_t warps = static_cast<uint64_t>(gridDim.x) * (blockDim.x >> 5);
    float zs[kMaxZMasks] = {}, zc[kMaxZMasks] = {};
    for (uint64_t w = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; w < nblocks; w += warps) {
        const uint64_t y0 = w * bsz;
        const float2* p = psi + y0;
        uint64_t s = 0;
        for (int j = lane; j < bsz; j += 32) {
            const float2 a = __ldcs(p + j);
            s += weight(a);
#pragma unroll
            for (int m = 0; m < kMaxZMasks; ++m) {
                if (m >= masks.n) break;
                const bool neg = __popcll((y0 + j) & masks.m[m]) & 1;
                acc_square(zs[m], zc[m], a.x, neg);
                acc_square(zs[m], zc[m], a.y, neg);
            }
        }
        s = warp_sum_u64(s);
        if (lane == 0) cum[w] = s;
    }
    __shared__ double ws[kRedThreads / 32];
    for (int m = 0; m < masks.n; ++m) {
        double acc = static_cast<double>(zs[m]) + static_cast<double>(zc[m]);
        acc = warp_sum_d(acc);
        if (lane == 0) ws[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x < 32) {
            double v = threadIdx.x < (kRedThreads / 32) ? ws[threadIdx.x] : 0.0;
            v = warp_sum_d(v);
            if (threadIdx.x == 0) partials[static_cast<uint64_t>(m) * gridDim.x + blockIdx.x] = v;
        }
        __syncthreads();
    }
}

// |x + iy|^2 as an unevaluated pair hi + lo: each square split exactly by the
// FMA two-product, the two high parts added by Knuth's two-sum, the low parts
// (about 2^-24 of hi) rounded into lo.
__device__ __forceinline__ void square_pair(float x, float y, float& hi, float& lo) {
    const float h1 = __fmul_rn(x, x), l1 = __fmaf_rn(x, x, -h1);
    const float h2 = __fmul_rn(y, y), l2 = __fmaf_rn(y, y, -h2);
    const float t = __fadd_rn(h1, h2);
    const float bp = __fsub_rn(t, h1);
    const float e = __fadd_rn(__fsub_rn(h1, __fsub_rn(t, bp)), __fsub_rn(h2, bp));
    hi = t;
    lo = __fadd_rn(e, __fadd_rn(l1, l2));
}

// Weight of one component from its bits when its biased exponent e is at most
// 127 (|v| < 2): floor(v^2 2^60) = floor(M^2 2^(2e - 240)) as (M 2^7)^2 =
// M^2 2^14 < 2^62 shifted right by 254 - 2e, the shift left unclamped (PTX
// shr.b64 takes shifts above 64 as 64 and gives 0, the exact result there).
// The implicit bit is set unconditionally; for e = 0 (zero, subnormals) the
// shift is 254, so the result is 0 as in sq_fixed60.  254 - 2e = 2e ^ 254
// since 2e is even and below 256.
__device__ __forceinline__ uint64_t sq_fixed60_small(uint32_t bits) {
    const uint32_t mq = ((bits & 0x7fffffu) | 0x800000u) << 7;
    const uint32_t sh = ((bits >> 22) & 0x1feu) ^ 0xfeu;
    const uint64_t prod = static_cast<uint64_t>(mq) * mq;
    uint64_t r;
    asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(prod), "r"(sh));
    return r;
}

// s + c += g (hi + lo) for g = +-1, in double-float: Knuth's two-sum of s and
// g hi (its rounding error to c with g lo), the sign taken inside FMAs (g hi
// and g lo are exact products, so each FMA rounds once, like an addition of
// the negated term).
__device__ __forceinline__ void add_scaled(float& s, float& c, float hi, float lo, float g) {
    const float t = __fmaf_rn(g, hi, s);
    const float bp = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fmaf_rn(g, hi, -bp));
    s = t;
    c = __fadd_rn(c, __fmaf_rn(g, lo, e));
}

// Blocks of 1024 amplitudes: the block weights and the <Z_mask> sums of NM
// masks in one read.  A warp takes a block; lane l loads the 16-byte pairs
// l + 32 k (k = 0..15) up front, so 8 KiB per warp are in flight.  Amplitude
// y = 1024 w + 2 (l + 32 k) + b has its index bits split over (w, l, k, b), so
// its sign parity is a per-block, a per-lane, a per-k and a per-b part.
// Weights: when no component of the block has |v| >= 2 (always, for a state
// of norm about 1) the warp takes sq_fixed60_small, else sq_fixed60 (equal
// values where both apply).  Sums: each thread keeps its mask-m pair in the
// frame of its own block-and-lane sign (the pair negated when that sign
// changes between blocks; round-to-nearest is symmetric, so the values are
// those of summing in the true signs, up to the sign of zeros), so the sign
// left per amplitude, of its k and b bits, is the same across the warp.  EVEN: no
// mask holds the lowest position, so a pair's two squares are added once for all
// masks (2^26 amplitudes, two masks: 126 us, 136 without).  Per CTA partials of
// mask m at m * gridDim.x.
template <int NM, bool EVEN>
__global__ void __launch_bounds__(kRedThreads, 2) k_weights_z1024(const float4* __restrict__ psi2, uint64_t nblocks,
                                                                  uint64_t* __restrict__ cum, ZMasks masks,
                                                                  double* partials, double* out,
                                                                  unsigned* count) {
    constexpr int NA = NM > 0 ? NM : 1;
    const int lane = threadIdx.x & 31;
    const uint64_t warps = static_cast<uint64_t>(gridDim.x) * (blockDim.x >> 5);
    float zs[NA] = {}, zc[NA] = {};
    uint32_t kb[NA] = {}, lb[NA] = {}, fr[NA] = {};
    float bf[NA] = {};
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        for (int k = 0; k < 16; ++k) kb[m] |= static_cast<uint32_t>(__popcll((64ull * k) & masks.m[m]) & 1) << k;
        lb[m] = __popcll((2ull * lane) & masks.m[m]) & 1;
        bf[m] = (masks.m[m] & 1ull) ? -1.f : 1.f;
    }
    for (uint64_t w = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; w < nblocks; w += warps) {
        const float4* p = psi2 + w * 512 + lane;
        float4 a[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) a[k] = __ldcs(p + 32 * k);
        if constexpr (NM > 0) {
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                // this thread's sign for the block; the pair follows it into the new frame
                const uint32_t f = (__popcll((w << 10) & masks.m[m]) & 1) ^ lb[m];
                if (f != fr[m]) {
                    zs[m] = -zs[m];
                    zc[m] = -zc[m];
                    fr[m] = f;
                }
            }
        }
        uint32_t any = 0;
        uint64_t s = 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const uint32_t x0 = __float_as_uint(a[k].x), y0 = __float_as_uint(a[k].y);
            const uint32_t x1 = __float_as_uint(a[k].z), y1 = __float_as_uint(a[k].w);
            any |= x0 | y0 | x1 | y1;
            s += sq_fixed60_small(x0) + sq_fixed60_small(y0) + sq_fixed60_small(x1) + sq_fixed60_small(y1);
            if constexpr (NM > 0) {
                float h0, l0, h1, l1;
                square_pair(a[k].x, a[k].y, h0, l0);
                square_pair(a[k].z, a[k].w, h1, l1);
                if constexpr (EVEN) {
                    // both amplitudes of a pair enter every sum with the same sign: added once
                    const float t = __fadd_rn(h0, h1), bp = __fsub_rn(t, h0);
                    const float e = __fadd_rn(__fsub_rn(h0, __fsub_rn(t, bp)), __fsub_rn(h1, bp));
                    const float l = __fadd_rn(e, __fadd_rn(l0, l1));
#pragma unroll
                    for (int m = 0; m < NM; ++m)
                        add_scaled(zs[m], zc[m], t, l, __uint_as_float(0x3f800000u | (((kb[m] >> k) & 1u) << 31)));
                } else {
#pragma unroll
                    for (int m = 0; m < NM; ++m) {
                        const float g0 = __uint_as_float(0x3f800000u | (((kb[m] >> k) & 1u) << 31));
                        add_scaled(zs[m], zc[m], h0, l0, g0);
                        add_scaled(zs[m], zc[m], h1, l1, g0 * bf[m]);
                    }
                }
            }
        }
        if (!__all_sync(0xffffffffu, (any & 0x40000000u) == 0u)) {
            // a component with |v| >= 2 (or not finite) in the block: the weights again, by sq_fixed60
            s = 0;
#pragma unroll 4
            for (int k = 0; k < 16; ++k) {
                const float4 v = __ldcs(p + 32 * k);
                s += sq_fixed60(v.x) + sq_fixed60(v.y) + sq_fixed60(v.z) + sq_fixed60(v.w);
            }
        }
        s = warp_sum_u64(s);
        if (lane == 0) cum[w] = s;
    }
    if constexpr (NM > 0) {
        __shared__ double ws[kRedThreads / 32];
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            // back from the thread's frame (the last block's sign)
            const double sg = fr[m] ? -1.0 : 1.0;
            double acc = sg * static_cast<double>(zs[m]) + sg * static_cast<double>(zc[m]);
            acc = warp_sum_d(acc);
            if (lane == 0) ws[threadIdx.x >> 5] = acc;
            __syncthreads();
            if (threadIdx.x < 32) {
                double v = threadIdx.x < (kRedThreads / 32) ? ws[threadIdx.x] : 0.0;
                v = warp_sum_d(v);
                if (threadIdx.x == 0) partials[static_cast<uint64_t>(m) * gridDim.x + blockIdx.x] = v;
            }
            __syncthreads();
        }
        sum_by_last_cta(partials, NM, out, count);
    }
}

// The sums alone, for states of at least one block of 1024 amplitudes: as
// k_weights_z1024 (each mask's terms in the same order whatever the other masks,
// so a mask's result does not depend on them), kZLoads 16-byte loads per lane in
// flight (64 KiB per SM).  N = 27: one mask 0.283 ms with one load per thread and
// the signs selected per component, 0.197 here (two / four masks 0.207 / 0.272;
// 0.158 ms at the copy rate).
constexpr int kZLoads = 4, kZCtas = 4;
template <int NM>
__global__ void __launch_bounds__(kRedThreads, NM <= 2 ? kZCtas : 1) k_zsums1024(const float4* __restrict__ psi2, uint64_t nblocks,
                                                           const __grid_constant__ ZMasks masks,
                                                           double* partials, double* out, unsigned* count) {
    const int lane = threadIdx.x & 31;
    const uint64_t warps = static_cast<uint64_t>(gridDim.x) * (blockDim.x >> 5);
    float zs[NM] = {}, zc[NM] = {};
    uint32_t kb[NM] = {}, lb[NM] = {}, fr[NM] = {};
    float bf[NM] = {};
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        for (int k = 0; k < 16; ++k) kb[m] |= static_cast<uint32_t>(__popcll((64ull * k) & masks.m[m]) & 1) << k;
        lb[m] = __popcll((2ull * lane) & masks.m[m]) & 1;
        bf[m] = (masks.m[m] & 1ull) ? -1.f : 1.f;
    }
    for (uint64_t w = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; w < nblocks; w += warps) {
        const float4* p = psi2 + w * 512 + lane;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const uint32_t f = (__popcll((w << 10) & masks.m[m]) & 1) ^ lb[m];
            if (f != fr[m]) {
                zs[m] = -zs[m];
                zc[m] = -zc[m];
                fr[m] = f;
            }
        }
#pragma unroll
        for (int k0 = 0; k0 < 16; k0 += kZLoads) {
            float4 a[kZLoads];
#pragma unroll
            for (int k = 0; k < kZLoads; ++k) a[k] = __ldcs(p + 32 * (k0 + k));
#pragma unroll
            for (int k = 0; k < kZLoads; ++k) {
                float h0, l0, h1, l1;
                square_pair(a[k].x, a[k].y, h0, l0);
                square_pair(a[k].z, a[k].w, h1, l1);
#pragma unroll
                for (int m = 0; m < NM; ++m) {
                    const float g0 = __uint_as_float(0x3f800000u | (((kb[m] >> (k0 + k)) & 1u) << 31));
                    add_scaled(zs[m], zc[m], h0, l0, g0);
                    add_scaled(zs[m], zc[m], h1, l1, g0 * bf[m]);
                }
            }
        }
    }
    __shared__ double ws[kRedThreads / 32];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        const double sg = fr[m] ? -1.0 : 1.0;   // back from the thread's frame
        double acc = sg * static_cast<double>(zs[m]) + sg * static_cast<double>(zc[m]);
        acc = warp_sum_d(acc);
        if (lane == 0) ws[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x < 32) {
            double v = threadIdx.x < (kRedThreads / 32) ? ws[threadIdx.x] : 0.0;
            v = warp_sum_d(v);
            if (threadIdx.x == 0) partials[static_cast<uint64_t>(m) * gridDim.x + blockIdx.x] = v;
        }
        __syncthreads();
    }
    sum_by_last_cta(partials, NM, out, count);
}

// In-place inclusive scan of cum[0..n-1] by one CTA of 1024 threads.
__global__ void __launch_bounds__(1024) k_scan_inclusive(uint64_t* __restrict__ cum, uint64_t n) {
    __shared__ uint64_t wsum[32];
    __shared__ uint64_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (uint64_t base = 0; base < n; base += blockDim.x) {
        const uint64_t i = base + threadIdx.x;
        uint64_t v = i < n ? cum[i] : 0;
        uint64_t inc = warp_incl_scan_u64(v);
        if (lane == 31) wsum[wid] = inc;
        __syncthreads();
        if (wid == 0) {
            uint64_t s = wsum[lane];
            wsum[lane] = warp_incl_scan_u64(s);
        }
        __syncthreads();
        const uint64_t off = carry + (wid ? wsum[wid - 1] : 0);
        if (i < n) cum[i] = inc + off;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = inc + off;
        __syncthreads();
    }
}


// Multi-CTA inclusive scan of cum[0..n-1]: each CTA scans one segment of
// kScanSeg entries in place and writes its total to parts[b]; parts is then
// scanned by k_scan_inclusive and k_scan_add adds parts[b - 1] to segment b.
// Integer sums, so the result is the same as the one-CTA scan.
constexpr int kScanSeg = 4096;

__global__ void __launch_bounds__(1024) k_scan_segments(uint64_t* __restrict__ cum, uint64_t n,
                                                        uint64_t* __restrict__ parts) {
    __shared__ uint64_t wsum[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t i0 = static_cast<uint64_t>(blockIdx.x) * kScanSeg + 4ull * threadIdx.x;
    uint64_t v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = i0 + k < n ? cum[i0 + k] : 0;
    v[1] += v[0];
    v[2] += v[1];
    v[3] += v[2];
    const uint64_t inc = warp_incl_scan_u64(v[3]);
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    if (wid == 0) wsum[lane] = warp_incl_scan_u64(wsum[lane]);
    __syncthreads();
    const uint64_t off = inc - v[3] + (wid ? wsum[wid - 1] : 0);
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (i0 + k < n) cum[i0 + k] = v[k] + off;
    if (threadIdx.x == 1023) parts[blockIdx.x] = wsum[31];
}

__global__ void k_scan_add(uint64_t* __restrict__ cum, uint64_t n, const uint64_t* __restrict__ parts) {
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
    for (uint64_t i = kScanSeg + static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride)
        cum[i] += parts[i / kScanSeg - 1];
}

// Shot s's draw u = floor(r * total / 2^64) and its block: the first with cum > u.
__device__ __forceinline__ uint64_t draw_u(uint64_t s, uint64_t stream_id, uint64_t seed, uint64_t total) {
    return __umul64hi(philox4x64_10_w0(s, stream_id, 0, 0, seed, 0), total);
}
__device__ __forceinline__ uint64_t find_block(const uint64_t* __restrict__ cum, uint64_t nblocks, uint64_t u) {
    uint64_t lo = 0, hi = nblocks - 1;
    while (lo < hi) {
        const uint64_t mid = lo + ((hi - lo) >> 1);
        if (cum[mid] > u) hi = mid; else lo = mid + 1;
    }
    return lo;
}

// One warp per shot on a state below one block of 1024 amplitudes: draw u, find
// the block (first cum > u), then the amplitude.
__global__ void k_draw(const float2* __restrict__ psi, const uint64_t* __restrict__ cum, uint64_t nblocks, int bsz,
                       Layout lay, uint64_t shots, uint64_t seed, uint64_t stream_id, uint64_t* __restrict__ keys) {
    const uint64_t s = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (s >= shots) return;
    const uint64_t total = cum[nblocks - 1];
    if (total == 0) {  // all-zero state: the host reports it; avoid the modulo by zero
        if (lane == 0) keys[s] = 0;
        return;
    }
    const uint64_t u = draw_u(s, stream_id, seed, total);
    const uint64_t b = find_block(cum, nblocks, u);
    const uint64_t ub = u - (b ? cum[b - 1] : 0);
    // lane l covers amplitudes [l*per, (l+1)*per) of the block
    const int per = (bsz + 31) >> 5;
    const float2* p = psi + b * static_cast<uint64_t>(bsz);
    uint64_t wl = 0;
    for (int j = 0; j < per; ++j) {
        int idx = lane * per + j;
        if (idx < bsz) wl += weight(p[idx]);
    }
    const uint64_t incl = warp_incl_scan_u64(wl);
    const uint64_t excl = incl - wl;
    const unsigned hit = __ballot_sync(0xffffffffu, excl <= ub && ub < incl);
    const int owner = __ffs(hit) - 1;   // exactly one lane: the weights sum to cum[b] - cum[b-1] > ub
    if (lane == owner) {
        uint64_t acc = excl;
        int j = 0;
        for (; j < per; ++j) {
            int idx = lane * per + j;
            if (idx >= bsz) break;
            acc += weight(p[idx]);
            if (acc > ub) break;
        }
        const uint64_t y = b * static_cast<uint64_t>(bsz) + static_cast<uint64_t>(lane * per + j);
        keys[s] = decode_physical(y, lay);
    }
}

// Many shots on blocks of 1024 amplitudes: the shots are sorted by block first
// (key: block << kShotBits | shot), so that a block's 8 KiB are read once for
// all of its shots instead of once per shot.
constexpr int kShotBits = 26;   // shots are at most 2^26, blocks at most 2^24

// `count` shots in all, `shots` of each state: state t (its nblocks blocks from
// block t nblocks on) has shots t * shots ... with stream stream_id + t.
__global__ void __launch_bounds__(256) k_draw_blocks(const uint64_t* __restrict__ cum, uint64_t nblocks, uint64_t shots,
                                                     uint64_t count, uint64_t seed, uint64_t stream_id,
                                                     uint64_t* __restrict__ out) {
    const uint64_t s = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (s >= count) return;
    const uint64_t t = s / shots;
    cum += t * nblocks;
    const uint64_t total = cum[nblocks - 1];
    const uint64_t b = total ? find_block(cum, nblocks, draw_u(s - t * shots, stream_id + t, seed, total)) : 0;
    out[s] = ((t * nblocks + b) << kShotBits) | s;
}

// The pair weights of a block of 1024 amplitudes into sums (pair i at i + i / 16:
// rows of 17), by one warp with the block's 8 KiB in flight; returns this
// lane's inclusive prefix, through pair 16 lane + 15, and its own 16 pairs' sum.
constexpr int kPairWords = 512 + 32;
__device__ __forceinline__ uint64_t block_pairs(const float4* __restrict__ block, uint64_t* sums, int lane, uint64_t* own) {
    const float4* p = block + lane;
    float4 a[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) a[k] = __ldg(p + 32 * k);
    uint32_t any = 0;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const uint32_t x0 = __float_as_uint(a[k].x), y0 = __float_as_uint(a[k].y);
        const uint32_t x1 = __float_as_uint(a[k].z), y1 = __float_as_uint(a[k].w);
        any |= x0 | y0 | x1 | y1;
        sums[lane + (lane >> 4) + 34 * k] =
            sq_fixed60_small(x0) + sq_fixed60_small(y0) + sq_fixed60_small(x1) + sq_fixed60_small(y1);
    }
    if (any & 0x40000000u) {   // a component with |v| >= 2 or not finite, as in k_weights_z1024
#pragma unroll 1
        for (int k = 0; k < 16; ++k) {
            const float4 v = __ldg(p + 32 * k);
            sums[lane + (lane >> 4) + 34 * k] = sq_fixed60(v.x) + sq_fixed60(v.y) + sq_fixed60(v.z) + sq_fixed60(v.w);
        }
    }
    __syncwarp();
    uint64_t s = 0;
#pragma unroll
    for (int j = 0; j < 16; ++j) s += sums[17 * lane + j];
    *own = s;
    return warp_incl_scan_u64(s);
}

constexpr int kResolveWarps = 4;

// find_block by a warp: 32 probes a step, so 65536 blocks take 4 dependent reads
// instead of 16.
__device__ __forceinline__ uint64_t find_block_warp(const uint64_t* __restrict__ cum, uint64_t nblocks, uint64_t u, int lane) {
    uint64_t lo = 0, hi = nblocks - 1;
    while (lo < hi) {
        const uint64_t step = (hi - lo) / 32 + 1;
        const uint64_t at = min(lo + static_cast<uint64_t>(lane + 1) * step - 1, hi);
        const int f = __ffs(__ballot_sync(0xffffffffu, cum[at] > u) | 0x80000000u) - 1;   // lane 31 reads cum[hi] > u
        hi = min(lo + static_cast<uint64_t>(f + 1) * step - 1, hi);
        lo = min(lo + static_cast<uint64_t>(f) * step, hi);
    }
    return lo;
}

// One warp per shot on blocks of 1024 amplitudes: the block, its pair sums as in
// k_draw_resolve, then the 16 pairs and the two amplitudes.  A serial chain of
// loads, so as few and as wide as they go: 1000 shots of 2^26 / 2^16 amplitudes
// 10.2 / 7.5 us, 18.5 / 15.3 with a binary search and 32 strided reads a lane.
__global__ void __launch_bounds__(32 * kResolveWarps) k_draw1024(const float4* __restrict__ psi2,
                                                                  const uint64_t* __restrict__ cum, uint64_t nblocks,
                                                                  const __grid_constant__ Layout lay, uint64_t shots,
                                                                  uint64_t seed, uint64_t stream_id,
                                                                  uint64_t* __restrict__ keys) {
    __shared__ uint64_t sums[kResolveWarps][kPairWords];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint64_t s = static_cast<uint64_t>(blockIdx.x) * kResolveWarps + w;
    if (s >= shots) return;
    const uint64_t total = cum[nblocks - 1];
    if (total == 0) {   // all-zero state: the host reports it
        if (lane == 0) keys[s] = 0;
        return;
    }
    const uint64_t u = draw_u(s, stream_id, seed, total);
    const uint64_t b = find_block_warp(cum, nblocks, u, lane);
    uint64_t rest = u - (b ? cum[b - 1] : 0), own;
    const float4* block = psi2 + b * 512;
    const uint64_t incl = block_pairs(block, sums[w], lane, &own);
    // the first lane whose prefix is above rest (the last one's is)
    const int row = __ffs(__ballot_sync(0xffffffffu, incl > rest) | 0x80000000u) - 1;
    rest -= __shfl_sync(0xffffffffu, incl - own, row);
    const uint64_t v = lane < 16 ? sums[w][17 * row + lane] : 0;
    const uint64_t in16 = warp_incl_scan_u64(v);
    const int col = __ffs(__ballot_sync(0xffffffffu, lane < 16 && in16 > rest) | 0x8000u) - 1;
    if (lane == col) {
        const float4 x = __ldg(block + 16 * row + col);
        const bool second = rest - (in16 - v) >= sq_fixed60(x.x) + sq_fixed60(x.y);
        keys[s] = decode_physical(b * 1024 + static_cast<uint64_t>(2 * (16 * row + col) + second), lay);
    }
}

// A warp takes `per` consecutive shots of the sorted list.  For each block among
// them it stores the weights of the block's 512 pairs in shared memory (lanes
// over 16-byte pairs, 64 amplitudes a step), lane l sums pairs 16 l .. 16 l + 15
// of them, one warp scan gives the prefixes at every 32nd amplitude, and every
// lane whose shot lies in the block searches those, then its 16 pairs, then the
// two amplitudes of its pair.  Scanning all 16 steps of a block instead (160
// shuffles a block) was bound by its instructions: 200,000 shots of 2^26
// amplitudes 221 us, this way 137 to 160 (reading the state once: 79).
__global__ void __launch_bounds__(32 * kResolveWarps) k_draw_resolve(const float4* __restrict__ psi2,
                                                                      const uint64_t* __restrict__ cum,
                                                                      uint64_t nblocks, const __grid_constant__ Layout lay,
                                                                      const uint64_t* __restrict__ draws, uint64_t shots,
                                                                      uint64_t count, uint64_t seed, uint64_t stream_id,
                                                                      int per, uint64_t* __restrict__ keys) {
    __shared__ uint64_t sums[kResolveWarps][kPairWords];
    __shared__ uint64_t pre[kResolveWarps][32];          // inclusive prefixes after pair 16 l + 15
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint64_t i = (static_cast<uint64_t>(blockIdx.x) * kResolveWarps + w) * per + lane;
    const bool valid = lane < per && i < count;
    const uint64_t d = valid ? draws[i] : 0;
    const uint64_t b = d >> kShotBits, sh = d & ((1ull << kShotBits) - 1), t = sh / shots, b0 = t * nblocks;
    const uint64_t total = cum[b0 + nblocks - 1];
    uint64_t ub = 0;
    if (valid && total) ub = draw_u(sh - t * shots, stream_id + t, seed, total) - (b > b0 ? cum[b - 1] : 0);
    bool open = valid && total;
    uint64_t key = lay.n ? 0 : b0 * 1024;   // a state of zero weight: its first index
    for (;;) {
        const unsigned left = __ballot_sync(0xffffffffu, open);
        if (!left) break;
        const uint64_t bb = __shfl_sync(0xffffffffu, b, __ffs(left) - 1);
        uint64_t own;
        pre[w][lane] = block_pairs(psi2 + bb * 512, sums[w], lane, &own);
        __syncwarp();
        if (open && b == bb) {
            int lo = 0, hi = 31;   // the first prefix above ub (the last one is: ub < cum[b] - cum[b - 1])
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const int mid = (lo + hi) >> 1;
                if (pre[w][mid] > ub) hi = mid; else lo = mid + 1;
            }
            uint64_t rest = ub - (lo ? pre[w][lo - 1] : 0);
            int pair = 0;   // the first pair whose prefix within the 16 is above rest
#pragma unroll
            for (int j = 0; j < 15; ++j) {
                const uint64_t v = sums[w][17 * lo + j];
                const bool past = pair == j && rest >= v;
                pair += past;
                rest -= past ? v : 0;
            }
            pair += 16 * lo;
            const float4 v = __ldg(psi2 + bb * 512 + pair);
            key = bb * 1024 + static_cast<uint64_t>(2 * pair + (rest >= sq_fixed60(v.x) + sq_fixed60(v.y)));
            if (lay.n) key = decode_physical(key, lay);   // else the index through all states
            open = false;
        }
        __syncwarp();
    }
    if (valid) keys[i] = key;
}

// Stable radix sort of 64-bit keys by one 8-bit digit (least significant digit
// first): per-tile digit counts (hist[digit][tile]), their prefixes per digit,
// and the scatter, where a warp ranks its keys by matching digits 32 at a time.
// Three launches a digit against (log2 P)^2 / 2 for a whole bitonic network:
// 200 000 26-bit outcomes 542 us in 171 global bitonic steps, about 60 us in the
// 12 launches here; their run-length encoding 294 us in one CTA, 17 us in tiles.
// Four keys a thread: the kernels are chains of latencies, so smaller tiles are
// faster until their number costs the scan more (whole calls with 2 / 4 / 8 keys:
// N = 26, 200 000 shots 457 / 471 / 488 us, 5 000 000 4.83 / 4.67 / 4.72 ms).
constexpr int kRadixThreads = 256, kRadixPer = 4, kRadixTile = kRadixThreads * kRadixPer;

__global__ void __launch_bounds__(kRadixThreads) k_radix_hist(const uint64_t* __restrict__ keys, uint64_t n, int shift,
                                                               uint32_t ntiles, uint32_t* __restrict__ hist) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRadixPer; ++j) {
        const uint64_t i = static_cast<uint64_t>(blockIdx.x) * kRadixTile + j * kRadixThreads + threadIdx.x;
        if (i < n) atomicAdd(&h[(keys[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    hist[static_cast<uint64_t>(threadIdx.x) * ntiles + blockIdx.x] = h[threadIdx.x];
}

// CTA d: exclusive prefixes of digit d's tile counts in place, their sum to totals[d].
__global__ void __launch_bounds__(kRadixThreads) k_radix_scan(uint32_t* __restrict__ hist, uint32_t ntiles,
                                                               uint32_t* __restrict__ totals) {
    __shared__ uint32_t ws[8];
    uint32_t* h = hist + static_cast<uint64_t>(blockIdx.x) * ntiles;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t run = 0;
    for (uint32_t t0 = 0; t0 < ntiles; t0 += kRadixThreads) {
        const uint32_t t = t0 + threadIdx.x;
        const uint32_t v = t < ntiles ? h[t] : 0;
        uint32_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += x;
        }
        if (lane == 31) ws[w] = inc;
        __syncthreads();
        uint32_t before = run, all = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k < w) before += ws[k];
            all += ws[k];
        }
        if (t < ntiles) h[t] = before + inc - v;
        run += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = run;
}

__global__ void __launch_bounds__(kRadixThreads) k_radix_scatter(const uint64_t* __restrict__ in, uint64_t n, int shift,
                                                                  uint32_t ntiles, const uint32_t* __restrict__ hist,
                                                                  const uint32_t* __restrict__ totals,
                                                                  uint64_t* __restrict__ out) {
    __shared__ uint32_t cnt[kRadixThreads / 32][256];
    __shared__ uint32_t ws[8];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int i = tid; i < 8 * 256; i += kRadixThreads) cnt[i >> 8][i & 255] = 0;
    // digit tid's first place: every smaller digit, then this digit's tiles before
    const uint32_t tot = totals[tid];
    uint32_t inc = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += x;
    }
    if (lane == 31) ws[w] = inc;
    __syncthreads();
    uint32_t place = inc - tot + hist[static_cast<uint64_t>(tid) * ntiles + blockIdx.x];
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (k < w) place += ws[k];
    // warp w ranks its 256 keys in order, 32 at a time
    const uint64_t i0 = static_cast<uint64_t>(blockIdx.x) * kRadixTile + w * 32 * kRadixPer + lane;
    uint64_t key[kRadixPer];
    uint32_t rank[kRadixPer];
#pragma unroll
    for (int j = 0; j < kRadixPer; ++j) key[j] = i0 + 32 * j < n ? in[i0 + 32 * j] : 0;
#pragma unroll
    for (int j = 0; j < kRadixPer; ++j) {
        const bool valid = i0 + 32 * j < n;
        const unsigned vm = __ballot_sync(0xffffffffu, valid);
        const uint32_t dg = static_cast<uint32_t>(key[j] >> shift) & 255u;
        unsigned peers = 0;
        if (valid) {
            peers = __match_any_sync(vm, dg);
            rank[j] = cnt[w][dg] + __popc(peers & ((1u << lane) - 1u));
        }
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) cnt[w][dg] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t c = cnt[k][tid];
        cnt[k][tid] = place;
        place += c;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRadixPer; ++j)
        if (i0 + 32 * j < n) out[cnt[w][static_cast<uint32_t>(key[j] >> shift) & 255u] + rank[j]] = key[j];
}

// Run-length encoding of sorted keys in tiles: heads per tile, (their prefix by
// k_scan_inclusive,) the distinct keys and where their runs start, the lengths.
__device__ __forceinline__ uint32_t tile_heads(const uint64_t* __restrict__ keys, uint64_t n, uint64_t i0, uint32_t* flags) {
    uint32_t c = 0, f = 0;
#pragma unroll
    for (int j = 0; j < kRadixPer; ++j) {   // this thread's kRadixPer consecutive keys
        const uint64_t i = i0 + j;
        const uint32_t head = i < n && (i == 0 || keys[i] != keys[i - 1]) ? 1u : 0u;
        f |= head << j;
        c += head;
    }
    *flags = f;
    return c;
}

__global__ void __launch_bounds__(kRadixThreads) k_rle_heads(const uint64_t* __restrict__ keys, uint64_t n,
                                                              uint64_t* __restrict__ tile_count) {
    __shared__ uint32_t ws[8];
    uint32_t f;
    uint32_t c = tile_heads(keys, n, static_cast<uint64_t>(blockIdx.x) * kRadixTile + threadIdx.x * kRadixPer, &f);
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int k = 0; k < 8; ++k) t += ws[k];
        tile_count[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(kRadixThreads) k_rle_write(const uint64_t* __restrict__ keys, uint64_t n,
                                                              const uint64_t* __restrict__ tile_incl,
                                                              uint64_t* __restrict__ out_keys, uint64_t* __restrict__ starts,
                                                              uint64_t* __restrict__ n_distinct) {
    __shared__ uint32_t ws[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint64_t i0 = static_cast<uint64_t>(blockIdx.x) * kRadixTile + threadIdx.x * kRadixPer;
    uint32_t f;
    const uint32_t c = tile_heads(keys, n, i0, &f);
    uint32_t inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += x;
    }
    if (lane == 31) ws[w] = inc;
    __syncthreads();
    uint64_t pos = (blockIdx.x ? tile_incl[blockIdx.x - 1] : 0) + inc - c;
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (k < w) pos += ws[k];
#pragma unroll
    for (int j = 0; j < kRadixPer; ++j)
        if ((f >> j) & 1u) {
            out_keys[pos] = keys[i0 + j];
            starts[pos++] = i0 + j;
        }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *n_distinct = tile_incl[blockIdx.x];
}

__global__ void k_rle_counts(const uint64_t* __restrict__ starts, uint64_t n, const uint64_t* __restrict__ n_distinct,
                             uint64_t* __restrict__ counts) {
    const uint64_t nd = *n_distinct;
    const uint64_t d = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (d < nd) counts[d] = (d + 1 < nd ? starts[d + 1] : n) - starts[d];
}

// Up to 4096 outcomes sorted and run-length encoded by one CTA: E keys a thread
// in registers, key e B + t of thread t of B.  A bitonic step exchanges them by
// shuffles below distance 32, through shared memory (two buffers in turn, one
// barrier a step) below B, and within the thread above.  A serial chain of
// steps: 1000 keys 8.8 us; with a barrier over all keys in shared memory for
// every step and launches of their own for padding and runs, 18.2.
// T holds an outcome (32 bits for N <= 32); the padding is the largest T, which
// sorts behind every other key and beside equal ones.
template <typename T>
__device__ __forceinline__ void order(T& a, T& b, bool up) {
    const T lo = a < b ? a : b, hi = a < b ? b : a;
    a = up ? lo : hi;
    b = up ? hi : lo;
}
template <typename T, int E>
__global__ void __launch_bounds__(1024) k_sort_rle(const uint64_t* __restrict__ in, uint32_t n,
                                                   uint64_t* __restrict__ out_keys, uint64_t* __restrict__ out_counts,
                                                   uint64_t* __restrict__ n_distinct) {
    extern __shared__ __align__(16) unsigned char sort_smem[];
    __shared__ uint32_t wsum[32];
    const uint32_t B = blockDim.x, t = threadIdx.x, N = E * B;
    T* cur = reinterpret_cast<T*>(sort_smem);
    T* nxt = cur + N;
    T v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = e * B + t < n ? static_cast<T>(in[e * B + t]) : static_cast<T>(~static_cast<T>(0));
    for (uint32_t k = 2; k <= N; k <<= 1) {
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            if (j >= B) {   // partner rows e ^ 1 or e ^ 2; k > j, so the direction is the row's
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const bool up = ((e * B) & k) == 0;
                    if (E > 1 && !(e & 1) && j == B) order(v[e], v[(e + 1) % E], up);
                    if (E > 2 && !(e & 2) && j != B) order(v[e], v[(e + 2) % E], up);
                }
            } else if (j >= 32) {
#pragma unroll
                for (int e = 0; e < E; ++e) cur[e * B + t] = v[e];
                __syncthreads();
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const uint32_t i = e * B + t;
                    const T c = cur[i ^ j];
                    const bool low = ((i & j) == 0) == ((i & k) == 0);   // keeps the smaller
                    v[e] = low ? (c < v[e] ? c : v[e]) : (c > v[e] ? c : v[e]);
                }
                T* x = cur;
                cur = nxt;
                nxt = x;
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const uint32_t i = e * B + t;
                    const T c = __shfl_xor_sync(0xffffffffu, v[e], j);
                    const bool low = ((i & j) == 0) == ((i & k) == 0);
                    v[e] = low ? (c < v[e] ? c : v[e]) : (c > v[e] ? c : v[e]);
                }
            }
        }
    }
    // the runs: thread t takes keys E t ..; the run starts go to the other buffer
#pragma unroll
    for (int e = 0; e < E; ++e) cur[e * B + t] = v[e];
    __syncthreads();
    uint32_t* starts = reinterpret_cast<uint32_t*>(nxt);
    uint32_t heads = 0, mask = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t i = E * t + e;
        v[e] = cur[i];
        const bool h = i < n && (i == 0 || v[e] != cur[i - 1]);
        mask |= static_cast<uint32_t>(h) << e;
        heads += h;
    }
    const uint32_t lane = t & 31, w = t >> 5;
    uint32_t inc = heads;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += x;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    uint32_t pos = inc - heads, nd = 0;
    for (uint32_t q = 0; q < B >> 5; ++q) {
        const uint32_t x = wsum[q];
        if (q < w) pos += x;
        nd += x;
    }
#pragma unroll
    for (int e = 0; e < E; ++e)
        if ((mask >> e) & 1u) {
            out_keys[pos] = v[e];
            starts[pos++] = E * t + e;
        }
    __syncthreads();
    for (uint32_t d = t; d < nd; d += B) out_counts[d] = (d + 1 < nd ? starts[d + 1] : n) - starts[d];
    if (t == 0) *n_distinct = nd;
}

template <typename T>
cudaError_t launch_sort_rle(const uint64_t* in, uint32_t n, uint32_t P, uint64_t* out_keys, uint64_t* out_counts,
                            uint64_t* n_distinct, cudaStream_t st, uint64_t* launches) {
    const uint32_t N = P < 32 ? 32 : P, B = N < 1024 ? N : 1024;   // N = E B, E = 1, 2 or 4
    auto kern = N <= 1024 ? k_sort_rle<T, 1> : N == 2048 ? k_sort_rle<T, 2> : k_sort_rle<T, 4>;
    const size_t smem = 2 * sizeof(T) * N;
    if (smem > 48 * 1024) {
        cudaError_t e = set_smem_attr(reinterpret_cast<const void*>(kern), static_cast<int>(smem));
        if (e != cudaSuccess) return e;
    }
    kern<<<1, B, smem, st>>>(in, n, out_keys, out_counts, n_distinct);
    ++*launches;
    return cudaGetLastError();
}

inline uint64_t next_pow2(uint64_t v) {
    uint64_t p = 1;
    while (p < v) p <<= 1;
    return p;
}

// Up to this many shots are sorted and counted by one CTA, more by radix sorts
// and tiles (whole calls at N = 12: 3000 shots 122 us, 5000 139).
constexpr uint64_t kSortSmemMax = 4096;

// Run-length encoding of one CTA's sorted keys (any indexable), wsum and carry
// in shared memory.
template <typename Keys>
__device__ __forceinline__ void rle_cta(const Keys& keys, uint32_t shots, uint32_t* wsum, uint32_t& carry, uint32_t* okeys,
                                        uint32_t* ocnt, uint32_t* n_distinct) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    // run-length encode: heads get their output slot; out_counts holds the
    // run starts until they are turned into counts
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (uint32_t base = 0; base < shots; base += blockDim.x) {
        const uint32_t i = base + threadIdx.x;
        const uint32_t head = (i < shots && (i == 0 || keys[i] != keys[i - 1])) ? 1u : 0u;
        uint32_t inc = head;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        if (warp == 0) {
            uint32_t v = lane < nw ? wsum[lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += t;
            }
            wsum[lane] = v;
        }
        __syncthreads();
        const uint32_t pos = carry + (warp ? wsum[warp - 1] : 0) + inc - head;
        if (head) {
            okeys[pos] = keys[i];
            ocnt[pos] = i;
        }
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = pos + head;
        __syncthreads();
    }
    const uint32_t nd = carry;
    for (uint32_t base = 0; base < nd; base += blockDim.x) {
        const uint32_t d = base + threadIdx.x;
        uint32_t c = 0;
        if (d < nd) c = (d + 1 < nd ? ocnt[d + 1] : shots) - ocnt[d];
        __syncthreads();
        if (d < nd) ocnt[d] = c;
        __syncthreads();
    }
    if (threadIdx.x == 0) *n_distinct = nd;
}

// Batched sampler: CTA t samples state t (identity layout) with Philox stream
// id t.  Shared memory: cum[nblocks] (uint64) then keys[P] (uint32).
constexpr int kBatchSampleThreads = 512;

__global__ void __launch_bounds__(kBatchSampleThreads)
    k_batch_sample(const float2* __restrict__ states, int n, uint32_t shots, uint32_t P, uint64_t seed,
                   uint32_t* __restrict__ out_keys, uint32_t* __restrict__ out_counts,
                   uint32_t* __restrict__ n_distinct) {
    extern __shared__ uint64_t sm64[];
    const int traj = blockIdx.x;
    const float2* psi = states + (static_cast<uint64_t>(traj) << n);
    const int bsz = n >= 10 ? 1024 : (1 << n);
    const int nb = (1 << n) / bsz;
    uint64_t* cum = sm64;
    uint32_t* keys = reinterpret_cast<uint32_t*>(cum + nb);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    __shared__ uint32_t wsum[32];
    __shared__ uint32_t carry;

    for (int b = warp; b < nb; b += nw) {
        uint64_t s = 0;
        for (int j = lane; j < bsz; j += 32) s += weight(psi[static_cast<uint64_t>(b) * bsz + j]);
        s = warp_sum_u64(s);
        if (lane == 0) cum[b] = s;
    }
    __syncthreads();
    if (warp == 0) {   // inclusive scan: lane l owns a contiguous range
        const int per = (nb + 31) / 32;
        const int lo = lane * per, hi = min(nb, lo + per);
        uint64_t s = 0;
        for (int i = lo; i < hi; ++i) s += cum[i];
        uint64_t run = warp_incl_scan_u64(s) - s;
        for (int i = lo; i < hi; ++i) {
            run += cum[i];
            cum[i] = run;
        }
    }
    __syncthreads();
    const uint64_t total = cum[nb - 1];
    const int per = (bsz + 31) >> 5;
    for (uint32_t s = warp; s < shots; s += nw) {
        const uint64_t r = philox4x64_10_w0(s, static_cast<uint64_t>(traj), 0, 0, seed, 0);
        const uint64_t u = __umul64hi(r, total);  // floor(r * total / 2^64)
        int lo = 0, hi = nb - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (cum[mid] > u) hi = mid; else lo = mid + 1;
        }
        const uint64_t ub = u - (lo ? cum[lo - 1] : 0);
        const float2* p = psi + static_cast<uint64_t>(lo) * bsz;
        uint64_t wl = 0;
        for (int j = 0; j < per; ++j) {
            const int idx = lane * per + j;
            if (idx < bsz) wl += weight(p[idx]);
        }
        const uint64_t incl = warp_incl_scan_u64(wl);
        const uint64_t excl = incl - wl;
        const unsigned hit = __ballot_sync(0xffffffffu, excl <= ub && ub < incl);
        const int owner = hit ? __ffs(hit) - 1 : 0;
        if (lane == owner) {
            uint64_t acc = excl;
            int j = 0;
            for (; j < per; ++j) {
                const int idx = lane * per + j;
                if (idx >= bsz) break;
                acc += weight(p[idx]);
                if (acc > ub) break;
            }
            keys[s] = static_cast<uint32_t>(lo * bsz + lane * per + j);
        }
    }
    for (uint32_t i = shots + threadIdx.x; i < P; i += blockDim.x) keys[i] = 0xFFFFFFFFu;
    __syncthreads();
    for (uint32_t k = 2; k <= P; k <<= 1)
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t i = threadIdx.x; i < P; i += blockDim.x) {
                const uint32_t l = i ^ j;
                if (l > i) {
                    const bool up = (i & k) == 0;
                    const uint32_t x = keys[i], y = keys[l];
                    if ((x > y) == up) {
                        keys[i] = y;
                        keys[l] = x;
                    }
                }
            }
            __syncthreads();
        }
    rle_cta(keys, shots, wsum, carry, out_keys + static_cast<uint64_t>(traj) * shots,
            out_counts + static_cast<uint64_t>(traj) * shots, n_distinct + traj);
}

// Samples of all trajectories sorted by (trajectory, outcome): CTA t encodes
// trajectory t's.
__global__ void __launch_bounds__(kBatchSampleThreads)
    k_batch_rle(const uint64_t* __restrict__ keys, int n, uint32_t shots, uint32_t* __restrict__ out_keys,
                uint32_t* __restrict__ out_counts, uint32_t* __restrict__ n_distinct) {
    __shared__ uint32_t wsum[32];
    __shared__ uint32_t carry;
    const uint64_t at = static_cast<uint64_t>(blockIdx.x) * shots;
    const uint64_t mask = (1ull << n) - 1;
    struct Outcomes {
        const uint64_t* k;
        uint64_t mask;
        __device__ uint32_t operator[](uint32_t i) const { return static_cast<uint32_t>(k[i] & mask); }
    };
    rle_cta(Outcomes{keys + at, mask}, shots, wsum, carry, out_keys + at, out_counts + at, n_distinct + blockIdx.x);
}

// Inclusive prefixes of the block weights of each state, a CTA per state of up
// to 4096 blocks.
__global__ void __launch_bounds__(1024) k_batch_scan(uint64_t* __restrict__ cum, int nblocks) {
    __shared__ uint64_t wsum[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t* c = cum + static_cast<uint64_t>(blockIdx.x) * nblocks;
    const int i0 = 4 * threadIdx.x;
    uint64_t v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = i0 + k < nblocks ? c[i0 + k] : 0;
    v[1] += v[0];
    v[2] += v[1];
    v[3] += v[2];
    const uint64_t inc = warp_incl_scan_u64(v[3]);
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    if (wid == 0) wsum[lane] = warp_incl_scan_u64(wsum[lane]);
    __syncthreads();
    const uint64_t off = inc - v[3] + (wid ? wsum[wid - 1] : 0);
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (i0 + k < nblocks) c[i0 + k] = v[k] + off;
}

}  // namespace

uint64_t next_pow2_u64(uint64_t v) { return next_pow2(v); }

namespace {

// Sorts n keys by their bits [lo, lo + bits), a digit of eight at a time, between
// the two arrays; returns the one they end in.  hist: 256 (tiles + 1) words.
uint64_t* radix_sort(uint64_t* from, uint64_t* other, uint64_t n, int lo, int bits, uint32_t* hist, cudaStream_t st,
                     uint64_t* launches) {
    const uint32_t ntiles = static_cast<uint32_t>((n + kRadixTile - 1) / kRadixTile);
    uint32_t* totals = hist + 256ull * ntiles;
    for (int sh = 0; sh < bits; sh += 8) {
        k_radix_hist<<<ntiles, kRadixThreads, 0, st>>>(from, n, lo + sh, ntiles, hist);
        k_radix_scan<<<256, kRadixThreads, 0, st>>>(hist, ntiles, totals);
        k_radix_scatter<<<ntiles, kRadixThreads, 0, st>>>(from, n, lo + sh, ntiles, hist, totals, other);
        std::swap(from, other);
        *launches += 3;
    }
    return from;
}

int bits_of(uint64_t count) {   // bits of 0 .. count - 1
    int b = 0;
    while ((1ull << b) < count) ++b;
    return b;
}

// shots per resolving warp: few when most lie in blocks of their own, which a
// warp reads one after another, many when they share blocks.  Whole calls with
// 8 / 16 / 32 at so many shots a block: N = 26, 1.5: 413 / 421 / 447 us, 2.5: 458 / 457
// / 475, 4: 501 / 485 / 492, 6: 552 / 524 / 509, 12: 721 / 633 / 600; N = 24, 3: 261 /
// 269 / 295, 4: 270 / 271 / 280, 8: 282 / 272 / 274, 30: 438 / 380 / 352; N = 22, 8: 202 /
// 195 / 201, 12: 203 / 197 / 197, 30: 232 / 212 / 206.
int resolve_per(uint64_t shots, uint64_t nblocks) { return shots >= 8 * nblocks ? 32 : shots >= 3 * nblocks ? 16 : 8; }

// The batch's samples of all trajectories at once, where the shots' numbers fit
// their keys: a CTA per trajectory reads a block of 8 KiB for every shot and sorts
// in one CTA, which is slower at every size measured (whole runs of shallow
// trajectories, N = 10 / 14 / 20: one with 100 shots 113 / 131 / 850 us against
// 57 / 85 / 468, 64 with 16 000 shots each 11.2 / 12.2 / 14.3 ms against 0.21 /
// 0.27 / 1.64).  It remains for states below one block of 1024 amplitudes and
// where the scratch could not be allocated.
bool batch_samples_together(int n, int n_traj, uint32_t shots) {
    const uint64_t total = static_cast<uint64_t>(n_traj) * shots;
    return n >= 10 && total <= (1ull << kShotBits);
}

}  // namespace

size_t batch_sample_scratch_bytes(int n, int n_traj, uint32_t shots) {
    if (!batch_samples_together(n, n_traj, shots)) return 0;
    const uint64_t total = static_cast<uint64_t>(n_traj) * shots, ntiles = (total + kRadixTile - 1) / kRadixTile;
    return sizeof(uint64_t) * ((static_cast<uint64_t>(n_traj) << (n - 10)) + 2 * total) + sizeof(uint32_t) * 256 * (ntiles + 1);
}

cudaError_t launch_batch_sample(const float2* states, int n, int n_traj, uint32_t shots, uint64_t seed,
                                uint32_t* out_keys, uint32_t* out_counts, uint32_t* n_distinct, void* d_scratch,
                                cudaStream_t st, uint64_t* launches) {
    if (d_scratch && batch_samples_together(n, n_traj, shots)) {
        const uint64_t nblocks = 1ull << (n - 10), all = nblocks * n_traj, total = static_cast<uint64_t>(n_traj) * shots;
        uint64_t* cum = static_cast<uint64_t*>(d_scratch);
        uint64_t* x = cum + all;
        uint64_t* y = x + total;
        uint32_t* hist = reinterpret_cast<uint32_t*>(y + total);
        const uint64_t nb = std::min<uint64_t>((all + 7) / 8, 2ull * num_sms());   // two CTAs of 8 warps fit an SM
        k_weights_z1024<0, true><<<static_cast<unsigned>(nb), kRedThreads, 0, st>>>(reinterpret_cast<const float4*>(states), all,
                                                                            cum, ZMasks{}, nullptr, nullptr, nullptr);
        k_batch_scan<<<n_traj, 1024, 0, st>>>(cum, static_cast<int>(nblocks));
        k_draw_blocks<<<static_cast<unsigned>((total + 255) / 256), 256, 0, st>>>(cum, nblocks, shots, total, seed, 0, x);
        uint64_t* d = radix_sort(x, y, total, kShotBits, bits_of(all), hist, st, launches);
        uint64_t* keys = d == x ? y : x;
        const int per = resolve_per(shots, nblocks);
        const uint64_t cta = static_cast<uint64_t>(per) * kResolveWarps;
        k_draw_resolve<<<static_cast<unsigned>((total + cta - 1) / cta), 32 * kResolveWarps, 0, st>>>(
            reinterpret_cast<const float4*>(states), cum, nblocks, Layout{}, d, shots, total, seed, 0, per, keys);
        keys = radix_sort(keys, d, total, 0, n + bits_of(n_traj), hist, st, launches);
        k_batch_rle<<<n_traj, kBatchSampleThreads, 0, st>>>(keys, n, shots, out_keys, out_counts, n_distinct);
        *launches += 5;
        return cudaGetLastError();
    }
    const int bsz = n >= 10 ? 1024 : (1 << n);
    const uint64_t nb = (1ull << n) / bsz;
    const uint32_t P = static_cast<uint32_t>(next_pow2(shots));
    const size_t smem = sizeof(uint64_t) * nb + sizeof(uint32_t) * P;
    {
        cudaError_t e = set_smem_attr(reinterpret_cast<const void*>(k_batch_sample), static_cast<int>(smem));
        if (e != cudaSuccess) return e;
    }
    k_batch_sample<<<n_traj, kBatchSampleThreads, smem, st>>>(states, n, shots, P, seed, out_keys, out_counts,
                                                              n_distinct);
    ++*launches;
    return cudaGetLastError();
}

// Diagonal of a vectorised density matrix (2n-qubit state, vec index
// x + 2^n x): optional copy of rho_xx (real part) to out[], and per-block
// FP64 partial sums of rho_xx (-1)^popc(x & mask) for the final reduction.
__global__ void __launch_bounds__(kRedThreads) k_dm_diag(const float2* __restrict__ psi, Layout lay, int n,
                                                          uint64_t mask, double* __restrict__ out,
                                                          double* __restrict__ partials) {
    const uint64_t dim = 1ull << n;
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
    double acc = 0.0;
    for (uint64_t x = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; x < dim; x += stride) {
        const double p = psi[encode_logical(x | (x << n), lay)].x;
        if (out) out[x] = p;
        acc += (__popcll(x & mask) & 1) ? -p : p;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    __shared__ double sh[kRedThreads / 32];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kRedThreads / 32; ++w) t += sh[w];
        partials[blockIdx.x] = t;
    }
}

int reduce_partials() { return num_sms() * kRedBlocksPerSM; }

namespace {

cudaError_t launch_zsums(const float2* psi, int n, const uint64_t* physmasks, int nmasks, double* d_partials, double* d_out,
                         unsigned* d_count, cudaStream_t st, uint64_t* launches) {
    const uint64_t nblocks = 1ull << (n - 10);
    ZMasks zm{};
    zm.n = nmasks;
    for (int m = 0; m < nmasks; ++m) zm.m[m] = physmasks[m];
    // the same grid for any number of masks: a mask's partial sums are the same in all of them
    const uint64_t nb = std::min<uint64_t>((nblocks + 7) / 8, static_cast<uint64_t>(kZCtas) * num_sms());
    auto kern = nmasks == 1 ? k_zsums1024<1> : nmasks == 2 ? k_zsums1024<2> : nmasks == 3 ? k_zsums1024<3> : k_zsums1024<4>;
    kern<<<static_cast<unsigned>(nb), kRedThreads, 0, st>>>(reinterpret_cast<const float4*>(psi), nblocks, zm, d_partials,
                                                             d_out, d_count);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_reduce_z(const float2* psi, int n, uint64_t physmask, double* d_partials, double* d_out,
                            unsigned* d_count, cudaStream_t st, uint64_t* launches) {
    const uint64_t npairs = (1ull << n) >> 1;
    const int nb = reduce_partials();
    if (npairs == 0) {
        // n = 1 is still >= one pair; n >= 1 always holds here
        return cudaErrorInvalidValue;
    }
    if (n >= 10) return launch_zsums(psi, n, &physmask, 1, d_partials, d_out, d_count, st, launches);
    k_reduce_z<<<nb, kRedThreads, 0, st>>>(reinterpret_cast<const float4*>(psi), npairs, physmask, d_partials);
    k_finalize_sum<<<1, kRedThreads, 0, st>>>(d_partials, nb, d_out);
    *launches += 2;
    return cudaGetLastError();
}

cudaError_t launch_reduce_z_multi(const float2* psi, int n, const uint64_t* physmasks, int nmasks,
                                  double* d_partials, double* d_out, unsigned* d_count, cudaStream_t st,
                                  uint64_t* launches) {
    if (nmasks < 1 || nmasks > kMaxZMasks || n < 1) return cudaErrorInvalidValue;
    if (n >= 10) return launch_zsums(psi, n, physmasks, nmasks, d_partials, d_out, d_count, st, launches);
    const uint64_t npairs = (1ull << n) >> 1;
    const int nb = reduce_partials();
    ZMasks zm{};
    zm.n = nmasks;
    for (int m = 0; m < nmasks; ++m) zm.m[m] = physmasks[m];
    k_reduce_z_multi<<<nb, kRedThreads, 0, st>>>(reinterpret_cast<const float4*>(psi), npairs, zm, d_partials);
    k_finalize_sum<<<nmasks, kRedThreads, 0, st>>>(d_partials, nb, d_out);
    *launches += 2;
    return cudaGetLastError();
}

cudaError_t launch_dm_diag(const float2* psi, int n, const int32_t* layout_host, uint64_t mask, double* d_out,
                           double* d_partials, double* d_sum, cudaStream_t st, uint64_t* launches) {
    Layout lay{};
    lay.n = 2 * n;
    for (int q = 0; q < 2 * n; ++q) lay.L[q] = layout_host[q];
    const int nb = reduce_partials();
    k_dm_diag<<<nb, kRedThreads, 0, st>>>(psi, lay, n, mask, d_out, d_partials);
    k_finalize_sum<<<1, kRedThreads, 0, st>>>(d_partials, nb, d_sum);
    *launches += 2;
    return cudaGetLastError();
}

cudaError_t launch_probs_logical(const float2* psi, int n, const int32_t* layout_host, double* out, double* d_partials,
                                 double* d_norm, unsigned* d_count, cudaStream_t st, uint64_t* launches) {
    if (n < kProbT || reinterpret_cast<uintptr_t>(out) % 16) {   // small, or an output that takes no 16-byte stores
        Layout lay{};
        lay.n = n;
        for (int q = 0; q < n; ++q) lay.L[q] = layout_host[q];
        const uint64_t dim = 1ull << n;
        k_probs_logical<<<static_cast<unsigned>((dim + 255) / 256), 256, 0, st>>>(psi, lay, out);
        ++*launches;
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess || !d_norm) return e;
        return launch_reduce_z(psi, n, 0, d_partials, d_norm, d_count, st, launches);
    }
    int inv[QSA_MAX_QUBITS];
    for (int q = 0; q < n; ++q) inv[layout_host[q]] = q;
    // tile: the six lowest positions, the positions of the six lowest qubits,
    // then the next lowest positions
    uint64_t tile = 63;
    for (int q = 0; q < 6; ++q) tile |= 1ull << layout_host[q];
    for (int p = 0; __builtin_popcountll(tile) < kProbT; ++p) tile |= 1ull << p;
    ProbArgs a{};
    a.psi = psi;
    a.out = out;
    a.partials = d_norm ? d_partials : nullptr;
    a.norm = d_norm;
    a.count = d_count;
    a.ntiles = 1ull << (n - kProbT);
    int tb[QSA_MAX_QUBITS], nt = 0;   // tile bit of a position
    for (int p = 0; p < n; ++p) {
        if ((tile >> p) & 1) {
            a.poff[nt] = 1ull << p;
            tb[p] = nt++;
        } else {
            a.opos[a.nouter] = static_cast<uint8_t>(p);
            a.oq[a.nouter++] = static_cast<uint8_t>(inv[p]);
        }
    }
    // The writing lanes vary the tile's logical qubits 1..4 (positions of the
    // tile bits lt[1..4]): those at tile bit 4 or above take slot bits 1..3 that
    // no other of them has.
    int lt[kProbT], nl = 0;
    for (int q = 0; q < n; ++q)
        if ((tile >> layout_host[q]) & 1) {
            a.loff[nl] = 1ull << q;
            lt[nl++] = tb[layout_host[q]];
        }
    uint32_t used = 0, vec[kProbT] = {};
    for (int i = 1; i <= 4; ++i)
        if (lt[i] >= 1 && lt[i] <= 3) used |= 1u << lt[i];
    for (int i = 1; i <= 4; ++i)
        if (lt[i] >= 4)
            for (int j = 1; j <= 3; ++j)
                if (!((used >> j) & 1)) {
                    used |= 1u << j;
                    vec[lt[i]] = 1u << j;
                    break;
                }
    for (int b = 0; b < kProbT; ++b) a.pslot[b] = static_cast<uint16_t>((1u << b) ^ vec[b]);
    for (int i = 0; i < kProbT; ++i) a.lslot[i] = a.pslot[lt[i]];
    // as many CTAs as stay resident; at most reduce_partials()
    const uint64_t nb = std::min<uint64_t>(a.ntiles, static_cast<uint64_t>(kProbCtas) * num_sms());
    k_probs_tile<<<static_cast<unsigned>(nb), kRedThreads, 0, st>>>(a);
    ++*launches;
    return cudaGetLastError();
}

size_t sample_scratch_bytes(int n, uint64_t shots) {
    const int bsz = n >= 10 ? 1024 : (1 << n);
    const uint64_t nblocks = (1ull << n) / bsz;
    const uint64_t P = next_pow2(shots);
    return sizeof(uint64_t) * (nblocks + P + shots) + 256;
}

cudaError_t launch_sample(const float2* psi, int n, const int32_t* layout_host, uint64_t shots, uint64_t seed,
                          uint64_t stream_id, void* d_scratch, uint64_t* d_out_keys, uint64_t* d_out_counts,
                          uint64_t* d_n_distinct, cudaStream_t st, uint64_t* launches) {
    return launch_sample_z(psi, n, layout_host, shots, seed, stream_id, d_scratch, d_out_keys, d_out_counts,
                           d_n_distinct, nullptr, 0, nullptr, nullptr, nullptr, st, launches);
}

cudaError_t launch_sample_z(const float2* psi, int n, const int32_t* layout_host, uint64_t shots, uint64_t seed,
                            uint64_t stream_id, void* d_scratch, uint64_t* d_out_keys, uint64_t* d_out_counts,
                            uint64_t* d_n_distinct, const uint64_t* physmasks, int nmasks, double* d_zpartials,
                            double* d_zout, unsigned* d_count, cudaStream_t st, uint64_t* launches) {
    if (nmasks < 0 || nmasks > kMaxZMasks) return cudaErrorInvalidValue;
    Layout lay{};
    lay.n = n;
    for (int q = 0; q < n; ++q) lay.L[q] = layout_host[q];
    const int bsz = n >= 10 ? 1024 : (1 << n);
    const uint64_t nblocks = (1ull << n) / bsz;
    const uint64_t P = next_pow2(shots);
    uint64_t* cum = reinterpret_cast<uint64_t*>(d_scratch);
    uint64_t* keys = cum + nblocks;
    uint64_t* starts = keys + P;

    const unsigned wpb = 8;  // warps per CTA
    if (bsz == 1024) {
        ZMasks zm{};
        zm.n = nmasks;
        for (int m = 0; m < nmasks; ++m) zm.m[m] = physmasks[m];
        bool even = true;   // no mask holds the lowest position
        for (int m = 0; m < nmasks; ++m) even = even && !(physmasks[m] & 1);
        auto kern = nmasks == 0   ? k_weights_z1024<0, true>
                    : nmasks == 1 ? (even ? k_weights_z1024<1, true> : k_weights_z1024<1, false>)
                    : nmasks == 2 ? (even ? k_weights_z1024<2, true> : k_weights_z1024<2, false>)
                    : nmasks == 3 ? (even ? k_weights_z1024<3, true> : k_weights_z1024<3, false>)
                                  : (even ? k_weights_z1024<4, true> : k_weights_z1024<4, false>);
        // as many CTAs as stay resident (at most reduce_partials(), the partials' size)
        int occ = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kRedThreads, 0);
        if (e != cudaSuccess) return e;
        occ = occ < 1 ? 1 : (occ > kRedBlocksPerSM ? kRedBlocksPerSM : occ);
        uint64_t nb = (nblocks + wpb - 1) / wpb;
        const uint64_t cap = static_cast<uint64_t>(num_sms()) * occ;
        if (nb > cap) nb = cap;
        kern<<<static_cast<unsigned>(nb), kRedThreads, 0, st>>>(reinterpret_cast<const float4*>(psi), nblocks, cum,
                                                                 zm, d_zpartials, d_zout, d_count);
    } else if (nmasks > 0) {
        ZMasks zm{};
        zm.n = nmasks;
        for (int m = 0; m < nmasks; ++m) zm.m[m] = physmasks[m];
        const int nb = reduce_partials();
        k_block_weights_z<<<nb, kRedThreads, 0, st>>>(psi, nblocks, bsz, cum, zm, d_zpartials);
        k_finalize_sum<<<nmasks, kRedThreads, 0, st>>>(d_zpartials, nb, d_zout);
        ++*launches;
    } else {
        k_block_weights<<<static_cast<unsigned>((nblocks + wpb - 1) / wpb), wpb * 32, 0, st>>>(psi, nblocks, bsz,
                                                                                                cum);
    }
    const uint64_t nseg = (nblocks + kScanSeg - 1) / kScanSeg;
    if (nseg > 1 && nseg <= P + shots) {
        // segment totals in the key area, which k_draw fills only afterwards
        k_scan_segments<<<static_cast<unsigned>(nseg), 1024, 0, st>>>(cum, nblocks, keys);
        k_scan_inclusive<<<1, 1024, 0, st>>>(keys, nseg);
        uint64_t ab = (nblocks - kScanSeg + 255) / 256;
        const uint64_t cap = static_cast<uint64_t>(num_sms()) * 8;
        if (ab > cap) ab = cap;
        k_scan_add<<<static_cast<unsigned>(ab), 256, 0, st>>>(cum, nblocks, keys);
        *launches += 2;
    } else {
        k_scan_inclusive<<<1, 1024, 0, st>>>(cum, nblocks);
    }
    auto draw = [&](uint64_t* to) {
        if (bsz == 1024)
            k_draw1024<<<static_cast<unsigned>((shots + kResolveWarps - 1) / kResolveWarps), 32 * kResolveWarps, 0, st>>>(
                reinterpret_cast<const float4*>(psi), cum, nblocks, lay, shots, seed, stream_id, to);
        else
            k_draw<<<static_cast<unsigned>((shots + wpb - 1) / wpb), wpb * 32, 0, st>>>(psi, cum, nblocks, bsz, lay, shots,
                                                                                         seed, stream_id, to);
    };
    if (P <= kSortSmemMax) {
        draw(keys);
        *launches += 3;
        const uint32_t m = static_cast<uint32_t>(shots), p2 = static_cast<uint32_t>(P);
        return n <= 32 ? launch_sort_rle<uint32_t>(keys, m, p2, d_out_keys, d_out_counts, d_n_distinct, st, launches)
                       : launch_sort_rle<uint64_t>(keys, m, p2, d_out_keys, d_out_counts, d_n_distinct, st, launches);
    }
    // Many shots: radix sorts between the arrays at hand (the digit counts go
    // where the outcome counts end up).  The outcomes must end in `keys`.
    const uint32_t ntiles = static_cast<uint32_t>((shots + kRadixTile - 1) / kRadixTile);
    uint32_t* hist = reinterpret_cast<uint32_t*>(d_out_counts);
    auto sort = [&](uint64_t* from, uint64_t* other, int lo, int bits) {
        return radix_sort(from, other, shots, lo, bits, hist, st, launches);
    };
    const bool odd = ((n + 7) / 8) & 1;
    uint64_t* first = odd ? d_out_keys : keys;    // the unsorted outcomes
    uint64_t* second = odd ? keys : d_out_keys;
    // Grouping by block costs a sort of the shots (about 40 us of launches) and a read of every block met;
    // shot by shot, each reads its block.  Where they meet grows with the root of the number of blocks
    // (whole calls, grouped against shot by shot: N = 16, 16 384 shots 153 and 157 us, 30 000 155 and 185;
    // N = 20, 16 384: 202 and 174, 60 000: 203 and 263; N = 26, 60 000: 420 and 382, 100 000: 445 and 460;
    // N = 28, 100 000: 742 and 693, 200 000: 861 and 901).
    if (bsz == 1024 && shots >= 16384 + (256ull << ((n - 10) / 2))) {
        uint64_t* d = starts;
        k_draw_blocks<<<static_cast<unsigned>((shots + 255) / 256), 256, 0, st>>>(cum, nblocks, shots, shots, seed, stream_id,
                                                                                  d);
        d = sort(d, second, kShotBits, n - 10);
        const int per = resolve_per(shots, nblocks);
        const uint64_t cta = static_cast<uint64_t>(per) * kResolveWarps;
        k_draw_resolve<<<static_cast<unsigned>((shots + cta - 1) / cta), 32 * kResolveWarps, 0, st>>>(
            reinterpret_cast<const float4*>(psi), cum, nblocks, lay, d, shots, shots, seed, stream_id, per, first);
        *launches += 2;
    } else {
        draw(first);
        ++*launches;
    }
    sort(first, second, 0, n);
    uint64_t* tiles = d_out_counts;
    k_rle_heads<<<ntiles, kRadixThreads, 0, st>>>(keys, shots, tiles);
    k_scan_inclusive<<<1, 1024, 0, st>>>(tiles, ntiles);
    k_rle_write<<<ntiles, kRadixThreads, 0, st>>>(keys, shots, tiles, d_out_keys, starts, d_n_distinct);
    k_rle_counts<<<static_cast<unsigned>((shots + 255) / 256), 256, 0, st>>>(starts, shots, d_n_distinct, d_out_counts);
    *launches += 6;
    return cudaGetLastError();
}

}  // namespace qsa

// ---------------------------------------------------------------------------
// Sampling without any device allocation.
//
// Some callers cannot let the library call cudaMalloc: a framework whose
// caching allocator owns the device memory budget (a stray cudaMalloc can fail
// or fragment the pool when the state fills most of HBM, as at N = 33/34), or
// a pipeline that must not stall, since cudaFree synchronises the whole
// device.  For them the sampler's scratch (block cumulative weights, the sort
// keys and the run starts) lives in one fixed, file-scope device array that
// every GPU loading this library holds until the process exits.
// ---------------------------------------------------------------------------
#include <mutex>
#include <string>

#include "qsa_runtime.h"

namespace {
constexpr uint64_t kNoAllocWords = QSA_NOALLOC_SCRATCH_WORDS;
static __device__ __align__(256) uint64_t g_noalloc_scratch[kNoAllocWords];

std::mutex g_noalloc_mu;
void* g_noalloc_addr[256] = {};

// Device address of the array for the current device, looked up once per
// device (host code only sees a host-side stand-in for the symbol).
cudaError_t noalloc_scratch_ptr(void** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> g(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_addr[dev] = p;
    }
    *out = g_noalloc_addr[dev];
    return cudaSuccess;
}
}  // namespace

extern "C" qsa_status qsa_sample_counts_noalloc(const void* dev_amplitudes, int n_qubits,
                                                const int32_t* phys_of_logical, uint64_t shots, uint64_t seed,
                                                uint64_t* out_outcomes_dev, uint64_t* out_counts_dev,
                                                uint64_t* out_n_distinct_dev, void* cuda_stream) {
    using qsa::fail;
    if (!dev_amplitudes || (reinterpret_cast<uintptr_t>(dev_amplitudes) % 16))
        return fail(QSA_E_ARG, "amplitudes must be a non-NULL, 16-byte aligned device pointer");
    if (n_qubits < 1 || n_qubits > QSA_MAX_QUBITS) return fail(QSA_E_ARG, "n_qubits must be in 1..34");
    if (!phys_of_logical) return fail(QSA_E_ARG, "layout is NULL");
    uint64_t seen = 0;
    for (int q = 0; q < n_qubits; ++q) {
        const int p = phys_of_logical[q];
        if (p < 0 || p >= n_qubits || ((seen >> p) & 1)) return fail(QSA_E_ARG, "layout is not a bijection");
        seen |= 1ull << p;
    }
    if (shots < 1 || shots > (1ull << 26)) return fail(QSA_E_ARG, "shots must be in 1..2^26");
    if (!out_outcomes_dev || !out_counts_dev || !out_n_distinct_dev) return fail(QSA_E_ARG, "output is NULL");
    const int bsz = n_qubits >= 10 ? 1024 : (1 << n_qubits);
    const uint64_t nblocks = (1ull << n_qubits) / bsz;
    const uint64_t need = nblocks + qsa::next_pow2_u64(shots) + shots;
    if (need > kNoAllocWords)
        return fail(QSA_E_RANGE, "request needs " + std::to_string(need) + " words of sampler scratch; the fixed "
                                 "no-allocation buffer holds " + std::to_string(kNoAllocWords) +
                                 " (2^(N-10) + next_pow2(shots) + shots must fit)");
    void* scratch = nullptr;
    cudaError_t e = noalloc_scratch_ptr(&scratch);
    if (e != cudaSuccess) return fail(QSA_E_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    uint64_t launches = 0;
    e = qsa::launch_sample(static_cast<const float2*>(dev_amplitudes), n_qubits, phys_of_logical, shots, seed, 0,
                           scratch, out_outcomes_dev, out_counts_dev, out_n_distinct_dev,
                           static_cast<cudaStream_t>(cuda_stream), &launches);
    if (e != cudaSuccess) return fail(QSA_E_CUDA, std::string("sampler kernels: ") + cudaGetErrorString(e));
    return QSA_OK;
}
