// FP32 fused dense update, product and qubit-permutation kernels (sm_103a).
//
// All three share one tile engine: a CTA walks tiles t0, t0 + stride, ...;
// each tile (2^T amplitudes = 2^nx contiguous runs of 2^m amplitudes) is
// staged into shared memory with 16-byte cp.async copies in an S-deep ring,
// transformed, and written back in place.  Tiles partition the index space,
// so the in-place update needs no second state buffer (the paper's CUDA path
// holds two, App. C "Capacity and execution profiles").
//
//   apply   (§IV-B, R2 apply; Eq. cost-formal): for every group of 2^k
//           amplitudes that differ only in the target bits,
//           psi'[x|spread(r)] = sum_c G[r][c] psi[x|spread(c)];
//   permute (§IV-D, Lemma "distributed promotion swap" with the rank bits read
//           as out-of-block bits): psi'[tau(y)] = psi[y] for a permutation tau
//           of the bit positions, in as few passes as its cycles allow.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>
#include <vector>

#include "qsa_bounds.cuh"
#include "qsa_device.cuh"
#include "qsa_internal.h"

namespace qsa {

namespace {

using namespace dev;

constexpr int kThreads = 256;
constexpr int kBeyondL2 = 24;   // states of 128 MiB and more do not stay in the L2 (129 MB)

struct TileArgs {
    float2* psi;
    uint64_t ntiles;
    int T, m, nx;
    int xpos[6];
};

__device__ __forceinline__ uint64_t tile_base(const TileArgs& a, uint64_t t) {
    uint64_t b = t << a.m;
#pragma unroll
    for (int e = 0; e < 6; ++e)
        if (e < a.nx) b = insert_zero(b, a.xpos[e]);
    return b;
}

// Global index of tile-local index j.
__device__ __forceinline__ uint64_t tile_global(const TileArgs& a, const uint64_t* runoff, uint64_t base,
                                                uint32_t j) {
    return base | (j & ((1u << a.m) - 1u)) | runoff[j >> a.m];
}

__device__ __forceinline__ void build_runoff(const TileArgs& a, uint64_t* runoff) {
    for (int r = threadIdx.x; r < (1 << a.nx); r += blockDim.x) {
        uint64_t off = 0;
#pragma unroll
        for (int e = 0; e < 6; ++e)
            if (e < a.nx && ((r >> e) & 1)) off |= 1ull << a.xpos[e];
        runoff[r] = off;
    }
}

// Issue the 16-byte copies of tile t into stage buffer `st`.
__device__ __forceinline__ void load_tile(const TileArgs& a, const uint64_t* runoff, uint64_t t, float2* st) {
    const uint64_t base = tile_base(a, t);
    const uint32_t chunks = 1u << (a.T - 1);
    for (uint32_t q = threadIdx.x; q < chunks; q += blockDim.x) {
        uint32_t j = q << 1;
        const uint64_t gi = tile_global(a, runoff, base, j);
        if (dbg::in_bounds(gi, 2, a.ntiles << a.T, 1)) cp_async16(st + j, a.psi + gi);
    }
}

// ---------------------------------------------------------------------------
// Apply
// ---------------------------------------------------------------------------
struct ApplyArgs {
    TileArgs t;
    const float* mat;   // 2 * 4^K floats
    int tl[6];          // tile-local position of target j (V order)
    int tls[6];         // the same positions, ascending
    uint8_t fv[16];     // stage layout: slot vector of tile-local position p >= 4 (k <= 4)
    // k <= 4 launches: the tile-local offsets of a group's D members in the plain (loffc) and the
    // swizzled (sloffc) stage, formed on the host and read at compile-time member indices from the
    // parameter bank
    int loffc[16];
    int sloffc[16];
};

// Stage layout of the k <= 4 kernels: tile-local element j sits at
// j ^ (h(j >> 4) << 1), h linear with h(bit i) = fv[4 + i].  Position 0 stays
// the element within a 16-byte unit and positions 1..3 its slot in a 128-byte
// line, so the copies in and out move whole 16-byte units with eight lanes on
// eight slots; the slot vectors of higher positions are chosen per launch so
// that the lowest non-target positions (the bits that vary across a
// half-warp's groups) land on distinct banks.
__device__ __forceinline__ uint32_t stage_xor(const uint8_t* htab, uint32_t j) {
    return static_cast<uint32_t>(htab[j >> 4]) << 1;
}

__device__ __forceinline__ void build_htab(const ApplyArgs& a, uint8_t* htab) {
    const int n = 1 << (a.t.T - 4);
    for (int x = threadIdx.x; x < n; x += blockDim.x) {
        uint32_t h = 0;
#pragma unroll
        for (int i = 0; i < 12; ++i)   // constant indices keep the arguments in parameter space
            if (i < a.t.T - 4 && ((x >> i) & 1)) h ^= a.fv[4 + i];
        htab[x] = static_cast<uint8_t>(h);
    }
}

__device__ __forceinline__ void load_tile_swz(const TileArgs& a, const uint64_t* runoff, const uint8_t* htab, uint64_t t,
                                              float2* st) {
    const uint64_t base = tile_base(a, t);
    const uint32_t chunks = 1u << (a.T - 1);
    for (uint32_t q = threadIdx.x; q < chunks; q += blockDim.x) {
        const uint32_t j = q << 1;
        const uint64_t gi = tile_global(a, runoff, base, j);
        if (dbg::in_bounds(gi, 2, a.ntiles << a.T, 2)) cp_async16(st + (j ^ stage_xor(htab, j)), a.psi + gi);
    }
}

// Write a transformed tile back in address order (16-byte units).  All of a
// thread's shared-memory reads come before its stores, which they could not
// pass otherwise.
template <int UNITS>
__device__ __forceinline__ void store_tile_swz(const TileArgs& a, const uint64_t* runoff, const uint8_t* htab,
                                               uint64_t t, const float2* st) {
    const uint64_t base = tile_base(a, t);
    float4 v[UNITS];
    uint64_t g[UNITS];
#pragma unroll
    for (int u = 0; u < UNITS; ++u) {
        const uint32_t j = (threadIdx.x + u * blockDim.x) << 1;
        v[u] = *reinterpret_cast<const float4*>(st + (j ^ stage_xor(htab, j)));
        g[u] = tile_global(a, runoff, base, j);
    }
#pragma unroll
    for (int u = 0; u < UNITS; ++u)
        if (dbg::in_bounds(g[u], 2, a.ntiles << a.T, 3)) __stcs(reinterpret_cast<float4*>(a.psi + g[u]), v[u]);
}

// The tile pipeline of one fused operator over tiles t0, t0 + stride, ...
// Ms (G as float2[D][D]), runoff and loff are set up in shared memory.
// SWZ (k <= 4): the stage takes the swizzled layout (htab; sloff holds the
// swizzled group offsets), so a half-warp's gathers meet at most two to a
// bank wherever the targets sit.  WB (with SWZ, one item per group): each
// item writes its outputs in place and the tile goes back in address order
// (16-byte units of 2^TB-amplitude tiles), for target sets whose direct
// stores would give every lane its own sector.
template <int K, int R, int S, bool SWZ = false, bool WB = false, int TB = 11, bool PO = false, int NG = 1, int TH = kThreads, bool SC = false>
__device__ __forceinline__ void apply_tiles(const ApplyArgs& a, float2* stage, const float2* Ms,
                                            const uint64_t* runoff, const int* loff, uint64_t t0, uint64_t stride,
                                            const uint8_t* htab = nullptr, const int* sloff = nullptr) {
    constexpr int D = 1 << K;
    static_assert(!WB || (SWZ && R == D), "in-place outputs: swizzled stage, the whole group in one item");
    // PO: member offsets from the parameter bank (k <= 4)
    static_assert(!PO || D <= 16, "parameter-bank member offsets: k <= 4");
    auto moff = [&](int c) { return PO ? a.loffc[c] : loff[c]; };
    auto msoff = [&](int c) { return PO ? a.sloffc[c] : sloff[c]; };
    const int tileAmps = 1 << a.t.T;
    auto load = [&](uint64_t t, float2* st) {
        if constexpr (SWZ)
            load_tile_swz(a.t, runoff, htab, t, st);
        else
            load_tile(a.t, runoff, t, st);
    };
#pragma unroll
    for (int s = 0; s < S - 1; ++s) {
        uint64_t t = t0 + s * stride;
        if (t < a.t.ntiles) load(t, stage + s * tileAmps);
        cp_async_commit();
    }
    const int G = tileAmps >> K;                  // groups per tile
    const int gshift = a.t.T - K;
    const int items = G * (D / R);
    int it_stage = 0;
    for (uint64_t t = t0; t < a.t.ntiles; t += stride) {
        uint64_t tn = t + (S - 1) * stride;
        int ld_stage = it_stage + (S - 1);
        if (ld_stage >= S) ld_stage -= S;
        if (tn < a.t.ntiles) load(tn, stage + ld_stage * tileAmps);
        cp_async_commit();
        cp_async_wait<S - 1>();
        __syncthreads();

        float2* st = stage + it_stage * tileAmps;
        const uint64_t base = tile_base(a.t, t);
        // NG groups per item share the matrix's loads (whole groups only: R = D, full tiles)
        for (int it = threadIdx.x; it < items / NG; it += blockDim.x) {
            const int g = it & (G - 1);
            const int rb = it >> gshift;
            uint32_t lb[NG], lbs[NG];   // the groups' bases, in the tile and in the stage
#pragma unroll
            for (int x = 0; x < NG; ++x) {
                lb[x] = static_cast<uint32_t>(g + x * (G / NG));
#pragma unroll
                for (int j = 0; j < K; ++j) lb[x] = static_cast<uint32_t>(insert_zero(lb[x], a.tls[j]));
                lbs[x] = SWZ ? (lb[x] ^ stage_xor(htab, lb[x])) : lb[x];
            }
            auto put = [&](int x, int r, float re, float im) {
                if constexpr (WB) {
                    st[lbs[x] ^ msoff(r)] = make_float2(re, im);   // in place: inputs are in registers
                } else {
                    const uint64_t gj = tile_global(a.t, runoff, base, lb[x] | moff(r));
                    if (dbg::in_bounds(gj, 1, a.t.ntiles << a.t.T, 4)) __stcs(a.t.psi + gj, make_float2(re, im));
                }
            };
            if constexpr (!SC) {
                // Packed FP32 pairs: with x2_c = (Re v_c, Re v_c), y2_c = (Im v_c, Im v_c)
                // and g = (Re G, Im G), p = sum x2_c * g and q = sum y2_c * g give
                // Re = p.x - q.y and Im = p.y + q.x; one 16-byte load of two G entries
                // feeds four f32x2 FMAs.
                uint64_t x2[NG][D], y2[NG][D];
#pragma unroll
                for (int x = 0; x < NG; ++x)
#pragma unroll
                    for (int c = 0; c < D; ++c) {
                        const float2 f = SWZ ? st[lbs[x] ^ msoff(c)] : st[lb[x] | moff(c)];
                        x2[x][c] = pack2(f.x, f.x);
                        y2[x][c] = pack2(f.y, f.y);
                    }
#pragma unroll
                for (int rr = 0; rr < R; ++rr) {
                    const int r = rb * R + rr;
                    const ulonglong2* mrow = reinterpret_cast<const ulonglong2*>(Ms + r * D);
                    uint64_t p[NG] = {}, qv[NG] = {};
#pragma unroll
                    for (int c = 0; c < D; c += 2) {
                        const ulonglong2 gg = mrow[c >> 1];  // G[r][c], G[r][c+1]
#pragma unroll
                        for (int x = 0; x < NG; ++x) {
                            p[x] = fma2(x2[x][c], gg.x, p[x]);
                            qv[x] = fma2(y2[x][c], gg.x, qv[x]);
                        }
#pragma unroll
                        for (int x = 0; x < NG; ++x) {
                            p[x] = fma2(x2[x][c + 1], gg.y, p[x]);
                            qv[x] = fma2(y2[x][c + 1], gg.y, qv[x]);
                        }
                    }
#pragma unroll
                    for (int x = 0; x < NG; ++x) {
                        const float2 P = unpack2(p[x]), Q = unpack2(qv[x]);
                        put(x, r, P.x - Q.y, P.y + Q.x);
                    }
                }
            } else {
                // Scalar FMAs: a packed pair reads six registers and issues every third
                // cycle when its operands change.
                float2 v[NG][D];
#pragma unroll
                for (int x = 0; x < NG; ++x)
#pragma unroll
                    for (int c = 0; c < D; ++c) v[x][c] = SWZ ? st[lbs[x] ^ msoff(c)] : st[lb[x] | moff(c)];
#pragma unroll
                for (int rr = 0; rr < R; ++rr) {
                    const int r = rb * R + rr;
                    const float4* mrow = reinterpret_cast<const float4*>(Ms + r * D);
                    // the products of the real and of the imaginary parts in sums of their own
                    float ar[NG] = {}, ai[NG] = {}, br[NG] = {}, bi[NG] = {};
#pragma unroll
                    for (int c = 0; c < D; c += 2) {
                        const float4 m2 = mrow[c >> 1];  // G[r][c], G[r][c+1]
#pragma unroll
                        for (int x = 0; x < NG; ++x) {
                            ar[x] = fmaf(m2.x, v[x][c].x, ar[x]);
                            ai[x] = fmaf(m2.x, v[x][c].y, ai[x]);
                            br[x] = fmaf(m2.y, v[x][c].y, br[x]);
                            bi[x] = fmaf(m2.y, v[x][c].x, bi[x]);
                            ar[x] = fmaf(m2.z, v[x][c + 1].x, ar[x]);
                            ai[x] = fmaf(m2.z, v[x][c + 1].y, ai[x]);
                            br[x] = fmaf(m2.w, v[x][c + 1].y, br[x]);
                            bi[x] = fmaf(m2.w, v[x][c + 1].x, bi[x]);
                        }
                    }
#pragma unroll
                    for (int x = 0; x < NG; ++x) put(x, r, ar[x] - br[x], ai[x] + bi[x]);
                }
            }
        }
        if constexpr (WB) {
            __syncthreads();
            store_tile_swz<(1 << (TB - 1)) / TH>(a.t, runoff, htab, t, st);
        }
        __syncthreads();
        if (++it_stage == S) it_stage = 0;
    }
    cp_async_wait<0>();
}

template <int K>
__device__ __forceinline__ void build_loff(const int* tl, int* loff) {
    constexpr int D = 1 << K;
    for (int c = threadIdx.x; c < D; c += blockDim.x) {
        int o = 0;
#pragma unroll
        for (int j = 0; j < K; ++j)
            if ((c >> j) & 1) o |= 1 << tl[j];
        loff[c] = o;
    }
}

template <int K, int R, int S, bool SWZ, bool WB, int TB, int NG, int TH, bool SC>
__global__ void __launch_bounds__(TH) k_apply_fp32(ApplyArgs a) {
    constexpr int D = 1 << K;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tileAmps = 1 << a.t.T;
    float2* stage = reinterpret_cast<float2*>(smem_raw);
    float2* Ms = stage + S * tileAmps;
    uint64_t* runoff = reinterpret_cast<uint64_t*>(Ms + D * D);
    int* loff = reinterpret_cast<int*>(runoff + 64);
    int* sloff = loff + 64;
    uint8_t* htab = reinterpret_cast<uint8_t*>(sloff + 64);

    const float2* gm = reinterpret_cast<const float2*>(a.mat);
    for (int i = threadIdx.x; i < D * D; i += blockDim.x) Ms[i] = gm[i];
    build_runoff(a.t, runoff);
    build_loff<K>(a.tl, loff);
    if constexpr (SWZ) {
        build_htab(a, htab);
        __syncthreads();
        for (int c = threadIdx.x; c < D; c += blockDim.x) sloff[c] = loff[c] ^ static_cast<int>(stage_xor(htab, loff[c]));
    }
    __syncthreads();
    apply_tiles<K, R, S, SWZ, WB, TB, (K <= 4), NG, TH, SC>(a, stage, Ms, runoff, loff, blockIdx.x, gridDim.x, htab, sloff);
}

template <int K>
struct ApplyCfg;
// SWZ: the swizzled stage and, where the targets call for it, in-place outputs
// with an address-order write-back are available (k <= 4).
template <> struct ApplyCfg<1> { static constexpr int NG = 1, TH = kThreads, T = 11, R = 2, S = 2; static constexpr bool SWZ = true; };
template <> struct ApplyCfg<2> { static constexpr int NG = 1, TH = kThreads, T = 11, R = 4, S = 2; static constexpr bool SWZ = true; };
template <> struct ApplyCfg<3> { static constexpr int NG = 1, TH = kThreads, T = 11, R = 8, S = 2; static constexpr bool SWZ = true; };
// k = 3: scalar FMAs beyond the L2 (N = 27: 0.349 ms, packed ones 0.367; N = 23:
// 28.3 us, packed 26.7).  k = 4: CTAs of 128
// threads with two groups per thread, which share the matrix's broadcast loads
// (N = 27: 0.406 ms; one group, 256 threads: 0.422; scalar FMAs 0.452 / 0.499 with
// one / two groups); 2^12-amplitude tiles, two stages so that three CTAs fit an SM
template <> struct ApplyCfg<4> { static constexpr int NG = 2, TH = 128, T = 12, R = 16, S = 2; static constexpr bool SWZ = true; };
// k = 5, 6: states below one tile of 2^12 amplitudes only (launch_apply_fp32)
template <> struct ApplyCfg<5> { static constexpr int NG = 1, TH = kThreads, T = 12, R = 8, S = 2; static constexpr bool SWZ = false; };
template <> struct ApplyCfg<6> { static constexpr int NG = 1, TH = kThreads, T = 12, R = 8, S = 2; static constexpr bool SWZ = false; };

// Form of a k <= 4 launch from its lowest non-target tile positions np[0..4]
// (the group-index bits that vary across a warp).  With the plain layout a
// half-warp's gathers spread over 2^(#np[0..3] below 4) of the 16 bank pairs,
// and a warp's direct 8-byte stores over 32 / 2^(#np[0..4] below 2) sectors.
// 0: plain layout, direct stores; 1: swizzled gathers, direct stores (gathers
// four or more to a bank); 2: swizzled gathers and in-place write-back (one
// sector per lane).  The thresholds follow CUDA-event timings of all three
// forms on target sets at N = 30.
int apply_form(int T, const int* tls, int k) {
    int np[5], nn = 0;
    for (int p = 0; p < T && nn < 5; ++p) {
        bool tgt = false;
        for (int j = 0; j < k; ++j) tgt = tgt || tls[j] == p;
        if (!tgt) np[nn++] = p;
    }
    int low4 = 0, low2 = 0;
    for (int b = 0; b < nn; ++b) {
        if (b < 4 && np[b] < 4) ++low4;
        if (np[b] < 2) ++low2;
    }
    if (low2 == 0) return 2;
    if (low4 <= 2) return 1;
    return 0;
}

// Slot vectors of the swizzled stage: the four lowest non-target tile
// positions take distinct slot bits where they can (positions 1..3 own theirs;
// a higher one takes a free one; position 0 is the element within a unit).
void stage_slots(int T, const int* tls, int k, uint8_t* fv) {
    for (int p = 0; p < 16; ++p) fv[p] = 0;
    int np[4], nn = 0;
    for (int p = 0; p < T && nn < 4; ++p) {
        bool tgt = false;
        for (int j = 0; j < k; ++j) tgt = tgt || tls[j] == p;
        if (!tgt) np[nn++] = p;
    }
    uint32_t used = 0;
    for (int b = 0; b < nn; ++b)
        if (np[b] >= 1 && np[b] <= 3) used |= 1u << (np[b] - 1);
    for (int b = 0; b < nn; ++b)
        if (np[b] >= 4) {
            int j = 0;
            while (j < 3 && ((used >> j) & 1u)) ++j;
            if (j < 3) {
                used |= 1u << j;
                fv[np[b]] = static_cast<uint8_t>(1u << j);
            }
        }
}

// Tile-local positions of the targets for geometry g.
void local_targets(const TileGeom& g, const int* phys, int k, int* tl, int* tls) {
    for (int j = 0; j < k; ++j) {
        int p = phys[j];
        int loc = p;
        if (p >= g.m) {
            int e = 0;
            while (g.xpos[e] != p) ++e;
            loc = g.m + e;
        }
        tl[j] = loc;
        tls[j] = loc;
    }
    std::sort(tls, tls + k);
}

template <int K>
cudaError_t launch_apply_k(float2* psi, int n, const int* phys, const float* d_mat, cudaStream_t st,
                           uint64_t* launches) {
    using C = ApplyCfg<K>;
    TileGeom g;
    if (!make_geom(n, phys, K, C::T, &g)) return cudaErrorInvalidValue;
    ApplyArgs a{};
    a.t.psi = psi;
    a.t.ntiles = g.ntiles;
    a.t.T = g.T;
    a.t.m = g.m;
    a.t.nx = g.nx;
    for (int e = 0; e < 6; ++e) a.t.xpos[e] = g.xpos[e];
    a.mat = d_mat;
    local_targets(g, phys, K, a.tl, a.tls);
    // the write-back is unrolled for full tiles (states of at least 2^T
    // amplitudes); smaller states take the plain form
    const int form = C::SWZ && g.T == C::T ? apply_form(g.T, a.tls, K) : 0;
    if (form) stage_slots(g.T, a.tls, K, a.fv);
    const int D = 1 << K;
    for (int c = 0; c < D && c < 16; ++c) {
        int o = 0;
        for (int j = 0; j < K; ++j)
            if ((c >> j) & 1) o |= 1 << a.tl[j];
        a.loffc[c] = o;
        // swizzled stage: o ^ (h(o >> 4) << 1), h the XOR of the slot vectors of o's bits from 4 on
        uint32_t h = 0;
        for (int i = 0; i < g.T - 4; ++i)
            if ((o >> (4 + i)) & 1) h ^= a.fv[4 + i];
        a.sloffc[c] = o ^ static_cast<int>(h << 1);
    }
    constexpr size_t tables = sizeof(uint64_t) * 64 + 2 * sizeof(int) * 64 + 256;
    const size_t smem = sizeof(float2) * (static_cast<size_t>(C::S) << g.T) + sizeof(float2) * D * D + tables;
    // several groups per item on full tiles only
    const bool whole = g.T == C::T;
    auto of_form = [&](auto scalar) {
        constexpr bool SC = decltype(scalar)::value;
        return form == 2   ? k_apply_fp32<K, C::R, C::S, C::SWZ, C::SWZ, C::T, C::NG, C::TH, SC>
               : form == 1 ? k_apply_fp32<K, C::R, C::S, C::SWZ, false, C::T, C::NG, C::TH, SC>
               : whole     ? k_apply_fp32<K, C::R, C::S, false, false, C::T, C::NG, C::TH, SC>
                           : k_apply_fp32<K, C::R, C::S, false, false, C::T, 1, C::TH, SC>;
    };
    auto kern = of_form(std::false_type{});
    if constexpr (K == 3) {
        if (n >= kBeyondL2) kern = of_form(std::true_type{});
    }
    {
        const size_t full = sizeof(float2) * (static_cast<size_t>(C::S) << C::T) + sizeof(float2) * D * D + tables;
        cudaError_t e = set_smem_attr(reinterpret_cast<const void*>(kern), static_cast<int>(full));
        if (e != cudaSuccess) return e;
    }
    int occ = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, C::TH, smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) occ = 1;
    // k = 1, 2 on states beyond the L2: two CTAs per SM, 32 KiB of loads in flight, which is all that the
    // memory's latency takes; more only turn its bus around more often (N = 26 / 29, k = 1: 182 / 1402 us
    // with the six that fit, 162 / 1269 with two).  In the L2 (N = 22: 10.3 and 12.3 us) and at k = 3,
    // whose arithmetic wants the warps (N = 26: 179 and 199 us), as many as fit.
    if (K <= 2 && n >= kBeyondL2 && occ > 2) occ = 2;
    uint64_t grid = static_cast<uint64_t>(num_sms()) * occ;
    if (grid > g.ntiles) grid = g.ntiles;
    kern<<<static_cast<unsigned>(grid), C::TH, smem, st>>>(a);
    ++*launches;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Apply, k = 5 and 6
// ---------------------------------------------------------------------------
// A 2^k x 2^k complex matrix on the tile's 2^(12-k) groups: bound by the FP32
// pipe (128 / 256 real FMAs per amplitude against 16 bytes), so what matters is
// how many FMAs each shared-memory load feeds.  A team of 128 threads takes a
// tile; a thread accumulates 8 rows x 4 groups, so that one column step is 128
// FMAs on 4 state loads (one amplitude of each group) and 4 matrix loads of 16
// bytes (two rows' entries).  Scalar FMAs: a packed pair reads six registers and
// issues every third cycle (84 FMAs per clock and SM with operands that change,
// 95 with one held, measured), scalar ones reach 104.  The two half-warps of a
// k = 6 team take neighbouring row pairs and read neighbouring 16-byte units.
// The teams of a CTA, one CTA per SM, share the matrix; two stages per team keep
// the next tile's copies under the arithmetic.  k = 5 adds the products of the
// real and of the imaginary parts in sums of their own (relative error of one
// operator 1.09e-7, 1.47e-7 with one running sum): 128 accumulators, so two teams
// with 255 registers a thread (N = 26: 381 us; three teams with 168 386, 428 with
// a target on position 0).  k = 6 keeps one running sum and three teams (641 us;
// two 686, four leave 128 registers and spill).  The matrix's index bits are put
// in ascending position order, so a target on position 0 (P0) is column bit 0
// and both columns of a pair come in one 16-byte load.  Outputs go back to the
// stage in place and leave in address order.
// N = 26, four target sets, k = 5 / 6: 412..596 / 902..1224 us with one row of the
// matrix read per group (the kernel above, 8 rows per thread), 381 / 623..648 us
// here, 0.56 / 0.66 of 128 FMAs per clock and SM.
constexpr int kWideT = 12, kWideTeam = 128, kWideR = 8, kWideG = 4;
template <int K>
constexpr int kWideTeams = K == 5 ? 2 : 3;
constexpr int kWideChunks = (1 << (kWideT - 1)) / kWideTeam;   // 16-byte units per thread

struct WideArgs {
    float2* psi;
    uint64_t ntiles;
    int m, nx;
    int xpos[6];
    const float* mat;
    int src[6];                    // sorted index bit i is the operator's index bit src[i]
    uint64_t poff[kWideT];         // global offset and slot of tile bit b
    uint16_t pslot[kWideT];
    uint64_t goff[kWideChunks];    // global offset and slot of tile-local 256 k
    uint16_t gslot[kWideChunks];
    uint16_t sloff[64];            // slot of column c (sorted index)
    uint16_t fslot[8];             // slot of each non-target tile bit, ascending
};

template <int K>
__host__ __device__ constexpr size_t wide_smem() {
    return sizeof(float2) * 2 * kWideTeams<K> * (1 << kWideT) + (8u << (2 * K));
}

template <int K, bool P0>
__global__ void __launch_bounds__(kWideTeam * kWideTeams<K>, 1) k_apply_wide(const __grid_constant__ WideArgs a) {
    constexpr int D = 1 << K, NRB = D / kWideR, NF = kWideT - K;
    static_assert((D / kWideR) * (1 << NF) / kWideG == kWideTeam, "a team covers the tile");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int team = threadIdx.x / kWideTeam, tid = threadIdx.x % kWideTeam;
    float2* stage = reinterpret_cast<float2*>(smem_raw) + team * 2 * (1 << kWideT);
    float2* Mt = reinterpret_cast<float2*>(smem_raw + sizeof(float2) * 2 * kWideTeams<K> * (1 << kWideT));   // [column][row]

    const float2* gm = reinterpret_cast<const float2*>(a.mat);
    for (int i = threadIdx.x; i < D * D; i += blockDim.x) {
        const int r = i & (D - 1), c = i >> K;
        int ro = 0, co = 0;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            ro |= ((r >> j) & 1) << a.src[j];
            co |= ((c >> j) & 1) << a.src[j];
        }
        Mt[i] = gm[ro * D + co];
    }
    // this thread's copies: tile-local 2 tid + 256 k
    uint64_t gld = 0;
    int sld = 0;
#pragma unroll
    for (int b = 0; b < 7; ++b)
        if ((tid >> b) & 1) {
            gld |= a.poff[b + 1];
            sld ^= a.pslot[b + 1];
        }
    // row block and groups of this thread: the lowest lane bits are groups
    constexpr int LB = NF - 2;                       // thread bits that choose groups (two more: its four groups)
    const int rb = tid >> LB;
    const int rslot = a.sloff[2 * rb];               // of its first row
    int gs[kWideG];
    gs[0] = 0;
#pragma unroll
    for (int i = 0; i < LB; ++i)
        if ((tid >> i) & 1) gs[0] ^= a.fslot[i];
    gs[1] = gs[0] ^ a.fslot[LB];
    gs[2] = gs[0] ^ a.fslot[LB + 1];
    gs[3] = gs[1] ^ a.fslot[LB + 1];
    __syncthreads();

    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * kWideTeams<K>;
    const uint64_t limit = a.ntiles << kWideT;
    auto team_sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(kWideTeam) : "memory"); };
    auto tile_at = [&](uint64_t t) {
        uint64_t base = t << a.m;
#pragma unroll
        for (int e = 0; e < 6; ++e)
            if (e < a.nx) base = insert_zero(base, a.xpos[e]);
        return base | gld;
    };
    auto load = [&](uint64_t base, float2* to) {
#pragma unroll
        for (int k = 0; k < kWideChunks; ++k)
            if (dbg::in_bounds(base | a.goff[k], 2, limit, 7)) cp_async16(to + (sld ^ a.gslot[k]), a.psi + (base | a.goff[k]));
    };
    const uint64_t t0 = blockIdx.x + static_cast<uint64_t>(gridDim.x) * team;
    uint64_t next = tile_at(t0);
    if (t0 < a.ntiles) load(next, stage);
    cp_async_commit();
    int cur = 0;
    for (uint64_t t = t0; t < a.ntiles; t += stride) {
        const uint64_t base = next;
        float2* st = stage + cur * (1 << kWideT);
        cur ^= 1;
        cp_async_wait<0>();
        team_sync();   // the tile has landed, and the team has written the other stage's tile out
        next = tile_at(t + stride);
        if (t + stride < a.ntiles) load(next, stage + cur * (1 << kWideT));
        cp_async_commit();
        // k = 5: the products of the real and of the imaginary parts in sums of their own
        constexpr bool TWO = K == 5;
        float2 acc[kWideR][kWideG], acc2[kWideR][kWideG];
#pragma unroll
        for (int r = 0; r < kWideR; ++r)
#pragma unroll
            for (int g = 0; g < kWideG; ++g) acc[r][g] = acc2[r][g] = make_float2(0.f, 0.f);
        auto column = [&](const float4* m, const float2 (&v)[kWideG]) {
            auto row = [&](int r, float re, float im) {
                float2 (&b)[kWideG] = TWO ? acc2[r] : acc[r];
#pragma unroll
                for (int g = 0; g < kWideG; ++g) {
                    acc[r][g].x = fmaf(re, v[g].x, acc[r][g].x);
                    acc[r][g].y = fmaf(re, v[g].y, acc[r][g].y);
                    b[g].x = fmaf(-im, v[g].y, b[g].x);
                    b[g].y = fmaf(im, v[g].x, b[g].y);
                }
            };
#pragma unroll
            for (int r = 0; r < kWideR; r += 2) {
                const float4 e = m[NRB * (r >> 1)];   // rows 2 (rb + NRB r / 2) and the next
                row(r, e.x, e.y);
                row(r + 1, e.z, e.w);
            }
        };
        // eight columns at a time: their low bits' slots enter from the parameter bank
        constexpr int kWC = 8;
#pragma unroll 1
        for (int o = 0; o < D; o += kWC) {
            const int hi = a.sloff[o];
            const float4* m = reinterpret_cast<const float4*>(Mt + o * D) + rb;
#pragma unroll
            for (int c = 0; c < kWC; c += 2) {
                float2 v0[kWideG], v1[kWideG];
#pragma unroll
                for (int g = 0; g < kWideG; ++g) {
                    if constexpr (P0) {
                        const float4 f = *reinterpret_cast<const float4*>(st + (gs[g] ^ hi ^ a.sloff[c]));
                        v0[g] = make_float2(f.x, f.y);
                        v1[g] = make_float2(f.z, f.w);
                    } else {
                        v0[g] = st[gs[g] ^ hi ^ a.sloff[c]];
                        v1[g] = st[gs[g] ^ hi ^ a.sloff[c + 1]];
                    }
                }
                column(m + c * (D / 2), v0);
                column(m + (c + 1) * (D / 2), v1);
            }
        }
        team_sync();   // every input of the tile has been read
#pragma unroll
        for (int r = 0; r < kWideR; ++r) {
            const int so = rslot ^ a.sloff[2 * NRB * (r >> 1) + (r & 1)];
#pragma unroll
            for (int g = 0; g < kWideG; ++g)
                st[gs[g] ^ so] = TWO ? make_float2(acc[r][g].x + acc2[r][g].x, acc[r][g].y + acc2[r][g].y) : acc[r][g];
        }
        team_sync();
#pragma unroll
        for (int k = 0; k < kWideChunks; ++k)
            if (dbg::in_bounds(base | a.goff[k], 2, limit, 8))
                __stcs(reinterpret_cast<float4*>(a.psi + (base | a.goff[k])),
                       *reinterpret_cast<const float4*>(st + (sld ^ a.gslot[k])));
    }
    cp_async_wait<0>();
}

template <int K>
cudaError_t launch_apply_wide(float2* psi, int n, const int* phys, const float* d_mat, cudaStream_t st,
                              uint64_t* launches) {
    TileGeom g;
    if (!make_geom(n, phys, K, kWideT, &g) || g.T != kWideT) return cudaErrorInvalidValue;
    WideArgs a{};
    a.psi = psi;
    a.ntiles = g.ntiles;
    a.m = g.m;
    a.nx = g.nx;
    for (int e = 0; e < 6; ++e) a.xpos[e] = g.xpos[e];
    a.mat = d_mat;
    int tl[6], tls[6];
    uint8_t fv[16];
    local_targets(g, phys, K, tl, tls);
    for (int i = 0; i < K; ++i) a.src[i] = static_cast<int>(std::find(tl, tl + K, tls[i]) - tl);
    stage_slots(g.T, tls, K, fv);
    int nf = 0;
    for (int b = 0; b < kWideT; ++b) {
        a.poff[b] = 1ull << (b < g.m ? b : g.xpos[b - g.m]);
        a.pslot[b] = static_cast<uint16_t>((1 << b) ^ (b >= 4 ? fv[b] << 1 : 0));
        if (std::find(tls, tls + K, b) == tls + K) a.fslot[nf++] = a.pslot[b];
    }
    for (int k = 0; k < kWideChunks; ++k)
        for (int b = 0; b < 4; ++b)
            if ((k >> b) & 1) {
                a.goff[k] |= a.poff[8 + b];
                a.gslot[k] = static_cast<uint16_t>(a.gslot[k] ^ a.pslot[8 + b]);
            }
    for (int c = 0; c < (1 << K); ++c)
        for (int j = 0; j < K; ++j)
            if ((c >> j) & 1) a.sloff[c] = static_cast<uint16_t>(a.sloff[c] ^ a.pslot[tls[j]]);
    auto kern = tls[0] == 0 ? k_apply_wide<K, true> : k_apply_wide<K, false>;
    cudaError_t e = set_smem_attr(reinterpret_cast<const void*>(kern), static_cast<int>(wide_smem<K>()));
    if (e != cudaSuccess) return e;
    const uint64_t grid = std::min<uint64_t>(g.ntiles, static_cast<uint64_t>(num_sms()));
    kern<<<static_cast<unsigned>(grid), kWideTeam * kWideTeams<K>, wide_smem<K>(), st>>>(a);
    ++*launches;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Product of one-qubit factors (a structured fused block, §IV-D)
// ---------------------------------------------------------------------------
constexpr int kProdT = 11, kProdS = 3, kProdHigh = 3;

struct ProdArgs {
    TileArgs t;
    const float* fac;          // 8 floats per factor: 2x2 complex, row-major
    int k;
    int tl[QSA_MAX_PROD];      // tile-local position of factor j
};

// a x + b y for complex a, b, x, y.
__device__ __forceinline__ float2 cfma2(float2 a, float2 x, float2 b, float2 y) {
    return make_float2(a.x * x.x - a.y * x.y + b.x * y.x - b.y * y.y, a.x * x.y + a.y * x.x + b.x * y.y + b.y * y.x);
}

// One round over the staged tile.  A warp covers 32 x 2^H amplitudes: its
// lanes are tile-local bits 0..4 (so every shared-memory access of the warp
// touches 32 consecutive amplitudes), and each lane holds the 2^H
// combinations of the round's H high targets (positions >= 5, ascending
// hpos[]).  High factors are butterflies in registers, low factors (targets
// below 5) butterflies across lanes with shuffles.  The last round stores
// straight to HBM (32 consecutive amplitudes per warp store).
template <int H>
__device__ __forceinline__ void prod_round(const ProdArgs& a, float2* st, const float2* F, const int* hpos,
                                           const int* hfi, int nlow, const int* lpos, const int* lfi, bool last,
                                           const uint64_t* runoff, uint64_t base) {
    constexpr int G = 1 << H;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int units = (1 << a.t.T) >> (5 + H);
    // per round: each high target's tile-local bit and the global offset of
    // that bit (tile indexing is bitwise linear, so offsets add)
    uint32_t hm[H > 0 ? H : 1];
    uint64_t gb[H > 0 ? H : 1];
#pragma unroll
    for (int j = 0; j < H; ++j) {
        hm[j] = 1u << hpos[j];
        gb[j] = tile_global(a.t, runoff, 0, hm[j]);
    }
    for (int u = warp; u < units; u += nw) {
        uint32_t ub = static_cast<uint32_t>(u) << 5;
#pragma unroll
        for (int j = 0; j < H; ++j) ub = static_cast<uint32_t>(insert_zero(ub, hpos[j]));
        ub |= static_cast<uint32_t>(lane);
        float2 v[G];
#pragma unroll
        for (int c = 0; c < G; ++c) {
            uint32_t o = ub;
#pragma unroll
            for (int j = 0; j < H; ++j)
                if ((c >> j) & 1) o |= hm[j];
            v[c] = st[o];
        }
#pragma unroll
        for (int j = 0; j < H; ++j) {
            const float2* U = F + 4 * hfi[j];
#pragma unroll
            for (int c = 0; c < G; ++c) {
                if ((c >> j) & 1) continue;
                const float2 x = v[c], y = v[c | (1 << j)];
                v[c] = cfma2(U[0], x, U[1], y);
                v[c | (1 << j)] = cfma2(U[3], y, U[2], x);
            }
        }
        for (int l = 0; l < nlow; ++l) {
            const int m = 1 << lpos[l];
            const float2* U = F + 4 * lfi[l];
            // bit clear: u00 x + u01 y; bit set: u11 x + u10 y (x own, y partner)
            const bool one = (lane & m) != 0;
            const float2 ua = one ? U[3] : U[0], ub2 = one ? U[2] : U[1];
#pragma unroll
            for (int c = 0; c < G; ++c) {
                float2 y;
                y.x = __shfl_xor_sync(0xffffffffu, v[c].x, m);
                y.y = __shfl_xor_sync(0xffffffffu, v[c].y, m);
                v[c] = cfma2(ua, v[c], ub2, y);
            }
        }
        if (last) {
            const uint64_t g0 = tile_global(a.t, runoff, base, ub);
#pragma unroll
            for (int c = 0; c < G; ++c) {
                uint64_t go = 0;
#pragma unroll
                for (int j = 0; j < H; ++j)
                    if ((c >> j) & 1) go += gb[j];
                if (dbg::in_bounds(g0 + go, 1, a.t.ntiles << a.t.T, 5)) __stcs(a.t.psi + g0 + go, v[c]);
            }
        } else {
#pragma unroll
            for (int c = 0; c < G; ++c) {
                uint32_t o = ub;
#pragma unroll
                for (int j = 0; j < H; ++j)
                    if ((c >> j) & 1) o |= hm[j];
                st[o] = v[c];
            }
        }
    }
}

__global__ void __launch_bounds__(kThreads) k_apply_prod(ProdArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tileAmps = 1 << a.t.T;
    float2* stage = reinterpret_cast<float2*>(smem_raw);
    float2* F = stage + kProdS * tileAmps;
    uint64_t* runoff = reinterpret_cast<uint64_t*>(F + 4 * QSA_MAX_PROD);
    const float2* gf = reinterpret_cast<const float2*>(a.fac);
    for (int i = threadIdx.x; i < 4 * a.k; i += blockDim.x) F[i] = gf[i];
    build_runoff(a.t, runoff);
    // factors on tile-local bits 0..4 act across lanes (all in round 0); the
    // others, ascending by position, go kProdHigh per round
    int hpos[QSA_MAX_PROD], hfi[QSA_MAX_PROD], lpos[5], lfi[5];
    int nh = 0, nl = 0;
    for (int j = 0; j < a.k; ++j) {
        if (a.tl[j] < 5) {
            lpos[nl] = a.tl[j];
            lfi[nl++] = j;
        } else {
            int x = nh++;
            while (x > 0 && hpos[x - 1] > a.tl[j]) {
                hpos[x] = hpos[x - 1];
                hfi[x] = hfi[x - 1];
                --x;
            }
            hpos[x] = a.tl[j];
            hfi[x] = j;
        }
    }
    const int rounds = nh > 0 ? (nh + kProdHigh - 1) / kProdHigh : 1;
    __syncthreads();

    const uint64_t t0 = blockIdx.x, stride = gridDim.x;
#pragma unroll
    for (int s = 0; s < kProdS - 1; ++s) {
        const uint64_t t = t0 + s * stride;
        if (t < a.t.ntiles) load_tile(a.t, runoff, t, stage + s * tileAmps);
        cp_async_commit();
    }
    int it_stage = 0;
    for (uint64_t t = t0; t < a.t.ntiles; t += stride) {
        const uint64_t tn = t + (kProdS - 1) * stride;
        int ld_stage = it_stage + (kProdS - 1);
        if (ld_stage >= kProdS) ld_stage -= kProdS;
        if (tn < a.t.ntiles) load_tile(a.t, runoff, tn, stage + ld_stage * tileAmps);
        cp_async_commit();
        cp_async_wait<kProdS - 1>();
        __syncthreads();
        float2* st = stage + it_stage * tileAmps;
        const uint64_t base = tile_base(a.t, t);
        for (int r = 0; r < rounds; ++r) {
            const int h0 = r * kProdHigh, hb = min(kProdHigh, nh - h0);
            const int nlr = r == 0 ? nl : 0;
            const bool last = r == rounds - 1;
            if (hb >= 3)
                prod_round<3>(a, st, F, hpos + h0, hfi + h0, nlr, lpos, lfi, last, runoff, base);
            else if (hb == 2)
                prod_round<2>(a, st, F, hpos + h0, hfi + h0, nlr, lpos, lfi, last, runoff, base);
            else if (hb == 1)
                prod_round<1>(a, st, F, hpos + h0, hfi + h0, nlr, lpos, lfi, last, runoff, base);
            else
                prod_round<0>(a, st, F, hpos + h0, hfi + h0, nlr, lpos, lfi, last, runoff, base);
            __syncthreads();
        }
        if (++it_stage == kProdS) it_stage = 0;
    }
    cp_async_wait<0>();
}

// ---------------------------------------------------------------------------
// Permute
// ---------------------------------------------------------------------------
// A permutation of the tile's bits, in place: the tile (2^T amplitudes, 16-byte
// copies) is in shared memory before any of it is written.  Bound by HBM; what
// counts is the number of passes a permutation of the state's positions takes,
// so tiles are wide (up to 2^13 amplitudes, runs of at least 64 bytes): ten
// positions above the lowest three can move in one pass (plan_permutation).  One
// stage per CTA; the CTAs of an SM, 128 KiB of stages, hide each other's latency
// (192 KiB was slower: 40 registers a thread, with spills).  Up to nine such
// positions: tiles of 2^12 and CTAs of 256 threads, whose shorter steps leave
// less of the last wave empty.  Beyond the L2 a CTA per tile: the loads of one
// start while the stores of another drain, which CTAs that walk tiles in step do
// not reach; in the L2 starting CTAs costs more than that.
// One pair at N = 22 / 23 / 24 / 28: 10.3 / 15.2 / 43.2 / 607 us here; in 2^13 tiles
// with three walking CTAs per SM 12.4 / 18.7 / 48.0 / 684; in 2^11 tiles with three
// stages and up to six positions (before) 10.3 / 17.6 / 46.1 / 708.  Two random
// layouts and five bit swaps at N = 28: 22 passes of that kind, 14.5 ms; 7 passes
// here, 4.4 ms.
constexpr int kPermT = 13, kPermLow = 3;

struct PermArgs {
    float2* psi;
    uint64_t ntiles;
    int T, m, nx;
    int xpos[kPermT];
    uint64_t poff[kPermT];    // global offset and slot of tile bit b
    uint16_t pslot[kPermT];
    uint16_t sslot[kPermT];   // slot of the tile bit whose content tile bit b receives
};

// LT: thread bits, CTAS: CTAs of an SM
template <int LT, int CTAS>
__global__ void __launch_bounds__(1 << LT, CTAS) k_permute(const __grid_constant__ PermArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* st = reinterpret_cast<float2*>(smem_raw);
    const int tid = threadIdx.x;
    uint64_t g0 = 0;
    uint32_t sl = 0, ss = 0;
#pragma unroll
    for (int b = 0; b < LT; ++b)
        if ((tid >> b) & 1) {
            g0 |= a.poff[b + 1];
            sl ^= a.pslot[b + 1];
            ss ^= a.sslot[b + 1];
        }
    const uint32_t chunks = 1u << (a.T - 1);
    const int nk = chunks > (1u << LT) ? static_cast<int>(chunks >> LT) : 1;
    const bool copies = static_cast<uint32_t>(tid) < chunks;
    const uint64_t limit = a.ntiles << a.T;
    const uint32_t s0 = a.sslot[0];
    for (uint64_t t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        uint64_t base = t << a.m;
#pragma unroll
        for (int e = 0; e < kPermT - kPermLow; ++e)
            if (e < a.nx) base = insert_zero(base, a.xpos[e]);
        base |= g0;
        uint64_t g[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            g[k] = base | (k & 1 ? a.poff[LT + 1] : 0ull) | (k & 2 ? a.poff[LT + 2] : 0ull) | (k & 4 ? a.poff[LT + 3] : 0ull);
            const uint32_t s = sl ^ (k & 1 ? a.pslot[LT + 1] : 0u) ^ (k & 2 ? a.pslot[LT + 2] : 0u) ^
                               (k & 4 ? a.pslot[LT + 3] : 0u);
            if (k < nk && copies && dbg::in_bounds(g[k], 2, limit, 6)) cp_async16(st + s, a.psi + g[k]);
        }
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t s = ss ^ (k & 1 ? a.sslot[LT + 1] : 0u) ^ (k & 2 ? a.sslot[LT + 2] : 0u) ^
                               (k & 4 ? a.sslot[LT + 3] : 0u);
            if (k < nk && copies && dbg::in_bounds(g[k], 2, limit, 6)) {
                const float2 v0 = st[s], v1 = st[s ^ s0];
                __stcs(reinterpret_cast<float4*>(a.psi + g[k]), make_float4(v0.x, v0.y, v1.x, v1.y));
            }
        }
        __syncthreads();
    }
}

__global__ void k_set_one(float2* psi) { psi[0] = make_float2(1.f, 0.f); }

}  // namespace

QSA_BOUNDS_READER(bounds_word_apply)

int num_sms() {
    static std::mutex mu;
    static std::map<int, int> cached;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    auto it = cached.find(dev);
    if (it != cached.end()) return it->second;
    int v = 0;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    if (v <= 0) v = 1;
    cached[dev] = v;
    return v;
}

cudaError_t set_smem_attr(const void* kernel, int bytes) {
    static std::mutex mu;
    static std::map<std::pair<int, const void*>, int> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_pair(dev, kernel);
    auto it = done.find(key);
    if (it != done.end() && it->second >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    done[key] = bytes;
    return cudaSuccess;
}

bool make_geom(int n, const int* special, int ns, int T_want, TileGeom* g) {
    g->n = n;
    g->T = std::min(T_want, n);
    int m = g->T;
    for (;;) {
        int cnt = 0;
        for (int i = 0; i < ns; ++i)
            if (special[i] >= m) ++cnt;
        if (m + cnt <= g->T) break;
        --m;
    }
    if (m < 1) return false;
    g->m = m;
    int nx = 0;
    int tmp[16];
    for (int i = 0; i < ns; ++i)
        if (special[i] >= m) {
            if (nx >= 6) return false;
            tmp[nx++] = special[i];
        }
    std::sort(tmp, tmp + nx);
    g->nx = nx;
    for (int e = 0; e < 6; ++e) g->xpos[e] = e < nx ? tmp[e] : 0;
    g->ntiles = 1ull << (n - g->T);
    return true;
}

__global__ void k_fill_one(float4* psi2, uint64_t npairs) {
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < npairs;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x)
        psi2[i] = make_float4(1.f, 0.f, 1.f, 0.f);
}

cudaError_t launch_fill_one(float2* psi, int n, cudaStream_t st, uint64_t* launches) {
    if (n < 1) return cudaErrorInvalidValue;
    const uint64_t npairs = (1ull << n) >> 1;
    uint64_t blocks = (npairs + 255) / 256;
    const uint64_t cap = static_cast<uint64_t>(num_sms()) * 16;
    if (blocks > cap) blocks = cap;
    k_fill_one<<<static_cast<unsigned>(blocks), 256, 0, st>>>(reinterpret_cast<float4*>(psi), npairs);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_init_zero(float2* psi, int n, cudaStream_t st, uint64_t* launches) {
    cudaError_t e = cudaMemsetAsync(psi, 0, sizeof(float2) << n, st);
    if (e != cudaSuccess) return e;
    k_set_one<<<1, 1, 0, st>>>(psi);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_apply_fp32(float2* psi, int n, const int* phys, int k, const float* d_mat, cudaStream_t st,
                              uint64_t* launches) {
    switch (k) {
        case 1: return launch_apply_k<1>(psi, n, phys, d_mat, st, launches);
        case 2: return launch_apply_k<2>(psi, n, phys, d_mat, st, launches);
        case 3: return launch_apply_k<3>(psi, n, phys, d_mat, st, launches);
        case 4: return launch_apply_k<4>(psi, n, phys, d_mat, st, launches);
        // states below one tile keep the kernel that takes any tile size
        case 5:
            return n >= kWideT ? launch_apply_wide<5>(psi, n, phys, d_mat, st, launches)
                               : launch_apply_k<5>(psi, n, phys, d_mat, st, launches);
        case 6:
            return n >= kWideT ? launch_apply_wide<6>(psi, n, phys, d_mat, st, launches)
                               : launch_apply_k<6>(psi, n, phys, d_mat, st, launches);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_apply_prod(float2* psi, int n, const int* phys, int k, const float* d_fac, cudaStream_t st,
                              uint64_t* launches) {
    if (n < 5) {
        // the product round maps warp lanes to 5 tile bits: tiny states apply
        // each factor as its own one-qubit update
        for (int j = 0; j < k; ++j) {
            cudaError_t e = launch_apply_k<1>(psi, n, phys + j, d_fac + 8 * j, st, launches);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    // a tile holds at most 6 high target bits: larger sets go in several passes
    int j0 = 0;
    while (j0 < k) {
        int j1 = k;
        TileGeom g;
        while (!make_geom(n, phys + j0, j1 - j0, kProdT, &g)) {
            if (j1 - j0 == 1) return cudaErrorInvalidValue;
            --j1;
        }
        ProdArgs a{};
        a.t.psi = psi;
        a.t.ntiles = g.ntiles;
        a.t.T = g.T;
        a.t.m = g.m;
        a.t.nx = g.nx;
        for (int e = 0; e < 6; ++e) a.t.xpos[e] = g.xpos[e];
        a.fac = d_fac + 8 * j0;
        a.k = j1 - j0;
        int tls[QSA_MAX_PROD];
        local_targets(g, phys + j0, a.k, a.tl, tls);
        const size_t smem = sizeof(float2) * (static_cast<size_t>(kProdS) << g.T) + sizeof(float2) * 4 * QSA_MAX_PROD +
                            sizeof(uint64_t) * 64;
        {
            const size_t full = sizeof(float2) * (static_cast<size_t>(kProdS) << kProdT) +
                                sizeof(float2) * 4 * QSA_MAX_PROD + sizeof(uint64_t) * 64;
            cudaError_t e = set_smem_attr(reinterpret_cast<const void*>(k_apply_prod), static_cast<int>(full));
            if (e != cudaSuccess) return e;
        }
        int occ = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_apply_prod, kThreads, smem);
        if (e != cudaSuccess) return e;
        if (occ < 1) occ = 1;
        uint64_t grid = static_cast<uint64_t>(num_sms()) * occ;
        if (grid > g.ntiles) grid = g.ntiles;
        k_apply_prod<<<static_cast<unsigned>(grid), kThreads, smem, st>>>(a);
        ++*launches;
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        j0 = j1;
    }
    return cudaSuccess;
}

std::vector<std::vector<int>> plan_permutation(int n, const int* dest, int T) {
    const int cap = T - kPermLow;   // positions at kPermLow or above in one pass
    std::vector<int> to(dest, dest + n);
    std::vector<std::vector<int>> passes;
    auto high = [](int p) { return p >= kPermLow ? 1 : 0; };
    for (;;) {
        // the cycles left, longest (in high positions) first
        std::vector<std::vector<int>> cyc;
        std::vector<char> seen(n, 0);
        for (int p = 0; p < n; ++p) {
            if (seen[p] || to[p] == p) continue;
            std::vector<int> c;
            for (int x = p; !seen[x]; x = to[x]) {
                seen[x] = 1;
                c.push_back(x);
            }
            cyc.push_back(c);
        }
        if (cyc.empty()) return passes;
        auto highs = [&](const std::vector<int>& c) {
            int h = 0;
            for (int p : c) h += high(p);
            return h;
        };
        std::stable_sort(cyc.begin(), cyc.end(),
                         [&](const std::vector<int>& x, const std::vector<int>& y) { return highs(x) > highs(y); });
        std::vector<int> pass(n);
        for (int p = 0; p < n; ++p) pass[p] = p;
        // contents of c[0..k) move one place along; the last one's goes back to c[0], from where it still has
        // to reach its destination
        int room = cap;
        auto move = [&](const std::vector<int>& c, size_t k) {
            for (size_t i = 0; i < k; ++i) {
                pass[c[i]] = c[(i + 1) % k];
                room -= high(c[i]);
            }
            const int last = to[c[k - 1]];
            for (size_t i = 0; i + 1 < k; ++i) to[c[i + 1]] = c[i + 1];
            to[c[0]] = k == c.size() ? c[0] : last;
        };
        std::vector<char> done(cyc.size(), 0);
        for (size_t i = 0; i < cyc.size(); ++i)   // whole cycles that fit
            if (highs(cyc[i]) <= room) {
                move(cyc[i], cyc[i].size());
                done[i] = 1;
            }
        for (size_t i = 0; i < cyc.size(); ++i) {   // then the first positions of others, from a low one if there is one
            if (done[i]) continue;
            std::vector<int> c = cyc[i];
            for (size_t r = 0; r < c.size(); ++r)
                if (!high(c[r])) {
                    std::rotate(c.begin(), c.begin() + static_cast<long>(r), c.end());
                    break;
                }
            size_t k = 0;
            for (int h = 0; k < c.size() && h + high(c[k]) <= room; ++k) h += high(c[k]);
            if (k >= 2) move(c, k);
        }
        passes.push_back(pass);
    }
}

namespace {

// One pass: the content of position p moves to dest[p], at most kPermT - kPermLow
// positions at kPermLow or above move.
cudaError_t permute_pass(float2* psi, int n, const int* dest, cudaStream_t st) {
    uint64_t moved = 0;
    for (int p = 0; p < n; ++p)
        if (dest[p] != p) moved |= 1ull << p;
    const bool wide = __builtin_popcountll(moved >> kPermLow) > kPermT - 1 - kPermLow;
    const int T = std::min(wide ? kPermT : kPermT - 1, n);
    PermArgs a{};
    a.psi = psi;
    a.T = T;
    a.ntiles = 1ull << (n - T);
    int m = T;
    while (m + __builtin_popcountll(moved >> m) > T) --m;
    if (m < 1) return cudaErrorInvalidValue;
    a.m = m;
    for (int p = m; p < n; ++p)
        if ((moved >> p) & 1) a.xpos[a.nx++] = p;
    auto position = [&](int b) { return b < m ? b : a.xpos[b - m]; };
    int bit_of[QSA_MAX_QUBITS] = {}, from[kPermT] = {};
    for (int b = 0; b < T; ++b) bit_of[position(b)] = b;
    for (int b = 0; b < T; ++b) from[bit_of[dest[position(b)]]] = b;
    // The reading lanes vary the destination's bits 1..4: their source bits at 4 or above take slot
    // bits 1..3 that no other of them has.
    uint32_t used = 0, vec[kPermT] = {};
    for (int b = 1; b <= 4 && b < T; ++b)
        if (from[b] >= 1 && from[b] <= 3) used |= 1u << from[b];
    for (int b = 1; b <= 4 && b < T; ++b)
        if (from[b] >= 4)
            for (int j = 1; j <= 3; ++j)
                if (!((used >> j) & 1)) {
                    used |= 1u << j;
                    vec[from[b]] = 1u << j;
                    break;
                }
    for (int b = 0; b < T; ++b) {
        a.poff[b] = 1ull << position(b);
        a.pslot[b] = static_cast<uint16_t>((1u << b) ^ vec[b]);
    }
    for (int b = 0; b < T; ++b) a.sslot[b] = a.pslot[from[b]];
    const size_t smem = sizeof(float2) << T;
    auto kern = wide ? k_permute<9, 2> : k_permute<8, 4>;
    if (wide) {
        cudaError_t e = set_smem_attr(reinterpret_cast<const void*>(kern), static_cast<int>(smem));
        if (e != cudaSuccess) return e;
    }
    const uint64_t grid = n >= kBeyondL2 ? a.ntiles : std::min<uint64_t>(a.ntiles, num_sms() * (wide ? 2ull : 4ull));
    kern<<<static_cast<unsigned>(grid), wide ? 512 : 256, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_permute(float2* psi, int n, const int* dest, cudaStream_t st, uint64_t* launches) {
    auto run = [&](const int* pass) {
        ++*launches;
        return permute_pass(psi, n, pass, st);
    };
    int moved = 0, high = 0;
    for (int p = 0; p < n; ++p)
        if (dest[p] != p) {
            ++moved;
            high += p >= kPermLow ? 1 : 0;
        }
    if (moved == 0) return cudaSuccess;
    if (high <= kPermT - kPermLow) return run(dest);   // what plan_permutation would find
    for (const std::vector<int>& pass : plan_permutation(n, dest, kPermT)) {
        cudaError_t e = run(pass.data());
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace qsa
