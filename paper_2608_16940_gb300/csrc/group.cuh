// Group passes: a run of fused blocks (dense k <= 4, diagonal k <= 8) applied in
// one pass over the state.
//
// A tile is 2^T amplitudes (T = min(12, N)): the m lowest positions and nx
// higher ones; every dense block of the pass has its targets inside the tile,
// diagonal blocks may sit anywhere (their bits outside the tile are constant
// per tile).  The tile stays in shared memory while the pass's blocks run in
// rounds: a round names four tile bits, each thread takes the 16 amplitudes
// that differ in them into registers and applies every block of the round
// there, so blocks on the same four bits cost no shared-memory traffic between
// them.
//
// What bounds a pass: instruction issue and the FP32 pipe, no longer HBM (a
// pass of its own over HBM is about 2800 SM cycles per tile at the copy rate).
// So unitary one-qubit blocks run as real rotations in two in-place shears, one
// FMA per amplitude (64 SM cycles per tile where the complex 2 x 2 took 256), and
// their phases share tables with the diagonal blocks around them
// (group_host.cpp); what a thread needs to find its places and entries comes
// from small tables in the program instead of bit arithmetic.
// Measured, one pass per block / group passes with complex 2 x 2 blocks / with
// rotations: QFT + 3 random layers at N = 25, DP plan of k <= 4 blocks, 24.5 /
// 4.58 / 3.36 ms; the 12-qubit brick circuit of 20 layers from |0...0> (one
// tile: one launch instead of about 250) with its probabilities and norm, 1.77
// / 0.159 / 0.100 ms; 128 trajectories at N = 20 of 10..40 layers with their
// samples, 295 / 45.9 / 22.8 ms.
// Dense 2- and 3-qubit blocks with scalar FMAs (3.63 ms at N = 25 against 3.30) and an
// operator's head read ahead of it (3.53) were slower: what counts is the
// number of instructions and registers.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "qsa_bounds.cuh"
#include "qsa_device.cuh"
#include "qsa_internal.h"

namespace qsa {
namespace group {

using namespace dev;

constexpr int kThreads = 256;
constexpr int kAmps = 1 << kGroupTileBits;

// Slot of tile-local amplitude j in the stage: position 0 stays the element of
// a 16-byte unit; the unit's place within its 128-byte line (slot bits 1..3) is
// XORed with a vector per higher tile bit.  The eleven vectors of bits 1..11
// (1, 2, 4 | 3, 5, 6, 7, 1, 2, 4, 7) leave at most five of them in any plane,
// so whichever four bits a round holds in registers, the others contain lane
// bits whose vectors are independent: the round's accesses are free of bank
// conflicts (group_build orders the thread bits accordingly).
__host__ __device__ constexpr int slot_vec(int bit) {
    return bit == 1 ? 1 : bit == 2 ? 2 : bit == 3 ? 4 : bit == 4 ? 3 : bit == 5 ? 5 : bit == 6 ? 6 : bit == 7 ? 7
         : bit == 8 ? 1 : bit == 9 ? 2 : bit == 10 ? 4 : bit == 11 ? 7 : 0;
}
__host__ __device__ constexpr int slot_of(int j) {
    int h = 0;
    for (int b = 4; b < kGroupTileBits; ++b)
        if ((j >> b) & 1) h ^= slot_vec(b);
    return j ^ (h << 1);
}

// Shared-memory tables of a pass, after its stages and its program.
struct Tables {
    uint64_t goff[8];        // global offsets of the copy loop's strides (tile-local 512 k)
    uint64_t runoff[512];    // global offset of the tile's bits m..T-1
};

__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// i v
__device__ __forceinline__ uint64_t rot90(uint64_t v) {
    const float2 f = unpack2(v);
    return pack2(-f.y, f.x);
}
// acc + g v with g = ((Re, Re), (Im, Im)), iv = i v
__device__ __forceinline__ uint64_t cfma(const ulonglong2& g, uint64_t v, uint64_t iv, uint64_t acc) {
    return fma2(g.y, iv, fma2(g.x, v, acc));
}

// p + i q
__device__ __forceinline__ uint64_t join(uint64_t p, uint64_t q) {
    const float2 P = unpack2(p), Q = unpack2(q);
    return pack2(P.x - Q.y, P.y + Q.x);
}

// The dense blocks on register bits B.. (ascending, as the matrix's index
// bits).  An amplitude is one packed pair (Re, Im); a matrix entry is stored
// as (Re, Re, Im, Im), so one complex multiply-add is two packed FMAs and the
// broadcast load of an entry is one 16-byte load.  One-qubit blocks run on (v, i v)
// in one sum of four products; wider ones sum the products with the real and
// with the imaginary parts apart (p += Re v, q += Im v), as the kernels of single
// blocks do: one sum of all had 1.10 / 1.21 times their error at k = 2 / 3, two
// cost an addition per output (QFT and random layers at N = 25 3.29 -> 3.36 ms,
// 128 trajectories at N = 20 22.5 -> 22.8 ms).  With two products a sum a
// one-qubit block's error is the same either way.
template <int B>
__device__ __forceinline__ void dense1(uint64_t (&v)[16], const ulonglong2* __restrict__ g) {
    const ulonglong2 g00 = g[0], g01 = g[1], g10 = g[2], g11 = g[3];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        if ((i >> B) & 1) continue;
        const uint64_t a = v[i], b = v[i | (1 << B)], ia = rot90(a), ib = rot90(b);
        v[i] = cfma(g01, b, ib, fma2(g00.y, ia, mul2(g00.x, a)));
        v[i | (1 << B)] = cfma(g11, b, ib, fma2(g10.y, ia, mul2(g10.x, a)));
    }
}

// Register index of local index c of the group with the free bits of f
template <int K, int B0, int B1, int B2>
__device__ constexpr int reg_of(int f, int c) {
    int r = 0, fi = 0, ci = 0;
    for (int b = 0; b < 4; ++b) {
        const bool t = b == B0 || b == B1 || (K == 3 && b == B2);
        if (t)
            r |= ((c >> ci++) & 1) << b;
        else
            r |= ((f >> fi++) & 1) << b;
    }
    return r;
}

template <int B0, int B1>
__device__ __forceinline__ void dense2(uint64_t (&v)[16], const ulonglong2* __restrict__ g) {
#pragma unroll
    for (int f0 = 0; f0 < 4; f0 += 2) {   // two groups at a time share the entries' loads
        uint64_t x[2][4];
#pragma unroll
        for (int f = 0; f < 2; ++f)
#pragma unroll
            for (int c = 0; c < 4; ++c) x[f][c] = v[reg_of<2, B0, B1, 0>(f0 + f, c)];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const ulonglong2 e0 = g[4 * r], e1 = g[4 * r + 1], e2 = g[4 * r + 2], e3 = g[4 * r + 3];
#pragma unroll
            for (int f = 0; f < 2; ++f)
                v[reg_of<2, B0, B1, 0>(f0 + f, r)] =
                    join(fma2(e3.x, x[f][3], fma2(e2.x, x[f][2], fma2(e1.x, x[f][1], mul2(e0.x, x[f][0])))),
                         fma2(e3.y, x[f][3], fma2(e2.y, x[f][2], fma2(e1.y, x[f][1], mul2(e0.y, x[f][0])))));
        }
    }
}

template <int B0, int B1, int B2>
__device__ __forceinline__ void dense3(uint64_t (&v)[16], const ulonglong2* __restrict__ g) {
    uint64_t x[2][8];
#pragma unroll
    for (int f = 0; f < 2; ++f)
#pragma unroll
        for (int c = 0; c < 8; ++c) x[f][c] = v[reg_of<3, B0, B1, B2>(f, c)];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        uint64_t p0 = 0, q0 = 0, p1 = 0, q1 = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const ulonglong2 e = g[8 * r + c];
            p0 = fma2(e.x, x[0][c], p0);
            q0 = fma2(e.y, x[0][c], q0);
            p1 = fma2(e.x, x[1][c], p1);
            q1 = fma2(e.y, x[1][c], q1);
        }
        v[reg_of<3, B0, B1, B2>(0, r)] = join(p0, q0);
        v[reg_of<3, B0, B1, B2>(1, r)] = join(p1, q1);
    }
}

// All four register bits: entries stored as (Re, Im), two to a 16-byte load,
// the inputs as (Re, Re) and (Im, Im) pairs (half the broadcast loads per FMA).
__device__ __forceinline__ void dense4(uint64_t (&v)[16], const ulonglong2* __restrict__ g) {
    uint64_t x2[16], y2[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        const float2 f = unpack2(v[c]);
        x2[c] = pack2(f.x, f.x);
        y2[c] = pack2(f.y, f.y);
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        uint64_t p = 0, q = 0;
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
            const ulonglong2 e = g[8 * r + (c >> 1)];
            p = fma2(x2[c], e.x, p);
            q = fma2(y2[c], e.x, q);
            p = fma2(x2[c + 1], e.y, p);
            q = fma2(y2[c + 1], e.y, q);
        }
        v[r] = join(p, q);
    }
}

// Real rotation by atan t on register bit B up to a factor per row, as two
// shears in place (no temporaries), one packed FMA per amplitude (both
// components share the real coefficient); a = t / (1 + t^2), kappa = 1 / sqrt(1 + t^2):
// first order x0 -= t x1, x1 += a x0 gives diag(1 / kappa, kappa) R, second order
// x1 += t x0, x0 -= a x1 gives diag(kappa, 1 / kappa) R.
template <int B, bool SECOND>
__device__ __forceinline__ void rotate(uint64_t (&v)[16], float t, float a) {
    const uint64_t t2 = SECOND ? pack2(t, t) : pack2(-t, -t), a2 = SECOND ? pack2(-a, -a) : pack2(a, a);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        if ((i >> B) & 1) continue;
        uint64_t& x = v[SECOND ? i | (1 << B) : i];
        uint64_t& y = v[SECOND ? i : i | (1 << B)];
        x = fma2(t2, y, x);
        y = fma2(a2, x, y);
    }
}

template <int B>
__device__ __forceinline__ void rotate_if(uint64_t (&v)[16], uint32_t head, float t, float a) {
    if (!((head >> (8 + B)) & 1)) return;
    if ((head >> (16 + B)) & 1)
        rotate<B, true>(v, t, a);
    else
        rotate<B, false>(v, t, a);
}

__device__ __forceinline__ uint64_t cmul(uint64_t v, float2 d) {
    const float2 x = unpack2(v);
    return pack2(fmaf(-x.y, d.y, x.x * d.x), fmaf(x.x, d.y, x.y * d.x));
}

// A diagonal block whose entry index takes the register bits of OM: base = the
// thread's entry, o[] the register bits' byte offsets.
template <int OM>
__device__ __forceinline__ void diagonal_om(uint64_t (&v)[16], const unsigned char* base, uint32_t ro01, uint32_t ro23) {
    const uint32_t o[4] = {ro01 & 0xffffu, ro01 >> 16, ro23 & 0xffffu, ro23 >> 16};
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        if (e & ~OM) continue;
        const float2 f = *reinterpret_cast<const float2*>(base + (e & 1 ? o[0] : 0u) + (e & 2 ? o[1] : 0u) +
                                                          (e & 4 ? o[2] : 0u) + (e & 8 ? o[3] : 0u));
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if ((i & OM) == e) v[i] = cmul(v[i], f);
    }
}

// w: the operator's first 16 bytes; d: the thread's entry.
__device__ __forceinline__ void diagonal(uint64_t (&v)[16], uint4 w, const unsigned char* d) {
    switch ((w.x >> 16) & 15u) {
        case 0: diagonal_om<0>(v, d, w.z, w.w); break;
        case 1: diagonal_om<1>(v, d, w.z, w.w); break;
        case 2: diagonal_om<2>(v, d, w.z, w.w); break;
        case 3: diagonal_om<3>(v, d, w.z, w.w); break;
        case 4: diagonal_om<4>(v, d, w.z, w.w); break;
        case 5: diagonal_om<5>(v, d, w.z, w.w); break;
        case 6: diagonal_om<6>(v, d, w.z, w.w); break;
        case 7: diagonal_om<7>(v, d, w.z, w.w); break;
        case 8: diagonal_om<8>(v, d, w.z, w.w); break;
        case 9: diagonal_om<9>(v, d, w.z, w.w); break;
        case 10: diagonal_om<10>(v, d, w.z, w.w); break;
        case 11: diagonal_om<11>(v, d, w.z, w.w); break;
        case 12: diagonal_om<12>(v, d, w.z, w.w); break;
        case 13: diagonal_om<13>(v, d, w.z, w.w); break;
        case 14: diagonal_om<14>(v, d, w.z, w.w); break;
        default: diagonal_om<15>(v, d, w.z, w.w); break;
    }
}

// w: the operator's first 16 bytes; t: the tile's number.
__device__ __forceinline__ void run_op(uint64_t (&v)[16], const GroupOp& op, uint4 w, const unsigned char* par, uint32_t t) {
    const float4 rt = *reinterpret_cast<const float4*>(op.t), ra = *reinterpret_cast<const float4*>(op.a);
    uint32_t x = op.lo[threadIdx.x & 15] + op.hi[threadIdx.x >> 4];
    const uint32_t code = w.x & 255u;
    if (code == kGroupRot) {
        rotate_if<0>(v, w.x, rt.x, ra.x);
        rotate_if<1>(v, w.x, rt.y, ra.y);
        rotate_if<2>(v, w.x, rt.z, ra.z);
        rotate_if<3>(v, w.x, rt.w, ra.w);
        return;
    }
    const ulonglong2* g = reinterpret_cast<const ulonglong2*>(par + w.y);
    switch (code) {
        case kGroupDiag: {
            const int k = (w.x >> 8) & 255u;
            for (int j = 0; j < k; ++j) x += ((t >> op.out[j]) & 1u) << op.obit[j];
            diagonal(v, w, par + w.y + x);
            break;
        }
        case 1: dense1<0>(v, g); break;
        case 2: dense1<1>(v, g); break;
        case 4: dense1<2>(v, g); break;
        case 8: dense1<3>(v, g); break;
        case 3: dense2<0, 1>(v, g); break;
        case 5: dense2<0, 2>(v, g); break;
        case 9: dense2<0, 3>(v, g); break;
        case 6: dense2<1, 2>(v, g); break;
        case 10: dense2<1, 3>(v, g); break;
        case 12: dense2<2, 3>(v, g); break;
        case 7: dense3<0, 1, 2>(v, g); break;
        case 11: dense3<0, 1, 3>(v, g); break;
        case 13: dense3<0, 2, 3>(v, g); break;
        case 14: dense3<1, 2, 3>(v, g); break;
        default: dense4(v, g); break;
    }
}

// One pass over tiles t0, t0 + stride, ... of psi.  prog: the pass's program in
// shared memory (rounds, ops, parameters); tb: the tables, built here.  zero:
// the state is taken as |0...0> and not read.
__device__ __forceinline__ void run_pass(const GroupPass& p, float2* psi, float2* stage, const unsigned char* prog,
                                         Tables& tb, uint64_t t0, uint64_t stride, bool zero) {
    const int tid = threadIdx.x;
    const int T = p.T, m = p.m, nx = p.nx;
    for (int r = tid; r < (1 << nx); r += kThreads) {
        uint64_t off = 0;
        for (int e = 0; e < nx; ++e)
            if ((r >> e) & 1) off |= 1ull << p.xpos[e];
        tb.runoff[r] = off;
    }
    __syncthreads();
    auto offset = [&](int j) { return static_cast<uint64_t>(j & ((1 << m) - 1)) | tb.runoff[j >> m]; };
    const uint32_t chunks = T == 0 ? 0u : 1u << (T - 1);      // 16-byte units of the tile
    const bool copies = static_cast<uint32_t>(tid) < chunks;
    const int nk = chunks > static_cast<uint32_t>(kThreads) ? static_cast<int>(chunks) / kThreads : 1;
    if (tid < 8) tb.goff[tid] = tid < nk ? offset(512 * tid) : 0;
    const uint64_t gld = copies ? offset(2 * tid) : 0;
    const int sld = slot_of(2 * tid);
    // the pass leaves some bits inverted: amplitude j stands in place j ^ flip
    const int sst = sld ^ slot_of(static_cast<int>(p.flip & ~1u));
    const bool swap = p.flip & 1u;
    if (T < 4)   // the registers' bits above the state's: amplitudes that stay zero
        for (int j = tid; j < 16; j += kThreads) stage[j] = stage[kAmps + j] = make_float2(0.f, 0.f);
    __syncthreads();
    const uint64_t limit = p.ntiles << T;
    auto tile_base = [&](uint64_t t) {
        uint64_t b = t << m;
        for (int e = 0; e < nx; ++e) b = insert_zero(b, p.xpos[e]);
        return b;
    };
    auto load = [&](uint64_t t, float2* st) {
        if (!copies) return;
        const uint64_t base = tile_base(t) | gld;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k >= nk) break;
            float2* s = st + (sld ^ slot_of(512 * k));
            const uint64_t gi = base | tb.goff[k];
            if (zero)
                *reinterpret_cast<float4*>(s) = make_float4(gi == 0 ? 1.f : 0.f, 0.f, 0.f, 0.f);
            else if (dbg::in_bounds(gi, 2, limit, 14))
                cp_async16(s, psi + gi);
        }
    };
    const GroupRound* rounds = reinterpret_cast<const GroupRound*>(prog);
    const GroupOp* ops = reinterpret_cast<const GroupOp*>(prog + p.ops_off);
    const unsigned char* par = prog + p.par_off;
    const int tbits = T > 4 ? T - 4 : 0;
    const bool active = tid < (1 << tbits);
    if (t0 < p.ntiles) load(t0, stage);
    cp_async_commit();
    int cur = 0;
    for (uint64_t t = t0; t < p.ntiles; t += stride) {
        cp_async_wait<0>();
        __syncthreads();   // the tile has landed; every thread is done with the other stage
        if (t + stride < p.ntiles) load(t + stride, stage + (cur ^ 1) * kAmps);
        cp_async_commit();
        float2* st = stage + cur * kAmps;
        for (int r = 0; r < p.nrounds; ++r) {
            const GroupRound& rd = rounds[r];
            if (active) {
                const int sb = rd.lo[tid & 15] ^ rd.hi[tid >> 4];
                const int s0 = rd.s[0], s1 = rd.s[1], s2 = rd.s[2], s3 = rd.s[3];
                uint64_t v[16];
                if (s0 == 1) {   // tile bit 0 is the first register bit: pairs in one 16-byte access
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const ulonglong2 f = *reinterpret_cast<const ulonglong2*>(
                            st + (sb ^ (i & 2 ? s1 : 0) ^ (i & 4 ? s2 : 0) ^ (i & 8 ? s3 : 0)));
                        v[i] = f.x;
                        v[i + 1] = f.y;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        v[i] = *reinterpret_cast<const uint64_t*>(
                            st + (sb ^ (i & 1 ? s0 : 0) ^ (i & 2 ? s1 : 0) ^ (i & 4 ? s2 : 0) ^ (i & 8 ? s3 : 0)));
                }
                const int o1 = rd.op1;
                for (int o = rd.op0; o < o1; ++o)
                    run_op(v, ops[o], *reinterpret_cast<const uint4*>(ops + o), par, static_cast<uint32_t>(t));
                if (s0 == 1) {
#pragma unroll
                    for (int i = 0; i < 16; i += 2)
                        *reinterpret_cast<ulonglong2*>(
                            st + (sb ^ (i & 2 ? s1 : 0) ^ (i & 4 ? s2 : 0) ^ (i & 8 ? s3 : 0))) =
                            make_ulonglong2(v[i], v[i + 1]);
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        *reinterpret_cast<uint64_t*>(
                            st + (sb ^ (i & 1 ? s0 : 0) ^ (i & 2 ? s1 : 0) ^ (i & 4 ? s2 : 0) ^ (i & 8 ? s3 : 0))) = v[i];
                }
            }
            __syncthreads();
        }
        if (copies) {
            const uint64_t base = tile_base(t) | gld;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k >= nk) break;
                const uint64_t gi = base | tb.goff[k];
                float4 x = *reinterpret_cast<const float4*>(st + (sst ^ slot_of(512 * k)));
                if (swap) x = make_float4(x.z, x.w, x.x, x.y);
                if (dbg::in_bounds(gi, 2, limit, 15)) *reinterpret_cast<float4*>(psi + gi) = x;
            }
        }
        cur ^= 1;
    }
    cp_async_wait<0>();
}

// Stages, then the program, then the tables.
__host__ __device__ constexpr size_t smem_bytes(size_t prog) { return sizeof(float2) * 2 * kAmps + prog + sizeof(Tables); }

// The pass's program from global to shared memory (16-byte units).
__device__ __forceinline__ void fetch_program(const unsigned char* src, uint32_t bytes, unsigned char* dst) {
    for (uint32_t i = threadIdx.x * 16u; i < bytes; i += kThreads * 16u)
        *reinterpret_cast<uint4*>(dst + i) = __ldg(reinterpret_cast<const uint4*>(src + i));
}

}  // namespace group
}  // namespace qsa
