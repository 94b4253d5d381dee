// Host side of the group passes (group.cuh): which blocks share a pass, in
// which rounds they run, and the program that the kernel reads.
//
// Operators are taken in order; one that does not fit is left for a later pass
// (or round), and an operator behind it is still taken when it acts on other
// positions than everything left behind, or when both are diagonal.  That is
// the reordering that the fusion planner may make (§IV-C: a gate moves only
// across disjoint or commuting neighbours).
#include <algorithm>
#include <cstring>
#include <vector>

#include "qsa_internal.h"

namespace qsa {

namespace {

int popc(uint64_t v) { return __builtin_popcountll(v); }

// slot vector of tile bits 1..11 (group.cuh); bit 0 is the element of a unit
constexpr int kSlotVec[kGroupTileBits] = {0, 1, 2, 4, 3, 5, 6, 7, 1, 2, 4, 7};
// Operators looked at past the first one left behind, so that building stays
// linear in the length of a long run.
constexpr size_t kLookahead = 512;
constexpr size_t kMaxOps = 512;

int slot_of_bit(int b) { return b < 4 ? 1 << b : (1 << b) ^ (kSlotVec[b] << 1); }

uint32_t dense_bytes(int k) { return k == 4 ? 2048u : 16u << (2 * k); }
uint32_t diag_bytes(int k) { return std::max(16u, 8u << k); }

struct Item {
    uint64_t mask;   // positions
    bool diag;
    int src;
};

// Orders the thread bits of a round: the lanes of one shared-memory phase (16
// lanes of 8 bytes, 8 lanes of 16 bytes when tile bit 0 is in registers) take
// tile bits whose slot vectors are independent, so the phase touches every bank once.
void order_threads(uint32_t reg, uint8_t* tb) {
    std::vector<int> rest;
    for (int b = 0; b < kGroupTileBits; ++b)
        if (!((reg >> b) & 1)) rest.push_back(b);
    int n = 0;
    if (!(reg & 1)) {
        tb[n++] = 0;
        rest.erase(rest.begin());
    }
    int basis[3] = {0, 0, 0}, rank = 0;
    for (size_t i = 0; i < rest.size() && rank < 3;) {
        int v = kSlotVec[rest[i]];
        for (int j = 2; j >= 0; --j)
            if (((v >> j) & 1) && basis[j]) v ^= basis[j];
        if (v) {
            int j = 2;
            while (!((v >> j) & 1)) --j;
            basis[j] = v;
            ++rank;
            tb[n++] = static_cast<uint8_t>(rest[i]);
            rest.erase(rest.begin() + static_cast<long>(i));
        } else {
            ++i;
        }
    }
    for (int b : rest) tb[n++] = static_cast<uint8_t>(b);
}

// A round's register bits when its dense blocks need only `reg`: the lowest
// free tile bits, so that tile bit 0 (16-byte accesses) is among them when it can be.
uint32_t fill_registers(uint32_t reg) {
    for (int b = 0; b < kGroupTileBits && popc(reg) < 4; ++b) reg |= 1u << b;
    return reg;
}

}  // namespace

bool group_takes(int k, bool diag) { return k >= 1 && (diag ? k <= kGroupDiagMax : k <= 4); }

std::vector<GroupPass> group_build(int n, const std::vector<GroupSrc>& src, std::vector<unsigned char>* progs) {
    std::vector<GroupPass> out;
    const int T = std::min(kGroupTileBits, n);
    const int max_high = kGroupTileBits - kGroupLowBits;
    std::vector<Item> left(src.size());
    for (size_t i = 0; i < src.size(); ++i) {
        uint64_t m = 0;
        for (int j = 0; j < src[i].k; ++j) m |= 1ull << src[i].pos[j];
        left[i] = {m, src[i].diag, static_cast<int>(i)};
    }
    while (!left.empty()) {
        // the operators of this pass
        std::vector<Item> take, later;
        uint64_t tile = 0, held_dense = 0, held_diag = 0;
        uint32_t bytes = 0;
        size_t i = 0;
        for (; i < left.size(); ++i) {
            const Item& it = left[i];
            if (later.size() >= kLookahead) break;
            const int k = src[it.src].k;
            const uint32_t b = (it.diag ? diag_bytes(k) : dense_bytes(k)) + sizeof(GroupOp) + sizeof(GroupRound);
            bool ok = !(it.mask & held_dense) && (it.diag || !(it.mask & held_diag));
            ok = ok && take.size() < kMaxOps && bytes + b + 64 <= kGroupProgBytes;
            if (ok && !it.diag && n > kGroupTileBits) ok = popc((tile | it.mask) >> kGroupLowBits) <= max_high;
            if (ok) {
                take.push_back(it);
                bytes += b;
                if (!it.diag) tile |= it.mask;
            } else {
                later.push_back(it);
                (it.diag ? held_diag : held_dense) |= it.mask;
            }
        }
        later.insert(later.end(), left.begin() + static_cast<long>(i), left.end());
        left.swap(later);

        // the tile: the positions of the dense operators, filled up from the lowest
        GroupPass p{};
        p.T = T;
        p.ntiles = 1ull << (n - T);
        int m = T;   // m + popc(tile >> m) falls by at most one a step, so it meets T
        while (m + popc(tile >> m) > T) --m;
        p.m = m;
        for (int q = m; q < n; ++q)
            if ((tile >> q) & 1) p.xpos[p.nx++] = q;
        uint64_t tmask = (1ull << m) - 1;
        for (int e = 0; e < p.nx; ++e) tmask |= 1ull << p.xpos[e];
        // bit of (tile number, tile-local index) that holds position q
        auto cbit = [&](int q) {
            if (q < m) return q;
            if ((tmask >> q) & 1) {
                int e = 0;
                while (p.xpos[e] != q) ++e;
                return m + e;
            }
            return T + popc(~tmask & ((1ull << q) - 1));
        };

        // rounds
        std::vector<GroupRound> rounds;
        std::vector<GroupOp> ops;
        std::vector<unsigned char> par;
        std::vector<Item> rest = take, nextr;
        while (!rest.empty()) {
            uint32_t reg = 0;
            uint64_t hd = 0, hg = 0;
            std::vector<Item> now;
            nextr.clear();
            for (const Item& it : rest) {
                bool ok = !(it.mask & hd) && (it.diag || !(it.mask & hg));
                uint32_t lm = 0;
                if (!it.diag)
                    for (int j = 0; j < src[it.src].k; ++j) lm |= 1u << cbit(src[it.src].pos[j]);
                ok = ok && popc(reg | lm) <= 4;
                if (ok) {
                    now.push_back(it);
                    reg |= lm;
                } else {
                    nextr.push_back(it);
                    (it.diag ? hg : hd) |= it.mask;
                }
            }
            rest.swap(nextr);
            reg = fill_registers(reg);
            int rb[4], nr = 0, reg_of[kGroupTileBits];
            for (int b = 0; b < kGroupTileBits; ++b)
                if ((reg >> b) & 1) {
                    reg_of[b] = nr;
                    rb[nr++] = b;
                }
            GroupRound rd{};
            for (int b = 0; b < 4; ++b) rd.s[b] = static_cast<uint16_t>(slot_of_bit(rb[b]));
            order_threads(reg, rd.tb);
            // a tile of fewer bits: its thread bits come first, the others are never set
            std::stable_partition(rd.tb, rd.tb + 8, [&](uint8_t b) { return b < std::max(T, 4); });
            rd.op0 = static_cast<uint16_t>(ops.size());
            for (const Item& it : now) {
                const GroupSrc& s = src[it.src];
                GroupOp op{};
                op.k = static_cast<uint8_t>(s.k);
                op.off = static_cast<uint32_t>(par.size());
                if (s.diag) {
                    op.code = kGroupDiag;
                    for (int j = 0; j < s.k; ++j) {
                        const int c = cbit(s.pos[j]);
                        op.c[j] = static_cast<uint8_t>(c);
                        if (c < kGroupTileBits && ((reg >> c) & 1)) {
                            op.ro[reg_of[c]] = static_cast<uint16_t>(1u << j);
                            op.om |= static_cast<uint8_t>(1u << reg_of[c]);
                        }
                    }
                    par.resize(op.off + diag_bytes(s.k));
                    std::memcpy(par.data() + op.off, s.mat, sizeof(float) * (2u << s.k));
                } else {
                    // index bits in ascending register-bit order
                    int rbit[4], ord[4];
                    for (int j = 0; j < s.k; ++j) {
                        rbit[j] = reg_of[cbit(s.pos[j])];
                        ord[j] = j;
                        op.code |= static_cast<uint8_t>(1u << rbit[j]);
                    }
                    std::sort(ord, ord + s.k, [&](int a, int b) { return rbit[a] < rbit[b]; });
                    const int D = 1 << s.k;
                    auto from = [&](int x) {   // sorted index -> the operator's own
                        int y = 0;
                        for (int j = 0; j < s.k; ++j)
                            if ((x >> j) & 1) y |= 1 << ord[j];
                        return y;
                    };
                    par.resize(op.off + dense_bytes(s.k));
                    float* g = reinterpret_cast<float*>(par.data() + op.off);
                    for (int r = 0; r < D; ++r)
                        for (int c = 0; c < D; ++c) {
                            const float* e = s.mat + 2 * (from(r) * D + from(c));
                            if (s.k == 4) {
                                *g++ = e[0];
                                *g++ = e[1];
                            } else {
                                *g++ = e[0];
                                *g++ = e[0];
                                *g++ = e[1];
                                *g++ = e[1];
                            }
                        }
                }
                ops.push_back(op);
            }
            rd.op1 = static_cast<uint16_t>(ops.size());
            rounds.push_back(rd);
        }

        p.nrounds = static_cast<int32_t>(rounds.size());
        p.only = take.size() == 1 ? take[0].src : -1;
        auto up16 = [](size_t v) { return static_cast<uint32_t>((v + 15) & ~static_cast<size_t>(15)); };
        p.ops_off = up16(rounds.size() * sizeof(GroupRound));
        p.par_off = up16(p.ops_off + ops.size() * sizeof(GroupOp));
        p.bytes = up16(p.par_off + par.size());
        p.prog = static_cast<uint32_t>(progs->size());
        progs->resize(p.prog + p.bytes);
        unsigned char* d = progs->data() + p.prog;
        std::memcpy(d, rounds.data(), rounds.size() * sizeof(GroupRound));
        std::memcpy(d + p.ops_off, ops.data(), ops.size() * sizeof(GroupOp));
        if (!par.empty()) std::memcpy(d + p.par_off, par.data(), par.size());
        out.push_back(p);
    }
    return out;
}

}  // namespace qsa
