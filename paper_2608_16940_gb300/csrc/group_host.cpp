// Host side of the group passes (group.cuh): which blocks share a pass, in
// which rounds they run, and the program that the kernel reads.
//
// Operators are taken in order; one that does not fit is left for a later pass
// (or round), and an operator behind it is still taken when it acts on other
// positions than everything left behind, or when both are diagonal.  That is
// the reordering that the fusion planner may make (§IV-C: a gate moves only
// across disjoint or commuting neighbours).
#include <algorithm>
#include <array>
#include <cmath>
#include <complex>
#include <cstring>
#include <deque>
#include <utility>
#include <vector>

#include "qsa_internal.h"
#include "qsa_runtime.h"

namespace qsa {

namespace {

int popc(uint64_t v) { return __builtin_popcountll(v); }

// slot vector of tile bits 1..11 (group.cuh); bit 0 is the element of a unit
constexpr int kSlotVec[kGroupTileBits] = {0, 1, 2, 4, 3, 5, 6, 7, 1, 2, 4, 7};
// Operators looked at past the first one left behind, so that building stays
// linear in the length of a long run.
constexpr size_t kLookahead = 512;
constexpr size_t kMaxOps = 2048;

int slot_of_bit(int b) { return b < 4 ? 1 << b : (1 << b) ^ (kSlotVec[b] << 1); }

uint32_t dense_bytes(int k) { return k == 4 ? 2048u : 16u << (2 * k); }
uint32_t diag_bytes(int k) { return std::max(16u, 8u << k); }
static_assert(sizeof(GroupOp) == 112 && sizeof(GroupRound) % 16 == 0, "16-byte aligned program");

using Cx = std::complex<double>;

// Plain products and moduli: the library's complex product tests for NaN and its
// modulus guards against overflow, several times the cost of the arithmetic here.
Cx mul(Cx a, Cx b) { return {a.real() * b.real() - a.imag() * b.imag(), a.real() * b.imag() + a.imag() * b.real()}; }
double modulus(Cx z) { return std::sqrt(std::norm(z)); }

// What the passes are made of.  A unitary one-qubit operator is split as
// diag(p) R diag(q) with a real rotation R: diag(q) becomes a diagonal operator
// before R, and diag(p) waits for the next operator on its qubit that is not
// diagonal and joins its matrix, so the phases between two operators of a qubit
// are one diagonal, which shares a table with other diagonal operators, and the
// rotation is one FMA per amplitude.  It runs as two shears (group.cuh), which
// leave the rows scaled by 1 / kappa and kappa: their inverses join p.  An angle
// above 45 degrees is one below times X Z: Z joins q, and the pass keeps the
// qubit's bit inverted (X) from there on, in the operators that follow and in
// the places where it stores.
struct Fine {
    enum Kind { kRot, kDense, kDiag } kind;
    uint64_t mask;           // positions
    int k;
    int pos[kGroupDiagMax];
    float t = 0.f;           // rotation: tangent, and whether the bit is inverted after it
    bool flip = false;
    // dense: row-major; diagonal: entries.  In m, or the source operator's as they are (own), or the
    // two of a diagonal on one position (two): most operators need no memory of their own
    std::vector<Cx> m;
    const double* own = nullptr;
    Cx two[2];
    Cx entry(size_t i) const { return own ? Cx(own[2 * i], own[2 * i + 1]) : m.empty() ? two[i] : m[i]; }
    Fine* next = nullptr;    // in the block of diagonal operators that it is part of
    int src = -1;            // the source operator it is all of, unchanged
    uint32_t inv = 0;        // index bits on positions that are inverted when it runs
};

std::vector<Fine> split_operators(int n, const std::vector<GroupSrc>& src) {
    std::vector<Fine> out;
    out.reserve(2 * src.size() + static_cast<size_t>(n));
    std::vector<std::array<Cx, 2>> wait(n, {1.0, 1.0});   // phases that wait on a position
    auto waiting = [&](int q) { return wait[q][0] != 1.0 || wait[q][1] != 1.0; };
    auto diag1 = [&](int q, Cx d0, Cx d1) {
        Fine f{Fine::kDiag, 1ull << q, 1, {q}};
        f.two[0] = d0;
        f.two[1] = d1;
        out.push_back(std::move(f));
    };
    for (size_t i = 0; i < src.size(); ++i) {
        const GroupSrc& s = src[i];
        Fine f{s.diag ? Fine::kDiag : Fine::kDense, 0, s.k, {}};
        f.src = static_cast<int>(i);
        for (int j = 0; j < s.k; ++j) {
            f.pos[j] = s.pos[j];
            f.mask |= 1ull << s.pos[j];
        }
        const size_t D = size_t(1) << s.k, cnt = s.diag ? D : D * D;
        f.own = s.mat;
        if (!s.diag && s.k == 1) {
            const int at = s.pos[0];
            // the phases that wait join the operator, their moduli (the factors of a rotation's rows) stay
            // with the diagonal before it, so that it is still unitary
            const double m0 = modulus(wait[at][0]), m1 = modulus(wait[at][1]);
            const Cx w0 = wait[at][0] / m0, w1 = wait[at][1] / m1;
            const Cx e[4] = {f.entry(0), f.entry(1), f.entry(2), f.entry(3)};
            double scale = 0.0;
            for (const Cx& z : e) scale = std::max(scale, modulus(z));
            double c = 0.0, sn = 0.0;
            Cx p[2], q[2];
            if (m0 > 0.0 && m1 > 0.0 && scale > 0.0 && scale < 1e30 &&
                split_rotation({mul(e[0], w0) / scale, mul(e[1], w1) / scale, mul(e[2], w0) / scale,
                                mul(e[3], w1) / scale}, &c, &sn, p, q)) {
                if (sn == 0.0) {   // diagonal after all
                    wait[at] = {scale * c * p[0] * m0, scale * c * p[1] * m1};
                    continue;
                }
                const bool flip = sn > c;
                f.t = static_cast<float>(flip ? c / sn : sn / c);
                // exact for the rounded tangent: what is left over is a common factor
                const double t = f.t, kappa = 1.0 / std::sqrt(1.0 + t * t), norm = scale * std::sqrt(c * c + sn * sn);
                wait[at] = {p[0] * norm * (flip ? 1.0 / kappa : kappa), p[1] * norm * (flip ? kappa : 1.0 / kappa)};
                const Cx q0 = m0, q1 = (flip ? -q[1] : q[1]) * m1;
                if (std::norm(q0 - 1.0) > 1e-28 || std::norm(q1 - 1.0) > 1e-28) diag1(at, q0, q1);
                f.kind = Fine::kRot;
                f.flip = flip;
                f.src = -1;
                f.own = nullptr;
                out.push_back(std::move(f));
                continue;
            }
        }
        if (!s.diag)
            for (int j = 0; j < s.k; ++j) {
                if (!waiting(s.pos[j])) continue;
                if (f.own) {
                    f.m.resize(cnt);
                    for (size_t e = 0; e < cnt; ++e) f.m[e] = f.entry(e);
                    f.own = nullptr;
                }
                for (size_t r = 0; r < D; ++r)
                    for (size_t c = 0; c < D; ++c) f.m[r * D + c] *= wait[s.pos[j]][(c >> j) & 1];
                wait[s.pos[j]] = {1.0, 1.0};
                f.src = -1;
            }
        out.push_back(std::move(f));
    }
    for (int q = 0; q < n; ++q)
        if (waiting(q)) diag1(q, wait[q][0], wait[q][1]);
    return out;
}

// A pass's operators with their diagonal ones multiplied into blocks of up to
// `cap` positions.  A block stands right before the first operator that acts on
// one of its positions without being diagonal; until then it is open.  It still
// takes an operator afterwards, on positions that nothing but diagonal operators
// has touched since where it stands.
// New blocks are kept in *made.
std::vector<Fine*> merge_diagonals(const std::vector<Fine*>& ops, int cap, std::deque<Fine>* made) {
    int diagonal = 0;
    for (const Fine* f : ops) diagonal += f->kind == Fine::kDiag ? 1 : 0;
    if (diagonal < 2) return ops;
    struct Block {
        uint64_t mask = 0, closed = 0;
        int64_t place = -1;          // index in seq, -1: not placed yet
        Fine *first = nullptr, *last = nullptr;
    };
    std::vector<Block> blocks;
    std::vector<std::pair<Fine*, int>> seq;         // an operator, or a block's index
    blocks.reserve(static_cast<size_t>(diagonal));
    seq.reserve(ops.size());
    int64_t last[64];                               // per position: the last operator that is not diagonal
    std::fill(last, last + 64, int64_t(-1));
    size_t open = 0;   // blocks before this one are closed on every position
    for (Fine* fp : ops) {
        Fine& f = *fp;
        if (f.kind != Fine::kDiag) {
            while (open < blocks.size() && blocks[open].closed == blocks[open].mask) ++open;
            for (size_t b = open; b < blocks.size(); ++b) {
                if (!(blocks[b].mask & f.mask)) continue;
                if (blocks[b].place < 0) {
                    blocks[b].place = static_cast<int64_t>(seq.size());
                    seq.push_back({nullptr, static_cast<int>(b)});
                }
                blocks[b].closed |= blocks[b].mask & f.mask;
            }
            for (int j = 0; j < f.k; ++j) last[f.pos[j]] = static_cast<int64_t>(seq.size());
            seq.push_back({fp, -1});
            continue;
        }
        int best = -1, gain = -1;
        for (size_t b = blocks.size() > 24 ? blocks.size() - 24 : 0; b < blocks.size(); ++b) {
            Block& B = blocks[b];
            if ((B.closed & f.mask) || popc(B.mask | f.mask) > cap) continue;
            bool ok = true;
            for (int j = 0; j < f.k; ++j) ok = ok && (B.place < 0 || last[f.pos[j]] < B.place);
            if (ok && popc(B.mask & f.mask) > gain) {
                best = static_cast<int>(b);
                gain = popc(B.mask & f.mask);
            }
        }
        if (best < 0) {
            best = static_cast<int>(blocks.size());
            blocks.emplace_back();
        }
        blocks[best].mask |= f.mask;
        Block& B = blocks[best];
        (B.last ? B.last->next : B.first) = fp;
        B.last = fp;
        fp->next = nullptr;
    }
    for (size_t b = 0; b < blocks.size(); ++b)
        if (blocks[b].place < 0) seq.push_back({nullptr, static_cast<int>(b)});
    std::vector<Fine*> out;
    out.reserve(seq.size());
    for (const auto& it : seq) {
        if (it.first) {
            out.push_back(it.first);
            continue;
        }
        const Block& B = blocks[it.second];
        if (B.first == B.last) {
            out.push_back(B.first);
            continue;
        }
        made->push_back(Fine{Fine::kDiag, B.mask, 0, {}});
        Fine& f = made->back();
        int bit_of[64];
        for (int q = 0; q < 64; ++q)
            if ((B.mask >> q) & 1) {
                bit_of[q] = f.k;
                f.pos[f.k++] = q;
            }
        // one-qubit members as an outer product, then the others
        std::array<std::array<Cx, 2>, kGroupDiagMax> one;
        one.fill({1.0, 1.0});
        for (const Fine* o = B.first; o; o = o->next)
            if (o->k == 1)
                for (int v = 0; v < 2; ++v) one[bit_of[o->pos[0]]][v] = mul(one[bit_of[o->pos[0]]][v], o->entry(v));
        f.m.resize(size_t(1) << f.k);
        f.m[0] = 1.0;
        for (int j = 0; j < f.k; ++j)
            for (size_t c = 0; c < (size_t(1) << j); ++c) {
                f.m[c | size_t(1) << j] = mul(f.m[c], one[j][1]);
                f.m[c] = mul(f.m[c], one[j][0]);
            }
        for (const Fine* o = B.first; o; o = o->next) {
            if (o->k == 1) continue;
            uint8_t part[kGroupDiagMax] = {}, at[1 << kGroupDiagMax] = {};   // index parts of f's bits, its indices
            for (int j = 0; j < o->k; ++j) part[bit_of[o->pos[j]]] = static_cast<uint8_t>(1u << j);
            for (size_t c = 0; c < f.m.size(); ++c) {
                if (c) at[c] = static_cast<uint8_t>(at[c & (c - 1)] | part[__builtin_ctzll(c)]);
                f.m[c] = mul(f.m[c], o->entry(at[c]));
            }
        }
        out.push_back(&f);
    }
    return out;
}

// Parameter bytes of an operator.
uint32_t op_bytes(const Fine& f) {
    return f.kind == Fine::kRot ? 0u : f.kind == Fine::kDiag ? diag_bytes(f.k) : dense_bytes(f.k);
}

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
    std::vector<Fine> fine = split_operators(n, src);
    std::vector<Fine*> left(fine.size());
    for (size_t i = 0; i < fine.size(); ++i) left[i] = &fine[i];
    // Small tables round to nearest until the plan's constants would change the norm by 5e-8, then with
    // error feedback.  Feedback alone takes entries up to an ulp and a half away: two one-qubit
    // operators (a plan of blocks of one qubit) 8.8e-8 from 64 bits, 6.5e-8 this way, 6.7e-8 as passes
    // of their own; a slack of 2e-8 left 7.0e-8.
    ModulusCarry carry;
    carry.slack = 1e-7;
    const uint64_t all = n < 64 ? (1ull << n) - 1 : ~0ull;
    // What a pass may take, by the sizes before diagonal operators share tables and rotations share
    // entries; less of it where the program comes out too long after all.
    constexpr double kRoom = 2.0 * kGroupProgBytes;
    double room = kRoom;
    while (!left.empty()) {
        // the operators of this pass
        std::vector<Fine*> take, later;
        uint64_t tile = 0, held_dense = 0, held_diag = 0;
        double bytes = 0.0;
        size_t i = 0;
        for (; i < left.size(); ++i) {
            const Fine& f = *left[i];
            // nothing behind can be taken once every position is held
            if (later.size() >= kLookahead || held_dense == all) break;
            const bool dg = f.kind == Fine::kDiag;
            const double b = op_bytes(f) + (dg && f.k < 3 ? 16.0 : 64.0);
            bool ok = !(f.mask & held_dense) && (dg || !(f.mask & held_diag));
            ok = ok && take.size() < kMaxOps && bytes + b <= room;
            if (ok && !dg && n > kGroupTileBits) ok = popc((tile | f.mask) >> kGroupLowBits) <= max_high;
            if (ok) {
                take.push_back(left[i]);
                bytes += b;
                if (!dg) tile |= f.mask;
            } else {
                later.push_back(left[i]);
                (dg ? held_diag : held_dense) |= f.mask;
            }
        }
        later.insert(later.end(), left.begin() + static_cast<long>(i), left.end());

        GroupPass p{};
        p.only = take.size() == 1 ? take[0]->src : -1;
        // the tile: the positions of the dense operators, filled up from the lowest
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
        int cbit[64];
        for (int q = 0, e = 0; q < n; ++q)
            cbit[q] = q < m ? q : (tmask >> q) & 1 ? m + e++ : T + popc(~tmask & ((1ull << q) - 1));

        // diagonal operators share tables of up to 2^6 entries (lanes read 512 bytes)
        std::deque<Fine> made;
        const std::vector<Fine*> ops = merge_diagonals(take, 6, &made);

        // inverted bits, as the operators in order leave them
        uint64_t flipped = 0;
        for (Fine* fp : ops) {
            Fine& f = *fp;
            f.inv = 0;
            for (int j = 0; j < f.k; ++j) f.inv |= static_cast<uint32_t>((flipped >> f.pos[j]) & 1) << j;
            if (f.flip) flipped ^= f.mask;
        }
        for (int q = 0; q < n; ++q)
            if ((flipped >> q) & 1) p.flip |= 1u << cbit[q];

        // rounds
        std::vector<GroupRound> rounds;
        std::vector<GroupOp> code;
        std::vector<unsigned char> par;
        std::vector<const Fine*> rest(ops.begin(), ops.end()), nextr;
        while (!rest.empty()) {
            uint32_t reg = 0;
            uint64_t hd = 0, hg = 0;
            std::vector<const Fine*> now;
            nextr.clear();
            for (size_t x = 0; x < rest.size(); ++x) {
                const Fine* f = rest[x];
                if (!(tile & ~hd) && tile) {   // every position that a dense operator acts on is held
                    nextr.insert(nextr.end(), rest.begin() + static_cast<long>(x), rest.end());
                    break;
                }
                const bool dg = f->kind == Fine::kDiag;
                bool ok = !(f->mask & hd) && (dg || !(f->mask & hg));
                uint32_t lm = 0;
                if (!dg)
                    for (int j = 0; j < f->k; ++j) lm |= 1u << cbit[f->pos[j]];
                ok = ok && popc(reg | lm) <= 4;
                if (ok) {
                    now.push_back(f);
                    reg |= lm;
                } else {
                    nextr.push_back(f);
                    (dg ? hg : hd) |= f->mask;
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
            uint8_t tb[8];
            order_threads(reg, tb);
            // a tile of fewer bits: its thread bits come first, the others are never set
            std::stable_partition(tb, tb + 8, [&](uint8_t b) { return b < std::max(T, 4); });
            for (int x = 0; x < 16; ++x)
                for (int b = 0; b < 4; ++b)
                    if ((x >> b) & 1) {
                        rd.lo[x] = static_cast<uint16_t>(rd.lo[x] ^ slot_of_bit(tb[b]));
                        rd.hi[x] = static_cast<uint16_t>(rd.hi[x] ^ slot_of_bit(tb[4 + b]));
                    }
            rd.op0 = static_cast<uint16_t>(code.size());
            std::vector<uint64_t> masks;   // positions of this round's codes
            for (const Fine* f : now) {
                GroupOp op{};
                if (f->kind == Fine::kRot) {
                    // joins the last rotations when nothing after them acts on its position
                    const int r = reg_of[cbit[f->pos[0]]];
                    size_t x = masks.size();
                    bool joined = false;
                    while (x > 0 && !joined && !(masks[x - 1] & f->mask)) {
                        --x;
                        joined = code[rd.op0 + x].code == kGroupRot;
                    }
                    if (!joined) {
                        op.code = kGroupRot;
                        code.push_back(op);
                        masks.push_back(0);
                        x = masks.size() - 1;
                    }
                    GroupOp& g = code[rd.op0 + x];
                    g.k |= static_cast<uint8_t>(1u << r);
                    // on an inverted bit: the other way round, the rows' factors exchanged
                    const bool inv = f->inv != 0;
                    if (inv) g.om |= static_cast<uint8_t>(1u << r);
                    const double t = inv ? -f->t : f->t;
                    g.t[r] = static_cast<float>(t);
                    g.a[r] = static_cast<float>(t / (1.0 + t * t));
                    masks[x] |= f->mask;
                    continue;
                }
                op.off = static_cast<uint32_t>(par.size());
                par.resize(op.off + op_bytes(*f));
                if (f->kind == Fine::kDiag) {
                    // index bits: the thread bits in lane order (neighbouring lanes read neighbouring
                    // entries), then the register bits, then the bits outside the tile
                    op.code = kGroupDiag;
                    int ord[kGroupDiagMax], key[kGroupDiagMax];
                    for (int j = 0; j < f->k; ++j) {
                        const int c = cbit[f->pos[j]];
                        ord[j] = j;
                        key[j] = c >= kGroupTileBits ? 64 + c : (reg >> c) & 1 ? 32 + c
                                 : static_cast<int>(std::find(tb, tb + 8, c) - tb);
                    }
                    std::sort(ord, ord + f->k, [&](int x, int y) { return key[x] < key[y]; });
                    for (int j = 0; j < f->k; ++j) {
                        const int key_j = key[ord[j]];
                        if (key_j >= 64) {
                            op.out[op.k] = static_cast<uint8_t>(key_j - 64 - T);
                            op.obit[op.k++] = static_cast<uint8_t>(j + 3);
                        } else if (key_j >= 32) {
                            op.ro[reg_of[key_j - 32]] = static_cast<uint16_t>(8u << j);
                            op.om |= static_cast<uint8_t>(1u << reg_of[key_j - 32]);
                        } else {
                            for (int x = 0; x < 16; ++x)
                                if ((x >> (key_j & 3)) & 1) {
                                    uint16_t& o = key_j < 4 ? op.lo[x] : op.hi[x];
                                    o = static_cast<uint16_t>(o + (8u << j));
                                }
                        }
                    }
                    float* g = reinterpret_cast<float*>(par.data() + op.off);
                    const size_t entries = size_t(1) << f->k;
                    const double share = 1.0 / static_cast<double>(entries);
                    uint8_t own[1 << kGroupDiagMax] = {static_cast<uint8_t>(f->inv)};   // the operator's own index
                    for (size_t x = 0; x < entries; ++x) {
                        if (x) own[x] = static_cast<uint8_t>(own[x & (x - 1)] ^ 1u << ord[__builtin_ctzll(x)]);
                        const Cx z = f->entry(own[x]);
                        const double m2 = std::norm(z);
                        // small tables repeat over the state: the carry bounds what they do to the modulus,
                        // relative to the entry's own (in a large one the entries' errors average out)
                        const float2 e = entries <= 8 && m2 > 1e-30 && m2 < 1e30
                                             ? f2_modulus(z, m2, share / m2, &carry)
                                             : make_float2(static_cast<float>(z.real()), static_cast<float>(z.imag()));
                        g[2 * x] = e.x;
                        g[2 * x + 1] = e.y;
                    }
                } else {
                    // index bits in ascending register-bit order
                    float* g = reinterpret_cast<float*>(par.data() + op.off);
                    int rbit[4], ord[4];
                    for (int j = 0; j < f->k; ++j) {
                        rbit[j] = reg_of[cbit[f->pos[j]]];
                        ord[j] = j;
                        op.code |= static_cast<uint8_t>(1u << rbit[j]);
                    }
                    std::sort(ord, ord + f->k, [&](int x, int y) { return rbit[x] < rbit[y]; });
                    const int D = 1 << f->k;
                    int from[16];   // sorted index -> the operator's own
                    for (int x = 0; x < D; ++x) {
                        from[x] = static_cast<int>(f->inv);
                        for (int j = 0; j < f->k; ++j)
                            if ((x >> j) & 1) from[x] ^= 1 << ord[j];
                    }
                    for (int r = 0; r < D; ++r)
                        for (int c = 0; c < D; ++c) {
                            const Cx e = f->entry(static_cast<size_t>(from[r]) * D + from[c]);
                            const float re = static_cast<float>(e.real()), im = static_cast<float>(e.imag());
                            *g++ = re;
                            if (f->k < 4) *g++ = re;
                            *g++ = im;
                            if (f->k < 4) *g++ = im;
                        }
                }
                code.push_back(op);
                masks.push_back(f->mask);
            }
            rd.op1 = static_cast<uint16_t>(code.size());
            rounds.push_back(rd);
        }

        p.nrounds = static_cast<int32_t>(rounds.size());
        auto up16 = [](size_t v) { return static_cast<uint32_t>((v + 15) & ~static_cast<size_t>(15)); };
        p.ops_off = up16(rounds.size() * sizeof(GroupRound));
        p.par_off = up16(p.ops_off + code.size() * sizeof(GroupOp));
        p.bytes = up16(p.par_off + par.size());
        if (p.bytes > kGroupProgBytes) {   // the same operators again, as many fewer as it was too long
            room = std::min(bytes, room) * std::min(0.95, 0.98 * kGroupProgBytes / p.bytes);
            continue;
        }
        // the operators to come are much like these: as much again, or more where the program is short
        if (p.bytes < 0.9 * kGroupProgBytes) room = std::min(kRoom, room * 0.95 * kGroupProgBytes / p.bytes);
        left.swap(later);
        p.prog = static_cast<uint32_t>(progs->size());
        progs->resize(p.prog + p.bytes);
        unsigned char* d = progs->data() + p.prog;
        std::memcpy(d, rounds.data(), rounds.size() * sizeof(GroupRound));
        std::memcpy(d + p.ops_off, code.data(), code.size() * sizeof(GroupOp));
        if (!par.empty()) std::memcpy(d + p.par_off, par.data(), par.size());
        out.push_back(p);
    }
    return out;
}

}  // namespace qsa
