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
constexpr size_t kMaxOps = 512;

int slot_of_bit(int b) { return b < 4 ? 1 << b : (1 << b) ^ (kSlotVec[b] << 1); }

uint32_t dense_bytes(int k) { return k == 4 ? 2048u : 16u << (2 * k); }
uint32_t diag_bytes(int k) { return std::max(16u, 8u << k); }

using Cx = std::complex<double>;

// What the passes are made of.  A unitary one-qubit operator is split as
// diag(p) R diag(q) with a real rotation R: diag(q) becomes a diagonal operator
// before R, and diag(p) waits for the next operator on its qubit that is not
// diagonal and joins its matrix, so the phases between two operators of a qubit
// are one diagonal, which shares a table with other diagonal operators, and the
// rotation is one FMA per amplitude: R = kappa M with one coefficient of each
// row of M equal to 1 (tangent form when c >= s, else cotangent, whose first row
// is negated into p), kappa in the diagonal.
struct Fine {
    enum Kind { kRot, kDense, kDiag } kind;
    uint64_t mask;           // positions
    int k;
    int pos[kGroupDiagMax];
    float t = 0.f;           // rotation
    bool cot = false;
    std::vector<Cx> m;       // dense: row-major; diagonal: entries
    int src = -1;            // the source operator it is all of, unchanged
};

std::vector<Fine> split_operators(int n, const std::vector<GroupSrc>& src) {
    std::vector<Fine> out;
    std::vector<std::array<Cx, 2>> wait(n, {1.0, 1.0});   // phases that wait on a position
    auto waiting = [&](int q) { return wait[q][0] != 1.0 || wait[q][1] != 1.0; };
    auto diag1 = [&](int q, Cx d0, Cx d1) {
        Fine f{Fine::kDiag, 1ull << q, 1, {q}};
        f.m = {d0, d1};
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
        f.m.resize(cnt);
        for (size_t e = 0; e < cnt; ++e) f.m[e] = Cx(s.mat[2 * e], s.mat[2 * e + 1]);
        if (!s.diag) {
            for (int j = 0; j < s.k; ++j) {
                if (!waiting(s.pos[j])) continue;
                for (size_t r = 0; r < D; ++r)
                    for (size_t c = 0; c < D; ++c) f.m[r * D + c] *= wait[s.pos[j]][(c >> j) & 1];
                wait[s.pos[j]] = {1.0, 1.0};
                f.src = -1;
            }
            double scale = 0.0;
            for (const Cx& z : f.m) scale = std::max(scale, std::abs(z));
            double c = 0.0, sn = 0.0;
            Cx p[2], q[2];
            if (s.k == 1 && scale > 0.0 && scale < 1e30 &&
                split_rotation({f.m[0] / scale, f.m[1] / scale, f.m[2] / scale, f.m[3] / scale}, &c, &sn, p, q)) {
                const int at = s.pos[0];
                if (sn == 0.0) {   // diagonal after all
                    wait[at] = {scale * c * p[0], scale * c * p[1]};
                    continue;
                }
                const bool cot = sn > c;
                const double t = cot ? c / sn : sn / c;
                const float tf = static_cast<float>(t);
                // kappa for the rounded coefficient: the pass applies an exact multiple of a rotation
                const double kappa =
                    scale * std::sqrt((c * c + sn * sn) / (1.0 + static_cast<double>(tf) * static_cast<double>(tf)));
                wait[at] = {cot ? -p[0] : p[0], p[1]};
                if (std::abs(q[1] - 1.0) > 1e-14) {
                    diag1(at, kappa, kappa * q[1]);
                } else {
                    wait[at][0] *= kappa;
                    wait[at][1] *= kappa;
                }
                f.kind = Fine::kRot;
                f.t = tf;
                f.cot = cot;
                f.src = -1;
                f.m.clear();
            }
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
std::vector<Fine> merge_diagonals(const std::vector<Fine>& ops, int cap) {
    struct Block {
        uint64_t mask = 0, closed = 0;
        int64_t place = -1;          // index in seq, -1: not placed yet
        std::vector<const Fine*> of;
    };
    std::vector<Block> blocks;
    std::vector<std::pair<const Fine*, int>> seq;   // an operator, or a block's index
    std::vector<int64_t> last(64, -1);              // per position: the last operator that is not diagonal
    for (const Fine& f : ops) {
        if (f.kind != Fine::kDiag) {
            for (size_t b = 0; b < blocks.size(); ++b) {
                if (!(blocks[b].mask & f.mask)) continue;
                if (blocks[b].place < 0) {
                    blocks[b].place = static_cast<int64_t>(seq.size());
                    seq.push_back({nullptr, static_cast<int>(b)});
                }
                blocks[b].closed |= blocks[b].mask & f.mask;
            }
            for (int j = 0; j < f.k; ++j) last[f.pos[j]] = static_cast<int64_t>(seq.size());
            seq.push_back({&f, -1});
            continue;
        }
        int best = -1, gain = -1;
        for (size_t b = 0; b < blocks.size(); ++b) {
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
        blocks[best].of.push_back(&f);
    }
    for (size_t b = 0; b < blocks.size(); ++b)
        if (blocks[b].place < 0) seq.push_back({nullptr, static_cast<int>(b)});
    std::vector<Fine> out;
    for (const auto& it : seq) {
        if (it.first) {
            out.push_back(*it.first);
            continue;
        }
        const Block& B = blocks[it.second];
        if (B.of.size() == 1) {
            out.push_back(*B.of[0]);
            continue;
        }
        Fine f{Fine::kDiag, B.mask, 0, {}};
        for (int q = 0; q < 64; ++q)
            if ((B.mask >> q) & 1) f.pos[f.k++] = q;
        f.m.assign(size_t(1) << f.k, 1.0);
        for (const Fine* o : B.of) {
            int bit[kGroupDiagMax];
            for (int j = 0; j < o->k; ++j) bit[j] = static_cast<int>(std::find(f.pos, f.pos + f.k, o->pos[j]) - f.pos);
            for (size_t c = 0; c < f.m.size(); ++c) {
                size_t x = 0;
                for (int j = 0; j < o->k; ++j) x |= ((c >> bit[j]) & 1) << j;
                f.m[c] *= o->m[x];
            }
        }
        out.push_back(std::move(f));
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
    std::vector<const Fine*> left(fine.size());
    for (size_t i = 0; i < fine.size(); ++i) left[i] = &fine[i];
    ModulusCarry carry;
    while (!left.empty()) {
        // the operators of this pass
        std::vector<Fine> take;
        std::vector<const Fine*> later;
        uint64_t tile = 0, held_dense = 0, held_diag = 0;
        uint32_t bytes = 0;
        size_t i = 0;
        for (; i < left.size(); ++i) {
            const Fine& f = *left[i];
            if (later.size() >= kLookahead) break;
            const bool dg = f.kind == Fine::kDiag;
            const uint32_t b = op_bytes(f) + sizeof(GroupOp) + sizeof(GroupRound);
            bool ok = !(f.mask & held_dense) && (dg || !(f.mask & held_diag));
            ok = ok && take.size() < kMaxOps && bytes + b + 64 <= kGroupProgBytes;
            if (ok && !dg && n > kGroupTileBits) ok = popc((tile | f.mask) >> kGroupLowBits) <= max_high;
            if (ok) {
                take.push_back(f);
                bytes += b;
                if (!dg) tile |= f.mask;
            } else {
                later.push_back(left[i]);
                (dg ? held_diag : held_dense) |= f.mask;
            }
        }
        later.insert(later.end(), left.begin() + static_cast<long>(i), left.end());
        left.swap(later);

        GroupPass p{};
        p.only = take.size() == 1 ? take[0].src : -1;
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
        auto cbit = [&](int q) {
            if (q < m) return q;
            if ((tmask >> q) & 1) {
                int e = 0;
                while (p.xpos[e] != q) ++e;
                return m + e;
            }
            return T + popc(~tmask & ((1ull << q) - 1));
        };

        // diagonal operators share tables of 2^6 entries (lanes read 512 bytes); smaller ones where the
        // program would not fit
        std::vector<Fine> ops;
        for (int cap : {6, 4, 0}) {
            ops = cap ? merge_diagonals(take, cap) : take;
            uint32_t total = 64;
            for (const Fine& f : ops) total += op_bytes(f) + sizeof(GroupOp) + sizeof(GroupRound);
            if (total <= kGroupProgBytes) break;
        }

        // rounds
        std::vector<GroupRound> rounds;
        std::vector<GroupOp> code;
        std::vector<unsigned char> par;
        std::vector<const Fine*> rest(ops.size()), nextr;
        for (size_t x = 0; x < ops.size(); ++x) rest[x] = &ops[x];
        while (!rest.empty()) {
            uint32_t reg = 0;
            uint64_t hd = 0, hg = 0;
            std::vector<const Fine*> now;
            nextr.clear();
            for (const Fine* f : rest) {
                const bool dg = f->kind == Fine::kDiag;
                bool ok = !(f->mask & hd) && (dg || !(f->mask & hg));
                uint32_t lm = 0;
                if (!dg)
                    for (int j = 0; j < f->k; ++j) lm |= 1u << cbit(f->pos[j]);
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
            order_threads(reg, rd.tb);
            // a tile of fewer bits: its thread bits come first, the others are never set
            std::stable_partition(rd.tb, rd.tb + 8, [&](uint8_t b) { return b < std::max(T, 4); });
            rd.op0 = static_cast<uint16_t>(code.size());
            std::vector<uint64_t> masks;   // positions of this round's codes
            for (const Fine* f : now) {
                GroupOp op{};
                if (f->kind == Fine::kRot) {
                    // joins the last rotations when nothing after them acts on its position
                    const int r = reg_of[cbit(f->pos[0])];
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
                    if (f->cot) g.om |= static_cast<uint8_t>(1u << r);
                    g.t[r] = f->t;
                    masks[x] |= f->mask;
                    continue;
                }
                op.k = static_cast<uint8_t>(f->k);
                op.off = static_cast<uint32_t>(par.size());
                par.resize(op.off + op_bytes(*f));
                float* g = reinterpret_cast<float*>(par.data() + op.off);
                if (f->kind == Fine::kDiag) {
                    // index bits: the thread bits in lane order (neighbouring lanes read neighbouring
                    // entries), then the register bits, then the bits outside the tile
                    op.code = kGroupDiag;
                    int ord[kGroupDiagMax], key[kGroupDiagMax];
                    for (int j = 0; j < f->k; ++j) {
                        const int c = cbit(f->pos[j]);
                        ord[j] = j;
                        key[j] = c >= kGroupTileBits ? 64 + c : (reg >> c) & 1 ? 32 + c
                                 : static_cast<int>(std::find(rd.tb, rd.tb + 8, c) - rd.tb);
                    }
                    std::sort(ord, ord + f->k, [&](int x, int y) { return key[x] < key[y]; });
                    for (int j = 0; j < kGroupDiagMax; ++j) op.c[j] = 31;   // no bit
                    for (int j = 0; j < f->k; ++j) {
                        const int c = cbit(f->pos[ord[j]]);
                        op.c[j] = static_cast<uint8_t>(c);
                        if (c < kGroupTileBits && ((reg >> c) & 1)) {
                            op.ro[reg_of[c]] = static_cast<uint16_t>(8u << j);
                            op.om |= static_cast<uint8_t>(1u << reg_of[c]);
                        }
                    }
                    const double share = 1.0 / static_cast<double>(f->m.size());
                    for (size_t x = 0; x < f->m.size(); ++x) {
                        size_t y = 0;
                        for (int j = 0; j < f->k; ++j) y |= ((x >> j) & 1) << ord[j];
                        const double m2 = std::norm(f->m[y]);
                        // rounded with error feedback on the modulus, relative to the entry's own
                        const float2 e = m2 > 1e-30 && m2 < 1e30
                                             ? f2_modulus(f->m[y], m2, share / m2, &carry)
                                             : make_float2(static_cast<float>(f->m[y].real()),
                                                           static_cast<float>(f->m[y].imag()));
                        g[2 * x] = e.x;
                        g[2 * x + 1] = e.y;
                    }
                } else {
                    // index bits in ascending register-bit order
                    int rbit[4], ord[4];
                    for (int j = 0; j < f->k; ++j) {
                        rbit[j] = reg_of[cbit(f->pos[j])];
                        ord[j] = j;
                        op.code |= static_cast<uint8_t>(1u << rbit[j]);
                    }
                    std::sort(ord, ord + f->k, [&](int x, int y) { return rbit[x] < rbit[y]; });
                    const int D = 1 << f->k;
                    auto from = [&](int x) {   // sorted index -> the operator's own
                        int y = 0;
                        for (int j = 0; j < f->k; ++j)
                            if ((x >> j) & 1) y |= 1 << ord[j];
                        return y;
                    };
                    for (int r = 0; r < D; ++r)
                        for (int c = 0; c < D; ++c) {
                            const Cx e = f->m[static_cast<size_t>(from(r)) * D + from(c)];
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
