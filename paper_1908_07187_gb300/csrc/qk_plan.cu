// Planner for the fused mode: groups queued gates into tile passes (K3).
//
// Two gates commute when neither one's non-diagonal qubit (the target of a 2x2
// gate) is touched by the other; diagonal gates and the control qubits of a
// controlled gate act diagonally.  A pass picks a set S of 13 physical qubits
// (always 0 .. kTileContig-1, for coalesced access) and takes, in order, every
// queued gate that
//   - is diagonal, or is a 2x2 gate whose target is in S (controls may be
//     anywhere: a control outside S is constant over a tile), and
//   - commutes with every earlier gate the pass leaves behind.
// Qubits join S greedily as 2x2 targets are met.  Inside the pass the taken
// gates are list-scheduled over the three register arrangements of the tile
// kernel, inserting a transpose when no ready gate fits the current one.
//
// A last walk over the program (fold_program) turns each layer gate into pivot
// form (LayerGate in qk_kernels.cuh) and keeps, in double precision, every
// pending factor that is the same for all threads -- per local qubit (a phase and
// a magnitude), plus a constant phase -- and the pass's real scale: those fold
// into later gates' coefficients and the final flush, so the device never sees
// them.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <complex>
#include <cstring>
#include <deque>
#include <vector>

#include "qk_plan.h"

namespace qk {

struct TilePlanner {
    bool log = false;  // QK_PLAN_LOG=1: one line per tile pass on stderr
};

TilePlanner *make_planner() {
    TilePlanner *p = new TilePlanner();
    const char *e = std::getenv("QK_PLAN_LOG");
    p->log = e && e[0] == '1';
    return p;
}
void free_planner(TilePlanner *p) { delete p; }

namespace {

struct POp {
    const FusedOp *op;
    uint64_t nd;   // non-diagonal qubits
    uint64_t all;  // every qubit the op depends on
};

POp classify(const FusedOp &op) {
    POp p;
    p.op = &op;
    if (op.kind == FusedOp::U2) {
        p.nd = 1ull << op.q;
        p.all = p.nd | op.cmask;
    } else {
        p.nd = 0;
        p.all = op.mask;
    }
    return p;
}

bool commute(const POp &a, const POp &b) { return !(a.nd & b.all) && !(b.nd & a.all); }

bool same_cond(const Cond &a, const Cond &b) {
    if (a.n != b.n) return false;
    for (int k = 0; k < a.n; ++k)
        if (a.idx[k] != b.idx[k]) return false;
    return true;
}

// slot of a local bit in an arrangement: 0 = register, 1 = lane, 2 = warp; *pos = index
int slot_of(int arr, int lb, int *pos) {
    if (arr == ARR_IO) {
        if (lb < 5) { *pos = lb; return 1; }
        if (lb < 10) { *pos = lb - 5; return 0; }
        *pos = lb - 10;
        return 2;
    }
    if (arr == ARR_LO) {
        if (lb < 5) { *pos = lb; return 0; }
        if (lb < 10) { *pos = lb - 5; return 1; }
        *pos = lb - 10;
        return 2;
    }
    // ARR_HI
    if (lb < 5) { *pos = lb; return 1; }
    if (lb < 8) { *pos = lb - 5; return 2; }
    *pos = lb - 8;
    return 0;
}

bool executable(const POp &p, int arr, const int *local_of) {
    if (p.op->kind != FusedOp::U2) return true;
    int pos;
    return slot_of(arr, local_of[p.op->q], &pos) == 0;
}

// Encode a mask/value condition over physical qubits into register / thread /
// fixed-bit parts for an arrangement.
void encode_cond(uint64_t mask, uint64_t val, int arr, const int *local_of, TileOp &t) {
    t.rmask = t.rval = 0;
    t.tmask = t.tval = 0;
    t.gmask = t.gval = 0;
    for (int b = 0; b < 64; ++b) {
        if (!((mask >> b) & 1)) continue;
        const int bit = (int)((val >> b) & 1);
        const int lb = local_of[b];
        if (lb < 0) {
            t.gmask |= 1ull << b;
            t.gval |= (uint64_t)bit << b;
            continue;
        }
        int pos;
        const int s = slot_of(arr, lb, &pos);
        if (s == 0) {
            t.rmask |= (uint8_t)(1 << pos);
            t.rval |= (uint8_t)(bit << pos);
        } else if (s == 1) {
            t.tmask |= (uint16_t)(1 << pos);
            t.tval |= (uint16_t)(bit << pos);
        } else {
            t.tmask |= (uint16_t)(1 << (5 + pos));
            t.tval |= (uint16_t)(bit << (5 + pos));
        }
    }
}

uint32_t angle_turns(double x) {
    double frac = x / (2.0 * M_PI);
    frac -= std::floor(frac);
    return (uint32_t)(uint64_t)std::llround(frac * 4294967296.0);
}
double turns_angle(uint32_t t) { return 2.0 * M_PI * (double)t / 4294967296.0; }

// local qubit of register bit k in an arrangement
int local_of_reg(int arr, int k) { return arr == ARR_IO ? 5 + k : arr == ARR_LO ? k : 8 + k; }

// Planner-only op kind: a diagonal term that is the same for every thread and
// tile (no thread or fixed-bit condition) on register bit k (k == 5: constant),
// ph.turns; fold_program absorbs it and it never reaches the device.
constexpr uint8_t TOP_HOSTPH = 0x40;

using cdm = std::complex<double>;
struct Mat2 {
    cdm m[4];
};

// The program's pending state that is the same for every thread, in double
// precision: mag[q] e^{i u[q]} the factor of local qubit q's stored |1> relative
// to its stored |0>, u0 a constant phase, lam the real scale that the pivot form
// leaves over, flip[q] whether q's values are stored swapped.
struct UniformPending {
    double u[kTileQubits] = {};     // phase of the pending factor on a local qubit's stored |1>
    double mag[kTileQubits];        // its magnitude (in [1/2, 2])
    double u0 = 0.0;
    double lam = 1.0;
    int flip[kTileQubits] = {};   // local qubit stored with its two values swapped
    UniformPending() {
        for (double &m : mag) m = 1.0;
    }
};

// Pivot form of a layer gate on local qubit q (LayerGate in qk_kernels.cuh).  The
// gate in stored order is W = U X^f (f: q stored flipped); the output is stored
// flipped (f') when that puts the larger entries of M = X^f' W on the diagonal.
// F = mag[q] e^{i u[q]} is the pending factor of q's stored |1>.  Returns zf, the
// value of the pair the device updates first: the one that keeps the pending
// magnitude of q's |1> within [1/2, 2] (zf = 0 multiplies it by s <= 1, zf = 1
// divides it by s >= 1/2).
int pivot_gate(const Mat2 &g, UniformPending &st, int q, LayerGate &out) {
    cdm W[4] = {g.m[0], g.m[1], g.m[2], g.m[3]};
    if (st.flip[q]) {  // U X: swap the columns
        std::swap(W[0], W[1]);
        std::swap(W[2], W[3]);
    }
    const bool fout = std::abs(W[0]) < std::abs(W[2]);
    if (fout) {        // X W: swap the rows
        std::swap(W[0], W[2]);
        std::swap(W[1], W[3]);
    }
    const cdm m00 = W[0], m01 = W[1], m10 = W[2], m11 = W[3];
    const cdm F = std::polar(st.mag[q], st.u[q]);
    const cdm A0 = m01 * F / m00, A1 = m10 / (m11 * F);
    // y1 += a1 y0 then y0 += s a0 y1 leaves y0 = s z0 (and the other order y1 =
    // s z1) for s = 1 / (1 - a0 a1), real and in [1/2, 1] for a unitary gate
    const cdm s = 1.0 / (1.0 - A0 * A1);
    const int zf = st.mag[q] < 1.0 ? 1 : 0;
    const cdm C0 = zf ? A0 : s * A0, C1 = zf ? s * A1 : A1;
    const cdm P0 = zf ? m00 : m00 / s, P1 = zf ? m11 * F / s : m11 * F;   // the true outputs' factors
    st.u0 += std::arg(P0);
    st.lam *= std::abs(P0);
    const cdm R = P1 / P0;
    st.u[q] = std::arg(R);
    st.mag[q] = std::abs(R);
    st.flip[q] = fout ? 1 : 0;
    const float a0r = (float)C0.real(), a0i = (float)C0.imag(), a1r = (float)C1.real(), a1i = (float)C1.imag();
    out.c[0] = make_float2(a0r, a0r);
    out.c[1] = make_float2(a0i, a0i);
    out.c[2] = make_float2(-a0i, -a0i);
    out.c[3] = make_float2(a1r, a1r);
    out.c[4] = make_float2(a1i, a1i);
    out.c[5] = make_float2(-a1i, -a1i);
    return zf;
}

// local qubits of the thread bits (0..4 lanes, 5..7 warps) in an arrangement
int local_of_tbit(int arr, int t) {
    if (t < 5) return arr == ARR_LO ? 5 + t : t;
    return arr == ARR_HI ? 5 + (t - 5) : 10 + (t - 5);
}
// The gates one pass takes from rem for a qubit set S: in order, each gate
// that commutes with every gate left behind before it, whose 2x2 target is in
// S (with grow, a target joins S while S has room) and whose classical
// condition fits the condition table.  Counts only when tk is null.
// Once every qubit carries a left-behind 2x2 gate, no later gate commutes with
// them all, so the walk stops there (the rest is left behind as a whole).
struct TakeLimits {
    int tile_qubits, max_u2, max_ph;
};
void take_gates(const std::vector<POp> &rem, int n, const TakeLimits &lim, uint64_t S0, bool grow,
                std::vector<Cond> &conds, std::vector<POp> *tk, std::vector<POp> *lf, uint64_t *S_out, int *n_u2_out,
                int *n_ph_out) {
    const uint64_t all_qubits = n >= 64 ? ~0ull : (1ull << n) - 1;
    uint64_t S = S0;
    int cnt = __builtin_popcountll(S0);
    uint64_t ndb = 0, allb = 0;
    int n_u2 = 0, n_ph = 0;
    conds.clear();
    for (auto it = rem.begin(); it != rem.end(); ++it) {
        if (ndb == all_qubits) {
            if (lf) lf->insert(lf->end(), it, rem.end());
            break;
        }
        const POp &p = *it;
        const bool is_u2 = p.op->kind == FusedOp::U2;
        bool ok = (is_u2 ? n_u2 < lim.max_u2 : n_ph < lim.max_ph) && !(p.nd & allb) && !(p.all & ndb);
        if (ok && is_u2) {
            const uint64_t t = 1ull << p.op->q;
            if (!(S & t)) {
                if (grow && cnt < lim.tile_qubits) {
                    S |= t;
                    ++cnt;
                } else {
                    ok = false;
                }
            }
        }
        if (ok && p.op->cond.n) {
            bool found = false;
            for (const auto &cd : conds) found = found || same_cond(cd, p.op->cond);
            if (!found) {
                if ((int)conds.size() < kTileMaxConds) conds.push_back(p.op->cond);
                else ok = false;
            }
        }
        if (ok) {
            if (tk) tk->push_back(p);
            if (is_u2) ++n_u2; else ++n_ph;
        } else {
            if (lf) lf->push_back(p);
            ndb |= p.nd;
            allb |= p.all;
        }
    }
    *S_out = S;
    *n_u2_out = n_u2;
    *n_ph_out = n_ph;
}

// S and its gates for one pass: the set that the greedy walk builds, or the low
// contiguous qubits plus a window of consecutive qubits, whichever lets the pass take
// the most 2x2 gates (then the most gates); a circuit whose gates spread along the
// qubit line (layers of neighbour couplings) fills passes better with windows
uint64_t choose_pass(const std::vector<POp> &rem, int n, const TakeLimits &lim, int contig, std::vector<Cond> &conds,
                     std::vector<POp> &taken, std::vector<POp> &left, int *n_u2, int *n_ph) {
    const uint64_t low = (1ull << contig) - 1;
    uint64_t S = 0, best_S0 = low;
    bool best_grow = true;
    take_gates(rem, n, lim, low, true, conds, nullptr, nullptr, &S, n_u2, n_ph);
    int best_u2 = *n_u2, best_all = *n_u2 + *n_ph;
    const int wlen = lim.tile_qubits - contig;
    for (int w = contig; w + wlen <= n; ++w) {
        const uint64_t S0 = low | (((1ull << wlen) - 1) << w);
        uint64_t Sw;
        take_gates(rem, n, lim, S0, false, conds, nullptr, nullptr, &Sw, n_u2, n_ph);
        if (*n_u2 > best_u2 || (*n_u2 == best_u2 && *n_u2 + *n_ph > best_all)) {
            best_u2 = *n_u2;
            best_all = *n_u2 + *n_ph;
            best_S0 = S0;
            best_grow = false;
        }
    }
    left.clear();
    taken.clear();
    take_gates(rem, n, lim, best_S0, best_grow, conds, &taken, &left, &S, n_u2, n_ph);
    int cnt = __builtin_popcountll(S);
    // fill S up with the lowest unused qubits
    for (int b = contig; b < n && cnt < lim.tile_qubits; ++b)
        if (!((S >> b) & 1)) {
            S |= 1ull << b;
            ++cnt;
        }
    return S;
}

// ---------------------------------------------------------------------------
// passes over tiles in shared memory (SmemTileParams in qk_kernels.cuh)
// ---------------------------------------------------------------------------

// Tile width by state size: wide tiles carry more gates per read and write of a state
// in HBM; states that fit L2 are split over more CTAs instead, because one SM's two
// FP64 lanes take 6 us for one gate on 2^12 amplitudes.  Measured on U3 / CZ / QFT
// circuits (us at 8, 10 and 12 tile qubits): 12 qubits 263 / 384 / 879, 16 qubits 333 /
// 412 / 924, 18 qubits 609 / 599 / 1003, 20 qubits 1831 / 1616 / 1676, 22 qubits 6691 /
// 5677 / 5413.  complex64 (below 13 qubits, at 8, 9, 10 and 12 tile qubits): 10 qubits
// 159 / 158 / 172 / 174, 12 qubits 182 / 170 / 184 / 231.
int smem_tile_qubits(int n, int prec) {
    if (prec == 0) return std::min(n, 9);
    return std::min(n, n <= 16 ? 8 : n <= 20 ? 10 : kSmemTileMax);
}
// Qubits that every tile holds, for runs of 128 bytes in HBM; none for states in L2.
int smem_tile_contig(int n) { return n >= 18 ? 3 : 0; }

// A diagonal term that is not yet in a program: f where (index & mask) == val.
struct DTerm {
    uint64_t mask, val;
    cdm f;
    const Cond *cond;
    const FusedOp *src;      // the queued op that it is, if none of it became pending
};

// Builds one pass's program from its gates in order.  Single-qubit diagonal factors
// never reach the device: F[q] is the pending complex factor of physical qubit q's |1>,
// lam the one of every amplitude.  Diagonal terms on more qubits wait in terms until a
// gate acts on one of their qubits and go out together there.
struct SmemTileBuilder {
    SmemTileParams &P;
    cdm *F;
    cdm &lam;
    int local_of[64], tile_of[64];
    std::vector<DTerm> terms;
    bool overflow = false;

    SmemTileBuilder(SmemTileParams &p, cdm *f, cdm &l) : P(p), F(f), lam(l) {}

    SmemTileOp *add(uint8_t kind, uint8_t q) {
        if (P.nops >= kSmemTileOps) {
            overflow = true;
            P.nops = 0;      // the program is thrown away
        }
        SmemTileOp &o = P.ops[P.nops++];
        std::memset(static_cast<void *>(&o), 0, sizeof o);
        o.kind = kind;
        o.q = q;
        o.cond = kNoBit;
        return &o;
    }
    // mask and value over physical bits as local and tile-index conditions
    void conditions(SmemTileOp &o, uint64_t mask, uint64_t val) {
        for (uint64_t m = mask; m; m &= m - 1) {
            const int b = __builtin_ctzll(m);
            const uint32_t v = (uint32_t)(val >> b) & 1u;
            if (local_of[b] >= 0) {
                o.lmask |= (uint16_t)(1u << local_of[b]);
                o.lval |= (uint16_t)(v << local_of[b]);
            } else {
                o.tmask |= 1u << tile_of[b];
                o.tval |= v << tile_of[b];
            }
        }
    }
    uint8_t cond_index(const Cond &c) const {
        for (int k = 0; k < P.n_conds; ++k)
            if (same_cond(P.conds[k], c)) return (uint8_t)k;
        return kNoBit;
    }

    // a term of the queue: single-qubit and constant parts become pending factors, a
    // two-qubit term keeps only its (1, 1) pattern
    void diagonal(const POp &p) {
        const FusedOp &op = *p.op;
        DTerm t{op.mask, op.val, op.f, op.cond.n ? &op.cond : nullptr, &op};
        const int k = __builtin_popcountll(t.mask);
        if (t.cond || k > 2) {
            terms.push_back(t);
            return;
        }
        if (k == 0) {
            lam *= t.f;
            return;
        }
        const int a = __builtin_ctzll(t.mask), b = 63 - __builtin_clzll(t.mask);
        const int va = (int)(t.val >> a) & 1, vb = (int)(t.val >> b) & 1;
        const cdm inv = 1.0 / t.f;
        if (k == 1) {
            if (va) F[a] *= t.f;
            else {
                lam *= t.f;
                F[a] *= inv;
            }
            return;
        }
        if (va && !vb) F[a] *= t.f;
        if (!va && vb) F[b] *= t.f;
        if (!va && !vb) {
            lam *= t.f;
            F[a] *= inv;
            F[b] *= inv;
        }
        if (t.val != t.mask) t.src = nullptr;
        if (va != vb) t.f = inv;
        t.val = t.mask;
        terms.push_back(t);
    }
    static bool is_pair(const DTerm &t) { return !t.cond && t.val == t.mask && __builtin_popcountll(t.mask) == 2; }
    static bool is_sign(const DTerm &t) { return t.f == cdm(-1.0, 0.0); }

    void single_term(const DTerm &t) {
        SmemTileOp *o = add(ST_PH, kNoBit);
        conditions(*o, t.mask, t.val);
        if (t.cond) o->cond = cond_index(*t.cond);
        o->c[0] = t.f.real();
        o->c[1] = t.f.imag();
    }
    // an op on the amplitudes with physical bit b set: its local bit, or a tile-index condition
    void on_bit(SmemTileOp &o, int b) {
        if (local_of[b] >= 0) o.q = (uint8_t)local_of[b];
        else o.tval |= 1u << tile_of[b];
    }
    // factors fac[b] of the physical bits in bits, times c0, on the amplitudes with
    // physical bit at set (at < 0: on all)
    void table(int at, uint64_t bits, const cdm *fac, cdm c0) {
        SmemTileOp *o = add(ST_TABLE, kNoBit);
        if (at >= 0) {
            on_bit(*o, at);
            o->tmask = o->tval;
        }
        o->first = (uint32_t)P.nfac;
        o->c[0] = c0.real();
        o->c[1] = c0.imag();
        if (P.nfac + __builtin_popcountll(bits) > kSmemTileFacs) {
            overflow = true;
            return;
        }
        for (int pass = 0; pass < 2; ++pass)               // physical order is local and tile-index order
            for (uint64_t m = bits; m; m &= m - 1) {
                const int b = __builtin_ctzll(m);
                if ((local_of[b] >= 0) != (pass == 0)) continue;
                if (pass == 0) o->lmask |= (uint16_t)(1u << local_of[b]);
                else o->tfac |= 1u << tile_of[b];
                P.fac[P.nfac++] = make_double2(fac[b].real(), fac[b].imag());
            }
    }
    // emit the waiting terms on physical qubit b.  Sign flips of pairs go to *sl, *st
    // (local and tile-index parity masks of the other qubits), to an op of their own
    // when these are null.
    void emit_touching(int b, uint16_t *sl, uint32_t *st) {
        uint64_t bits = 0, signs = 0;
        cdm fac[64];
        size_t w = 0;
        const uint64_t bb = 1ull << b;
        for (size_t i = 0; i < terms.size(); ++i) {
            const DTerm &t = terms[i];
            if (!(t.mask & bb)) {
                terms[w++] = t;
                continue;
            }
            if (!is_pair(t)) {
                single_term(t);
                continue;
            }
            const int d = __builtin_ctzll(t.mask & ~bb);
            if (is_sign(t)) signs ^= 1ull << d;
            else if ((bits >> d) & 1) fac[d] *= t.f;
            else {
                bits |= 1ull << d;
                fac[d] = t.f;
            }
        }
        terms.resize(w);
        if (bits) table(b, bits, fac, cdm(1.0, 0.0));
        if (!signs) return;
        uint16_t l = 0;
        uint32_t g = 0;
        for (uint64_t m = signs; m; m &= m - 1) {
            const int d = __builtin_ctzll(m);
            if (local_of[d] >= 0) l |= (uint16_t)(1u << local_of[d]);
            else g |= 1u << tile_of[d];
        }
        if (sl) {
            *sl = l;
            *st = g;
            return;
        }
        SmemTileOp *o = add(ST_SIGN, kNoBit);
        on_bit(*o, b);
        o->lmask = l;
        o->tmask = g;
    }
    // every waiting term, grouped by the qubit that most pairs share
    void emit_all() {
        while (!terms.empty()) {
            int cnt[64] = {0}, best = -1;
            for (const DTerm &t : terms) {
                if (!is_pair(t)) continue;
                for (uint64_t m = t.mask; m; m &= m - 1) {
                    const int b = __builtin_ctzll(m);
                    if (best < 0 || ++cnt[b] > cnt[best]) best = b;
                }
            }
            if (best < 0) best = __builtin_ctzll(terms[0].mask);
            emit_touching(best, nullptr, nullptr);
            if (overflow) return;
        }
    }
    // the pending factor of qubit b onto the amplitudes
    void materialise(int b) {
        if (F[b] == cdm(1.0, 0.0)) return;
        DTerm t{1ull << b, 1ull << b, F[b], nullptr, nullptr};
        single_term(t);
        F[b] = 1.0;
    }

    // A 2x2 gate on physical qubit op.q.  Uncontrolled: with M = W or X W (rows
    // exchanged when that puts the larger entries on the diagonal) and F the pending
    // factor, the outputs are W00 (y0 + a0 y1) and W11 F (y1 + a1 y0) with a0 = W01 F /
    // W00, a1 = W10 / (W11 F), and a0 a1 = -r0 r1 is real for a unitary M.  Turning y1
    // (or y0) by psi = arg a0 makes both updates real; of e^{i psi} = i^k cos(phi) (1 +
    // i tan(phi)), |phi| <= pi/4, only i^k (1 + i tan) is applied and the cosine stays
    // pending.  Updating one value from the other in place leaves s = 1 / (1 + r0 r1)
    // on the second one.  Which value is turned and which is updated first is chosen so
    // that the pending magnitude stays near 1.
    void gate(const POp &p) {
        const FusedOp &op = *p.op;
        const int b = op.q;
        const uint8_t q = (uint8_t)local_of[b];
        const cdm *M = op.m;
        const bool is_x = M[0] == 0.0 && M[3] == 0.0 && M[1] == 1.0 && M[2] == 1.0;
        // the update form below takes a0 a1 for real, which a matrix defined with a loose
        // tolerance need not have
        const cdm pr = M[1] * M[2] * std::conj(M[0] * M[3]);
        const bool unitary = std::abs(pr.imag()) <= 0x1p-50 * std::abs(pr) && pr.real() <= 0.0;
        if (op.cmask || op.cond.n || !unitary) {
            emit_touching(b, nullptr, nullptr);
            materialise(b);
            SmemTileOp *o = add(is_x ? ST_X : ST_CU2, q);
            conditions(*o, op.cmask, op.cmask);
            if (op.cond.n) o->cond = cond_index(op.cond);
            for (int e = 0; e < 4; ++e) {
                o->c[2 * e] = M[e].real();
                o->c[2 * e + 1] = M[e].imag();
            }
            return;
        }
        uint16_t sl = 0;
        uint32_t sg = 0;
        emit_touching(b, &sl, &sg);
        SmemTileOp *o = add(ST_U2, q);
        o->lmask = sl;
        o->tmask = sg;
        cdm W[4] = {M[0], M[1], M[2], M[3]};
        const bool sw = std::abs(W[0]) < std::abs(W[2]);
        if (sw) {
            std::swap(W[0], W[2]);
            std::swap(W[1], W[3]);
            o->flags |= kU2Swap;
        }
        const cdm f = F[b], a0 = W[1] * f / W[0], a1 = W[2] / (W[3] * f);
        const double r0 = std::abs(a0), r1 = std::abs(a1), s = 1.0 / (1.0 + r0 * r1);
        cdm p0 = W[0], p1 = W[3] * f;
        if (r0 != 0.0 || r1 != 0.0) {
            const double psi = std::arg(a0);
            const int k = (int)std::lround(psi / (M_PI / 2));
            const double phi = psi - k * (M_PI / 2), cs = std::cos(phi), tn = std::tan(phi);
            const cdm e = std::polar(1.0, psi);
            double best = 0.0;
            int side = -1, first0 = 0;
            for (int c = 0; c < 4; ++c) {                 // bit 0: y0 is turned; bit 1: y0 is updated first
                double r = std::abs(p1 / p0) * ((c & 1) ? 1.0 / cs : cs) * ((c & 2) ? 1.0 / s : s);
                if (sw) r = 1.0 / r;
                r = std::abs(std::log(r));
                if (side < 0 || r < best) {
                    best = r;
                    side = c & 1;
                    first0 = c >> 1;
                }
            }
            double b0, b1;
            if (side == 0) {
                b0 = r0 * cs;
                b1 = -r1 / cs;
                p1 *= std::conj(e) * cs;
            } else {
                b0 = r0 / cs;
                b1 = -r1 * cs;
                p0 *= e * cs;
                o->flags |= kU2On0;
            }
            if (first0) {
                b1 *= s;
                p1 /= s;
                o->flags |= kU2First0;
            } else {
                b0 *= s;
                p0 /= s;
            }
            o->flags |= (uint8_t)((k & 3) | kU2Lift);
            if (std::abs(tn) > 0x1p-55) o->flags |= kU2Phase;   // below: less than a rounding error
            o->c[0] = tn;
            o->c[1] = b0;
            o->c[2] = b1;
        }
        if (sw) std::swap(p0, p1);
        lam *= p0;
        F[b] = p1 / p0;
    }
};

}  // namespace

qk_status plan_smem_passes(TilePlanner *planner, int n, int prec, const std::vector<FusedOp> &ops,
                           const SmemPassSink &sink, const char **err) {
    *err = "";
    static thread_local std::vector<POp> rem, left, taken, next;
    rem.clear();
    for (const auto &op : ops) rem.push_back(classify(op));
    const int m = smem_tile_qubits(n, prec);
    TakeLimits lim{m, kSmemTileOps, 4096};
    const int contig = std::min(smem_tile_contig(n), m);
    std::vector<Cond> conds;
    const double far = prec == 0 ? 0x1p24 : 0x1p200;   // how far the stored amplitudes may drift from the true ones
    cdm F[64], lam = 1.0;
    for (cdm &f : F) f = 1.0;
    std::deque<FusedOp> rewritten;   // pair terms handed on without their single-qubit parts
    while (!rem.empty()) {
        int n_u2 = 0, n_ph = 0;
        const uint64_t S = choose_pass(rem, n, lim, contig, conds, taken, left, &n_u2, &n_ph);
        static thread_local SmemTileParams P;
        cdm F1[64], lam1 = lam;
        std::copy(F, F + 64, F1);
        SmemTileBuilder B(P, F1, lam1);
        P.n = n;
        P.m = m;
        P.n_tiles = 1u << (n - m);
        P.nfix = 0;
        P.nops = P.nfac = 0;
        for (int b = 0, lb = 0; b < 64; ++b) {
            B.local_of[b] = B.tile_of[b] = -1;
            if (b >= n) continue;
            if ((S >> b) & 1) {
                P.S[lb] = (int8_t)b;
                B.local_of[b] = lb++;
            } else {
                P.fixed[P.nfix] = (int8_t)b;
                B.tile_of[b] = P.nfix++;
            }
        }
        P.n_conds = (int)conds.size();
        for (int k = 0; k < P.n_conds; ++k) P.conds[k] = conds[k];
        for (const POp &p : taken) {
            if (p.op->kind == FusedOp::U2) B.gate(p);
            else B.diagonal(p);
            if (B.overflow) break;
        }
        // Terms that no gate of this pass called for go to the front of what is left:
        // they commute with everything taken after them, and with what was left
        // behind before them.  (Their single-qubit parts are pending already.)
        if (!B.overflow && (left.empty() || n_u2 == 0)) B.emit_all();
        if (!B.overflow && left.empty()) {
            // the plan's last pass applies what is pending
            uint64_t bits = 0;
            for (int b = 0; b < n; ++b)
                if (F1[b] != cdm(1.0, 0.0)) bits |= 1ull << b;
            if (!B.overflow && (bits || lam1 != cdm(1.0, 0.0))) B.table(-1, bits, F1, lam1);
        } else if (!B.overflow && !(std::abs(lam1) > 1.0 / far && std::abs(lam1) < far)) {
            // a factor in [2^-1/2, 2] per gate: keep the stored amplitudes in range
            B.table(-1, 0, F1, lam1);
            lam1 = 1.0;
        }
        if (B.overflow) {
            if (lim.max_u2 <= 1 && lim.max_ph <= 1) {
                *err = "internal: tile program overflow";
                return QK_EINVAL;
            }
            lim.max_u2 = std::max(1, lim.max_u2 / 2);
            lim.max_ph = std::max(1, lim.max_ph / 2);
            continue;
        }
        next.clear();
        for (const DTerm &t : B.terms) {
            if (t.src) {
                next.push_back(classify(*t.src));
                continue;
            }
            FusedOp o;
            o.kind = FusedOp::PHASE;
            o.mask = t.mask;
            o.val = t.val;
            o.f = t.f;
            rewritten.push_back(o);
            next.push_back(classify(rewritten.back()));
        }
        next.insert(next.end(), left.begin(), left.end());
        if (planner->log)
            std::fprintf(stderr, "[qk plan] c128 pass S=%#llx gates=%zu (u2 %d, phase %d) ops=%d factors=%d kept=%zu\n",
                         (unsigned long long)S, taken.size(), n_u2, n_ph, P.nops, P.nfac, B.terms.size());
        if (prec == 0) {   // coefficients and factors in the working precision
            for (int i = 0; i < P.nops; ++i)
                for (int e = 0; e < 8; ++e) P.ops[i].cf[e] = (float)P.ops[i].c[e];
            for (int i = 0; i < P.nfac; ++i) P.facf[i] = make_float2((float)P.fac[i].x, (float)P.fac[i].y);
        }
        if (P.nops > 0) {
            const qk_status st = sink(P);
            if (st != QK_OK) return st;
        }
        std::copy(F1, F1 + 64, F);
        lam = lam1;
        rem.swap(next);
        lim = TakeLimits{m, kSmemTileOps, 4096};
    }
    return QK_OK;
}

namespace {
}  // namespace

qk_status plan_passes(TilePlanner *planner, int n, const std::vector<FusedOp> &ops, const PassSink &sink,
                      const char **err) {
    *err = "";
    std::vector<POp> rem;
    rem.reserve(ops.size());
    for (const auto &op : ops) rem.push_back(classify(op));

    // take limits per pass; halved and retried when a program overflows the
    // kernel-parameter budget (ops and grouped phase entries)
    int max_u2 = 100, max_ph = 300;
    std::vector<POp> left, taken;
    // the uniform pending factors one pass leaves to the next (FP64): per physical
    // qubit, on its |1> (a phase and a magnitude), plus a constant phase and a real
    // scale; only the plan's last pass applies them to the amplitudes
    double carry[64] = {0.0};
    double carry_mag[64];
    for (double &m : carry_mag) m = 1.0;
    double carry_u0 = 0.0, carry_lam = 1.0;
    std::vector<Cond> conds;
    while (!rem.empty()) {
        int n_u2 = 0, n_ph = 0;
        const uint64_t S = choose_pass(rem, n, TakeLimits{kTileQubits, max_u2, max_ph}, kTileContig, conds, taken, left,
                                       &n_u2, &n_ph);

        static thread_local TileParams P;
        std::memset(static_cast<TileHead *>(&P), 0, sizeof(TileHead));
        P.n = n;
        P.n_tiles = 1ull << (n - kTileQubits);
        int local_of[64];
        for (int b = 0; b < 64; ++b) local_of[b] = -1;
        {
            int lb = 0, fb = 0;
            for (int b = 0; b < n; ++b) {
                if ((S >> b) & 1) {
                    P.S[lb] = (int8_t)b;
                    local_of[b] = lb++;
                } else {
                    P.fixed[fb++] = (int8_t)b;
                }
            }
            P.nfix = fb;
            // runs of consecutive fixed qubits
            P.nruns = 0;
            for (int b = 0; b < fb;) {
                int e = b + 1;
                while (e < fb && P.fixed[e] == P.fixed[e - 1] + 1) ++e;
                if (P.nruns >= kTileMaxRuns) {
                    *err = "internal: too many fixed-qubit runs";
                    return QK_EINVAL;
                }
                P.run_tlo[P.nruns] = (uint8_t)b;
                P.run_len[P.nruns] = (uint8_t)(e - b);
                P.run_plo[P.nruns] = (uint8_t)P.fixed[b];
                ++P.nruns;
                b = e;
            }
        }
        P.n_conds = (int)conds.size();
        for (int k = 0; k < P.n_conds; ++k) P.conds[k] = conds[k];

        // ---- list-schedule the taken gates over the arrangements
        const int m = (int)taken.size();
        // dependency edges i -> j (i < j, not commuting) as flat successor lists:
        // the successors of i are succ[succ_at[i] .. succ_at[i + 1])
        static thread_local std::vector<int> npred, succ_at, succ, edge_i, edge_j;
        npred.assign(m, 0);
        succ_at.assign(m + 1, 0);
        edge_i.clear();
        edge_j.clear();
        for (int j = 0; j < m; ++j)
            for (int i = 0; i < j; ++i)
                if (!commute(taken[i], taken[j])) {
                    npred[j]++;
                    succ_at[i + 1]++;
                    edge_i.push_back(i);
                    edge_j.push_back(j);
                }
        for (int i = 0; i < m; ++i) succ_at[i + 1] += succ_at[i];
        succ.resize(edge_i.size());
        {
            static thread_local std::vector<int> fill;
            fill.assign(succ_at.begin(), succ_at.end() - 1);
            for (size_t e = 0; e < edge_i.size(); ++e) succ[fill[edge_i[e]]++] = edge_j[e];   // ascending j per i
        }
        std::vector<char> done(m, 0);
        int ndone = 0, cur = ARR_IO, nops = 0;
        static thread_local std::vector<TileOp> prog;
        prog.assign(2 * (size_t)m + 2, TileOp{});
        auto emit = [&](int j, int arr) {
            const FusedOp &op = *taken[j].op;
            TileOp &t = prog[nops++];
            std::memset(&t, 0, sizeof t);
            t.cond = 0xffff;
            if (op.cond.n)
                for (int k = 0; k < P.n_conds; ++k)
                    if (same_cond(P.conds[k], op.cond)) t.cond = (uint16_t)k;
            if (op.kind == FusedOp::U2) {
                t.kind = TOP_U2;
                int pos;
                slot_of(arr, local_of[op.q], &pos);
                t.k = (uint8_t)pos;
                t.first = (uint16_t)j;   // the FP64 matrix: taken[j]
                encode_cond(op.cmask, op.cmask, arr, local_of, t);
                for (int e = 0; e < 4; ++e) {
                    t.m[2 * e] = (float)op.m[e].real();
                    t.m[2 * e + 1] = (float)op.m[e].imag();
                }
            } else {
                t.kind = TOP_PHASE;
                encode_cond(op.mask, op.val, arr, local_of, t);
                t.ph.re = (float)op.f.real();
                t.ph.im = (float)op.f.imag();
                // the factor's angle as a fraction of a turn in 32-bit fixed point
                double frac = std::arg(op.f) / (2.0 * M_PI);
                if (frac < 0) frac += 1.0;
                t.ph.turns = (uint32_t)(uint64_t)std::llround(frac * 4294967296.0);
            }
            done[j] = 1;
            ++ndone;
            for (int e = succ_at[j]; e < succ_at[j + 1]; ++e) npred[succ[e]]--;
        };
        while (ndone < m) {
            bool progress = false;
            for (int j = 0; j < m; ++j)
                if (!done[j] && npred[j] == 0 && executable(taken[j], cur, local_of)) {
                    emit(j, cur);
                    progress = true;
                }
            if (ndone == m) break;
            if (!progress) {
                int best = -1, best_cnt = -1;
                for (int a = 0; a < 3; ++a) {
                    if (a == cur) continue;
                    int cntr = 0;
                    for (int j = 0; j < m; ++j)
                        if (!done[j] && npred[j] == 0 && executable(taken[j], a, local_of)) ++cntr;
                    if (cntr > best_cnt) {
                        best_cnt = cntr;
                        best = a;
                    }
                }
                TileOp &t = prog[nops++];
                std::memset(&t, 0, sizeof t);
                t.kind = TOP_XPOSE;
                t.k = (uint8_t)best;
                t.cond = 0xffff;
                cur = best;
            }
        }
        if (cur == ARR_LO) {
            TileOp &t = prog[nops++];
            std::memset(&t, 0, sizeof t);
            t.kind = TOP_XPOSE;
            t.k = ARR_IO;
            t.cond = 0xffff;
            cur = ARR_IO;
        }
        // group runs of consecutive diagonal terms by the pending sum they feed
        {
            static thread_local TileOp out[2 * kTileMaxOps + 8];
            int nout = 0, nlin = 0;
            int fixed_index[64];   // physical qubit -> bit of the tile index
            for (int b = 0; b < 64; ++b) fixed_index[b] = -1;
            for (int b = 0; b < P.nfix; ++b) fixed_index[(int)P.fixed[b]] = b;
            bool overflow = false;
            for (int i = 0; i < nops && !overflow;) {
                if (nout >= 2 * kTileMaxOps) {
                    overflow = true;
                    break;
                }
                if (prog[i].kind != TOP_PHASE) {
                    out[nout++] = prog[i++];
                    continue;
                }
                int j = i;
                while (j < nops && prog[j].kind == TOP_PHASE) ++j;
                // per pending sum (register bit 0..4, constant 5): entries that add turns
                struct Term {
                    uint16_t tmask, tval;
                    uint32_t turns;
                    uint64_t gmask, gval;
                };
                std::vector<Term> grp[6];
                // terms on two register bits, reduced to the (1,1) pattern: key -> turns
                struct PairKey {
                    int code;
                    uint16_t tmask, tval;
                    uint64_t gmask, gval;
                    uint32_t turns;
                };
                std::vector<PairKey> pairs;
                auto add_entry = [&](int g, const TileOp &o, uint32_t turns) {
                    Term e;
                    e.tmask = o.tmask;
                    e.tval = o.tval;
                    e.gmask = o.gmask;
                    e.gval = o.gval;
                    e.turns = turns;
                    grp[g].push_back(e);
                };
                for (int t = i; t < j; ++t) {
                    const TileOp &o = prog[t];
                    if (nout >= 2 * kTileMaxOps) {
                        overflow = true;
                        break;
                    }
                    const int pc = __builtin_popcount(o.rmask);
                    const uint32_t T = o.ph.turns;
                    if (o.cond != 0xffff || pc >= 3) {
                        out[nout++] = o;   // applied directly
                        continue;
                    }
                    if (pc == 0) {
                        add_entry(5, o, T);
                    } else if (pc == 1) {
                        const int k = __builtin_ctz(o.rmask);
                        if (o.rval) {
                            add_entry(k, o, T);
                        } else {  // f on bit k = 0:  f * (f^-1 on bit k = 1)
                            add_entry(5, o, T);
                            add_entry(k, o, 0u - T);
                        }
                    } else {
                        // pattern (vk, vl) on register bits k < l as exact sums of a constant,
                        // single-bit terms and a (1,1) pair term
                        const int k = __builtin_ctz(o.rmask), l = 31 - __builtin_clz(o.rmask);
                        const int vk = (o.rval >> k) & 1, vl = (o.rval >> l) & 1;
                        uint32_t pair = T;
                        if (vk && !vl) {
                            add_entry(k, o, T);
                            pair = 0u - T;
                        } else if (!vk && vl) {
                            add_entry(l, o, T);
                            pair = 0u - T;
                        } else if (!vk && !vl) {
                            add_entry(5, o, T);
                            add_entry(k, o, 0u - T);
                            add_entry(l, o, 0u - T);
                        }
                        const int code = k | (l << 3);
                        bool merged = false;
                        for (auto &pk : pairs)
                            if (pk.code == code && pk.tmask == o.tmask && pk.tval == o.tval && pk.gmask == o.gmask &&
                                pk.gval == o.gval) {
                                pk.turns += pair;
                                merged = true;
                                break;
                            }
                        if (!merged) pairs.push_back({code, o.tmask, o.tval, o.gmask, o.gval, pair});
                    }
                }
                for (const auto &pk : pairs) {
                    if (pk.turns == 0) continue;
                    if (nout >= 2 * kTileMaxOps) {
                        overflow = true;
                        break;
                    }
                    TileOp &t = out[nout++];
                    std::memset(&t, 0, sizeof t);
                    t.cond = 0xffff;
                    t.k = (uint8_t)pk.code;
                    if (pk.tmask == 0 && pk.gmask == 0 && pk.turns == 0x80000000u) {
                        t.kind = TOP_PAIRNEG;   // a CZ between two register bits
                        continue;
                    }
                    t.kind = TOP_PAIR;
                    t.rval = 3;   // both bits 1
                    t.tmask = pk.tmask;
                    t.tval = pk.tval;
                    t.gmask = pk.gmask;
                    t.gval = pk.gval;
                    const double ang = 2.0 * M_PI * (double)pk.turns / 4294967296.0;
                    t.ph.re = (float)std::cos(ang);
                    t.ph.im = (float)std::sin(ang);
                    t.ph.turns = pk.turns;
                }
                for (int g = 0; g < 6 && !overflow; ++g) {
                    if (grp[g].empty()) continue;
                    // split the group's terms: the same for every thread and tile
                    // (kept by the planner), and the rest, each a linear term with
                    // its thread-bit and tile-index conditions (TOP_PHASEL)
                    uint32_t host_turns = 0;
                    std::vector<LinTerm> lins;
                    for (const Term &t : grp[g]) {
                        if (t.gmask == 0 && t.tmask == 0) {
                            host_turns += t.turns;
                            continue;
                        }
                        uint32_t fm = 0, fv = 0;   // the fixed-qubit condition on tile-index bits
                        for (uint64_t mk = t.gmask; mk; mk &= mk - 1) {
                            const int pb = __builtin_ctzll(mk), tb = fixed_index[pb];
                            fm |= 1u << tb;
                            if ((t.gval >> pb) & 1) fv |= 1u << tb;
                        }
                        bool merged = false;
                        for (auto &l : lins)
                            if (l.tmask == t.tmask && l.tval == t.tval && l.fmask == fm && l.fval == fv) {
                                l.turns += t.turns;
                                merged = true;
                                break;
                            }
                        if (!merged) {
                            LinTerm l{};
                            l.tmask = t.tmask;
                            l.tval = t.tval;
                            l.fmask = fm;
                            l.fval = fv;
                            l.turns = t.turns;
                            lins.push_back(l);
                        }
                    }
                    if (host_turns != 0) {
                        if (nout >= 2 * kTileMaxOps) { overflow = true; break; }
                        TileOp &t = out[nout++];
                        std::memset(&t, 0, sizeof t);
                        t.kind = TOP_HOSTPH;
                        t.k = (uint8_t)g;
                        t.cond = 0xffff;
                        t.ph.turns = host_turns;
                    }
                    int nl = 0;
                    for (const auto &l : lins) nl += l.turns != 0;
                    if (nl) {
                        if (nout >= 2 * kTileMaxOps || nlin + nl > kTileMaxLin) { overflow = true; break; }
                        TileOp &t = out[nout++];
                        std::memset(&t, 0, sizeof t);
                        t.kind = TOP_PHASEL;
                        t.k = (uint8_t)g;
                        t.cond = 0xffff;
                        t.first = (uint16_t)nlin;
                        for (const auto &l : lins)
                            if (l.turns != 0) P.lin[nlin++] = l;
                        t.count = (uint16_t)(nlin - t.first);
                    }
                }
                i = j;
            }
            if (overflow || nout > kTileMaxOps) {
                // too large for one launch: plan this pass again with fewer gates
                if (max_u2 <= 1 && max_ph <= 1) {
                    *err = "internal: tile program overflow";
                    return QK_EINVAL;
                }
                max_u2 = std::max(1, max_u2 / 2);
                max_ph = std::max(1, max_ph / 2);
                continue;
            }
            // merge runs of consecutive uncontrolled 2x2 gates on distinct
            // register bits into layer ops (they commute with each other)
            int nfin = 0, nmat = 0;
            static thread_local uint16_t lg_mat[kTileMaxMats];   // layer gate -> taken[] index
            for (int i = 0; i < nout && !overflow;) {
                const TileOp &o = out[i];
                const bool plain_u2 = o.kind == TOP_U2 && o.rmask == 0 && o.tmask == 0 && o.gmask == 0 &&
                                      o.cond == 0xffff;
                if (!plain_u2) {
                    if (nfin >= kTileMaxOps) { overflow = true; break; }
                    P.ops[nfin++] = out[i++];
                    continue;
                }
                int bits = 0, j = i;
                while (j < nout) {
                    const TileOp &q = out[j];
                    const bool ok = q.kind == TOP_U2 && q.rmask == 0 && q.tmask == 0 && q.gmask == 0 &&
                                    q.cond == 0xffff && !(bits & (1 << q.k));
                    if (!ok) break;
                    bits |= 1 << q.k;
                    ++j;
                }
                if (nfin >= kTileMaxOps || nmat + (j - i) > kTileMaxMats) { overflow = true; break; }
                TileOp &t = P.ops[nfin++];
                std::memset(&t, 0, sizeof t);
                t.kind = TOP_U2L;
                t.k = (uint8_t)bits;
                t.cond = 0xffff;
                t.first = (uint16_t)nmat;
                t.count = (uint16_t)(j - i);
                // the gates' FP64 matrices in register-bit order; fold_program turns
                // them into pivot coefficients
                for (int b = 0; b < 5; ++b)
                    for (int q = i; q < j; ++q)
                        if (out[q].k == b) lg_mat[nmat++] = out[q].first;
                i = j;
            }
            if (overflow) {
                if (max_u2 <= 1 && max_ph <= 1) {
                    *err = "internal: tile program overflow";
                    return QK_EINVAL;
                }
                max_u2 = std::max(1, max_u2 / 2);
                max_ph = std::max(1, max_ph / 2);
                continue;
            }
            // fold_program: walk the program in order, keeping the pending phases
            // that are the same for every thread (and the scale and the stored bit
            // order of each local qubit) in FP64; layer gates get their pivot
            // coefficients, every other op's conditions are rewritten to the stored
            // order, general gates take their target's uniform phase along to the
            // device, and what is left goes to the final flush
            {
                UniformPending st;
                for (int q = 0; q < kTileQubits; ++q) {
                    st.u[q] = carry[(int)P.S[q]];
                    st.mag[q] = carry_mag[(int)P.S[q]];
                }
                st.u0 = carry_u0;
                st.lam = carry_lam;
                int arr = ARR_IO, w = 0;
                const double pi = M_PI;
                for (int i = 0; i < nfin; ++i) {
                    TileOp o = P.ops[i];
                    // flipped register and thread bits in the current arrangement
                    int rflip = 0, tflip = 0;
                    for (int k = 0; k < 5; ++k) rflip |= st.flip[local_of_reg(arr, k)] << k;
                    for (int t = 0; t < 8; ++t) tflip |= st.flip[local_of_tbit(arr, t)] << t;
                    auto qk_of = [&](int k) { return local_of_reg(arr, k); };
                    switch (o.kind) {
                        case TOP_HOSTPH: {
                            const double ang = turns_angle(o.ph.turns);
                            if (o.k == 5) {
                                st.u0 += ang;
                            } else if (st.flip[qk_of(o.k)]) {  // on the stored |0>
                                st.u0 += ang;
                                st.u[qk_of(o.k)] -= ang;
                            } else {
                                st.u[qk_of(o.k)] += ang;
                            }
                            continue;   // never reaches the device
                        }
                        case TOP_XPOSE:
                            arr = o.k;
                            break;
                        case TOP_U2L: {
                            int idx = o.first;
                            for (int b = 0; b < 5; ++b) {
                                if (!((o.k >> b) & 1)) continue;
                                const FusedOp &fo = *taken[lg_mat[idx]].op;
                                const Mat2 g{{fo.m[0], fo.m[1], fo.m[2], fo.m[3]}};
                                if (pivot_gate(g, st, qk_of(b), P.lg[idx])) o.rmask |= (uint8_t)(1u << b);
                                ++idx;
                            }
                            break;
                        }
                        case TOP_PAIRNEG: {
                            // (-1)^((a^fa)(b^fb)) = (-1)^(ab) (-1)^(fb a) (-1)^(fa b) (-1)^(fa fb)
                            const int ka = o.k & 7, kb = o.k >> 3;
                            const int fa = (rflip >> ka) & 1, fb = (rflip >> kb) & 1;
                            if (fb) st.u[qk_of(ka)] += pi;
                            if (fa) st.u[qk_of(kb)] += pi;
                            if (fa && fb) st.u0 += pi;
                            break;
                        }
                        case TOP_PAIR: {
                            const int ka = o.k & 7, kb = o.k >> 3;
                            const int fa = (rflip >> ka) & 1, fb = (rflip >> kb) & 1;
                            o.tval ^= (uint16_t)(o.tmask & tflip);
                            if (o.tmask == 0 && o.gmask == 0 && o.cond == 0xffff) {
                                // e^{i th} where the true bits a = sa ^ fa, b = sb ^ fb are both
                                // 1, in stored bits: (sa ^ fa)(sb ^ fb) = fa fb + fa (1 - 2 fb) sb
                                // + fb (1 - 2 fa) sa + (1 - 2 fa)(1 - 2 fb) sa sb.  The stored
                                // pattern (1, 1) takes +-th on the device; the constant and the
                                // single-bit parts are uniform phases kept here.
                                const double th = turns_angle(o.ph.turns);
                                if (fa && fb) st.u0 += th;
                                if (fa) st.u[qk_of(kb)] += fb ? -th : th;
                                if (fb) st.u[qk_of(ka)] += fa ? -th : th;
                                if (fa ^ fb) {
                                    o.ph.turns = 0u - o.ph.turns;
                                    o.ph.im = -o.ph.im;
                                }
                                o.rval = 3;
                                o.kind = TOP_PAIRU;
                            } else {
                                o.rval = (uint8_t)(3 ^ (fa | (fb << 1)));
                            }
                            break;
                        }
                        case TOP_PHASEL: {
                            for (int e = o.first; e < o.first + o.count; ++e)
                                P.lin[e].tval ^= (uint16_t)(P.lin[e].tmask & tflip);
                            o.rval = (uint8_t)(o.k < 5 ? (rflip >> o.k) & 1 : 0);
                            // every term tests one bit: "turns where the bit is 1" terms
                            // (TOP_PHASEB), a term on a bit being 0 split into a
                            // constant kept here and a negated bit-1 term
                            bool single = true;
                            for (int e = o.first; e < o.first + o.count; ++e)
                                single = single && __builtin_popcount(P.lin[e].tmask) + __builtin_popcount(P.lin[e].fmask) == 1;
                            if (!single) break;
                            std::vector<BitTerm> th, ti;
                            uint32_t cst = 0;
                            for (int e = o.first; e < o.first + o.count; ++e) {
                                const LinTerm &L = P.lin[e];
                                const bool thread = L.tmask != 0;
                                const uint32_t b = thread ? (uint32_t)__builtin_ctz(L.tmask) : (uint32_t)__builtin_ctz(L.fmask);
                                const uint32_t v = thread ? ((uint32_t)L.tval >> b) & 1u : (L.fval >> b) & 1u;
                                uint32_t t = L.turns;
                                if (!v) {
                                    cst += t;
                                    t = 0u - t;
                                }
                                (thread ? th : ti).push_back(BitTerm{b, t});
                            }
                            BitTerm *bt = reinterpret_cast<BitTerm *>(&P.lin[o.first]);
                            for (size_t q = 0; q < th.size(); ++q) bt[q] = th[q];
                            for (size_t q = 0; q < ti.size(); ++q) bt[th.size() + q] = ti[q];
                            o.kind = TOP_PHASEB;
                            o.first = (uint16_t)(2 * o.first);
                            o.count = (uint16_t)th.size();
                            o.count2 = (uint16_t)ti.size();
                            if (cst) {   // the same for every thread and tile: kept here
                                const double ang = turns_angle(cst);
                                if (o.k == 5) {
                                    st.u0 += ang;
                                } else if (st.flip[qk_of(o.k)]) {
                                    st.u0 += ang;
                                    st.u[qk_of(o.k)] -= ang;
                                } else {
                                    st.u[qk_of(o.k)] += ang;
                                }
                            }
                            break;
                        }
                        case TOP_PHASE:
                            o.rval ^= (uint8_t)(o.rmask & rflip);
                            o.tval ^= (uint16_t)(o.tmask & tflip);
                            break;
                        case TOP_U2: {
                            const int q = qk_of(o.k);
                            o.rval ^= (uint8_t)(o.rmask & rflip);
                            o.tval ^= (uint16_t)(o.tmask & tflip);
                            if (st.flip[q]) {  // X U X in stored order
                                float t[8];
                                std::memcpy(t, o.m, sizeof t);
                                const int perm[4] = {3, 2, 1, 0};
                                for (int e = 0; e < 4; ++e) {
                                    o.m[2 * e] = t[2 * perm[e]];
                                    o.m[2 * e + 1] = t[2 * perm[e] + 1];
                                }
                            }
                            o.hturns = angle_turns(st.u[q]);
                            o.hmag = (float)st.mag[q];
                            st.u[q] = 0.0;
                            st.mag[q] = 1.0;
                            break;
                        }
                        default:
                            break;
                    }
                    P.ops[w++] = o;
                }
                nfin = w;
                // a CZ between register bits right after a layer op (nothing between
                // them) becomes a bit of that op's CZ mask: one dispatch fewer
                w = 0;
                for (int i = 0; i < nfin; ++i) {
                    const TileOp &o = P.ops[i];
                    if (o.kind == TOP_PAIRNEG && w > 0 && P.ops[w - 1].kind == TOP_U2L) {
                        P.ops[w - 1].tmask |= (uint16_t)(1u << cz_index(o.k & 7, o.k >> 3));
                        continue;
                    }
                    P.ops[w++] = o;
                }
                nfin = w;
                P.fin_flip = 0;
                for (int q = 0; q < kTileQubits; ++q) P.fin_flip |= st.flip[q] << q;
                P.fin_fixed_mask = 0;
                if (left.empty()) {   // the plan's last pass applies everything pending
                    for (int q = 0; q < kTileQubits; ++q) {
                        P.fin_turns[q] = angle_turns(st.u[q]);
                        P.fin_mag[q] = (float)st.mag[q];
                    }
                    P.fin_turns[13] = angle_turns(st.u0);
                    P.fin_scale = (float)st.lam;
                    for (int b = 0; b < P.nfix; ++b) {
                        const uint32_t t = angle_turns(carry[(int)P.fixed[b]]);
                        P.fin_fixed[b] = t;
                        P.fin_fixed_mag[b] = (float)carry_mag[(int)P.fixed[b]];
                        if (t || P.fin_fixed_mag[b] != 1.f) P.fin_fixed_mask |= 1ull << b;
                    }
                } else {              // hand the uniform part to the next pass
                    for (int q = 0; q < kTileQubits; ++q) {
                        // a qubit stored flipped has its factor F on |0>: F on |0> is F
                        // overall times 1 / F on |1>
                        const int pq = (int)P.S[q];
                        if (st.flip[q]) {
                            carry[pq] = -st.u[q];
                            carry_mag[pq] = 1.0 / st.mag[q];
                            st.u0 += st.u[q];
                            st.lam *= st.mag[q];
                        } else {
                            carry[pq] = st.u[q];
                            carry_mag[pq] = st.mag[q];
                        }
                        P.fin_turns[q] = 0;
                        P.fin_mag[q] = 1.f;
                    }
                    carry_u0 = st.u0;
                    P.fin_turns[13] = 0;
                    // the stored amplitudes are the true ones divided by the scale
                    // (a factor in [2^-1/2, 2] per gate): keep them within 2^24 of it
                    // in FP32
                    if (st.lam < 0x1p-24 || st.lam > 0x1p24) {
                        P.fin_scale = (float)st.lam;
                        carry_lam = 1.0;
                    } else {
                        P.fin_scale = 1.f;
                        carry_lam = st.lam;
                    }
                }
            }
            nops = nfin;
            P.nlg = nmat;
            P.nlin = nlin;
            // whether any phase factor the pass forms can be other than 1 or -1 (the
            // kernel fills its phase table only then)
            {
                auto general = [](uint32_t t) { return t != 0u && t != 0x80000000u; };
                bool need = false;
                for (int i = 0; i < nops && !need; ++i) {
                    const TileOp &o = P.ops[i];
                    if (o.kind == TOP_U2 || o.kind == TOP_PHASE) need = true;
                    if (o.kind == TOP_PHASEL)
                        for (int e = o.first; e < o.first + o.count; ++e) need = need || general(P.lin[e].turns);
                    if (o.kind == TOP_PHASEB) {
                        const BitTerm *bt = reinterpret_cast<const BitTerm *>(&P.lin[0]) + o.first;
                        for (int e = 0; e < o.count + o.count2; ++e) need = need || general(bt[e].turns);
                    }
                }
                for (int q = 0; q < 14; ++q) need = need || general(P.fin_turns[q]);
                for (int b = 0; b < P.nfix; ++b)
                    if ((P.fin_fixed_mask >> b) & 1) need = need || general(P.fin_fixed[b]);
                P.need_tab = need ? 1 : 0;
            }
        }
        P.nops = nops;
        P.store_arr = cur;
        if (planner->log) {
            int cnt_k[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // by TileOpKind
            for (int i = 0; i < nops; ++i) cnt_k[P.ops[i].kind]++;
            std::fprintf(stderr,
                         "[qk plan] pass S=%#llx gates=%d (u2 %d, phase %d) ops=%d u2=%d layers=%d phase_direct=%d "
                         "phase_groups=%d terms=%d pairs=%d pair_signs=%d xpose=%d store_arr=%d\n",
                         (unsigned long long)S, m, n_u2, n_ph, nops, cnt_k[TOP_U2], cnt_k[TOP_U2L], cnt_k[TOP_PHASE],
                         cnt_k[TOP_PHASEL], P.nlin, cnt_k[TOP_PAIR], cnt_k[TOP_PAIRNEG], cnt_k[TOP_XPOSE], cur);
        }

        const qk_status st = sink(P);
        if (st != QK_OK) return st;
        rem.swap(left);
        max_u2 = 100;
        max_ph = 300;
    }
    return QK_OK;
}

// A dense pass: S starts as the lowest qubits (runs of 128 bytes in HBM, 32 for states in
// L2) and takes the targets of every gate, in order, that commutes with the gates left
// behind, has the first one's k and still fits.  A pass of one controlled gate enumerates only the tiles whose
// control bits are set.  Fewer amplitudes per tile for small states, so that there are
// tiles for all SMs.
qk_status plan_dense(int n, int prec, const std::vector<DenseItem> &ops, const DenseSink &sink) {
    std::vector<const DenseItem *> rem, left, taken;
    for (const DenseItem &it : ops) rem.push_back(&it);
    while (!rem.empty()) {
        left.clear();
        taken.clear();
        static thread_local DenseParams P;
        std::memset(static_cast<void *>(&P), 0, offsetof(DenseParams, ops));
        // complex64 gates of 5 and 6 qubits form 8 rows per thread, which takes 2^13
        // amplitudes to give every thread columns
        int m = prec != 0 ? 11 : rem[0]->k >= 5 ? 13 : 12;
        if (n < 20) m = std::min(m, n >= 18 ? 11 : n >= 16 ? 10 : 9);
        m = std::min(m, n);
        const int contig = std::min(m, n >= 23 ? 4 : 2);
        uint64_t S = 0, left_t = 0, left_all = 0;
        int elems = 0;
        const uint64_t low = (1ull << contig) - 1;
        for (const DenseItem *it : rem) {
            const uint64_t all = it->tmask | it->cmask;
            bool ok = (int)taken.size() < kDenseOps && it->k == rem[0]->k &&
                      elems + (1 << (2 * it->k)) <= kDenseElems &&
                      !(it->tmask & left_all) && !(all & left_t);
            // the first gate may use the room of the low qubits
            if (ok && __builtin_popcountll(S | it->tmask | (taken.empty() ? 0 : low)) > m) ok = false;
            int ci = -1;
            if (ok && it->cond.n) {
                for (int k = 0; k < P.n_conds; ++k)
                    if (same_cond(P.conds[k], it->cond)) ci = k;
                if (ci < 0 && P.n_conds >= kTileMaxConds) ok = false;
                else if (ci < 0) {
                    ci = P.n_conds++;
                    P.conds[ci] = it->cond;
                }
            }
            if (!ok) {
                left.push_back(it);
                left_t |= it->tmask;
                left_all |= all;
                continue;
            }
            S |= it->tmask;
            elems += 1 << (2 * it->k);
            taken.push_back(it);
        }
        const uint64_t lone = taken.size() == 1 ? taken[0]->cmask : 0;   // enumerated only where set
        for (int b = 0; b < n && __builtin_popcountll(S) < m; ++b)
            if (!((S | lone) >> b & 1)) S |= 1ull << b;
        P.m = __builtin_popcountll(S);
        P.base = lone;
        int local_of[64], tile_of[64];
        for (int b = 0, lb = 0; b < n; ++b) {
            local_of[b] = tile_of[b] = -1;
            if ((S >> b) & 1) {
                P.S[lb] = (int8_t)b;
                local_of[b] = lb++;
            } else if (!((lone >> b) & 1)) {
                P.fixed[P.nfix] = (int8_t)b;
                tile_of[b] = P.nfix++;
            }
        }
        P.n_tiles = 1ull << P.nfix;
        P.k = rem[0]->k;
        for (const DenseItem *const &it : taken) {
            DenseOp &o = P.ops[P.nops++];
            std::memset(static_cast<void *>(&o), 0, sizeof o);
            uint32_t used = 0;
            for (int b = 0; b < it->k; ++b) {
                const int lb = local_of[it->tpos[it->k - 1 - b]];
                o.ts[b] = (uint16_t)dense_slot(1u << lb);
                used |= 1u << lb;
            }
            o.cond = 0xff;
            if (it->cond.n)
                for (int k = 0; k < P.n_conds; ++k)
                    if (same_cond(P.conds[k], it->cond)) o.cond = (uint8_t)k;
            for (uint64_t c = it->cmask & ~lone; c; c &= c - 1) {
                const int b = __builtin_ctzll(c);
                if (local_of[b] >= 0) {
                    o.ls ^= (uint16_t)dense_slot(1u << local_of[b]);
                    used |= 1u << local_of[b];
                } else {
                    o.tmask |= 1u << tile_of[b];
                }
            }
            // two 2-qubit gates in a row on other qubits, both unconditional: one round trip
            // through shared memory.  The first one's column bits are the second's register
            // bits (or, for one gate alone, its last free bits).
            const bool joined = P.nops >= 2 && P.ops[P.nops - 2].pair;
            const bool free2 = it->k == 2 && !it->cmask && !it->cond.n;
            o.pair = 0;
            if (free2 && !joined && &it != &taken.back()) {
                const DenseItem *nx = (&it)[1];
                if (!nx->cmask && !nx->cond.n && !(nx->tmask & it->tmask)) {
                    o.pair = 1;
                    o.ncs = 2;
                    for (int b = 0; b < 2; ++b) {
                        const int lb = local_of[nx->tpos[1 - b]];
                        o.cs[b] = (uint16_t)dense_slot(1u << lb);
                        used |= 1u << lb;
                    }
                }
            }
            // free bits: lanes walk the first ones, so those go to distinct banks (bit mod 4)
            uint32_t banks = 0, placed = used;
            for (int pass = 0; pass < 2; ++pass)
                for (int b = 0; b < P.m; ++b) {
                    if ((placed >> b) & 1u) continue;
                    if (pass == 0 && ((banks >> (b & 3)) & 1u)) continue;
                    banks |= 1u << (b & 3);
                    placed |= 1u << b;
                    o.fs[o.nfree++] = (uint16_t)dense_slot(1u << b);
                }
            if (it->k == 2 && !o.pair)
                while (o.ncs < 2 && o.nfree > 0) o.cs[o.ncs++] = o.fs[--o.nfree];
            o.mat = it->mat;
        }
        const qk_status st = sink(P);
        if (st != QK_OK) return st;
        rem.swap(left);
    }
    return QK_OK;
}

qk_status run_fused(TilePlanner *planner, qk_ctx *c, const std::vector<FusedOp> &ops) {
    const int n = ctx_n(c);
    const int prec = ctx_prec(c);
    if (prec != 0 || n < kTileQubits) {
        const SmemPassSink launch = [&](SmemTileParams &P) -> qk_status {
            void *tok = nullptr;
            ctx_launch_begin(c, 0, (prec == 0 ? 2.0 * 8.0 : 2.0 * 16.0) * (double)(1ull << n), &tok);
            const cudaError_t e = launch_smem_tile(prec, ctx_state(c), P, ctx_cbits(c), ctx_stream(c));
            ctx_launch_end(tok);
            return e == cudaSuccess ? QK_OK : ctx_fail(c, QK_ECUDA, cudaGetErrorString(e));
        };
        const char *err = "";
        const qk_status st = plan_smem_passes(planner, n, prec, ops, launch, &err);
        if (st != QK_OK && err[0]) return ctx_fail(c, st, err);
        return st;
    }
    const PassSink launch = [&](TileParams &P) -> qk_status {
        void *tok = nullptr;
        cudaEvent_t ev0 = nullptr, ev1 = nullptr;
        if (planner->log) {  // trace mode: time this pass on its own (synchronous)
            cudaEventCreate(&ev0);
            cudaEventCreate(&ev1);
            cudaEventRecord(ev0, ctx_stream(c));
        }
        ctx_launch_begin(c, 0, 2.0 * 8.0 * (double)(1ull << n), &tok);
        cudaError_t e = launch_tile(ctx_state(c), P, ctx_cbits(c), ctx_stream(c));
        ctx_launch_end(tok);
        if (e != cudaSuccess) return ctx_fail(c, QK_ECUDA, cudaGetErrorString(e));
        if (planner->log) {
            float ms = 0.f;
            cudaEventRecord(ev1, ctx_stream(c));
            cudaEventSynchronize(ev1);
            cudaEventElapsedTime(&ms, ev0, ev1);
            std::fprintf(stderr, "[qk plan]   %.3f ms\n", ms);
            cudaEventDestroy(ev0);
            cudaEventDestroy(ev1);
        }
        return QK_OK;
    };
    const char *err = "";
    const qk_status st = plan_passes(planner, n, ops, launch, &err);
    if (st != QK_OK && err[0]) return ctx_fail(c, st, err);
    return st;
}

}  // namespace qk
