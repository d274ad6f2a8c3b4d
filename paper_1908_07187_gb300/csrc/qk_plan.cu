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
// The program's builder (TileBuilder) keeps, in double precision, every single-qubit
// diagonal factor -- one complex factor per qubit, and one for all amplitudes -- and the
// diagonal terms on two qubits: a term waits until a gate acts on one of its qubits and
// is applied there, so the device carries no phases from op to op.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <complex>
#include <cstring>
#include <deque>
#include <tuple>
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

// Storage that a thread keeps from plan to plan is given back after a queue far beyond the
// default length of 4096 ops.
template <typename... V>
struct GiveBack {
    std::tuple<V &...> kept;
    explicit GiveBack(V &...v) : kept(v...) {}
    ~GiveBack() {
        std::apply([](V &...v) { ((v.capacity() > (1u << 16) ? V().swap(v) : void()), ...); }, kept);
    }
};

struct POp {
    const FusedOp *op;
    uint64_t nd;   // non-diagonal qubits
    uint64_t all;  // every qubit the op depends on
    bool u2, cond; // what the walks over long lists ask, without touching the op
};

POp classify(const FusedOp &op) {
    POp p;
    p.op = &op;
    p.u2 = op.kind == FusedOp::U2;
    p.cond = op.cond.n != 0;
    if (op.kind == FusedOp::U2) {
        p.nd = 1ull << op.q;
        p.all = p.nd | op.cmask;
    } else {
        p.nd = 0;
        p.all = op.mask;
    }
    return p;
}

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

using cdm = std::complex<double>;

// Double-double complex numbers (Dekker; products by FMA) for the factors that a complex128
// plan keeps pending: they go through a product per gate, and in plain doubles the rounding
// errors of that chain, the same for every amplitude, were most of a fused circuit's error.
// Layers, 290 gates on 12 qubits, against the same matrices in extended precision: 2.2e-15 in
// doubles, 1.6e-15 with these, 1.2e-15 with a gate's direction taken from both off-diagonal
// entries (SmemTileBuilder::gate); gate by gate 1.0e-15.  Planning takes the same time: the
// form needs no trigonometric functions.
struct DD {
    double h = 0.0, l = 0.0;
};
inline DD quick_sum(double a, double b) {      // |a| >= |b|
    const double s = a + b;
    return {s, b - (s - a)};
}
inline DD operator+(DD a, DD b) {
    const double s = a.h + b.h, t = s - a.h;
    return quick_sum(s, (a.h - (s - t)) + (b.h - t) + (a.l + b.l));
}
inline DD operator-(DD a) { return {-a.h, -a.l}; }
inline DD operator-(DD a, DD b) { return a + -b; }
inline DD operator*(DD a, DD b) {
    const double p = a.h * b.h;
    return quick_sum(p, std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
inline DD operator/(DD a, DD b) {
    const double q = a.h / b.h;
    const DD r = a - b * DD{q, 0.0};
    return quick_sum(q, r.h / b.h);
}
struct DDC {
    DD re, im;
    DDC(double r = 0.0) : re{r, 0.0} {}
    DDC(DD r, DD i) : re(r), im(i) {}
    explicit DDC(cdm z) : re{z.real(), 0.0}, im{z.imag(), 0.0} {}
    explicit operator cdm() const { return {re.h, im.h}; }
    DDC &operator/=(DD x) {
        re = re / x;
        im = im / x;
        return *this;
    }
    DDC &operator*=(const DDC &b) {
        const DD r = re * b.re - im * b.im;
        im = re * b.im + im * b.re;
        re = r;
        return *this;
    }
    DDC &operator/=(const DDC &b) {
        const DD n = b.re * b.re + b.im * b.im;
        *this *= DDC(b.re, -b.im);
        return *this /= n;
    }
};
inline DDC operator*(DDC a, const DDC &b) { return a *= b; }
inline DDC operator/(DDC a, const DDC &b) { return a /= b; }
// the same for either kind of factor: parts, rounding, making one of parts
inline DD real_of(const DDC &z) { return z.re; }
inline DD imag_of(const DDC &z) { return z.im; }
inline double real_of(const cdm &z) { return z.real(); }
inline double imag_of(const cdm &z) { return z.imag(); }
inline double rounded(DD x) { return x.h; }
inline double rounded(double x) { return x; }
template <typename X> struct RealOf { using T = double; };
template <> struct RealOf<DDC> { using T = DD; };
inline DD real_from(double x, DD) { return {x, 0.0}; }
inline double real_from(double x, double) { return x; }
template <typename X> X turned(const X &z, int k) {   // i^k z
    const auto r = real_of(z), m = imag_of(z);
    return (k & 3) == 0 ? z : (k & 3) == 1 ? X(-m, r) : (k & 3) == 2 ? X(-r, -m) : X(m, -r);
}

// A diagonal term that is not yet in a program: f where (index & mask) == val.
struct DTerm {
    uint64_t mask, val;
    cdm f;
    const Cond *cond;
    const FusedOp *src;      // the queued op that it is, if none of it became pending
};

// What a pass program's builder keeps off the device.  Single-qubit diagonal factors
// never reach it: F[q] is the pending complex factor of physical qubit q's |1>, lam the
// one of every amplitude.  Diagonal terms on more qubits wait in terms until a gate
// acts on one of their qubits and go out together there.  Pending factors are divided
// by, and a matrix defined with a wide tolerance may hold any entry, 0 among them: a
// factor far from magnitude 1, or one that would take F[q] far from it, waits in terms
// as it is, also on a single qubit.
template <typename X>      // cdm or DDC
struct PendingTerms {
    X *F;
    X &lam;
    std::vector<DTerm> terms;

    PendingTerms(X *f, X &l) : F(f), lam(l) {}

    // a term of the queue: single-qubit and constant parts become pending factors, a
    // two-qubit term keeps only its (1, 1) pattern
    void diagonal(const POp &p) {
        const FusedOp &op = *p.op;
        DTerm t{op.mask, op.val, op.f, op.cond.n ? &op.cond : nullptr, &op};
        const int k = __builtin_popcountll(t.mask);
        if (t.cond || k > 2 || (k == 2 && t.val == t.mask) || !moderate(t.f, 0x1p8) || !room(t.mask)) {
            terms.push_back(t);
            return;
        }
        const X f(t.f);
        if (k == 0) {
            lam *= f;
            return;
        }
        const int a = __builtin_ctzll(t.mask), b = 63 - __builtin_clzll(t.mask);
        const int va = (int)(t.val >> a) & 1, vb = (int)(t.val >> b) & 1;
        if (k == 1) {
            if (va) F[a] *= f;
            else {
                lam *= f;
                F[a] /= f;
            }
            return;
        }
        if (va && !vb) F[a] *= f;
        if (!va && vb) F[b] *= f;
        if (!va && !vb) {
            lam *= f;
            F[a] /= f;
            F[b] /= f;
        }
        t.src = nullptr;
        if (va != vb) t.f = 1.0 / t.f;
        t.val = t.mask;
        terms.push_back(t);
    }
    // |f| within [1 / lim, lim]; not so for 0 and NaN
    static bool moderate(cdm f, double lim) {
        const double a = std::norm(f);
        return a >= 1.0 / (lim * lim) && a <= lim * lim;
    }
    // whether the pending factors of these qubits can take one more factor
    bool room(uint64_t qubits) const {
        for (; qubits; qubits &= qubits - 1)
            if (!moderate(cdm(F[__builtin_ctzll(qubits)]), 0x1p40)) return false;
        return moderate(cdm(lam), 0x1p300);
    }
    static bool is_pair(const DTerm &t) { return !t.cond && t.val == t.mask && __builtin_popcountll(t.mask) == 2; }
    static bool is_sign(const DTerm &t) { return t.f == cdm(-1.0, 0.0); }
    // the waiting terms as queue entries for a later pass; rewritten holds those that
    // are not queued ops as they stand
    void hand_on(std::vector<POp> &next, std::deque<FusedOp> &rewritten) const {
        for (const DTerm &t : terms) {
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
    }
};

// How a 2x2 gate M on a qubit with pending factor f (on the stored |1>) is run: W is M
// or, with sw, X M (the rows exchanged so that the larger entries are on the diagonal);
// the true outputs are p0 and p1 times the values the device leaves.  a0 = W01 f / W00,
// a1 = W10 / (W11 f); r0 = |a0|, r1 = |a1|, a0 = r0 e^{i psi} and a1 = -r1 e^{-i psi} for a
// unitary M.  s = 1 / (1 + r0 r1) is what updating one value from the other in place
// leaves on the value updated second.
struct GateForm {
    bool sw;
    cdm p0, p1;
    double r0, r1, psi, s;
};
GateForm gate_form(const cdm *M, cdm f) {
    cdm W[4] = {M[0], M[1], M[2], M[3]};
    GateForm g;
    g.sw = std::abs(W[0]) < std::abs(W[2]);
    if (g.sw) {
        std::swap(W[0], W[2]);
        std::swap(W[1], W[3]);
    }
    const cdm a0 = W[1] * f / W[0], a1 = W[2] / (W[3] * f);
    g.r0 = std::abs(a0);
    g.r1 = std::abs(a1);
    // the mean of what the two say (real_form: not far apart), so that either is off by half
    // of what a matrix lacks
    g.psi = g.r0 != 0.0 && g.r1 != 0.0 ? std::arg(a0 * g.r1 - std::conj(a1) * g.r0) : 0.0;
    g.s = 1.0 / (1.0 + g.r0 * g.r1);
    g.p0 = W[0];
    g.p1 = W[3] * f;
    return g;
}
// whether a0 a1 is real and not positive, and both of them or neither is 0 (a phase taken
// from a0 alone says nothing of a1 then): GateForm holds only so, and a matrix defined
// with a loose tolerance need not be so
bool real_form(const cdm *M, double tol) {
    if ((M[1] == 0.0) != (M[2] == 0.0)) return false;
    const cdm pr = M[1] * M[2] * std::conj(M[0] * M[3]);
    return std::abs(pr.imag()) <= tol * std::abs(pr) && pr.real() <= 0.0;
}

// Whether M on a qubit with pending factor f can run in GateForm: its larger entries are
// divided by, and their ratio becomes the next pending factor.  Not so for a singular
// matrix, or one whose rows differ widely.  flipped: the two values are stored exchanged.
bool has_pivots(const cdm *M, cdm f, bool flipped) {
    const cdm a = flipped ? M[1] : M[0], b = flipped ? M[3] : M[2];
    const bool sw = std::norm(a) < std::norm(b);
    const double p = std::norm(sw ? b : a), nf = std::norm(f);
    double d = std::norm(flipped ? (sw ? M[0] : M[2]) : (sw ? M[1] : M[3]));
    d = flipped ? d / nf : d * nf;
    return p > 0x1p-200 && d >= p * 0x1p-16 && d <= p * 0x1p16;
}

// M = V diag(e[0], e[1]) V^+ for a unitary M that is not a multiple of 1; false when M is
// not unitary to rounding (or is such a multiple).
bool eigen_form(const cdm *M, cdm *V, cdm *e) {
    const cdm h = 0.5 * (M[0] + M[3]), t0 = 0.5 * (M[0] - M[3]);
    const cdm mu = std::sqrt(t0 * t0 + M[1] * M[2]);
    if (!(std::abs(mu) > 1e-6)) return false;
    // (M - h) / mu is Hermitian with eigenvalues 1 and -1: z on the diagonal, w below it
    double z = (t0 / mu).real();
    cdm w = 0.5 * (M[2] / mu + std::conj(M[1] / mu));
    const double len = std::sqrt(z * z + std::norm(w));
    z /= len;
    w /= len;
    const double r = 1.0 / std::sqrt(2.0 * (1.0 + std::abs(z)));
    if (z >= 0.0) {
        V[0] = V[3] = (1.0 + z) * r;
        V[2] = w * r;
        V[1] = -std::conj(V[2]);
    } else {
        V[1] = V[2] = (1.0 - z) * r;
        V[0] = std::conj(w) * r;
        V[3] = -std::conj(V[0]);
        // the columns as they stand: (conj(w), 1 - z) for 1 and (1 - z, -w) for -1
    }
    e[0] = h + mu;
    e[1] = h - mu;
    for (int k = 0; k < 2; ++k)
        if (std::abs(std::abs(e[k]) - 1.0) > 4e-15) return false;
    for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 2; ++j) {
            const cdm x = V[2 * i] * e[0] * std::conj(V[2 * j]) + V[2 * i + 1] * e[1] * std::conj(V[2 * j + 1]);
            if (std::abs(x - M[2 * i + j]) > 4e-15) return false;
        }
    return true;
}

// The queue rewritten for complex64 passes: 2x2 gates that follow one another on a qubit
// become one, and a controlled gate becomes V^+ on its target, phases on its controls and
// target, and V (eigen_form).  A tile pass runs an uncontrolled gate in 7 FMAs per pair
// beside the other gates of its layer and a phase almost for free, but a controlled one
// takes 16, in an op of its own behind another for the pending factor.  Gates that only
// permute (X, Y) are left alone on a qubit that no other 2x2 gate has touched: they are
// exact there.
// Measured, complex64, U3 / CNOT chains (440 gates) on 24 qubits: 3.12 -> 1.42 ms on the device; random built-in
// gates with up to two controls (379, QFT) on 26 qubits: 8.79 -> 7.44 ms.
struct Rewriter {
    std::vector<FusedOp> &out;
    int last[64];                    // the uncontrolled gate on the qubit that nothing has followed
    uint64_t mixed = 0;              // qubits that a 2x2 gate with no zeros has acted on

    explicit Rewriter(std::vector<FusedOp> &o) : out(o) {
        out.clear();
        for (int &l : last) l = -1;
    }
    void touch(uint64_t qubits) {
        for (; qubits; qubits &= qubits - 1) last[__builtin_ctzll(qubits)] = -1;
    }
    void single(int q, const cdm *m) {
        if (last[q] < 0) {
            last[q] = (int)out.size();
            FusedOp o;
            o.kind = FusedOp::U2;
            o.q = q;
            for (int e = 0; e < 4; ++e) o.m[e] = m[e];
            out.push_back(o);
        } else {
            cdm *a = out[last[q]].m;
            const auto dot = [](cdm x0, cdm y0, cdm x1, cdm y1) {   // 0 where the products cancel
                const cdm u = x0 * y0, v = x1 * y1, p = u + v;
                return std::norm(p) < 1e-30 * (std::norm(u) + std::norm(v)) ? cdm(0.0) : p;
            };
            const cdm p[4] = {dot(m[0], a[0], m[1], a[2]), dot(m[0], a[1], m[1], a[3]),
                              dot(m[2], a[0], m[3], a[2]), dot(m[2], a[1], m[3], a[3])};
            for (int e = 0; e < 4; ++e) a[e] = p[e];
        }
        const cdm *a = out[last[q]].m;
        if (a[0] != 0.0 && a[1] != 0.0 && a[2] != 0.0 && a[3] != 0.0) mixed |= 1ull << q;
    }
    void phase(uint64_t mask, cdm f) {
        if (std::abs(f - 1.0) < 1e-15) return;
        if (std::abs(f + 1.0) < 1e-15) f = -1.0;
        FusedOp o;
        o.kind = FusedOp::PHASE;
        o.mask = o.val = mask;
        o.f = f;
        out.push_back(o);
        touch(mask);
    }
    void add(const FusedOp &op) {
        if (op.kind == FusedOp::PHASE) {
            const int q = op.mask ? __builtin_ctzll(op.mask) : 0;
            if (!op.cond.n && op.mask == 1ull << q && last[q] >= 0) {
                const cdm d[4] = {op.val ? 1.0 : op.f, 0.0, 0.0, op.val ? op.f : 1.0};
                single(q, d);
                return;
            }
            touch(op.mask);
        } else {
            cdm V[4], e[2];
            if (!op.cond.n && !op.cmask) {
                single(op.q, op.m);
                return;
            }
            const bool permutes = op.m[0] == 0.0 && op.m[3] == 0.0;
            if (!op.cond.n && (!permutes || ((mixed >> op.q) & 1)) && eigen_form(op.m, V, e)) {
                const cdm Vt[4] = {std::conj(V[0]), std::conj(V[2]), std::conj(V[1]), std::conj(V[3])};
                single(op.q, Vt);
                phase(op.cmask, e[0]);
                phase(op.cmask | 1ull << op.q, e[1] / e[0]);
                single(op.q, V);
                return;
            }
            touch(op.cmask | 1ull << op.q);
            if (!permutes) mixed |= 1ull << op.q;
        }
        out.push_back(op);
    }
};
// Whether the queue is worth rewriting: any controlled gate, or enough gates that follow
// another on their qubit.  Rewriting takes 0.03 us per op of the queue, a gate less saves
// 0.2 ms of a pass over 30 qubits and in proportion (21-qubit layers and QFT, 744 ops and
// a handful of such gates: 298 us, with rewriting 320).
bool rewrites(const std::vector<FusedOp> &ops, int n) {
    uint64_t open = 0, merges = 0;
    for (const FusedOp &op : ops) {
        if (op.kind == FusedOp::PHASE) {
            open &= ~op.mask;
            continue;
        }
        if (op.cond.n) {
            open &= ~(op.cmask | 1ull << op.q);
            continue;
        }
        if (op.cmask) return true;
        merges += (open >> op.q) & 1;
        open |= 1ull << op.q;
    }
    return (merges << n) > ((uint64_t)ops.size() << 17);
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
        const bool is_u2 = p.u2;
        bool ok = (is_u2 ? n_u2 < lim.max_u2 : n_ph < lim.max_ph) && !(p.nd & allb) && !(p.all & ndb);
        if (ok && is_u2) {
            const uint64_t t = p.nd;
            if (!(S & t)) {
                if (grow && cnt < lim.tile_qubits) {
                    S |= t;
                    ++cnt;
                } else {
                    ok = false;
                }
            }
        }
        if (ok && p.cond) {
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

// Builds one pass's program from its gates in order.
template <typename X>
struct SmemTileBuilder : PendingTerms<X> {
    using Base = PendingTerms<X>;
    using Base::F;
    using Base::lam;
    using Base::terms;
    using Base::is_pair;
    using Base::is_sign;
    SmemTileParams &P;
    int local_of[64], tile_of[64];
    bool overflow = false;

    SmemTileBuilder(SmemTileParams &p, X *f, X &l) : Base(f, l), P(p) {}

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
        const cdm f(F[b]);
        if (f == cdm(1.0, 0.0)) return;
        DTerm t{1ull << b, 1ull << b, f, nullptr, nullptr};
        single_term(t);
        F[b] = 1.0;
    }

    // A 2x2 gate on physical qubit op.q.  Uncontrolled (GateForm): turning y1 (or y0) by
    // psi makes both updates real; of e^{i psi} = i^k cos(phi) (1 + i tan(phi)), |phi| <=
    // pi/4, only u = i^k (1 + i tan) is applied and the cosine stays pending.  Which value
    // is turned and which is updated first is chosen so that the pending magnitude stays
    // near 1.  The pending factors are then those that make the device's coefficients, as
    // rounded, leave the diagonal of the gate exact.
    void gate(const POp &p) {
        const FusedOp &op = *p.op;
        const int b = op.q;
        const uint8_t q = (uint8_t)local_of[b];
        const cdm *M = op.m;
        const bool is_x = M[0] == 0.0 && M[3] == 0.0 && M[1] == 1.0 && M[2] == 1.0;
        if (op.cmask || op.cond.n || !real_form(M, 0x1p-50) || !has_pivots(M, cdm(F[b]), false)) {
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
        const bool sw = std::norm(W[0]) < std::norm(W[2]);
        if (sw) {
            std::swap(W[0], W[2]);
            std::swap(W[1], W[3]);
            o->flags |= kU2Swap;
        }
        X p0(W[0]), p1 = X(W[3]) * F[b];
        if (W[1] != 0.0) {                                // and W[2], or it has no real form
            using R = typename RealOf<X>::T;
            const auto num = [](double x) { return real_from(x, R()); };
            X a0 = X(W[1]) * F[b] / p0, a1 = X(W[2]) / p1;
            const cdm dir(a0);
            const int k = std::abs(dir.real()) >= std::abs(dir.imag()) ? (dir.real() >= 0.0 ? 0 : 2) : dir.imag() > 0.0 ? 1 : 3;
            a0 = turned(a0, 4 - k);
            a1 = turned(a1, k);
            // a0 = i^k c (1 + i t), a1 = i^-k g (1 - i t): t from the mean of both directions,
            // since a matrix is unitary only to rounding, and c and g along it
            const double w0 = 1.0 / std::sqrt(std::norm(cdm(a0))), w1 = 1.0 / std::sqrt(std::norm(cdm(a1)));
            double t = rounded((imag_of(a0) * num(w0) + imag_of(a1) * num(w1)) /
                               (real_of(a0) * num(w0) - real_of(a1) * num(w1)));
            if (std::abs(t) > 0x1p-55) o->flags |= kU2Phase;   // below: less than a rounding error
            else t = 0.0;
            const R sq = num(1.0) + num(t) * num(t);
            const R c = (real_of(a0) + imag_of(a0) * num(t)) / sq, g = (real_of(a1) - imag_of(a1) * num(t)) / sq;
            const R s = num(1.0) / (num(1.0) - c * g * sq);
            const double cs = 1.0 / std::sqrt(rounded(sq)), sd = rounded(s);
            const double ratio = std::sqrt(std::norm(cdm(p1)) / std::norm(W[0]));
            double best = 0.0;
            int side = -1, first0 = 0;
            for (int e = 0; e < 4; ++e) {                 // bit 0: y0 is turned; bit 1: y0 is updated first
                double r = ratio * ((e & 1) ? 1.0 / cs : cs) * ((e & 2) ? 1.0 / sd : sd);
                if (sw) r = 1.0 / r;
                if (r < 1.0) r = 1.0 / r;
                if (side < 0 || r < best) {
                    best = r;
                    side = e & 1;
                    first0 = e >> 1;
                }
            }
            R b0 = side == 0 ? c : c * sq, b1 = side == 0 ? g * sq : g;
            if (first0) b1 = b1 * s;
            else b0 = b0 * s;
            o->c[0] = t;
            o->c[1] = rounded(b0);
            o->c[2] = rounded(b1);
            // 1 / u = i^-k (1 - i t) / (1 + t^2)
            if (side == 0) p1 = turned(p1 * X(cdm(1.0, -t)), 4 - k) /= sq;
            else p0 = turned(p0 * X(cdm(1.0, t)), k) /= sq;
            const R left = num(1.0) + num(o->c[1]) * num(o->c[2]);
            if (first0) p1 /= left;
            else p0 /= left;
            o->flags |= (uint8_t)(k | kU2Lift);
            if (side) o->flags |= kU2On0;
            if (first0) o->flags |= kU2First0;
        }
        if (sw) std::swap(p0, p1);
        lam *= p0;
        F[b] = p1 / p0;
    }
};

// ---------------------------------------------------------------------------
// register tiles (TileParams in qk_kernels.cuh)
// ---------------------------------------------------------------------------

constexpr uint32_t kHalf = 0x80000000u;   // half a turn

// Builds one pass's program in the order the scheduler emits its gates (PendingTerms
// holds what waits).  F is in terms of the qubits' true values; a local qubit may be
// stored with its two values exchanged (flip).
struct TileBuilder : PendingTerms<cdm> {
    TileParams &P;
    int local_of[64], tile_of[64];
    int flip[kTileQubits] = {};
    int arr = ARR_IO;
    // Index of the layer op that further gates may join, -1: none, and the register bits
    // that ops after it depend on (a gate on one of them cannot go before those ops) and
    // act on.
    int open = -1, since = 0, since_u2 = 0;
    int slots = 0;           // of the kernel's tables of turns, in use
    bool overflow = false;

    TileBuilder(TileParams &p, cdm *f, cdm &l) : PendingTerms<cdm>(f, l), P(p) {}

    TileOp &add(uint8_t kind) {
        if (P.nops >= kTileMaxOps) {
            overflow = true;
            open = -1;
            P.nops = 0;      // the program is thrown away
        }
        TileOp &o = P.ops[P.nops++];
        std::memset(static_cast<void *>(&o), 0, sizeof o);
        o.kind = kind;
        o.cond = 0xffff;
        return o;
    }
    void add_term(uint32_t bit, uint32_t turns) {
        if (P.nbt >= kTileMaxTerms) {
            overflow = true;
            P.nbt = 0;
        }
        P.bt[P.nbt++] = BitTerm{bit, turns};
    }
    void transpose_to(int a) {
        add(TOP_XPOSE).k = (uint8_t)a;
        arr = a;
        open = -1;
    }
    int flip_of(int b) const { return local_of[b] >= 0 ? flip[local_of[b]] : 0; }
    // where physical qubit b is: 0 a register bit, 1 a thread bit, 2 a tile-index bit
    int place(int b, int *pos) const {
        if (local_of[b] < 0) {
            *pos = tile_of[b];
            return 2;
        }
        const int s = slot_of(arr, local_of[b], pos);
        if (s == 2) *pos += 5;
        return s == 0 ? 0 : 1;
    }
    // a phase on the stored |1> of qubit b
    void stored_phase(int b, double x) {
        if (flip_of(b)) {
            lam *= std::polar(1.0, x);
            F[b] *= std::polar(1.0, -x);
        } else {
            F[b] *= std::polar(1.0, x);
        }
    }
    // Waiting pairs are kept as turns, which hold no magnitude: a pair from a diagonal
    // matrix that is not unitary to an FP32 rounding error (defined with a wide tolerance)
    // goes out as a direct factor instead.
    static bool is_turn(const DTerm &t) { return is_pair(t) && std::abs(std::norm(t.f) - 1.0) <= 0x1p-23; }
    // e^{i th} where the true values of a and b are both 1, in stored values sa, sb: (sa ^
    // fa)(sb ^ fb) = fa fb + fa (1 - 2 fb) sb + fb (1 - 2 fa) sa + (1 - 2 fa)(1 - 2 fb) sa
    // sb.  The constant and the single-bit parts become pending; returns the turns left
    // on the stored pattern (1, 1).
    uint32_t stored_pair(int a, int b, const DTerm &t) {
        const uint32_t T = is_sign(t) ? kHalf : angle_turns(std::arg(t.f));
        const double th = turns_angle(T);
        const int fa = flip_of(a), fb = flip_of(b);
        if (fa && fb) lam *= std::polar(1.0, th);
        if (fa) stored_phase(b, fb ? -th : th);
        if (fb) stored_phase(a, fa ? -th : th);
        return fa != fb ? 0u - T : T;
    }
    // an op's conditions in stored values
    void conditions(TileOp &o, uint64_t mask, uint64_t val) {
        for (uint64_t m = mask; m; m &= m - 1) {
            const int b = __builtin_ctzll(m);
            if (flip_of(b)) val ^= 1ull << b;
        }
        encode_cond(mask, val, arr, local_of, o);
        since |= o.rmask;
    }
    void set_cond(TileOp &o, const Cond &c) {
        for (int k = 0; k < P.n_conds; ++k)
            if (same_cond(P.conds[k], c)) o.cond = (uint16_t)k;
    }
    void direct(uint64_t mask, uint64_t val, cdm f, const Cond *c) {
        TileOp &o = add(TOP_PHASE);
        conditions(o, mask, val);
        if (c) set_cond(o, *c);
        o.ph.re = (float)f.real();
        o.ph.im = (float)f.imag();
    }
    void pair_op(int k, int l, uint32_t turns) {
        if (turns == 0) return;
        if (k > l) std::swap(k, l);
        TileOp &o = add(turns == kHalf ? TOP_PAIRNEG : TOP_PAIRU);
        since |= 1 << k | 1 << l;
        o.k = (uint8_t)(k | (l << 3));
        const double x = turns_angle(turns);
        o.ph.re = (float)std::cos(x);
        o.ph.im = (float)std::sin(x);
    }

    // what waits on qubit b (a register bit now), taken out of terms: register pairs
    // (other bit, turns), thread and tile-index terms, and everything else
    struct Touching {
        std::vector<std::pair<int, uint32_t>> reg;
        std::vector<BitTerm> thread, tile;
        std::vector<DTerm> other;
    };
    void take_touching(int b, Touching &out) {
        out.reg.clear();
        out.thread.clear();
        out.tile.clear();
        out.other.clear();
        size_t w = 0;
        const uint64_t bb = 1ull << b;
        auto put = [](std::vector<BitTerm> &v, uint32_t bit, uint32_t turns) {
            for (BitTerm &t : v)
                if (t.bit == bit) {
                    t.turns += turns;
                    return;
                }
            v.push_back(BitTerm{bit, turns});
        };
        for (size_t i = 0; i < terms.size(); ++i) {
            const DTerm t = terms[i];
            if (!(t.mask & bb)) {
                terms[w++] = t;
                continue;
            }
            if (!is_turn(t)) {
                out.other.push_back(t);
                continue;
            }
            const int d = __builtin_ctzll(t.mask & ~bb);
            const uint32_t T = stored_pair(b, d, t);
            int pos;
            const int where = place(d, &pos);
            if (where == 0) out.reg.push_back({pos, T});
            else put(where == 1 ? out.thread : out.tile, (uint32_t)pos, T);
        }
        terms.resize(w);
    }

    // a phase on register bit k from thread and tile-index terms, as an op
    void phase_op(int k, Touching &T) {
        if (T.thread.empty() && T.tile.empty()) return;
        TileOp &o = add(TOP_PHQ);
        since |= 1 << k;
        o.k = (uint8_t)k;
        o.first = (uint16_t)P.nbt;
        o.count = (uint16_t)T.thread.size();
        o.count2 = (uint16_t)T.tile.size();
        for (const BitTerm &t : T.thread) add_term(t.bit, t.turns);
        for (const BitTerm &t : T.tile) add_term(t.bit, t.turns);
        T.thread.clear();
        T.tile.clear();
    }
    // a 2x2 gate whose target is a register bit of the current arrangement
    void gate(const POp &p) {
        const FusedOp &op = *p.op;
        const int b = op.q, lq = local_of[b];
        int k;
        place(b, &k);
        static thread_local Touching T;
        take_touching(b, T);
        if (op.cmask || op.cond.n || !real_form(op.m, 1e-7) || !has_pivots(op.m, F[b], flip[lq])) {
            for (const DTerm &t : T.other) direct(t.mask, t.val, t.f, t.cond);
            for (const auto &r : T.reg) pair_op(k, r.first, r.second);
            phase_op(k, T);
            if (F[b] != cdm(1.0, 0.0)) {
                direct(1ull << b, 1ull << b, F[b], nullptr);
                F[b] = 1.0;
            }
            TileOp &o = add(TOP_U2);
            since |= 1 << k;
            since_u2 |= 1 << k;
            conditions(o, op.cmask, op.cmask);
            if (op.cond.n) set_cond(o, op.cond);
            o.k = (uint8_t)k;
            for (int e = 0; e < 4; ++e) {   // X M X in stored order when the qubit is flipped
                const cdm m = op.m[flip[lq] ? 3 - e : e];
                o.m[2 * e] = (float)m.real();
                o.m[2 * e + 1] = (float)m.imag();
            }
            return;
        }
        // its waiting terms: signs by parity when they are all it has, else a phase
        bool signs = true;
        for (const BitTerm &t : T.thread) signs = signs && (t.turns == kHalf || t.turns == 0);
        for (const BitTerm &t : T.tile) signs = signs && (t.turns == kHalf || t.turns == 0);
        if (!signs && slots == kTileSlots) {   // no room in the tables
            phase_op(k, T);
            signs = true;
        }
        // joins the open layer unless its bit is in it or in a later op, or a term with
        // one of the layer's bits (put there after that bit's gate) or a factor has to
        // come first
        bool join = open >= 0 && !(((P.ops[open].k | since) >> k) & 1) && T.other.empty();
        for (const auto &r : T.reg)
            join = join && (r.second == kHalf || r.second == 0) && !(((P.ops[open].k | since_u2) >> r.first) & 1);
        if (!join) {
            for (const DTerm &t : T.other) direct(t.mask, t.val, t.f, t.cond);
            for (const auto &r : T.reg)
                if (r.second != kHalf) pair_op(k, r.first, r.second);
            TileOp &o = add(TOP_U2L);
            o.first = (uint16_t)P.nlg;
            open = P.nops - 1;
            since = since_u2 = 0;
        }
        if (overflow || P.nlg >= kTileMaxMats) {
            overflow = true;
            return;
        }
        TileOp &o = P.ops[open];
        for (const auto &r : T.reg)
            if (r.second == kHalf) o.tmask ^= (uint16_t)(1u << cz_index(std::min(k, r.first), std::max(k, r.first)));
        // the layer is the last one in lg: keep its gates in bit order
        const int at = o.first + __builtin_popcount(o.k & ((1u << k) - 1));
        for (int i = P.nlg; i > at; --i) P.lg[i] = P.lg[i - 1];
        ++P.nlg;
        o.k |= (uint8_t)(1u << k);
        LayerGate &g = P.lg[at];
        std::memset(static_cast<void *>(&g), 0, sizeof g);
        g.slot = 0xff;
        g.first = (uint16_t)P.nbt;
        for (const BitTerm &t : T.thread) {
            if (t.turns == 0) continue;
            if (signs) {
                g.ts ^= (uint16_t)(1u << t.bit);
                continue;
            }
            add_term(t.bit, t.turns);
            ++g.nt;
        }
        for (const BitTerm &t : T.tile) {
            if (t.turns == 0) continue;
            if (signs) {
                g.fs ^= 1u << t.bit;
                continue;
            }
            add_term(t.bit, t.turns);
            ++g.ni;
        }
        if (g.ts || g.fs) o.tval |= (uint16_t)(1u << k);
        if (!signs) {
            o.count |= (uint16_t)(1u << k);
            g.slot = (uint8_t)slots++;
        }
        pivot(op.m, b, lq, k, o, g);
    }

    // LayerGate's coefficients.  zf is chosen so that the pending magnitude of the qubit's
    // |1> stays within [1/2, 2].
    void pivot(const cdm *M, int b, int lq, int k, TileOp &o, LayerGate &g) {
        cdm Ms[4] = {M[0], M[1], M[2], M[3]}, f = F[b];
        if (flip[lq]) {                       // the stored input is the true one exchanged
            std::swap(Ms[0], Ms[1]);
            std::swap(Ms[2], Ms[3]);
            lam *= f;
            f = 1.0 / f;
        }
        const GateForm w = gate_form(Ms, f);
        cdm p0 = w.p0, p1 = w.p1;
        if (w.r0 != 0.0 || w.r1 != 0.0) {
            const int turns = (int)std::lround(w.psi / M_PI);
            const double phi = w.psi - turns * M_PI, sg = turns & 1 ? -1.0 : 1.0;
            p1 *= std::polar(1.0, -phi);
            double b0 = sg * w.r0, b1 = -sg * w.r1;
            double r = std::abs(p1 / p0);
            if (w.sw) r = 1.0 / r;
            const bool zf = (r < 1.0) != w.sw;   // divide the smaller factor by s, or multiply the larger
            if (zf) {
                b1 *= w.s;
                p1 /= w.s;
                o.rmask |= (uint8_t)(1u << k);
            } else {
                b0 *= w.s;
                p0 /= w.s;
            }
            auto splat = [](double x) { return make_float2((float)x, (float)x); };
            if ((o.count >> k) & 1) {
                const uint32_t t = angle_turns(phi);
                std::memcpy(&g.h.x, &t, sizeof t);
            } else {
                if (std::abs(phi) > 0x1p-27) o.rval |= (uint8_t)(1u << k);   // below: less than a rounding error
                g.h = splat(-std::tan(phi / 2));
                g.s = splat(std::sin(phi));
            }
            g.c0 = splat(b0);
            g.c1 = splat(b1);
        }
        flip[lq] = w.sw ? 1 : 0;
        if (w.sw) std::swap(p0, p1);          // the true |0> and |1>
        lam *= p0;
        F[b] = p1 / p0;
    }

    // every waiting term as ops and as the final flush's terms
    void finish_terms() {
        std::vector<BitTerm> th[5], ti[5], two;
        for (const DTerm &t : terms) {
            if (!is_turn(t)) {
                direct(t.mask, t.val, t.f, t.cond);
                continue;
            }
            const int a = __builtin_ctzll(t.mask), b = 63 - __builtin_clzll(t.mask);
            const uint32_t T = stored_pair(a, b, t);
            int pa, pb;
            const int wa = place(a, &pa), wb = place(b, &pb);
            if (wa == 0 && wb == 0) pair_op(pa, pb, T);
            else if (wa == 0) (wb == 1 ? th : ti)[pa].push_back(BitTerm{(uint32_t)pb, T});
            else if (wb == 0) (wa == 1 ? th : ti)[pb].push_back(BitTerm{(uint32_t)pa, T});
            else
                two.push_back(BitTerm{(uint32_t)(wa == 2 ? pa + 8 : pa) | (uint32_t)(wb == 2 ? pb + 8 : pb) << 8, T});
        }
        terms.clear();
        for (int k = 0; k < 5; ++k) {
            if (th[k].size() > 255 || ti[k].size() > 255) overflow = true;
            P.fin_first[k] = (uint16_t)P.nbt;
            P.fin_nt[k] = (uint8_t)th[k].size();
            P.fin_ni[k] = (uint8_t)ti[k].size();
            for (const BitTerm &t : th[k]) add_term(t.bit, t.turns);
            for (const BitTerm &t : ti[k]) add_term(t.bit, t.turns);
        }
        P.fin2_first = (uint16_t)P.nbt;
        P.fin2_n = (uint16_t)two.size();
        for (const BitTerm &t : two) add_term(t.bit, t.turns);
    }
};

}  // namespace

qk_status plan_passes(TilePlanner *planner, int n, const std::vector<FusedOp> &ops, const PassSink &sink,
                      const char **err) {
    *err = "";
    std::vector<POp> rem;
    static thread_local std::vector<FusedOp> rewritten_ops;
    const std::vector<FusedOp> *list = &ops;
    if (rewrites(ops, n)) {
        Rewriter rw(rewritten_ops);
        for (const FusedOp &op : ops) rw.add(op);
        list = &rewritten_ops;
    }
    rem.reserve(list->size());
    for (const auto &op : *list) rem.push_back(classify(op));

    // take limits per pass; halved and retried when a program overflows the
    // kernel-parameter budget (ops and grouped phase entries)
    int max_u2 = 100, max_ph = 300;
    static thread_local std::vector<POp> left, taken, next;
    const GiveBack trim(rewritten_ops, left, taken, next);
    std::deque<FusedOp> rewritten;   // pair terms handed on without their single-qubit parts
    // per physical qubit the pending factor of its |1>, and the one of all amplitudes,
    // handed from pass to pass in FP64; only the plan's last pass applies them
    cdm F[64], lam = 1.0;
    for (cdm &f : F) f = 1.0;
    std::vector<Cond> conds;
    while (!rem.empty()) {
        int n_u2 = 0, n_ph = 0;
        const uint64_t S = choose_pass(rem, n, TakeLimits{kTileQubits, max_u2, max_ph}, kTileContig, conds, taken, left,
                                       &n_u2, &n_ph);

        static thread_local TileParams P;
        std::memset(static_cast<TileHead *>(&P), 0, sizeof(TileHead));
        P.n = n;
        P.n_tiles = 1ull << (n - kTileQubits);
        cdm F1[64], lam1 = lam;
        std::copy(F, F + 64, F1);
        TileBuilder B(P, F1, lam1);
        int *const local_of = B.local_of;
        for (int b = 0; b < 64; ++b) local_of[b] = B.tile_of[b] = -1;
        {
            int lb = 0, fb = 0;
            for (int b = 0; b < n; ++b) {
                if ((S >> b) & 1) {
                    P.S[lb] = (int8_t)b;
                    local_of[b] = lb++;
                } else {
                    B.tile_of[b] = fb;
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
        // What each op has to follow, qubit by qubit: a 2x2 gate comes after everything
        // on its target since the last gate on it, any other touch after that gate.
        // Successors of op i as a list in edges (next index in edges, or -1).
        struct Edge {
            int to, next;
        };
        static thread_local std::vector<Edge> edges;
        static thread_local std::vector<int> npred, head, touch_next, ready;
        edges.clear();
        npred.assign(m, 0);
        head.assign(m, -1);
        int last_gate[64], touched[64];      // per qubit: the last gate on it; ops since then (a list)
        for (int b = 0; b < 64; ++b) last_gate[b] = touched[b] = -1;
        std::vector<Edge> &E = edges;
        static thread_local std::vector<Edge> touches;
        touches.clear();
        auto edge = [&](int i, int j) {
            E.push_back({j, head[i]});
            head[i] = (int)E.size() - 1;
            ++npred[j];
        };
        for (int j = 0; j < m; ++j) {
            for (uint64_t q = taken[j].all; q; q &= q - 1) {
                const int b = __builtin_ctzll(q);
                if ((taken[j].nd >> b) & 1) {
                    if (touched[b] < 0 && last_gate[b] >= 0) edge(last_gate[b], j);
                    for (int t = touched[b]; t >= 0; t = touches[t].next) edge(touches[t].to, j);
                    last_gate[b] = j;
                    touched[b] = -1;
                } else {
                    if (last_gate[b] >= 0) edge(last_gate[b], j);
                    touches.push_back({j, touched[b]});
                    touched[b] = (int)touches.size() - 1;
                }
            }
        }
        // A diagonal term that is ready only starts to wait in the builder; a ready gate
        // (at most one per qubit) is emitted when its target is a register bit.
        ready.clear();
        int ndone = 0;
        static thread_local std::vector<int> stack;
        auto settle = [&](int j) {           // op j has no predecessors left
            stack.clear();
            stack.push_back(j);
            while (!stack.empty()) {
                const int i = stack.back();
                stack.pop_back();
                if (taken[i].op->kind == FusedOp::U2) {
                    ready.push_back(i);
                    continue;
                }
                B.diagonal(taken[i]);
                ++ndone;
                for (int e = head[i]; e >= 0; e = E[e].next)
                    if (--npred[E[e].to] == 0) stack.push_back(E[e].to);
            }
        };
        static thread_local std::vector<int> start;
        start.clear();
        for (int j = 0; j < m; ++j)
            if (npred[j] == 0) start.push_back(j);
        for (int j : start) settle(j);
        while (ndone < m && !B.overflow) {
            bool progress = false;
            for (size_t r = 0; r < ready.size();) {
                const int j = ready[r];
                if (!executable(taken[j], B.arr, local_of)) {
                    ++r;
                    continue;
                }
                ready.erase(ready.begin() + (long)r);
                B.gate(taken[j]);
                ++ndone;
                progress = true;
                for (int e = head[j]; e >= 0; e = E[e].next)
                    if (--npred[E[e].to] == 0) settle(E[e].to);
            }
            if (ndone == m || progress) continue;
            int best = -1, best_cnt = -1;
            for (int a = 0; a < 3; ++a) {
                if (a == B.arr) continue;
                int cntr = 0;
                for (int j : ready) cntr += executable(taken[j], a, local_of);
                if (cntr > best_cnt) {
                    best_cnt = cntr;
                    best = a;
                }
            }
            B.transpose_to(best);
        }
        const bool last = left.empty();
        if (B.arr == ARR_LO) B.transpose_to(ARR_IO);   // stores take ARR_IO or ARR_HI
        // Terms that no gate of this pass called for go to the front of what is left:
        // they commute with everything taken after them, and with what was left behind
        // before them.  (Their single-qubit parts are pending already.)
        if (last || n_u2 == 0) B.finish_terms();
        if (B.overflow) {
            // too large for one launch: plan this pass again with fewer gates
            if (max_u2 <= 1 && max_ph <= 1) {
                *err = "internal: tile program overflow";
                return QK_EINVAL;
            }
            max_u2 = std::max(1, max_u2 / 2);
            max_ph = std::max(1, max_ph / 2);
            continue;
        }
        P.fin_flip = 0;
        for (int q = 0; q < kTileQubits; ++q) P.fin_flip |= B.flip[q] << q;
        P.fin_fixed_mask = 0;
        if (last) {   // everything pending, on the stored values
            for (int q = 0; q < kTileQubits; ++q) {
                cdm f = F1[(int)P.S[q]];
                if (B.flip[q]) {
                    lam1 *= f;
                    f = 1.0 / f;
                }
                P.fin_turns[q] = angle_turns(std::arg(f));
                P.fin_mag[q] = (float)std::abs(f);
            }
            for (int b = 0; b < P.nfix; ++b) {
                const cdm f = F1[(int)P.fixed[b]];
                P.fin_fixed[b] = angle_turns(std::arg(f));
                P.fin_fixed_mag[b] = (float)std::abs(f);
                if (P.fin_fixed[b] || P.fin_fixed_mag[b] != 1.f) P.fin_fixed_mask |= 1ull << b;
            }
            P.fin_turns[13] = angle_turns(std::arg(lam1));
            P.fin_scale = (float)std::abs(lam1);
        } else {
            for (int q = 0; q < kTileQubits; ++q) {
                P.fin_turns[q] = 0;
                P.fin_mag[q] = 1.f;
            }
            P.fin_turns[13] = 0;
            // the stored amplitudes are the true ones divided by lam: keep them within
            // 2^24 of the true ones in FP32 (a factor in [2^-1/2, 2] per gate)
            P.fin_scale = 1.f;
            const double x = std::abs(lam1);
            if (x < 0x1p-24 || x > 0x1p24) {
                P.fin_scale = (float)x;
                lam1 /= x;
            }
        }
        // whether any phase factor the pass forms can be other than 1 or -1 (the kernel
        // fills its phase table only then)
        {
            auto general = [](uint32_t t) { return t != 0u && t != kHalf; };
            bool need = false;
            for (int e = 0; e < P.nbt && !need; ++e) need = general(P.bt[e].turns);
            for (int q = 0; q < 14; ++q) need = need || general(P.fin_turns[q]);
            for (int b = 0; b < P.nfix; ++b)
                if ((P.fin_fixed_mask >> b) & 1) need = need || general(P.fin_fixed[b]);
            P.need_tab = need ? 1 : 0;
        }
        next.clear();
        B.hand_on(next, rewritten);
        next.insert(next.end(), left.begin(), left.end());
        if (planner->log) {
            int cnt_k[9] = {0};  // by TileOpKind
            for (int i = 0; i < P.nops; ++i) cnt_k[P.ops[i].kind]++;
            std::fprintf(stderr,
                         "[qk plan] pass S=%#llx gates=%d (u2 %d, phase %d) ops=%d u2=%d layers=%d layer_gates=%d "
                         "phase_direct=%d phase_ops=%d terms=%d pairs=%d pair_signs=%d xpose=%d kept=%zu\n",
                         (unsigned long long)S, m, n_u2, n_ph, P.nops, cnt_k[TOP_U2], cnt_k[TOP_U2L], P.nlg,
                         cnt_k[TOP_PHASE], cnt_k[TOP_PHQ], P.nbt, cnt_k[TOP_PAIRU], cnt_k[TOP_PAIRNEG],
                         cnt_k[TOP_XPOSE], B.terms.size());
        }

        const qk_status st = sink(P);
        if (st != QK_OK) return st;
        std::copy(F1, F1 + 64, F);
        lam = lam1;
        rem.swap(next);
        max_u2 = 100;
        max_ph = 300;
    }
    return QK_OK;
}

namespace {
template <typename X>      // of the pending factors
qk_status smem_passes(TilePlanner *planner, int n, int prec, const std::vector<FusedOp> &ops, const SmemPassSink &sink,
                      const char **err) {
    *err = "";
    static thread_local std::vector<POp> rem, left, taken, next;
    const GiveBack trim(rem, left, taken, next);
    rem.clear();
    for (const auto &op : ops) rem.push_back(classify(op));
    const int m = smem_tile_qubits(n, prec);
    TakeLimits lim{m, kSmemTileOps, 4096};
    const int contig = std::min(smem_tile_contig(n), m);
    std::vector<Cond> conds;
    const double far = prec == 0 ? 0x1p24 : 0x1p200;   // how far the stored amplitudes may drift from the true ones
    X F[64], lam = 1.0;
    for (X &f : F) f = 1.0;
    std::deque<FusedOp> rewritten;   // pair terms handed on without their single-qubit parts
    while (!rem.empty()) {
        int n_u2 = 0, n_ph = 0;
        const uint64_t S = choose_pass(rem, n, lim, contig, conds, taken, left, &n_u2, &n_ph);
        static thread_local SmemTileParams P;
        X F1[64], lam1 = lam;
        std::copy(F, F + 64, F1);
        SmemTileBuilder<X> B(P, F1, lam1);
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
            cdm fac[64];
            for (int b = 0; b < n; ++b) {
                fac[b] = cdm(F1[b]);
                if (fac[b] != cdm(1.0, 0.0)) bits |= 1ull << b;
            }
            const cdm c0(lam1);
            if (bits || c0 != cdm(1.0, 0.0)) B.table(-1, bits, fac, c0);
        } else if (!B.overflow && !(std::abs(cdm(lam1)) > 1.0 / far && std::abs(cdm(lam1)) < far)) {
            // a factor in [2^-1/2, 2] per gate: keep the stored amplitudes in range
            B.table(-1, 0, nullptr, cdm(lam1));
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
        B.hand_on(next, rewritten);
        next.insert(next.end(), left.begin(), left.end());
        if (planner->log)
            std::fprintf(stderr, "[qk plan] smem pass S=%#llx gates=%zu (u2 %d, phase %d) ops=%d factors=%d kept=%zu\n",
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
}  // namespace

qk_status plan_smem_passes(TilePlanner *planner, int n, int prec, const std::vector<FusedOp> &ops,
                           const SmemPassSink &sink, const char **err) {
    return prec == 0 ? smem_passes<cdm>(planner, n, prec, ops, sink, err)
                     : smem_passes<DDC>(planner, n, prec, ops, sink, err);
}

namespace {

// Tile qubits of a dense pass that enumerates n qubits: complex64 gates of 5 and 6 qubits
// form 8 rows per thread, which takes 2^13 amplitudes to give every thread columns;
// smaller tiles for small states, so that there are tiles for all SMs (in complex128 a
// tile's FP64 work is the time).  One 6-qubit gate with a control on 20 qubits 24 us in
// tiles of 2^13, 36 in 2^11; two of them with controls inside the tile on 18 qubits 24 and 17.
int dense_tile_qubits(int n, int prec, int k, bool alone) {
    if (prec != 0) return n >= 20 ? 11 : n >= 18 ? 10 : 8;
    if (k >= 5 && n >= (alone ? 18 : 20)) return 13;
    return n >= 20 ? 12 : n >= 18 ? 11 : n >= 16 ? 10 : 9;
}
// its qubits: the gates' targets and the lowest others that are not enumerated away
uint64_t dense_tile_set(int n, int prec, int k, bool alone, uint64_t targets, uint64_t lone) {
    const int m = dense_tile_qubits(n - __builtin_popcountll(lone), prec, k, alone);
    uint64_t S = targets;
    for (int b = 0; b < n && __builtin_popcountll(S) < m; ++b)
        if (!((S | lone) >> b & 1)) S |= 1ull << b;
    return S;
}

// The program of one dense pass over the given gates.  A pass of one controlled gate
// enumerates only the tiles whose control bits are set.
void dense_program(int n, int prec, const std::vector<const DenseItem *> &taken, DenseParams &P) {
    std::memset(static_cast<void *>(&P), 0, offsetof(DenseParams, ops));
    uint64_t S = 0;
    for (const DenseItem *it : taken) {
        S |= it->tmask;
        bool known = !it->cond.n;
        for (int k = 0; k < P.n_conds; ++k) known = known || same_cond(P.conds[k], it->cond);
        if (!known) P.conds[P.n_conds++] = it->cond;
    }
    const uint64_t lone = taken.size() == 1 ? taken[0]->cmask : 0;   // enumerated only where set
    S = dense_tile_set(n, prec, taken[0]->k, taken.size() == 1, S, lone);
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
    P.k = taken[0]->k;
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
        const bool free2 = prec == 0 && it->k == 2 && !it->cmask && !it->cond.n;
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
        if (prec == 0 && it->k == 2 && !o.pair)
            while (o.ncs < 2 && o.nfree > 0) o.cs[o.ncs++] = o.fs[--o.nfree];
        o.mat = it->mat;
    }
}

// Whether the gates of a pass are cheaper in a pass each, which enumerates only the tiles
// whose control bits are set, than in one over the whole state.  Estimates in us, from 24
// qubits: traffic 45 (complex64) and 90, of which complex128's arithmetic hides most, and
// which follows control bits only down to runs of 64 bytes; a gate of k qubits 10 + 2^k *
// 3.4 and 2^k * 112; another launch 5.5.  In a shared pass a controlled gate keeps half its
// time in complex64 (threads without columns); in complex128 its time follows the controls
// inside the tile, but controls on tile-index bits leave it to few of an SM's CTAs, and the
// tile with all of them set runs every gate in turn (chain).  Eight gates with four
// controls on 24 qubits, gate by gate before / one pass / a pass each: complex64 k = 2 84 /
// 149 / 71, k = 4 552 / 214 / 102, complex128 k = 4 1543 / 2875 / 1086 us; with one control,
// complex64 k = 2, 394 / 180 in one pass.
bool dense_apart(int n, int prec, const std::vector<const DenseItem *> &taken) {
    uint64_t targets = 0, controls = 0;
    for (const DenseItem *it : taken) {
        targets |= it->tmask;
        controls |= it->cmask;
    }
    if (taken.size() < 2 || !controls) return false;
    const int k = taken[0]->k;
    const uint64_t S = dense_tile_set(n, prec, k, false, targets, 0), run = prec == 0 ? 7u : 3u;
    const double unit = std::ldexp(1.0, n - 24), traffic = unit * (prec == 0 ? 45.0 : 40.0);
    const double gate = unit * (prec == 0 ? 10.0 + std::ldexp(3.4, k) : std::ldexp(112.0, k));
    // complex128: a gate on one tile, beside others on its SM or by itself
    const auto tile = [&](int bits, double rate) { return std::ldexp(1.0 / rate, bits + k + 2); };
    const int m = __builtin_popcountll(S);
    double joint = 2.5 + traffic, apart = 0.0, chain = 0.0;
    for (const DenseItem *it : taken) {
        const int nc = __builtin_popcountll(it->cmask), tc = __builtin_popcountll(it->cmask & ~S);
        const double part = std::ldexp(traffic, -__builtin_popcountll(it->cmask & ~run)) + std::ldexp(gate, -nc);
        apart += prec == 0 ? 5.5 + part
                           : std::max(5.5 + part, 2.5 + tile(dense_tile_qubits(n - nc, prec, k, true), 2600.0));
        if (prec == 0) {
            joint += gate * (nc > 0 ? 0.5 : 1.0);
        } else {
            joint += std::ldexp(gate, tc - nc) * std::min(1.0, tc > 0 ? std::ldexp(5.0, -tc) : 1.0);
            chain += std::ldexp(tile(m, tc > 0 ? 1300.0 : 2600.0), tc - nc);
        }
    }
    return apart < 0.8 * std::max(joint, chain);
}
}  // namespace

// A dense pass: S starts as the lowest qubits (runs of 128 bytes in HBM, 32 for states in
// L2) and takes the targets of every gate, in order, that commutes with the gates left
// behind, has the first one's k and still fits; they go in one pass, or in one each where
// that is cheaper (dense_apart).
qk_status plan_dense(int n, int prec, const std::vector<DenseItem> &ops, const DenseSink &sink) {
    static thread_local std::vector<const DenseItem *> rem, left, taken, one(1);
    static thread_local std::vector<Cond> conds;
    const GiveBack trim(rem, left, taken);
    rem.clear();
    for (const DenseItem &it : ops) rem.push_back(&it);
    while (!rem.empty()) {
        left.clear();
        taken.clear();
        conds.clear();
        static thread_local DenseParams P;
        const int m = std::min(dense_tile_qubits(n, prec, rem[0]->k, false), n);
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
            if (ok && it->cond.n) {
                bool known = false;
                for (const Cond &c : conds) known = known || same_cond(c, it->cond);
                if (!known && (int)conds.size() >= kTileMaxConds) ok = false;
                else if (!known) conds.push_back(it->cond);
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
        if (dense_apart(n, prec, taken)) {
            for (const DenseItem *it : taken) {
                one[0] = it;
                dense_program(n, prec, one, P);
                const qk_status st = sink(P);
                if (st != QK_OK) return st;
            }
        } else {
            dense_program(n, prec, taken, P);
            const qk_status st = sink(P);
            if (st != QK_OK) return st;
        }
        rem.swap(left);
    }
    return QK_OK;
}

// Whether a queue that would go through tiles in shared memory is cheaper as one launch per
// op: a pass reads and writes the whole state, a launch only the amplitudes that match its
// controls, or its phase's bits.  Estimates in us, from complex128 on 26 qubits (2 GiB):
// a pass 370, half as much again with a gate or phase on one qubit (FP64), a phase 500 and
// a 2x2 gate 1030 times the fraction they match.  A launch takes 2.6, that of a pass, with
// its program of 20 KB, 4.4.  One launch per op / one pass, complex128: CZ on 26 qubits 141 /
// 380, T 253 / 582, X with two controls 264 / 371, with five 40 / 370, H 1034 / 743, three CZ
// 453 / 395; one gate on 10 qubits, either type, 6.3 / 8.2, two 11.6 / 11.1.
bool single_launches(int n, int prec, const std::vector<FusedOp> &ops) {
    const double unit = std::ldexp(prec == 0 ? 0.5 : 1.0, n - 26);   // of the 2 GiB
    double singles = 0.0;
    bool wide = false;
    for (const FusedOp &op : ops) {
        const bool u2 = op.kind == FusedOp::U2;
        const int bits = __builtin_popcountll(u2 ? op.cmask : op.mask);
        wide = wide || bits + (u2 ? 1 : 0) <= 1;
        singles += 2.6 + unit * std::ldexp(u2 ? 1030.0 : 500.0, -bits);
        if (singles >= 4.4 + unit * 555.0) return false;
    }
    return singles < 4.4 + unit * (wide ? 555.0 : 370.0);
}

qk_status run_fused(TilePlanner *planner, qk_ctx *c, const std::vector<FusedOp> &ops) {
    const int n = ctx_n(c);
    const int prec = ctx_prec(c);
    if (prec != 0 || n < kTileQubits) {
        if (single_launches(n, prec, ops)) {
            for (const FusedOp &op : ops) {
                const qk_status st = ctx_run_plain(c, op);
                if (st != QK_OK) return st;
            }
            return QK_OK;
        }
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
        cudaError_t e = launch_tile(ctx_state(c), P, ctx_cbits(c), ctx_sms(c), ctx_stream(c));
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
