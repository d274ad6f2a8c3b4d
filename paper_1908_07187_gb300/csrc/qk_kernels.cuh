// Internal declarations shared by the libqk host code and its CUDA kernels.
// Nothing here is part of the public ABI (include/qk.h).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

namespace qk {

// The dynamic shared-memory limit of a kernel belongs to the function on its device and
// not to the calling thread: set before a launch to that launch's size, a second thread
// lowers it in between and the first one's launch is refused.  So it is set once per
// device, to the most that any launch of the kernel asks for (twice by two threads at
// once is harmless: the value is the same).
struct SmemLimit {
    std::atomic<bool> set[64] = {};
};
template <typename F>
inline cudaError_t smem_limit(F *f, size_t most, SmemLimit &l) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (l.set[dev].load(std::memory_order_acquire)) return cudaSuccess;
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (e == cudaSuccess) l.set[dev].store(true, std::memory_order_release);
    return e;
}

constexpr int kMaxPos = 24;        // sorted bit positions a launch may insert
constexpr int kMaxCond = 16;       // classical-condition cbits per gate
constexpr int kMaxRphase = 62;     // cbits feeding one semiclassical phase
constexpr int kMaxPermW = 30;      // permutation register width

// Classical condition: the launch acts only if every listed cbit is 1.
struct Cond {
    int n;
    int idx[kMaxCond];
};

// Sorted ascending bit positions, used to enumerate a subspace by inserting a
// bit at each position into a dense counter.
struct Positions {
    int n;
    int pos[kMaxPos];
};

// 2x2 update on target bit q where all control bits (cmask) are 1.
struct U2Args {
    double m[8];          // m00, m01, m10, m11 as (re, im) pairs, FP64 master
    uint64_t cmask;
    int q;
    Positions ins;        // q and every control, sorted
    uint64_t n_units;     // work units in the subspace
    Cond cond;
};

// Multiply amplitudes whose index satisfies (i & mask) == val by f.
struct PhaseArgs {
    double f_re, f_im;
    uint64_t mask, val;
    Positions ins;        // bits of mask, sorted
    uint64_t n_units;
    Cond cond;
    // semiclassical phase (rphase): when n_rphase > 0, f is computed on the
    // device as exp(-2 pi i sum_l c[rphase_idx[l-1]] / 2^(l+1)).
    int n_rphase;
    int rphase_idx[kMaxRphase];
};

// Controlled permutation of a w-bit register, out-of-place gather.
// A register whose qubits sit on consecutive physical bits p0 .. p0 + w - 1 is a bit
// field of the index: its value is the field itself (first-listed qubit highest,
// rev = 0) or the field bit-reversed (first-listed qubit lowest, rev = 1).  Kernels
// use the field form when contig is set and the per-bit gather otherwise.
struct RegField {
    int contig, p0, rev;
};
inline RegField reg_field_of(const int *rpos, int w) {
    RegField f{0, 0, 0};
    bool asc = true, desc = true;
    for (int t = 0; t < w; ++t) {
        asc = asc && rpos[t] == rpos[0] + t;
        desc = desc && rpos[t] == rpos[0] - t;
    }
    if (w >= 1 && asc) f = RegField{1, rpos[0], 1};
    else if (w >= 1 && desc) f = RegField{1, rpos[w - 1], 0};
    return f;
}
#ifdef __CUDACC__
// I: the index type, 32 bits where the state allows; register values have at most 30
template <typename I>
__device__ __forceinline__ uint32_t field_get(I i, const RegField &f, int w) {
    const uint32_t v = (uint32_t)(i >> f.p0) & ((1u << w) - 1);
    return f.rev ? __brev(v) >> (32 - w) : v;
}
template <typename I>
__device__ __forceinline__ I field_put(I i, uint32_t x, const RegField &f, int w) {
    const uint32_t v = f.rev ? __brev(x) >> (32 - w) : x;
    const I m = (I)((1u << w) - 1) << f.p0;
    return (i & ~m) | ((I)v << f.p0);
}
// the value of a register on any bits (rpos[0] the most significant), and the index with
// that value replaced
template <typename I>
__device__ __forceinline__ uint32_t reg_get(I i, const RegField &f, const int *rpos, int w) {
    if (f.contig) return field_get<I>(i, f, w);
    uint32_t y = 0;
    for (int b = 0; b < w; ++b) y = (y << 1) | ((uint32_t)(i >> rpos[b]) & 1u);
    return y;
}
template <typename I>
__device__ __forceinline__ I reg_put(I i, uint32_t x, const RegField &f, const int *rpos, int w) {
    if (f.contig) return field_put<I>(i, x, f, w);
    for (int b = 0; b < w; ++b) {
        const I bit = (x >> (w - 1 - b)) & 1u;
        i = (i & ~((I)1 << rpos[b])) | (bit << rpos[b]);
    }
    return i;
}
#endif

// x -> c x mod N by a constant c, for 32-bit x (Shoup's form: with s = floor(2^32 c / N),
// q = floor(x s / 2^32) is the quotient or one less): two multiplies, a high multiply
// and a subtraction, where a Barrett step on 64-bit products takes some thirty.
struct MulConst {
    uint32_t c, s, N;
};
inline MulConst mul_const(uint64_t c, uint64_t N) {   // c < N <= 2^30
    return MulConst{(uint32_t)c, (uint32_t)((c << 32) / N), (uint32_t)N};
}
#ifdef __CUDACC__
__device__ __forceinline__ uint32_t mul_mod(uint32_t x, const MulConst &m) {
    uint32_t r = x * m.c - __umulhi(x, m.s) * m.N;    // exact modulo 2^32, below 2 N
    return r >= m.N ? r - m.N : r;
}
#endif

struct PermArgs {
    int w;
    int rpos[kMaxPermW];  // physical bit of register list entry a (a = 0 is the MSB)
    RegField field;       // zero (per-bit gather) unless set from rpos
    uint64_t cmask;
    uint64_t n_amps;
    int kind;             // 0 = mul-mod, 1 = table
    MulConst mul;         // mul-mod: y -> cinv * y mod N for y < N
    const uint32_t *finv; // table: inverse permutation
    Cond cond;
};

// Modular exponentiation of a register by a control register: for each basis
// state, the register value x < N becomes M x mod N, M the product of the
// multipliers whose control qubits are 1 (x >= N is left alone).  The controls go
// in groups of 8; tab[g][v] is the inverse of the product of group g's
// multipliers selected by the bits of v (the gather reads x = M^-1 y).
constexpr int kModExpMaxControls = 48;
constexpr int kModExpGroups = kModExpMaxControls / 8;
struct ModExpArgs {
    int w;
    int rpos[kMaxPermW];  // physical bit of register list entry a (a = 0 is the MSB)
    RegField field;       // zero (per-bit gather) unless set from rpos
    int nctl, ngroups;
    int cpos[kModExpMaxControls];   // physical bit of control j (group j / 8, bit j % 8)
    uint64_t n_amps;
    uint64_t N, mu;       // mu = floor((2^64-1)/N)
    Cond cond;
    uint32_t inv[kModExpMaxControls];   // inverse of multiplier j
    uint32_t tab[kModExpGroups][256];
};

// Device-side record of one single-qubit measurement decision.
struct MeasSlot {
    double p0;            // probability of reading 0
    double scale;         // 1/sqrt(P_m)
    int m;                // outcome
    int pad;
};

// Where a reduction's decision goes.  Every block of the reduction stores its
// (S0, S1) partials; the last block to finish (an atomic ticket, no waiting) adds
// all partials in a fixed order, so the result does not depend on timing, and
// records P0 = S0 / (S0 + S1), the outcome m = (u >= P0), 1/sqrt(S_m) and the cbit.
struct Decide {
    unsigned *counter;    // zero between launches; the deciding block resets it
    double u;
    MeasSlot *slot;
    uint8_t *cbits;
    int dest;             // destination cbit, -1: none
};
#ifdef __CUDACC__
// Running sum of FP32 terms kept as an unevaluated pair hi + lo (Knuth's TwoSum:
// the rounding error of each addition is carried in lo): about twice float's
// precision at the FP32 rate.  GB300's FP64 rate is too low for an FP64 add per
// term (2 FP64 lanes per SM per clock).
struct FSum {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float s = hi + x;
        const float bp = s - hi;
        const float e = (hi - (s - bp)) + (x - bp);
        hi = s;
        lo += e;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// The semiclassical phase exp(i theta), theta = -2 pi sum_l c_l / 2^(l+1) over the listed
// cbits, l = 1..n (64-bit fixed point), by one whole warp: a lane per cbit, so that
// their loads are one latency and not n of them.  Valid in lane 0.
__device__ __forceinline__ double2 warp_rphase(const int *idx, int n, const uint8_t *cbits) {
    const int lane = (int)(threadIdx.x & 31);
    uint32_t hi = 0, lo = 0;   // turns = sum of 2^(63 - l): bits 62 down to 1
    for (int l = lane + 1; l <= n; l += 32)
        if (cbits[idx[l - 1]]) {
            if (l < 32) hi |= 1u << (31 - l);
            else lo |= 1u << (63 - l);
        }
    hi = __reduce_or_sync(0xffffffffu, hi);
    lo = __reduce_or_sync(0xffffffffu, lo);
    double2 r = make_double2(1.0, 0.0);
    if (lane == 0) {
        const uint64_t turns = ((uint64_t)hi << 32) | lo;
        double s, c;
        sincospi(-2.0 * ((double)turns * 0x1p-64), &s, &c);
        r = make_double2(c, s);
    }
    return r;
}

// Sum over the block of one double per thread, the FP64 additions done by warp 0
// alone; sh holds blockDim.x doubles.  The result is valid in thread 0.
__device__ __forceinline__ double block_sum_w0(double v, double *sh) {
    __syncthreads();
    sh[threadIdx.x] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) {
        for (int k = threadIdx.x; k < (int)blockDim.x; k += 32) t += sh[k];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    }
    return t;
}

// Called by every thread of every block after thread 0 stored the block's
// partials[2 * blockIdx.x + {0, 1}].
__device__ __forceinline__ void last_block_decides(double *partials, const Decide &d) {
    __shared__ unsigned s_last;
    __shared__ double s_sum[2][32];
    if (threadIdx.x == 0) {
        __threadfence();                     // the partials before the ticket
        s_last = atomicAdd(d.counter, 1u) == gridDim.x - 1 ? 1u : 0u;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double a0 = 0.0, a1 = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
        a0 += __ldcg(&partials[2 * b]);
        a1 += __ldcg(&partials[2 * b + 1]);
    }
    for (int o = 16; o > 0; o >>= 1) {
        a0 += __shfl_xor_sync(0xffffffffu, a0, o);
        a1 += __shfl_xor_sync(0xffffffffu, a1, o);
    }
    if ((threadIdx.x & 31) == 0) {
        s_sum[0][threadIdx.x >> 5] = a0;
        s_sum[1][threadIdx.x >> 5] = a1;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s0 = 0.0, s1 = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            s0 += s_sum[0][w];
            s1 += s_sum[1][w];
        }
        const double tot = s0 + s1;
        const double p0 = tot > 0.0 ? s0 / tot : 1.0;
        const int m = (d.u >= p0) ? 1 : 0;
        const double pm = m ? s1 : s0;
        d.slot->p0 = p0;
        d.slot->m = m;
        d.slot->scale = pm > 0.0 ? 1.0 / sqrt(pm) : 0.0;
        if (d.dest >= 0) d.cbits[d.dest] = (uint8_t)m;
        *d.counter = 0;
    }
}
#endif

// Measurement of a list of qubits, up to kMeasRound decisions per round.  A round
// sums |a_i|^2 over the indices whose earlier measured bits equal the outcomes
// already decided (read from the slots on the device), into one bin per value of
// the round's qubits; the decisions then follow one qubit at a time from the bins.
constexpr int kMaxMeasure = 64;
constexpr int kMeasRound = 8;
// index bits below this are told apart by lane (and by the two amplitudes of a
// lane's 16-byte vector in complex64); the bits above select rows
__host__ __device__ constexpr int meas_low_bits(int prec) { return prec == 0 ? 6 : 5; }
struct MeasArgs {
    int n;
    int k;                // decisions already taken (prefix length); collapse: all decisions
    int nb;               // qubits decided in this round
    int pos[64];          // physical bit of measured qubit j (list order), j < k + nb
    int nins;             // row bits that are fixed (decided or a bin's), sorted ascending, for enumeration
    int ins[40];
    uint64_t n_rows;      // rows per bin value of the high qubits
    int bh;               // the round's qubits at or above the low bits: physical bit hpos[t] is
    int hpos[kMeasRound]; // bit t of the high bin
    uint32_t lmask;       // the round's qubits among the low bits
    int per_bin;          // blocks per high bin
    uint8_t src[kMeasRound];   // round qubit j: bit t of the high bin, or 64 + bit of the low bin
    double u[kMeasRound];      // its uniform
    int dest[kMeasRound];      // its destination cbit, -1: none
};
inline int meas_max_blocks(int sms) { return sms * 2 > (1 << kMeasRound) ? sms * 2 : 1 << kMeasRound; }
// doubles of partial sums a round may need
inline size_t meas_partials(int sms) { return (size_t)meas_max_blocks(sms) << 6; }

// One fused Kitaev stage (kernels_kitaev.cu): control qubit at physical bit
// cpos, register of w qubits at rpos[] (rpos[0] = MSB), permutation f given by
// its inverse (mul-mod: mul; table: finv), phase from cbits.
struct KitaevArgs {
    int cpos;
    int w;
    int rpos[kMaxPermW];
    RegField field;
    int kind;             // 0 = mul-mod, 1 = table
    MulConst mul;
    const uint32_t *finv;
    int n_rphase;
    int rphase_idx[kMaxRphase];
    uint64_t n_half;      // 2^(n-1): amplitudes with the control bit 0
};

// Qubit-relabelling gather: out[logical index] = in[physical index].
struct RelabelArgs {
    int n;
    int phys_of[40];      // physical bit of logical qubit
    uint64_t n_amps;
};

// ---------------------------------------------------------------------------
// fused tile pass (K3), complex64.  A tile is 2^13 amplitudes over 13 physical
// qubits S[0..12] (S[b] = b for b < 5, so 32 consecutive amplitudes form the
// lane dimension of every global access).  256 threads hold 32 amplitudes each
// in registers; three fixed "arrangements" say which local bits are register,
// lane and warp bits:
//   ARR_IO: lanes = local 0..4, registers = local 5..9,  warps = local 10..12
//   ARR_LO: registers = local 0..4, lanes = local 5..9,  warps = local 10..12
//   ARR_HI: lanes = local 0..4, registers = local 8..12, warps = local 5..7
// Gates act on register bits only; switching arrangement is a transpose through
// shared memory.  Loads use ARR_IO, stores use ARR_IO or ARR_HI.
// ---------------------------------------------------------------------------
constexpr int kTileQubits = 13;
// Physical qubits 0 .. kTileContig-1 belong to every tile pass, so a warp's loads
// and stores touch runs of 2^kTileContig contiguous amplitudes; the other tile
// qubits are chosen freely by the planner.  With 4 or 3 passes hold more gates but
// cost more transposes: the layered 30-qubit step 56.7 and 54.4 ms against 51.1, a
// 26-qubit request 4.53 and 4.60 against 4.42; better only without a QFT (28 qubits 8.27
// and 8.10 against 8.70).
constexpr int kTileContig = 5;
constexpr int kTileThreads = 256;
constexpr int kTileMaxOps = 192;
constexpr int kTileMaxTerms = 768;
// runs of consecutive fixed qubits: S holds 0..4 and eight more bits, which
// split the rest into at most nine runs
constexpr int kTileMaxRuns = 12;
constexpr int kTileMaxMats = 160;
constexpr int kTileMaxConds = 4;
enum TileArr : uint8_t { ARR_IO = 0, ARR_LO = 1, ARR_HI = 2 };
// TOP_U2L: a layer of uncontrolled 2x2 gates on distinct register bits (k is
// the bit mask); their descriptions are lg[first...] in bit order.  Before the gates, a
// CZ between register bits (k, l) for every bit set in tmask (bit cz_index(k, l) over
// the ten pairs, see below).  Bit b of rmask: the gate on register bit b updates the
// pair's stored |0> value first; of rval: it turns the |1> value; of tval: a sign by
// parity comes first; of count: phase terms come first (LayerGate).
// TOP_PAIRNEG: an unconditional sign flip of the amplitudes whose register bits k
// and l are both 1 (code k | l << 3): a CZ between two register bits.
// TOP_PAIRU: factor on the amplitudes whose register bits k and l (code k | l << 3)
// are both 1: a controlled phase between two register bits.
// TOP_PHQ: a thread- and tile-dependent phase on register bit k = 1, from the BitTerms
// [first, first + count) on thread bits and count2 more on tile-index bits (before a
// general gate; layer gates carry their own).
// TOP_U2, TOP_PHASE: controlled or conditioned 2x2 gate; factor on the amplitudes that
// match the op's register, thread, tile and classical conditions.
enum TileOpKind : uint8_t {
    TOP_U2 = 0, TOP_PHASE = 1, TOP_XPOSE = 2, TOP_PHQ = 3, TOP_U2L = 4, TOP_PAIRNEG = 7, TOP_PAIRU = 8
};
// "add turns (2^-32 of a turn) where the bit is 1": a thread-bit index (lane 0..4, warp
// 5..7) or a tile-index bit; in the final two-bit list b1 | b2 << 8, both bits of the
// index thread bits + 256 * tile index
struct BitTerm {
    uint32_t bit;
    uint32_t turns;
};
// the pairs k < l of register bits in the order (0,1) (0,2) (0,3) (0,4) (1,2)
// (1,3) (1,4) (2,3) (2,4) (3,4): the bit of a TOP_U2L op's CZ mask
__host__ __device__ constexpr int cz_index(int k, int l) { return k == 0 ? l - 1 : k == 1 ? l + 2 : k == 2 ? l + 4 : 9; }

// One gate of a TOP_U2L layer.  The planner may keep a local qubit's two values stored
// swapped ("flipped"); it picks the stored order of the gate's output so that, with M
// the gate in stored order and F the pending factor of the bit, the larger entries are
// on the diagonal.  With a0 = M01 F / M00 and a1 = M10 / (M11 F) the true outputs are
// M00 (y0 + a0 y1) and M11 F (y1 + a1 y0), and a0 a1 is real and negative.  Turning y1
// by e^{i phi} -- psi = arg a0 modulo pi, the sign goes into the updates -- makes both
// updates real: three shears of (re, im) for the turn (3 FMAs per pair, none when phi =
// 0), then, in place,
//   zf = 0:  y1 += c1 y0,  then y0 += c0 y1;   zf = 1: the other order
// (4 FMAs per pair).  7 FMAs per pair, against 8 for the same updates with complex
// coefficients, every one in place.  (A turn as 1 + i tan(phi), its cosine kept pending,
// is 2 FMAs but not in place: its register moves cost more, 103.8 ms of tile passes for
// the 30-qubit step.)  The updates leave s = 1 / (1 - a0 a1) in [1/2, 1] on one value;
// the planner picks zf so that the bit's pending magnitude stays near 1.
// The diagonal terms that wait on the qubit (the other qubit a thread or tile-index
// bit) come first, on the bit's |1>: when all are signs, by the parity of the thread bits
// ts and tile-index bits fs; else a phase from nt + ni BitTerms.  The turn is part of that
// phase then (h.x holds its 2^-32 turns as an integer, and the op's rval bit is clear).
struct LayerGate {
    float2 h, s;           // -tan(phi / 2), sin(phi), splatted
    float2 c0, c1;
    uint32_t fs;
    uint16_t ts, first;
    uint8_t nt, ni;
    uint8_t slot;          // of the phase in the kernel's tables, 0xff: no phase
    uint8_t pad;
};
constexpr int kTileSlots = 48;   // 7.5 KB: three CTAs still share an SM
static_assert(sizeof(LayerGate) == 48, "LayerGate layout");

struct TileOp {
    uint8_t kind;          // TileOpKind
    uint8_t k;             // U2: target register bit; XPOSE: new arrangement
    uint8_t rmask, rval;   // condition on register bits (5-bit register index space)
    uint16_t tmask, tval;  // condition on thread bits: bits 0..4 lane, 5..7 warp
    uint16_t cond;         // index into TileParams::conds, 0xffff = unconditional
    uint16_t count;
    uint16_t first;        // TOP_U2L: gates from lg[first]; TOP_PHQ: terms from bt[first]
    uint16_t count2;
    uint64_t gmask, gval;  // condition on the tile's fixed (non-tile) physical bits
    union {
        float m[8];        // U2: m00, m01, m10, m11 as (re, im)
        struct {
            float re, im;  // PHASE, PAIRU: factor
        } ph;
    };
};
// The tile kernel reads the fields the common op kinds need (kind, k, rmask, rval,
// tmask, tval, count, first, count2) as the op's first two 8-byte words, one op ahead.
static_assert(offsetof(TileOp, kind) == 0 && offsetof(TileOp, k) == 1 && offsetof(TileOp, rmask) == 2 &&
                  offsetof(TileOp, rval) == 3 && offsetof(TileOp, tmask) == 4 && offsetof(TileOp, tval) == 6 &&
                  offsetof(TileOp, count) == 10 && offsetof(TileOp, first) == 12 && offsetof(TileOp, count2) == 14,
              "TileOp head layout");
static_assert(alignof(TileOp) >= 8, "TileOp head is read as 8-byte words");

// The scalar part of a tile-pass program (the arrays follow in TileParams, or
// sit in device pools for a batched launch, see TileProg).
struct TileHead {
    uint64_t n_tiles;
    int n;
    int nfix;
    int8_t S[16];          // physical qubit of local bit b
    int8_t fixed[40];      // physical bits of the tile index, ascending
    // the same as runs of consecutive physical bits: tile-index bits [tlo, tlo +
    // len) land on physical bits [plo, plo + len)
    int nruns;
    uint8_t run_tlo[kTileMaxRuns], run_len[kTileMaxRuns], run_plo[kTileMaxRuns];
    int n_conds;
    Cond conds[kTileMaxConds];
    int nops;
    // final flush: the uniform pending factor of each local qubit's |1> (phase in
    // turns and magnitude), the uniform constant phase (fin_turns[13]) and the real
    // scale; a plan's last pass also applies the factors that earlier passes left on
    // qubits outside its S: fin_fixed[b] turns and fin_fixed_mag[b] where tile-index
    // bit b (qubit fixed[b]) is 1, for the bits set in fin_fixed_mask
    uint32_t fin_turns[14];
    float fin_mag[kTileQubits];
    float fin_scale;
    int need_tab;          // 0: every phase the pass can form is 0 or half a turn
    uint64_t fin_fixed_mask;
    uint32_t fin_fixed[40];
    float fin_fixed_mag[40];
    int fin_flip;          // local qubits stored flipped at the end (bit b: local qubit b)
    // diagonal terms that no gate of the plan called for (its last pass only): per
    // register bit BitTerms from bt[fin_first[k]], fin_nt[k] on thread bits, then fin_ni[k]
    // on tile-index bits; two-bit terms bt[fin2_first ...]
    uint16_t fin_first[5], fin2_first, fin2_n;
    uint8_t fin_nt[5], fin_ni[5];
    int nlg, nbt;          // entries of lg[] and bt[] in use
};

// A whole pass program, passed as kernel parameters for one state.
struct TileParams : TileHead {
    TileOp ops[kTileMaxOps];
    LayerGate lg[kTileMaxMats];
    BitTerm bt[kTileMaxTerms];
};

// A pass program of one circuit in a batched launch: the header plus offsets
// of its ops, layer gates and phase terms in device pools, and its state.
struct TileProg : TileHead {
    uint32_t op0, lg0, bt0, pad;
    float2 *psi;
};
static_assert(sizeof(TileParams) <= 32764, "tile program must fit in the kernel parameter space");

cudaError_t launch_tile(void *psi, const TileParams &p, const uint8_t *cbits, int sms, cudaStream_t s);
// Pass k of many circuits in one launch: CTA b runs tile (b - first[c]) of
// program c, where first[] (n_progs + 1 entries, ascending, first[0] = 0) splits
// the grid; programs are in n-qubit order so that the 32-bit offset kernel serves
// every circuit below 33 qubits.
// general: some program holds general ops (see tile_ops_need_general); without
// them a leaner instance of the kernel runs.
cudaError_t launch_tile_batch(const TileProg *progs, const uint32_t *first, int n_progs, uint32_t n_ctas,
                              const TileOp *ops, const LayerGate *lg, const BitTerm *bt, bool general,
                              int sms, cudaStream_t s);
// whether a pass program holds ops of the kinds TOP_U2, TOP_PHASE or TOP_PHQ
bool tile_ops_need_general(const TileOp *ops, size_t n);

// ---------------------------------------------------------------------------
// fused pass over tiles in shared memory (kernels_smem_tile.cu): complex128 states of
// any size, and complex64 states below the register tile's 13 qubits.  A tile is 2^m
// amplitudes over m physical qubits S[0..m-1] (ascending); the other n - m bits are the
// tile index.  GB300 does 2 FP64 lane operations per SM and clock, so in complex128 a
// pass is bound by its FP64 operations alone and the program is built to need few; in
// complex64 the states are small and the time goes to the latency of one op after
// another:
//   ST_U2    an uncontrolled 2x2 gate on local bit q, left-multiplied by a diagonal
//              that the planner keeps: y1 times i^k (1 + i t) (or y0 times its
//              conjugate), then two real in-place updates of one value from the
//              other: 6 FMAs per pair instead of the 16 operations of a complex 2x2
//              product; controlled-Z terms on q are sign flips on the way in
//   ST_X     exchange of the pair where the controls match (no arithmetic)
//   ST_CU2   controlled or conditioned 2x2 gate, 16 operations per matching pair
//   ST_SIGN  sign flips of the amplitudes with bit q set by a parity (no arithmetic)
//   ST_PH    one diagonal term on the matching amplitudes
//   ST_TABLE a product of factors, one per set local and tile-index bit, on the
//              amplitudes with bit q set (q = kNoBit: on all): two tables of 64
// ---------------------------------------------------------------------------
constexpr int kSmemTileMax = 12;      // local qubits
constexpr int kSmemTileOps = 144;
constexpr int kSmemTileFacs = 576;
constexpr uint8_t kNoBit = 0xff;
enum SmemTileKind : uint8_t { ST_U2 = 0, ST_X = 1, ST_CU2 = 2, ST_SIGN = 3, ST_PH = 4, ST_TABLE = 5 };
// ST_U2 flags: quarter turns in bits 0..1, then
constexpr uint8_t kU2Phase = 4;      // t != 0
constexpr uint8_t kU2On0 = 8;        // the phase goes on y0
constexpr uint8_t kU2First0 = 16;    // y0 is updated first
constexpr uint8_t kU2Swap = 32;      // the results are stored exchanged
constexpr uint8_t kU2Lift = 64;      // b0, b1 not both zero
struct SmemTileOp {
    uint8_t kind, q, flags, cond;    // cond: index into conds, kNoBit: none
    uint16_t lmask, lval;            // local-bit condition; U2, SIGN: parity mask in lmask; TABLE: bits with a factor
    uint32_t tmask, tval;            // the same on the tile index (U2, SIGN: parity mask in tmask)
    uint32_t tfac;                   // TABLE: tile-index bits with a factor
    uint32_t first;                  // TABLE: its factors, local bits ascending, then tile-index bits
    union {                          // U2: t, b0, b1; CU2: matrix; PH, TABLE: factor (re, im)
        double c[8];                 // (as the planner forms them, and in complex128 programs)
        float cf[8];                 // in complex64 programs
    };
};
static_assert(sizeof(SmemTileOp) % 8 == 0, "copied as 8-byte words");
struct SmemTileParams {
    uint32_t n_tiles;
    int n, m, nfix;
    int8_t S[kSmemTileMax + 4];
    int8_t fixed[32];                // physical bits of the tile index, ascending
    int n_conds;
    Cond conds[kTileMaxConds];
    int nops, nfac;
    SmemTileOp ops[kSmemTileOps];
    union {
        double2 fac[kSmemTileFacs];
        float2 facf[kSmemTileFacs];
    };
    SmemTileParams() {}
};
static_assert(sizeof(SmemTileParams) <= 32764, "tile program must fit in the kernel parameter space");
cudaError_t launch_smem_tile(int prec, void *psi, const SmemTileParams &p, const uint8_t *cbits, cudaStream_t s);

// ---------------------------------------------------------------------------
// dense k-qubit gates on CUDA cores (kernels_dense.cu): a pass keeps a tile of 2^m
// amplitudes over m physical qubits S[0..m-1] (ascending) in shared memory and applies
// a run of dense gates whose targets all lie in S.
// ---------------------------------------------------------------------------
constexpr int kDenseMaxK = 6;
constexpr int kDenseOps = 48;
constexpr int kDenseElems = 4096;    // matrix entries of one pass in shared memory
constexpr int kDenseMaxBits = 13;
// Shared-memory slot of local index i, linear over GF(2): index bits b, b + 4, b + 8 and
// b + 12 fold onto bank bit b
__host__ __device__ constexpr uint32_t dense_slot(uint32_t i) {
    return i ^ ((i >> 4) & 15u) ^ ((i >> 8) & 15u) ^ ((i >> 12) & 15u);
}
struct DenseOp {
    int8_t nfree;                // local bits that are neither targets nor local controls
    uint8_t cond;                // index into conds, 0xff: none
    uint16_t ls;                 // slot of the local control bits set
    uint16_t ts[kDenseMaxK];     // slot of register bit b (b = 0: the last-listed target)
    uint16_t fs[kDenseMaxBits];  // slots of the free bits; the first four on distinct banks where possible
    // k = 2: a thread's 16 amplitudes are the register values times ncs column bits (slots
    // cs); with pair set those are the next op's register bits, and both gates are applied
    // while the amplitudes are in registers (that op is then skipped)
    uint8_t pair, ncs;
    uint16_t cs[2];
    uint32_t tmask;              // tile-index control bits
    const void *mat;             // device matrix, 2^k x 2^k, row-major, amplitude type
};
struct DenseParams {
    uint64_t n_tiles;
    uint64_t base;               // physical control bits that every tile has set (not in S, not enumerated)
    int m, nfix;
    int8_t S[16];
    int8_t fixed[36];            // physical bits of the tile index, ascending
    int nops, k;                 // every gate of a pass has the same k
    int n_conds;
    Cond conds[kTileMaxConds];
    DenseOp ops[kDenseOps];
};
cudaError_t launch_dense(int prec, void *psi, const DenseParams &p, const uint8_t *cbits, int sms, cudaStream_t s);

// ---------------------------------------------------------------------------
// launchers (kernels_basic.cu); prec: 0 = complex64, 1 = complex128
// ---------------------------------------------------------------------------
cudaError_t launch_u2(int prec, void *psi, const U2Args &a, const uint8_t *cbits, int n, int sms,
                      cudaStream_t s);
cudaError_t launch_phase(int prec, void *psi, const PhaseArgs &a, const uint8_t *cbits, int sms,
                         cudaStream_t s);
cudaError_t launch_modexp(int prec, const void *in, void *out, const ModExpArgs &a, const uint8_t *cbits, int sms,
                          cudaStream_t s);
cudaError_t launch_perm(int prec, const void *in, void *out, const PermArgs &a, const uint8_t *cbits,
                        int sms, cudaStream_t s);
cudaError_t launch_measure_round(int prec, const void *psi, const MeasArgs &a, MeasSlot *slots, double *partials,
                                 unsigned *counter, uint8_t *cbits, int sms, cudaStream_t s);
cudaError_t launch_measure_collapse(int prec, void *psi, int n, const MeasArgs &a, const MeasSlot *slots, int sms,
                                    cudaStream_t s);
// one stage in one cooperative launch, for states that fit the register files; bar: two
// words, zero before the first launch (a ticket and a generation); err receives 1 if the
// grid barrier's bounded wait gave up
bool kitaev_stage_fits(int prec, uint64_t n_half, int sms);
cudaError_t launch_kitaev_stage(int prec, const void *psi, void *out, const KitaevArgs &a, const uint8_t *cbits,
                                double *partials, unsigned *bar, const Decide &d, int *err, int sms, cudaStream_t s);
cudaError_t launch_kitaev_reduce(int prec, const void *psi, const KitaevArgs &a, const uint8_t *cbits,
                                 double *partials, int nblocks, const Decide &d, cudaStream_t s);
cudaError_t launch_kitaev_update(int prec, const void *psi, void *out, const KitaevArgs &a, const uint8_t *cbits,
                                 const MeasSlot *slot, int sms, cudaStream_t s);
// K4 on tensor cores (kernels_block_tc.cu): dense 5-qubit complex64 unitary on
// physical qubits 0..4; bh/bl are the 64 x 64 split real embedding (row = output
// column); err receives 1 if a bounded wait gave up.
cudaError_t launch_block_tc(void *psi, int n, const float *bh, const float *bl, int *err, int sms, cudaStream_t s);
// one bounded mbarrier wait that runs out; sets *err (the timeout path's self-test)
cudaError_t launch_wait_selftest(int *err, cudaStream_t s);
cudaError_t launch_set_basis(int prec, void *psi, uint64_t index, cudaStream_t s);
cudaError_t launch_relabel(int prec, const void *in, void *out, const RelabelArgs &a, int sms,
                           cudaStream_t s);

}  // namespace qk
