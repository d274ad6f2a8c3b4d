// One-pass-per-gate kernels of libqk: 2x2 pair updates (K1), diagonal phases
// (K2), permutation gathers (K5), measurement (K6), and
// small helpers.  Every kernel streams the amplitudes it touches once, with
// 16-byte vector accesses where the qubit layout allows.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "qk_kernels.cuh"

namespace qk {
namespace {

constexpr int kThreads = 256;

template <typename R> struct Amp;
template <> struct Amp<float> { using T = float2; };
template <> struct Amp<double> { using T = double2; };

template <typename T>
__device__ __forceinline__ T cmul(T a, T b) {
    T r;
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
    return r;
}

// out = m0 * a + m1 * b
template <typename T>
__device__ __forceinline__ T cmac2(T m0, T a, T m1, T b) {
    T r;
    r.x = m0.x * a.x - m0.y * a.y + m1.x * b.x - m1.y * b.y;
    r.y = m0.x * a.y + m0.y * a.x + m1.x * b.y + m1.y * b.x;
    return r;
}

__device__ __forceinline__ bool cond_ok(const Cond &c, const uint8_t *cbits) {
    for (int k = 0; k < c.n; ++k)
        if (cbits[c.idx[k]] == 0) return false;
    return true;
}

// Insert a zero bit at each sorted position (ascending) of p into j.
__device__ __forceinline__ uint64_t insert_zeros(uint64_t j, const Positions &p) {
    for (int k = 0; k < p.n; ++k) {
        const uint64_t lo = j & ((1ull << p.pos[k]) - 1);
        j = ((j - lo) << 1) | lo;
    }
    return j;
}

// an index whose bits sit on arbitrary positions: lane t's bit at position p, over the warp
__device__ __forceinline__ uint64_t warp_deposit(bool bit, int p) {
    const uint64_t v = bit ? 1ull << p : 0ull;
    const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)v);
    const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(v >> 32));
    return ((uint64_t)hi << 32) | lo;
}

inline unsigned grid_for(uint64_t units, int sms, int per_sm = 16) {
    uint64_t b = (units + kThreads - 1) / kThreads;
    uint64_t cap = (uint64_t)sms * per_sm;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (unsigned)b;
}

// ---------------------------------------------------------------------------
// K1: 2x2 update on pairs (i0, i0 + 2^q) where every control bit is 1.
// V = 0: generic, one pair per unit, scalar amplitude accesses.
// V = 1: complex64, q == 0: the pair is one 16-byte vector.
// V = 2: complex64, q >= 1 and bit 0 free: two adjacent pairs per unit, two
//        16-byte vectors.
// ---------------------------------------------------------------------------
template <typename R, int V>
__global__ void __launch_bounds__(kThreads) k_u2(typename Amp<R>::T *psi, U2Args a, const uint8_t *cbits) {
    using T = typename Amp<R>::T;
    if (a.cond.n && !cond_ok(a.cond, cbits)) return;
    T m00, m01, m10, m11;
    m00.x = (R)a.m[0]; m00.y = (R)a.m[1];
    m01.x = (R)a.m[2]; m01.y = (R)a.m[3];
    m10.x = (R)a.m[4]; m10.y = (R)a.m[5];
    m11.x = (R)a.m[6]; m11.y = (R)a.m[7];
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t qbit = 1ull << a.q;
    for (uint64_t u = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; u < a.n_units; u += stride) {
        if constexpr (V == 1) {
            const uint64_t i0 = insert_zeros(u, a.ins) | a.cmask;
            float4 *p = reinterpret_cast<float4 *>(psi + i0);
            float4 v = *p;
            T x0 = make_float2(v.x, v.y), x1 = make_float2(v.z, v.w);
            T y0 = cmac2(m00, x0, m01, x1), y1 = cmac2(m10, x0, m11, x1);
            *p = make_float4(y0.x, y0.y, y1.x, y1.y);
        } else if constexpr (V == 2) {
            const uint64_t i0 = insert_zeros(u << 1, a.ins) | a.cmask;
            float4 *p0 = reinterpret_cast<float4 *>(psi + i0);
            float4 *p1 = reinterpret_cast<float4 *>(psi + (i0 | qbit));
            float4 v0 = *p0, v1 = *p1;
            T a0 = make_float2(v0.x, v0.y), b0 = make_float2(v1.x, v1.y);
            T a1 = make_float2(v0.z, v0.w), b1 = make_float2(v1.z, v1.w);
            T ya0 = cmac2(m00, a0, m01, b0), yb0 = cmac2(m10, a0, m11, b0);
            T ya1 = cmac2(m00, a1, m01, b1), yb1 = cmac2(m10, a1, m11, b1);
            *p0 = make_float4(ya0.x, ya0.y, ya1.x, ya1.y);
            *p1 = make_float4(yb0.x, yb0.y, yb1.x, yb1.y);
        } else {
            const uint64_t i0 = insert_zeros(u, a.ins) | a.cmask;
            const uint64_t i1 = i0 | qbit;
            T x0 = psi[i0], x1 = psi[i1];
            psi[i0] = cmac2(m00, x0, m01, x1);
            psi[i1] = cmac2(m10, x0, m11, x1);
        }
    }
}

// ---------------------------------------------------------------------------
// K2: multiply amplitudes with (i & mask) == val by a phase factor.
// V = 0 generic (one amplitude per unit); V = 1 complex64 with bit 0 outside
// the mask (two adjacent amplitudes per unit, one 16-byte vector).
// With n_rphase > 0 the factor is exp(-2 pi i sum_l c_l / 2^(l+1)) from cbits.
// ---------------------------------------------------------------------------
template <typename R, int V>
__global__ void __launch_bounds__(kThreads) k_phase(typename Amp<R>::T *psi, PhaseArgs a, const uint8_t *cbits) {
    using T = typename Amp<R>::T;
    if (a.cond.n && !cond_ok(a.cond, cbits)) return;
    // an angle from cbits is formed in FP64 once per block (GB300's FP64 rate is low)
    __shared__ double2 s_om;
    if (threadIdx.x < 32) {
        double2 om = make_double2(a.f_re, a.f_im);
        if (a.n_rphase) om = warp_rphase(a.rphase_idx, a.n_rphase, cbits);
        if (threadIdx.x == 0) s_om = om;
    }
    __syncthreads();
    T f;
    f.x = (R)s_om.x;
    f.y = (R)s_om.y;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t u = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; u < a.n_units; u += stride) {
        if constexpr (V == 1) {
            const uint64_t i = insert_zeros(u << 1, a.ins) | a.val;
            float4 *p = reinterpret_cast<float4 *>(psi + i);
            float4 v = *p;
            T x0 = cmul(make_float2(v.x, v.y), f), x1 = cmul(make_float2(v.z, v.w), f);
            *p = make_float4(x0.x, x0.y, x1.x, x1.y);
        } else {
            const uint64_t i = insert_zeros(u, a.ins) | a.val;
            psi[i] = cmul(psi[i], f);
        }
    }
}

// ---------------------------------------------------------------------------
// K5: controlled register permutation as an out-of-place gather:
// out[i] = in[src(i)], src replacing the register value y by f^-1(y).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t mulmod_barrett(uint64_t x, uint64_t y, uint64_t N, uint64_t mu) {
    const uint64_t p = x * y;                  // x, y < 2^30: exact
    const uint64_t q = __umul64hi(p, mu);      // floor(p / N) - {0, 1, 2}
    uint64_t r = p - q * N;
    while (r >= N) r -= N;
    return r;
}

template <typename R>
__global__ void __launch_bounds__(kThreads) k_perm(const typename Amp<R>::T *__restrict__ in,
                                                   typename Amp<R>::T *__restrict__ out, PermArgs a,
                                                   const uint8_t *cbits) {
    const bool active = (a.cond.n == 0) || cond_ok(a.cond, cbits);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n_amps; i += stride) {
        uint64_t src = i;
        if (active && (i & a.cmask) == a.cmask) {
            const uint32_t y = reg_get<uint64_t>(i, a.field, a.rpos, a.w);
            uint32_t x = y;
            if (a.kind != 0) x = a.finv[y];
            else if (y < a.mul.N) x = mul_mod(y, a.mul);
            src = reg_put<uint64_t>(i, x, a.field, a.rpos, a.w);
        }
        out[i] = in[src];
    }
}

// Modular exponentiation (ModExpArgs): one out-of-place gather for a whole run of
// controlled multiplications on one register.  The group tables go to shared
// memory once per block (their indices differ from lane to lane).
template <typename R>
__global__ void __launch_bounds__(kThreads) k_modexp(const typename Amp<R>::T *__restrict__ in,
                                                     typename Amp<R>::T *__restrict__ out,
                                                     const __grid_constant__ ModExpArgs a, const uint8_t *cbits) {
    __shared__ uint32_t tab[kModExpGroups * 256];
    for (int k = threadIdx.x; k < a.ngroups * 256; k += blockDim.x) tab[k] = a.tab[k >> 8][k & 255];
    __syncthreads();
    const bool active = (a.cond.n == 0) || cond_ok(a.cond, cbits);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n_amps; i += stride) {
        uint64_t src = i;
        if (active) {
            const uint32_t y = reg_get<uint64_t>(i, a.field, a.rpos, a.w);
            if (y < a.N) {
                uint64_t m = 1;
                for (int g = 0; g < a.ngroups; ++g) {
                    uint32_t v = 0;
                    const int j0 = 8 * g, j1 = min(a.nctl, j0 + 8);
                    for (int j = j0; j < j1; ++j) v |= (uint32_t)((i >> a.cpos[j]) & 1u) << (j - j0);
                    const uint64_t t = tab[(g << 8) | v];
                    m = g == 0 ? t : mulmod_barrett(m, t, a.N, a.mu);
                }
                const uint64_t x = mulmod_barrett(m, y, a.N, a.mu);
                src = reg_put<uint64_t>(i, (uint32_t)x, a.field, a.rpos, a.w);
            }
        }
        out[i] = in[src];
    }
}

// The same gather through shared memory, for a register on consecutive physical
// bits that is narrow enough: a tile is every register value times the lowest other
// bits (c of them, so that reads and writes are runs of at least 32 bytes).  The
// control register of the order-finding circuit holds the lowest bits, so
// neighbouring amplitudes take different multipliers: k_modexp's lanes each read
// another sector and use 8 of its 32 bytes, here every sector is read once.  The
// multiplier of each of the tile's 2^c control patterns is formed once per tile.
// HBM-bound by bytes: at 27 qubits (9-bit register above 18 controls,
// complex64) 2.64 -> 0.45 ms, 4.8 TB/s.
constexpr int kModExpMaxLow = 8;   // at most 2^8 control patterns per tile
struct ModExpTiled {
    int w, cb, n_other;
    int lp0, rev;                  // the register is local bits lp0 .. lp0 + w - 1
    uint64_t n_tiles;
    uint32_t N, mu;                // N <= 2^14: products stay below 2^28; mu = floor((2^32-1)/N)
    uint8_t bit[16];               // local bit -> physical bit, ascending
    uint8_t other[36];             // tile-index bit -> physical bit
    int nctl;
    uint8_t cpos[kModExpMaxControls];
    uint32_t inv[kModExpMaxControls];
    Cond cond;
};

__device__ __forceinline__ uint32_t mulmod_small(uint32_t x, uint32_t y, uint32_t N, uint32_t mu) {
    const uint32_t p = x * y;                  // x, y < 2^14: exact
    uint32_t r = p - __umulhi(p, mu) * N;      // the quotient is low by at most 2
    while (r >= N) r -= N;
    return r;
}

template <typename R>
__global__ void __launch_bounds__(kThreads) k_modexp_tiled(const typename Amp<R>::T *__restrict__ in,
                                                           typename Amp<R>::T *__restrict__ out,
                                                           const __grid_constant__ ModExpTiled a,
                                                           const uint8_t *cbits) {
    using T = typename Amp<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *buf = reinterpret_cast<T *>(smem_raw);
    __shared__ uint32_t mtab[1 << kModExpMaxLow];
    __shared__ uint64_t offj[64];              // offsets of the local bits from 8 on
    const int tid = threadIdx.x, lane = tid & 31;
    const int tb = a.w + a.cb, M = 1 << tb;
    const int rounds = M > kThreads ? M / kThreads : 1;
    const bool active = (a.cond.n == 0) || cond_ok(a.cond, cbits);
    uint64_t off0 = 0;
    for (int k = 0; k < 8 && k < tb; ++k)
        if ((tid >> k) & 1) off0 |= 1ull << a.bit[k];
    if (tid < rounds) {
        uint64_t o = 0;
        for (int k = 8; k < tb; ++k)
            if ((tid >> (k - 8)) & 1) o |= 1ull << a.bit[k];
        offj[tid] = o;
    }
    const uint32_t rmask = (1u << a.w) - 1, lomask = (1u << a.lp0) - 1;
    // thread t < 2^cb: the offset of control pattern t (the local bits outside the register)
    uint64_t coff = 0;
    for (int k = 0; k < a.cb; ++k)
        if ((tid >> k) & 1) coff |= 1ull << a.bit[k < a.lp0 ? k : k + a.w];
    __syncthreads();
    const bool live = tid < M;
    for (uint64_t tile = blockIdx.x; tile < a.n_tiles; tile += gridDim.x) {
        // the tile's base; tile-index bits above 32 (never at sizes that fit) by hand
        uint64_t base = warp_deposit(lane < a.n_other && ((tile >> lane) & 1u), lane < a.n_other ? a.other[lane] : 0);
        for (int t = 32; t < a.n_other; ++t)
            if ((tile >> t) & 1u) base |= 1ull << a.other[t];
        const T *src = in + (base | off0);
        if (live) {
            for (int j0 = 0; j0 < rounds; j0 += 8) {
                T v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (j0 + j < rounds) v[j] = src[offj[j0 + j]];
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (j0 + j < rounds) buf[tid + (j0 + j) * kThreads] = v[j];
            }
        }
        if (tid < (1 << a.cb)) {
            const uint64_t i = base | coff;
            uint32_t m = 1u % a.N;
            for (int j = 0; j < a.nctl; ++j)
                if ((i >> a.cpos[j]) & 1u) m = mulmod_small(m, a.inv[j], a.N, a.mu);
            mtab[tid] = m;
        }
        __syncthreads();
        if (live) {
            T *dst = out + (base | off0);
#pragma unroll 4
            for (int j = 0; j < rounds; ++j) {
                const uint32_t L = (uint32_t)(tid + j * kThreads);
                uint32_t y = (L >> a.lp0) & rmask;
                if (a.rev) y = __brev(y) >> (32 - a.w);
                uint32_t s = L;
                if (active && y < a.N) {
                    const uint32_t c = (L & lomask) | ((L >> (a.lp0 + a.w)) << a.lp0);
                    uint32_t x = mulmod_small(mtab[c], y, a.N, a.mu);
                    if (a.rev) x = __brev(x) >> (32 - a.w);
                    s = (L & ~(rmask << a.lp0)) | (x << a.lp0);
                }
                dst[offj[j]] = buf[s];
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// K6: measurement, up to kMeasRound qubits per read of the state.  One qubit at a
// time, P0 of the next qubit needs only sums of |a|^2 over the amplitudes that
// match the outcomes so far, and the sums over every value of eight qubits give all
// of those for eight decisions: one pass over 2^n amplitudes, then one over 2^(n-8),
// instead of passes over 2^n, 2^(n-1), ... with a launch and a deciding block each.
// A row is 2^L consecutive amplitudes, one 16-byte vector per lane, so measured bits
// below L never mix across lanes and need no branch; a block sums rows of one value
// of the round's higher bits.  The last block to finish (an atomic ticket, no
// waiting) adds the block partials in a fixed order, so results do not depend on
// timing.  complex64 sums run in compensated FP32 (a float pair that carries each
// addition's rounding error, about twice float's precision) and reach FP64 once per
// thread: GB300 has 2 FP64 lanes per SM per clock.  HBM-bound on large states,
// launch-bound on small ones: 8 qubits of a 30-qubit complex64 state 2.90 -> 1.25 ms
// (6.9 TB/s), 9 of 27 qubits 458 -> 194 us, 12 of 12 (complex128) 119 -> 24 us, one
// qubit of 26 108 -> 101 us.
// ---------------------------------------------------------------------------
// prefix value of the decided outcomes: sum_j m_j << pos[j], j < k (whole warps)
__device__ __forceinline__ uint64_t prefix_value(const MeasArgs &a, const MeasSlot *slots, int k) {
    uint64_t v = 0;
    for (int j0 = 0; j0 < k; j0 += 32) {
        const int j = j0 + (int)(threadIdx.x & 31);
        v |= warp_deposit(j < k && (slots[j].m & 1), j < k ? a.pos[j] : 0);
    }
    return v;
}

constexpr int kMeasThreads = 512;

template <typename R>
__global__ void __launch_bounds__(kMeasThreads, 2)
    k_meas_round(const typename Amp<R>::T *__restrict__ psi, const __grid_constant__ MeasArgs a, MeasSlot *slots,
                 double *partials, unsigned *counter, uint8_t *cbits) {
    constexpr bool kF = sizeof(R) == 4;
    constexpr int L = meas_low_bits(kF ? 0 : 1), W = 1 << L, kWarps = kMeasThreads / 32;
    __shared__ double sh[kWarps * W];
    __shared__ unsigned s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t pv = prefix_value(a, slots, a.k);
    uint64_t pm = 0;
    for (int j = 0; j < a.k; ++j) pm |= 1ull << a.pos[j];
    const uint32_t plm = (uint32_t)pm & (W - 1), plv = (uint32_t)pv & (W - 1);
    const int hb = (int)(blockIdx.x / a.per_bin), p = (int)(blockIdx.x % a.per_bin);
    uint64_t base = pv & ~(uint64_t)(W - 1);
    for (int t = 0; t < a.bh; ++t) base |= (uint64_t)((hb >> t) & 1) << a.hpos[t];
    // this lane's amplitudes of a row and whether the decided low bits let them in
    const uint32_t i0 = kF ? 2 * lane : lane;
    const uint32_t lim = a.n < L ? 1u << a.n : (uint32_t)W;
    const bool in0 = i0 < lim && (i0 & plm) == plv, in1 = kF && i0 + 1 < lim && ((i0 + 1) & plm) == plv;
    double d0 = 0.0, d1 = 0.0;
    if (in0 || in1) {
        FSum g0, g1;
        const uint64_t stride = (uint64_t)a.per_bin * kWarps, r0 = (uint64_t)p * kWarps + warp;
        // the free row bits count up around the fixed ones: a carry runs through the
        // fixed bits when they are set for the addition
        uint64_t fixed = 0, at = r0, step = stride;
        for (int t = 0; t < a.nins; ++t) {
            const uint64_t m = (1ull << a.ins[t]) - 1;
            at += at & ~m;
            step += step & ~m;
            fixed |= m + 1;
        }
        at <<= L;
        step <<= L;
        fixed <<= L;
        const typename Amp<R>::T *q = psi + (base | i0);
        // several rows' loads in flight per lane before the first is added
        constexpr int U = 8;
        const int64_t todo = r0 < a.n_rows ? (int64_t)((a.n_rows - r0 + stride - 1) / stride) : 0;
        for (int64_t left = todo; left > 0; left -= U) {
            typename std::conditional<kF, float4, double2>::type v[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                v[k].x = v[k].y = 0;
                if constexpr (kF) v[k].z = v[k].w = 0.f;
                if (k < left) {
                    if constexpr (kF) v[k] = *reinterpret_cast<const float4 *>(q + at);
                    else v[k] = q[at];
                    at = ((at | fixed) + step) & ~fixed;
                }
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                if constexpr (kF) {
                    g0.add(v[k].x * v[k].x + v[k].y * v[k].y);
                    g1.add(v[k].z * v[k].z + v[k].w * v[k].w);
                } else {
                    d0 += v[k].x * v[k].x + v[k].y * v[k].y;
                }
            }
        }
        if constexpr (kF) {
            d0 = g0.value();
            d1 = g1.value();
        }
    }
    if constexpr (kF) {
        sh[warp * W + 2 * lane] = in0 ? d0 : 0.0;
        sh[warp * W + 2 * lane + 1] = in1 ? d1 : 0.0;
    } else {
        sh[warp * W + lane] = d0;
    }
    __syncthreads();
    const int bl = __popc(a.lmask);
    if (warp == 0) {
        // over the warps, then over the low bits that this round does not decide
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            s0 += sh[w * W + lane];
            if (kF) s1 += sh[w * W + 32 + lane];
        }
        for (int k = 0; k < 5; ++k)
            if (!((a.lmask >> k) & 1u)) {
                s0 += __shfl_xor_sync(0xffffffffu, s0, 1 << k);
                if (kF) s1 += __shfl_xor_sync(0xffffffffu, s1, 1 << k);
            }
        if (kF && !((a.lmask >> 5) & 1u)) s0 += s1;
        if ((lane & ~a.lmask) == 0) {   // one lane per value of the round's low bits
            int c = 0, k2 = 0;
            for (int k = 0; k < 5; ++k)
                if ((a.lmask >> k) & 1u) c |= ((lane >> k) & 1) << k2++;
            double *out = partials + ((size_t)blockIdx.x << bl);
            out[c] = s0;
            if (kF && ((a.lmask >> 5) & 1u)) out[c | (1 << k2)] = s1;
            __threadfence();            // the partials before the ticket
        }
        __syncwarp();
        if (lane == 0) s_last = atomicAdd(counter, 1u) == gridDim.x - 1 ? 1u : 0u;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // bin e holds the round's qubits in list order, the first as its highest bit:
    // a tree of pair sums (node x of level j at sh[2^j + x]) gives every decision
    const int bins = 1 << a.nb, parts = kMeasThreads >> a.nb;
    {
        const int e = tid & (bins - 1), part = tid >> a.nb;
        int h = 0, c = 0;
        for (int j = 0; j < a.nb; ++j) {
            const int bit = (e >> (a.nb - 1 - j)) & 1, s = a.src[j];
            if (s < 64) h |= bit << s;
            else c |= bit << (s - 64);
        }
        const double *in = partials + ((size_t)h * a.per_bin << bl) + c;
        double s = 0.0;
#pragma unroll 4
        for (int b = part; b < a.per_bin; b += parts) s += __ldcg(in + ((size_t)b << bl));
        __syncthreads();
        sh[tid] = s;                    // part-major: sh[part * bins + e]
    }
    for (int w = parts >> 1; w > 0; w >>= 1) {
        __syncthreads();
        if (tid < w * bins) sh[tid] += sh[tid + w * bins];
    }
    __syncthreads();
    {
        const double v = tid < bins ? sh[tid] : 0.0;
        __syncthreads();
        if (tid < bins) sh[bins + tid] = v;
    }
    for (int j = a.nb - 1; j >= 0; --j) {
        __syncthreads();
        if (tid < (1 << j)) sh[(1 << j) + tid] = sh[(2 << j) + 2 * tid] + sh[(2 << j) + 2 * tid + 1];
    }
    __syncthreads();
    if (warp == 0) {
        int node = 0;
        double mine = 0.0, p0_mine = 1.0;
        int m_mine = 0;
        for (int j = 0; j < a.nb; ++j) {
            const double s0 = sh[(2 << j) + 2 * node], s1 = sh[(2 << j) + 2 * node + 1];
            const double tot = s0 + s1;
            const double p0 = tot > 0.0 ? s0 / tot : 1.0;
            const int m = (a.u[j] >= p0) ? 1 : 0;
            if (lane == j) {
                mine = m ? s1 : s0;
                p0_mine = p0;
                m_mine = m;
            }
            node = 2 * node + m;
        }
        if (lane < a.nb) {
            MeasSlot *sl = slots + a.k + lane;
            sl->p0 = p0_mine;
            sl->m = m_mine;
            sl->scale = mine > 0.0 ? 1.0 / sqrt(mine) : 0.0;
            if (a.dest[lane] >= 0) cbits[a.dest[lane]] = (uint8_t)m_mine;
        }
        if (lane == 0) *counter = 0;
    }
}

// Project onto the decided outcomes of every measured qubit and renormalise:
// amplitudes that match keep a * 1/sqrt(P), the others are written as zero
// without being read.
template <typename R>
__global__ void __launch_bounds__(kThreads) k_meas_collapse(typename Amp<R>::T *psi, uint64_t n_amps, MeasArgs a,
                                                            const MeasSlot *slots) {
    uint64_t M = 0;
    for (int j = 0; j < a.k; ++j) M |= 1ull << a.pos[j];
    const uint64_t V = prefix_value(a, slots, a.k);
    const R sc = (R)slots[a.k - 1].scale;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (sizeof(R) == 4) {
        float4 *p = reinterpret_cast<float4 *>(psi);
        for (uint64_t u = tid; u < (n_amps >> 1); u += stride) {
            const uint64_t i = u << 1;
            const bool ka = (i & M) == V, kb = ((i + 1) & M) == V;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (ka || kb) {
                v = p[u];
                const float sa = ka ? sc : 0.f, sb = kb ? sc : 0.f;
                v.x *= sa; v.y *= sa; v.z *= sb; v.w *= sb;
            }
            p[u] = v;
        }
    } else {
        for (uint64_t i = tid; i < n_amps; i += stride) {
            typename Amp<R>::T v;
            v.x = 0;
            v.y = 0;
            if ((i & M) == V) {
                v = psi[i];
                v.x *= sc;
                v.y *= sc;
            }
            psi[i] = v;
        }
    }
}

template <typename R>
__global__ void k_set_basis(typename Amp<R>::T *psi, uint64_t index) {
    typename Amp<R>::T one;
    one.x = 1;
    one.y = 0;
    psi[index] = one;
}

// Qubit relabelling, tiled: out[index with bit j] = in[index with bit phys_of[j]].
// A tile is every value of up to ten bits: the output's five lowest, the bits that
// the input's five lowest go to, and the lowest others up to ten; its amplitudes
// are read as runs along the input low bits and written as runs along the output
// low bits (at least 32 amplitudes each), through shared memory.  HBM-bound (one
// read and one write of the state).  Every offset is a sum over the bits of an
// index, so a thread keeps the part its own index gives (in, out and shared slot)
// in registers and the few bits beyond the block size come from kernel
// parameters; a tile's base is formed by one warp, one bit per lane.  Before, each
// block first copied 18 KB of offset tables from the kernel parameters, whose
// lane-dependent reads serialise.  Measured (complex64, bits moved to the other end):
// 30 qubits 4.44 -> 2.70 ms (6.37 TB/s), 27 qubits 555 -> 325 us, 24 qubits 398 -> 41 us,
// 21 qubits 26 -> 5 us.
constexpr int kRelabelBits = 10;
struct RelabelTiled {
    int m, n_other;
    uint64_t n_tiles;
    // local bit k of a tile element in input order sits at input bit in_bit[k]; in
    // output order at output bit out_bit[k], and its bit k is input-local bit src_bit[k]
    uint8_t in_bit[kRelabelBits], out_bit[kRelabelBits], src_bit[kRelabelBits];
    uint8_t other_in[32], other_out[32];   // tile-index bit t -> input / output bit
};

// the tile buffer is XOR-swizzled on its low five index bits so that reads along
// either side's runs stay conflict-free; linear over GF(2)
__device__ __forceinline__ int relabel_slot(int u) { return u ^ ((u >> 5) & 31); }

// J = 2^m / kThreads elements per thread (1 when the tile is smaller)
template <typename R, int J>
__global__ void __launch_bounds__(kThreads) k_relabel_tiled(const typename Amp<R>::T *__restrict__ in,
                                                            typename Amp<R>::T *__restrict__ out,
                                                            const __grid_constant__ RelabelTiled a) {
    using T = typename Amp<R>::T;
    constexpr int kB = 8;                      // bits of the thread index
    static_assert(kThreads == 1 << kB, "thread bits");
    __shared__ T buf[2][J * kThreads];
    const int tid = threadIdx.x, lane = tid & 31;
    const bool live = tid < (1 << a.m);        // false only for tiles below the block size
    const int mb = a.m < kB ? a.m : kB;
    uint64_t in0 = 0, out0 = 0;                // the thread's part of the offsets and slots
    int src0 = 0;
    for (int k = 0; k < mb; ++k)
        if ((tid >> k) & 1) {
            in0 |= 1ull << a.in_bit[k];
            out0 |= 1ull << a.out_bit[k];
            src0 |= 1 << a.src_bit[k];
        }
    const int put0 = relabel_slot(tid), get0 = relabel_slot(src0);
    // the bits beyond the block size (J = 2: one, J = 4: two): offsets and slots per bit
    uint64_t in_hi[2] = {0, 0}, out_hi[2] = {0, 0};
    int get_hi[2] = {0, 0};
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if ((1 << k) < J) {
            in_hi[k] = 1ull << a.in_bit[kB + k];
            out_hi[k] = 1ull << a.out_bit[kB + k];
            get_hi[k] = relabel_slot(1 << a.src_bit[kB + k]);
        }
    const int p_in = lane < a.n_other ? a.other_in[lane] : 0, p_out = lane < a.n_other ? a.other_out[lane] : 0;
    int b = 0;
    for (uint64_t tile = blockIdx.x; tile < a.n_tiles; tile += gridDim.x, b ^= 1) {
        const bool bit = lane < a.n_other && ((tile >> lane) & 1u);
        const T *src = in + (warp_deposit(bit, p_in) | in0);
        T *dst = out + (warp_deposit(bit, p_out) | out0);
        if (live) {
            T v[J];
#pragma unroll
            for (int j = 0; j < J; ++j) v[j] = src[((j & 1) ? in_hi[0] : 0) + ((j & 2) ? in_hi[1] : 0)];
#pragma unroll
            for (int j = 0; j < J; ++j) buf[b][put0 ^ relabel_slot(j << kB)] = v[j];
        }
        // two buffers: the next tile's writes go to the other one, so one barrier per
        // tile separates a buffer's reads from its next writes as well
        __syncthreads();
        if (live) {
#pragma unroll
            for (int j = 0; j < J; ++j)
                dst[((j & 1) ? out_hi[0] : 0) + ((j & 2) ? out_hi[1] : 0)] =
                    buf[b][get0 ^ ((j & 1) ? get_hi[0] : 0) ^ ((j & 2) ? get_hi[1] : 0)];
        }
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_u2(int prec, void *psi, const U2Args &a, const uint8_t *cbits, int n, int sms,
                      cudaStream_t s) {
    (void)n;
    if (prec == 0) {
        const bool bit0_control = (a.cmask & 1ull) != 0;
        if (a.q == 0) {
            k_u2<float, 1><<<grid_for(a.n_units, sms), kThreads, 0, s>>>((float2 *)psi, a, cbits);
        } else if (!bit0_control && a.n_units >= 2) {
            U2Args b = a;
            b.n_units = a.n_units >> 1;
            k_u2<float, 2><<<grid_for(b.n_units, sms), kThreads, 0, s>>>((float2 *)psi, b, cbits);
        } else {
            k_u2<float, 0><<<grid_for(a.n_units, sms), kThreads, 0, s>>>((float2 *)psi, a, cbits);
        }
    } else {
        k_u2<double, 0><<<grid_for(a.n_units, sms), kThreads, 0, s>>>((double2 *)psi, a, cbits);
    }
    return cudaGetLastError();
}

cudaError_t launch_phase(int prec, void *psi, const PhaseArgs &a, const uint8_t *cbits, int sms,
                         cudaStream_t s) {
    if (prec == 0) {
        if ((a.mask & 1ull) == 0 && a.n_units >= 2) {
            PhaseArgs b = a;
            b.n_units = a.n_units >> 1;
            k_phase<float, 1><<<grid_for(b.n_units, sms), kThreads, 0, s>>>((float2 *)psi, b, cbits);
        } else {
            k_phase<float, 0><<<grid_for(a.n_units, sms), kThreads, 0, s>>>((float2 *)psi, a, cbits);
        }
    } else {
        k_phase<double, 0><<<grid_for(a.n_units, sms), kThreads, 0, s>>>((double2 *)psi, a, cbits);
    }
    return cudaGetLastError();
}

// k_modexp_tiled where the register is a field of at most 12 bits (complex64) whose
// tile keeps runs of 32 bytes; anything else goes to k_modexp
template <typename R>
static bool modexp_tile(const ModExpArgs &a, ModExpTiled &t) {
    int n = 0;
    while ((1ull << n) < a.n_amps) ++n;
    const int full = sizeof(R) == 4 ? 13 : 12;           // 64 KiB of amplitudes: three blocks per SM
    const int need = a.field.p0 == 0 ? 0 : (sizeof(R) == 4 ? 2 : 1);
    if (!a.field.contig || a.w > 14 || a.w + need > full + 1 || n - a.w < need) return false;
    int cb = full - a.w;
    if (cb < need) cb = need;                            // 128 KiB: one block per SM
    if (cb > kModExpMaxLow) cb = kModExpMaxLow;
    if (cb > n - a.w) cb = n - a.w;
    t.w = a.w;
    t.cb = cb;
    t.rev = a.field.rev;
    t.N = (uint32_t)a.N;
    t.mu = 0xffffffffu / t.N;
    t.nctl = a.nctl;
    for (int j = 0; j < a.nctl; ++j) {
        t.cpos[j] = (uint8_t)a.cpos[j];
        t.inv[j] = a.inv[j];
    }
    t.cond = a.cond;
    const int p0 = a.field.p0, p1 = p0 + a.w;            // the register's bits
    t.lp0 = p0 < cb ? p0 : cb;
    int k = 0, left = cb;
    for (int p = 0; p < n; ++p) {
        const bool reg = p >= p0 && p < p1;
        if (reg || left > 0) {
            t.bit[k++] = (uint8_t)p;
            left -= reg ? 0 : 1;
        } else {
            t.other[t.n_other++] = (uint8_t)p;
        }
    }
    t.n_tiles = 1ull << t.n_other;
    return true;
}

template <typename R>
static cudaError_t modexp_r(const void *in, void *out, const ModExpArgs &a, const uint8_t *cbits, int sms,
                            cudaStream_t s) {
    using T = typename Amp<R>::T;
    ModExpTiled t{};
    if (!modexp_tile<R>(a, t)) {
        k_modexp<R><<<grid_for(a.n_amps, sms), kThreads, 0, s>>>((const T *)in, (T *)out, a, cbits);
        return cudaGetLastError();
    }
    const size_t sm = sizeof(T) << (t.w + t.cb);
    static SmemLimit limit;
    const cudaError_t e = smem_limit(k_modexp_tiled<R>, (size_t)128 * 1024, limit);
    if (e != cudaSuccess) return e;
    const uint64_t cap = (uint64_t)sms * (sm > 100 * 1024 ? 1 : sm > 48 * 1024 ? 3 : 6);
    k_modexp_tiled<R><<<(unsigned)(t.n_tiles < cap ? t.n_tiles : cap), kThreads, sm, s>>>((const T *)in, (T *)out, t, cbits);
    return cudaGetLastError();
}

cudaError_t launch_modexp(int prec, const void *in, void *out, const ModExpArgs &a, const uint8_t *cbits, int sms,
                          cudaStream_t s) {
    return prec == 0 ? modexp_r<float>(in, out, a, cbits, sms, s) : modexp_r<double>(in, out, a, cbits, sms, s);
}

cudaError_t launch_perm(int prec, const void *in, void *out, const PermArgs &a, const uint8_t *cbits,
                        int sms, cudaStream_t s) {
    if (prec == 0)
        k_perm<float><<<grid_for(a.n_amps, sms), kThreads, 0, s>>>((const float2 *)in, (float2 *)out, a, cbits);
    else
        k_perm<double><<<grid_for(a.n_amps, sms), kThreads, 0, s>>>((const double2 *)in, (double2 *)out, a, cbits);
    return cudaGetLastError();
}

cudaError_t launch_measure_round(int prec, const void *psi, const MeasArgs &args, MeasSlot *slots, double *partials,
                                 unsigned *counter, uint8_t *cbits, int sms, cudaStream_t s) {
    MeasArgs a = args;
    const int L = meas_low_bits(prec);
    if (a.n < 1 || a.nb < 1 || a.nb > kMeasRound) return cudaErrorInvalidValue;
    bool fixed[64] = {false};
    a.bh = 0;
    a.lmask = 0;
    for (int j = 0; j < a.k + a.nb; ++j) {
        const int q = a.pos[j];
        if (q >= L) fixed[q] = true;
        if (j < a.k) continue;
        if (q >= L) {
            a.src[j - a.k] = (uint8_t)a.bh;
            a.hpos[a.bh++] = q;
        } else {
            a.lmask |= 1u << q;
        }
    }
    for (int j = 0; j < a.nb; ++j) {   // a low qubit's rank among the round's low qubits
        const int q = a.pos[a.k + j];
        if (q < L) a.src[j] = (uint8_t)(64 + __builtin_popcount(a.lmask & ((1u << q) - 1)));
    }
    a.nins = 0;
    for (int q = L; q < a.n; ++q)
        if (fixed[q]) a.ins[a.nins++] = q - L;
    a.n_rows = a.n > L ? 1ull << (a.n - L - a.nins) : 1;
    // enough blocks to fill the device, no more than one row per warp
    const int cap = sms * 2;
    const uint64_t row_blocks = (a.n_rows + kMeasThreads / 32 - 1) / (kMeasThreads / 32);
    int per = cap >> a.bh;
    if (per < 1) per = 1;
    if ((uint64_t)per > row_blocks) per = (int)row_blocks;
    a.per_bin = per;
    const unsigned grid = (unsigned)per << a.bh;
    if (prec == 0)
        k_meas_round<float><<<grid, kMeasThreads, 0, s>>>((const float2 *)psi, a, slots, partials, counter, cbits);
    else
        k_meas_round<double><<<grid, kMeasThreads, 0, s>>>((const double2 *)psi, a, slots, partials, counter, cbits);
    return cudaGetLastError();
}

cudaError_t launch_measure_collapse(int prec, void *psi, int n, const MeasArgs &a, const MeasSlot *slots, int sms,
                                    cudaStream_t s) {
    const uint64_t n_amps = 1ull << n;
    if (prec == 0)
        k_meas_collapse<float><<<grid_for(n_amps >> 1, sms), kThreads, 0, s>>>((float2 *)psi, n_amps, a, slots);
    else
        k_meas_collapse<double><<<grid_for(n_amps, sms), kThreads, 0, s>>>((double2 *)psi, n_amps, a, slots);
    return cudaGetLastError();
}

cudaError_t launch_set_basis(int prec, void *psi, uint64_t index, cudaStream_t s) {
    if (prec == 0)
        k_set_basis<float><<<1, 1, 0, s>>>((float2 *)psi, index);
    else
        k_set_basis<double><<<1, 1, 0, s>>>((double2 *)psi, index);
    return cudaGetLastError();
}

cudaError_t launch_relabel(int prec, const void *in, void *out, const RelabelArgs &a, int sms,
                           cudaStream_t s) {
    // tile bits: output bits 0..4, the output bits fed by input bits 0..4, then the
    // lowest others
    const int n = a.n, lo = n < 5 ? n : 5, m = n < kRelabelBits ? n : kRelabelBits;
    if (n < 1 || n - m > 32) return cudaErrorInvalidValue;
    int inv[64];
    for (int j = 0; j < n; ++j) inv[a.phys_of[j]] = j;   // input bit -> output bit
    bool in_tile[64] = {false};
    RelabelTiled t{};
    t.m = m;
    int k = 0;
    auto add = [&](int j) {
        if (k < m && !in_tile[j]) {
            in_tile[j] = true;
            t.out_bit[k++] = (uint8_t)j;
        }
    };
    for (int j = 0; j < lo; ++j) add(j);
    for (int i = 0; i < lo; ++i) add(inv[i]);
    for (int j = 0; j < n; ++j) add(j);
    for (int j = 0; j < n; ++j)
        if (!in_tile[j]) {
            t.other_out[t.n_other] = (uint8_t)j;
            t.other_in[t.n_other++] = (uint8_t)a.phys_of[j];
        }
    t.n_tiles = 1ull << t.n_other;
    // input-local order: the five lowest input bits first.  The swizzle folds local
    // bit 5 + x onto bit x, so an output low bit that comes from above them gets an
    // x that no other output low bit's source uses: lanes then hit distinct banks
    int pos[64];
    uint32_t used = 0, low_src = 0;
    auto place = [&](int i, int at) {
        t.in_bit[at] = (uint8_t)i;
        pos[i] = at;
        used |= 1u << at;
    };
    for (int i = 0; i < n; ++i) pos[i] = -1;
    for (int i = 0; i < lo; ++i) place(i, i);
    for (int j = 0; j < lo; ++j)
        if (a.phys_of[j] < lo) low_src |= 1u << a.phys_of[j];
    for (int j = 0; j < lo; ++j) {
        if (pos[a.phys_of[j]] >= 0) continue;
        int x = 0;
        while (lo + x < m && (((low_src >> x) & 1u) || ((used >> (lo + x)) & 1u))) ++x;
        if (lo + x < m) place(a.phys_of[j], lo + x);
    }
    for (int i = 0, at = 0; i < n; ++i)
        if (in_tile[inv[i]] && pos[i] < 0) {
            while ((used >> at) & 1u) ++at;
            place(i, at);
        }
    for (int q = 0; q < m; ++q) t.src_bit[q] = (uint8_t)pos[a.phys_of[t.out_bit[q]]];
    const uint64_t want = (uint64_t)sms * 8;
    const unsigned grid = (unsigned)(t.n_tiles < want ? t.n_tiles : want);
    const int J = m > 8 ? 1 << (m - 8) : 1;
    auto go = [&](auto r, auto j) {
        using R = decltype(r);
        using T = typename Amp<R>::T;
        k_relabel_tiled<R, decltype(j)::value><<<grid, kThreads, 0, s>>>((const T *)in, (T *)out, t);
    };
    auto by_j = [&](auto r) {
        if (J == 4) go(r, std::integral_constant<int, 4>{});
        else if (J == 2) go(r, std::integral_constant<int, 2>{});
        else go(r, std::integral_constant<int, 1>{});
    };
    if (prec == 0) by_j(0.f);
    else by_j(0.0);
    return cudaGetLastError();
}

}  // namespace qk
