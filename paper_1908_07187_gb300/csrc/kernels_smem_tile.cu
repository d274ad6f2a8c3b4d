// Fused pass over tiles in shared memory (SmemTileParams in qk_kernels.cuh): complex128
// states, and complex64 states below 13 qubits.
//
// One CTA owns one tile of 2^m amplitudes in shared memory: it is read once, a
// program of gates runs on it, and it is written back once.  In complex128, with 2
// FP64 lanes per SM and clock, a warp's FP64 instruction takes 16 cycles of the SM's
// FP64 unit, which is the bound (a gate's pair: 6 instructions, 96 cycles per warp,
// against 16 to 32 cycles of shared-memory traffic and about 10 of issue), so
// amplitudes stay in shared memory between gates -- no register arrangements, no
// transposes -- and the program does whatever it can by exchange, sign bit and index
// arithmetic.  The tile width falls with the state (planner) so that small states
// still spread over the SMs.  Measured against one pass per gate: a 23-qubit
// complex128 circuit of 161 U3, 139 CZ and the QFT 33.0 -> 10.7 ms (six passes; the
// FP64 unit's own time for its 5.2 G instructions per lane is 8.3 ms) and to 6.0 ms with
// tiles of zeros left alone, the 12-qubit complex128 circuit of 290 gates 1322 -> 318 us
// (bound by the latency of one short op after another), a 10-qubit complex64 circuit of
// 175 gates, viewed and measured, 828 -> 153 us.
#include <cuda_runtime.h>
#include <stdint.h>

#include "qk_kernels.cuh"

namespace qk {
namespace {

constexpr int kMaxThreads = 256;

template <typename R> struct Amp;
template <> struct Amp<float> { using T = float2; };
template <> struct Amp<double> { using T = double2; };
__device__ __forceinline__ float2 pair(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ double2 pair(double x, double y) { return make_double2(x, y); }
// an op's coefficients and a program's factors in the working precision
__device__ __forceinline__ const float *coef(const SmemTileOp &op, float) { return op.cf; }
__device__ __forceinline__ const double *coef(const SmemTileOp &op, double) { return op.c; }
__device__ __forceinline__ const float2 *factors(const SmemTileParams &P, float) { return P.facf; }
__device__ __forceinline__ const double2 *factors(const SmemTileParams &P, double) { return P.fac; }

template <typename T>
__device__ __forceinline__ T cmul(T a, T b) {
    return pair(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ uint32_t ins0(uint32_t j, int pos) {
    const uint32_t lo = j & ((1u << pos) - 1);
    return ((j - lo) << 1) | lo;
}
// j's bits spread over the positions outside mask
__device__ __forceinline__ uint32_t spread(uint32_t j, uint32_t mask) {
    for (uint32_t m = mask; m; m &= m - 1) j = ins0(j, __ffs(m) - 1);
    return j;
}
__device__ __forceinline__ double flip(double x, uint32_t s) {   // s = 0 or 0x80000000
    return __hiloint2double(__double2hiint(x) ^ (int)s, __double2loint(x));
}
// nonzero unless x is 0 or -0 (integer operations: a complex128 comparison would take
// one of the two FP64 lanes)
__device__ __forceinline__ uint32_t magnitude_bits(float x) { return __float_as_uint(x) << 1; }
__device__ __forceinline__ uint32_t magnitude_bits(double x) {
    return ((uint32_t)__double2hiint(x) << 1) | (uint32_t)__double2loint(x);
}
__device__ __forceinline__ float flip(float x, uint32_t s) { return __uint_as_float(__float_as_uint(x) ^ s); }

// One ST_U2 op.  The value that is turned and the one that is not are told apart by
// their shared-memory slots, and the two orders of update are separate loops: as
// branches inside one loop they became predicated instructions, which occupy the FP64
// pipe (12 issued for the 6 that count).
template <bool kFirst0, bool kPhase, typename T>
__device__ __forceinline__ void u2_sweep(T *A, const SmemTileOp &op, uint32_t tile, uint32_t half) {
    const int fl = op.flags, q = op.q;
    const bool on0 = fl & kU2On0, lift = fl & kU2Lift, swap = fl & kU2Swap;
    const int k = on0 ? (4 - fl) & 3 : fl & 3;
    using R = decltype(T().x);
    const R *c = coef(op, R());
    const R t = on0 ? -c[0] : c[0], c0 = c[1], c1 = c[2];
    const uint32_t smask = op.lmask, par = __popc(tile & op.tmask) & 1u, bit = 1u << q;
    // quarter turns: exchange of the parts, then signs
    const uint32_t kx = (k == 1 || k == 2) ? 0x80000000u : 0u, ky = (k & 2) ? 0x80000000u : 0u;
    const uint32_t x0 = on0 ? kx : 0u, y0s = on0 ? ky : 0u, x1 = on0 ? 0u : kx, y1s = on0 ? 0u : ky;
    const bool turn0 = on0 && (k & 1), turn1 = !on0 && (k & 1);
    for (uint32_t p = threadIdx.x; p < half; p += blockDim.x) {
        const uint32_t i0 = ins0(p, q), i1 = i0 | bit;
        const T v0 = A[i0], v1 = A[i1];
        const uint32_t s = ((__popc(i0 & smask) + par) & 1u) << 31;
        T z0 = pair(flip(turn0 ? v0.y : v0.x, x0), flip(turn0 ? v0.x : v0.y, y0s));
        T z1 = pair(flip(turn1 ? v1.y : v1.x, x1 ^ s), flip(turn1 ? v1.x : v1.y, y1s ^ s));
        if constexpr (kPhase) {
            const T w = on0 ? z0 : z1;
            const T r = pair(fma(-t, w.y, w.x), fma(t, w.x, w.y));
            if (on0) z0 = r;
            else z1 = r;
        }
        if (lift) {
            if constexpr (kFirst0) {
                z0.x = fma(c0, z1.x, z0.x);
                z0.y = fma(c0, z1.y, z0.y);
                z1.x = fma(c1, z0.x, z1.x);
                z1.y = fma(c1, z0.y, z1.y);
            } else {
                z1.x = fma(c1, z0.x, z1.x);
                z1.y = fma(c1, z0.y, z1.y);
                z0.x = fma(c0, z1.x, z0.x);
                z0.y = fma(c0, z1.y, z0.y);
            }
        }
        A[swap ? i1 : i0] = z0;
        A[swap ? i0 : i1] = z1;
    }
}

// factors of a ST_TABLE op: lo[j] over local bits 0..5, hi[j] over the others times
// the constant and the tile-index bits' factors; built by doubling, a warp each.
// Without factors on one side its table is left out (the constant goes to the other).
template <typename T>
__device__ __forceinline__ void build_tables(const SmemTileParams &P, const SmemTileOp &op, uint32_t tile, T *lo, T *hi,
                                             int warp, int lane) {
    using R = decltype(T().x);
    const T *fac = factors(P, R());
    const uint32_t lf = op.lmask;
    const bool use_hi = (lf >> 6) != 0;
    if (warp > 1) return;
    T *tab = warp == 0 ? lo : hi;
    if (warp == 1 && !use_hi) return;
    T c0 = pair(R(1), R(0));
    if ((warp == 1) == use_hi) {
        // the constant and the tile-index factors: one bit per lane, multiplied over the warp
        if (op.tfac) {
            if ((op.tfac >> lane) & (tile >> lane) & 1u)
                c0 = fac[op.first + __popc(lf) + __popc(op.tfac & ((1u << lane) - 1))];
            for (int o = 16; o > 0; o >>= 1) {
                const T x = pair(__shfl_xor_sync(0xffffffffu, c0.x, o), __shfl_xor_sync(0xffffffffu, c0.y, o));
                c0 = cmul(c0, x);
            }
        }
        c0 = cmul(c0, pair(coef(op, R())[0], coef(op, R())[1]));
    }
    const int b0 = warp == 0 ? 0 : 6, b1 = warp == 0 ? min(6, P.m) : P.m;
    if (lane == 0) tab[0] = c0;
    for (int b = b0; b < b1; ++b) {
        __syncwarp();
        const int half = 1 << (b - b0);
        if (lane < half) {
            T v = tab[lane];
            if ((lf >> b) & 1u) v = cmul(v, fac[op.first + __popc(lf & ((1u << b) - 1))]);
            tab[half + lane] = v;
        }
    }
}

template <typename R>
__global__ void __launch_bounds__(kMaxThreads, 3)
    k_smem_tile(typename Amp<R>::T *__restrict__ psi, const __grid_constant__ SmemTileParams P,
                const uint8_t *__restrict__ cbits) {
    using T = typename Amp<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *A = reinterpret_cast<T *>(smem_raw);
    const uint32_t dim = 1u << P.m, half = dim >> 1;
    T *lo = A + dim, *hi = lo + 64;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t tile = blockIdx.x;

    uint64_t base = 0;
    {
        const uint64_t v = lane < P.nfix && ((tile >> lane) & 1u) ? 1ull << P.fixed[lane] : 0ull;
        base = ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(v >> 32)) << 32) |
               __reduce_or_sync(0xffffffffu, (uint32_t)v);
    }
    const int tb = 31 - __clz(nt);               // bits of the thread index
    for (int k = 0; k < tb && k < P.m; ++k)
        if ((tid >> k) & 1) base |= 1ull << P.S[k];
    uint64_t st[4];                              // strides of the local bits above them
#pragma unroll
    for (int k = 0; k < 4; ++k) st[k] = tb + k < P.m ? 1ull << P.S[tb + k] : 0ull;
    const uint32_t rounds = dim > (uint32_t)nt ? dim >> tb : 1u;
    const bool live = (uint32_t)tid < dim;
    uint32_t seen = 0;                           // whether anything loaded is other than 0 or -0
    if (live) {
        for (uint32_t j0 = 0; j0 < rounds; j0 += 4) {
            T v[4];
            const uint64_t hi_off = ((j0 & 4) ? st[2] : 0) + ((j0 & 8) ? st[3] : 0);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j0 + j < rounds) v[j] = psi[base + hi_off + ((j & 1) ? st[0] : 0) + ((j & 2) ? st[1] : 0)];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j0 + j < rounds) {
                    A[tid + (j0 + j) * nt] = v[j];
                    seen |= magnitude_bits(v[j].x) | magnitude_bits(v[j].y);
                }
        }
    }
    // The ops go to shared memory while the tile's loads are in flight: read from the
    // kernel parameters, each one's first touch waited for the constant cache (12 qubits
    // complex128 333 -> 318 us, 10 qubits complex64 159 -> 153, 12 qubits 275 -> 259).
    // Through a generic address, so that lanes read neighbouring words.
    const uint2 *src = reinterpret_cast<const uint2 *>(P.ops);
    asm volatile("" : "+l"(src));
    uint2 *staged = reinterpret_cast<uint2 *>(hi + 64);
    for (int w = tid; w < P.nops * (int)(sizeof(SmemTileOp) / sizeof(uint2)); w += nt) staged[w] = src[w];
    const SmemTileOp *ops = reinterpret_cast<const SmemTileOp *>(staged);
    unsigned condok = 0;
    for (int c = 0; c < P.n_conds; ++c) {
        bool ok = true;
        for (int k = 0; k < P.conds[c].n; ++k) ok = ok && cbits[P.conds[c].idx[k]] != 0;
        condok |= (ok ? 1u : 0u) << c;
    }
    // A tile of zeros stays one whatever the program does, so it is left as it is: from
    // |0...0> the first passes' gates act on few tiles (a 23-qubit complex128 circuit of 300
    // layer gates, a QFT and three measurements: 10.2 -> 5.7 ms)
    if (!__syncthreads_or(seen != 0u)) return;

    for (int o = 0; o < P.nops; ++o) {
        const SmemTileOp &op = ops[o];
        const int q = op.q;
        switch (op.kind) {
            case ST_U2: {
                if (op.flags & kU2First0) {
                    if (op.flags & kU2Phase) u2_sweep<true, true>(A, op, tile, half);
                    else u2_sweep<true, false>(A, op, tile, half);
                } else {
                    if (op.flags & kU2Phase) u2_sweep<false, true>(A, op, tile, half);
                    else u2_sweep<false, false>(A, op, tile, half);
                }
                break;
            }
            case ST_X:
            case ST_CU2: {
                if ((tile & op.tmask) != op.tval || (op.cond != kNoBit && !((condok >> op.cond) & 1u))) continue;
                const uint32_t bit = 1u << q, cm = op.lmask, cnt = half >> __popc(cm);
                if (op.kind == ST_X) {
                    for (uint32_t u = tid; u < cnt; u += nt) {
                        const uint32_t i0 = spread(u, cm | bit) | op.lval, i1 = i0 | bit;
                        const T a = A[i0], b = A[i1];
                        A[i0] = b;
                        A[i1] = a;
                    }
                } else {
                    const R *c = coef(op, R());
                    const T m00 = pair(c[0], c[1]), m01 = pair(c[2], c[3]), m10 = pair(c[4], c[5]), m11 = pair(c[6], c[7]);
                    for (uint32_t u = tid; u < cnt; u += nt) {
                        const uint32_t i0 = spread(u, cm | bit) | op.lval, i1 = i0 | bit;
                        const T a = A[i0], b = A[i1];
                        A[i0] = pair(m00.x * a.x - m00.y * a.y + m01.x * b.x - m01.y * b.y,
                                     m00.x * a.y + m00.y * a.x + m01.x * b.y + m01.y * b.x);
                        A[i1] = pair(m10.x * a.x - m10.y * a.y + m11.x * b.x - m11.y * b.y,
                                     m10.x * a.y + m10.y * a.x + m11.x * b.y + m11.y * b.x);
                    }
                }
                break;
            }
            case ST_SIGN: {
                const uint32_t par = __popc(tile & op.tmask) & 1u;
                const uint32_t n_at = q == kNoBit ? dim : half;
                if (op.tval & ~tile) continue;   // the common bit is a tile-index bit that is 0
                for (uint32_t p = tid; p < n_at; p += nt) {
                    const uint32_t i = q == kNoBit ? p : ins0(p, q) | (1u << q);
                    if (((__popc(i & op.lmask) + par) & 1u) == 0) continue;
                    T a = A[i];
                    a.x = flip(a.x, 0x80000000u);
                    a.y = flip(a.y, 0x80000000u);
                    A[i] = a;
                }
                break;
            }
            case ST_PH: {
                if ((tile & op.tmask) != op.tval || (op.cond != kNoBit && !((condok >> op.cond) & 1u))) continue;
                const T f = pair(coef(op, R())[0], coef(op, R())[1]);
                const uint32_t cnt = dim >> __popc(op.lmask);
                for (uint32_t u = tid; u < cnt; u += nt) {
                    const uint32_t i = spread(u, op.lmask) | op.lval;
                    if (f.x == -1 && f.y == 0) A[i] = pair(-A[i].x, -A[i].y);
                    else if (f.y == 0) A[i] = pair(A[i].x * f.x, A[i].y * f.x);
                    else A[i] = cmul(A[i], f);
                }
                break;
            }
            default: {   // ST_TABLE
                if ((tile & op.tmask) != op.tval) continue;
                build_tables(P, op, tile, lo, hi, warp, lane);
                __syncthreads();
                const bool use_hi = (op.lmask >> 6) != 0, use_lo = (op.lmask & 63) != 0 || !use_hi;
                const uint32_t n_at = q == kNoBit ? dim : half;
                for (uint32_t p = tid; p < n_at; p += nt) {
                    const uint32_t i = q == kNoBit ? p : ins0(p, q) | (1u << q);
                    const T f = use_lo ? (use_hi ? cmul(lo[i & 63], hi[i >> 6]) : lo[i & 63]) : hi[i >> 6];
                    A[i] = cmul(A[i], f);
                }
                break;
            }
        }
        __syncthreads();
    }

    if (live) {
        for (uint32_t j0 = 0; j0 < rounds; j0 += 4) {
            const uint64_t hi_off = ((j0 & 4) ? st[2] : 0) + ((j0 & 8) ? st[3] : 0);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j0 + j < rounds)
                    psi[base + hi_off + ((j & 1) ? st[0] : 0) + ((j & 2) ? st[1] : 0)] = A[tid + (j0 + j) * nt];
        }
    }
}

}  // namespace

template <typename R>
static cudaError_t smem_tile_r(void *psi, const SmemTileParams &p, const uint8_t *cbits, unsigned nt, cudaStream_t s) {
    using T = typename Amp<R>::T;
    const size_t sm = sizeof(T) * (((size_t)1 << p.m) + 128) + sizeof(SmemTileOp) * (size_t)p.nops;
    static SmemLimit limit;
    const cudaError_t e = smem_limit(
        k_smem_tile<R>, sizeof(T) * (((size_t)1 << kSmemTileMax) + 128) + sizeof(SmemTileOp) * kSmemTileOps, limit);
    if (e != cudaSuccess) return e;
    k_smem_tile<R><<<p.n_tiles, nt, sm, s>>>((T *)psi, p, cbits);
    return cudaGetLastError();
}

cudaError_t launch_smem_tile(int prec, void *psi, const SmemTileParams &p, const uint8_t *cbits, cudaStream_t s) {
    if (p.m < 1 || p.m > kSmemTileMax || p.nops < 0 || p.nops > kSmemTileOps || p.nfix > 31) return cudaErrorInvalidValue;
    const uint32_t half = 1u << (p.m - 1);
    const unsigned nt = half < 64 ? 64u : half > kMaxThreads ? (unsigned)kMaxThreads : half;
    return prec == 0 ? smem_tile_r<float>(psi, p, cbits, nt, s) : smem_tile_r<double>(psi, p, cbits, nt, s);
}

}  // namespace qk
