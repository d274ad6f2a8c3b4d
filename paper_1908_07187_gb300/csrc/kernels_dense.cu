// Dense k-qubit gates (k = 2..6) in the working precision on CUDA cores (DenseParams in
// qk_kernels.cuh).
//
// A CTA holds a tile of 2^m amplitudes in shared memory and applies a run of gates of
// one k to it: one read and one write of the state however many gates the run has.  A
// gate is a small matrix product, Y = U X with X the 2^k x columns matrix of the tile's
// groups; a thread forms several rows of several columns in registers, so that each
// shared-memory load feeds several FMAs.  Bound by HBM for one gate of k <= 3, by FP32
// (4 * 2^k FMAs per amplitude) above, by FP64 throughout in complex128 (2 lanes per SM
// and clock).  Before, one thread formed one amplitude with two shared loads per
// complex product, one gate per pass.  Measured in complex64: one gate on 24 qubits, k =
// 2, 3, 4, 5, 6: 86, 84, 108, 144, 224 us (k = 6: 3670 before); a brickwork of 63 pair
// gates on 22 qubits: 1383 -> 278 us.  In complex128, nine gates, k = 2 / 4 / 6: 892 -> 486,
// 2154 -> 1364, 7006 -> 4876 us on 20 qubits and 98 -> 74, 130 -> 75, 342 -> 219 us on 8.
#include <cuda_runtime.h>
#include <stdint.h>

#include "qk_kernels.cuh"

namespace qk {
namespace {

constexpr int kThreads = 256;
template <typename R> struct Amp;
template <> struct Amp<float> { using T = float2; };
template <> struct Amp<double> { using T = double2; };

// acc += m x.  Scalar FMAs in complex64 too: packed ones want (re, re) and (-im, im)
// operand pairs, whose moves ran on the same FMA pipes and cost more than the packing
// saved (6 qubits at 24 qubits: 330 us packed).
template <typename T>
__device__ __forceinline__ void mac(T &acc, T m, T x) {
    acc.x = fma(m.x, x.x, acc.x);
    acc.y = fma(m.x, x.y, acc.y);
    acc.x = fma(-m.y, x.y, acc.x);
    acc.y = fma(m.y, x.x, acc.y);
}
// Slots read from the kernel parameters are the same for every lane, and left to itself
// the compiler keeps their sums in uniform registers; nvcc 13.0 then stored a thread's
// fourth column to the address of its second.  An opaque copy keeps them in ordinary
// registers.
__device__ __forceinline__ uint32_t lane_copy(uint32_t x) {
    asm volatile("" : "+r"(x));
    return x;
}
template <typename T, int RT>
__device__ __forceinline__ void load_rows(T (&u)[RT], const T *p) {
    if constexpr (sizeof(T) == 8 && RT > 1) {
#pragma unroll
        for (int i = 0; i < RT; i += 2) {
            const float4 a = *reinterpret_cast<const float4 *>(p + i);
            u[i] = make_float2(a.x, a.y);
            u[i + 1] = make_float2(a.z, a.w);
        }
    } else {
#pragma unroll
        for (int i = 0; i < RT; ++i) u[i] = p[i];
    }
}

// One or two 2-qubit gates in complex64 (DenseOp::pair): a thread takes 16 amplitudes at
// a time, so the state crosses shared memory once for both, and a gate's matrix is held
// in registers for the four columns (read as kernel parameters per column, it kept the
// constant path busy 60 % of the time).
struct Mat2 {
    float2 m[16];
    __device__ __forceinline__ explicit Mat2(const float2 *q) { load_rows(m, q); }
};
__device__ __forceinline__ void gate2(float2 &x0, float2 &x1, float2 &x2, float2 &x3, const Mat2 &m) {
    float2 y[4];
    const float2 x[4] = {x0, x1, x2, x3};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        y[r].x = y[r].y = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) mac(y[r], m.m[4 * r + c], x[c]);
    }
    x0 = y[0];
    x1 = y[1];
    x2 = y[2];
    x3 = y[3];
}
__device__ __forceinline__ void dense_two(float2 *A, const DenseOp &op, const float2 *mat, const float2 *next) {
    const int nf = op.nfree, ncol = 1 << op.ncs;
    const uint32_t t0 = lane_copy(op.ts[0]), t1 = lane_copy(op.ts[1]);
    const uint32_t c0 = lane_copy(op.cs[0]), c1 = lane_copy(op.cs[1]);
    for (int g = threadIdx.x; g < (1 << nf); g += kThreads) {
        uint32_t s = op.ls;
        for (int b = 0; b < nf; ++b)
            if ((g >> b) & 1) s ^= op.fs[b];
        float2 x[4][4];                              // [column][register value]
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (c < ncol) {
                const uint32_t o = s ^ ((c & 1) ? c0 : 0u) ^ ((c & 2) ? c1 : 0u);
#pragma unroll
                for (int r = 0; r < 4; ++r) x[c][r] = A[o ^ ((r & 1) ? t0 : 0u) ^ ((r & 2) ? t1 : 0u)];
            }
        {
            const Mat2 m(mat);
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c < ncol) gate2(x[c][0], x[c][1], x[c][2], x[c][3], m);
        }
        if (op.pair) {
            const Mat2 m(next);
#pragma unroll
            for (int r = 0; r < 4; ++r) gate2(x[0][r], x[1][r], x[2][r], x[3][r], m);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (c < ncol) {
                const uint32_t o = s ^ ((c & 1) ? c0 : 0u) ^ ((c & 2) ? c1 : 0u);
#pragma unroll
                for (int r = 0; r < 4; ++r) A[o ^ ((r & 1) ? t0 : 0u) ^ ((r & 2) ? t1 : 0u)] = x[c][r];
            }
    }
}

// One gate (complex64: of k >= 3).  Column bits run over the op's free bits in their order: the
// thread's column group takes the first ones, then the columns of one thread, then
// rounds.  Ut holds the matrix transposed (Ut[c * G + r]).  A thread forms RT rows of CT
// columns: with 4 x 4 the shared-memory loads of a step (their 128 bytes per clock into
// registers) take as long as its FMAs, with 8 x 4 three quarters of it.  1 x 1 where the
// tile has few columns, or threads would form rows and columns that are not there, and
// in complex128, where a product's four FP64 FMAs take 64 cycles against 8 for its loads.
template <typename R, int K, int RT, int CT>
__device__ __forceinline__ void dense_gate(typename Amp<R>::T *A, const typename Amp<R>::T *Ut, const DenseOp &op) {
    using T = typename Amp<R>::T;
    constexpr int LRT = RT == 8 ? 3 : RT == 4 ? 2 : 0, LCT = CT == 4 ? 2 : CT == 2 ? 1 : 0;
    constexpr int G = 1 << K, RG = G / RT, CG = kThreads / RG, LCG = 8 - (K - LRT);
    static_assert(CG == 1 << LCG, "column groups");
    const int nf = op.nfree;
    // fewer columns than column groups: the threads that have work stay in whole warps
    const int lcg = nf < LCG ? nf : LCG;
    const int rg = threadIdx.x >> lcg, cg = threadIdx.x & ((1 << lcg) - 1);
    const bool live = rg < RG;
    uint32_t sb = op.ls;
#pragma unroll
    for (int b = 0; b < LCG; ++b)
        if (b < lcg && ((cg >> b) & 1)) sb ^= op.fs[b];
    uint32_t ts[K];
#pragma unroll
    for (int b = 0; b < K; ++b) ts[b] = lane_copy(op.ts[b]);
    uint32_t cs[CT];                                 // the thread's columns
    cs[0] = 0;
#pragma unroll
    for (int j = 1; j < CT; ++j) cs[j] = 0;
    const int ncol = CT == 1 || nf <= LCG ? 1 : nf == LCG + 1 ? 2 : CT;
    if (CT > 1 && nf > LCG) {
        cs[CT > 1 ? 1 : 0] = lane_copy(op.fs[LCG]);
        if constexpr (CT == 4)
            if (nf > LCG + 1) {
                cs[2] = lane_copy(op.fs[LCG + 1]);
                cs[3] = cs[1] ^ cs[2];
            }
    }
    const int lr = nf > LCG + LCT ? nf - LCG - LCT : 0;
    for (int it = 0; it < (1 << lr); ++it) {
        uint32_t s0 = sb;
        for (int b = 0; b < lr; ++b)
            if ((it >> b) & 1) s0 ^= op.fs[LCG + LCT + b];
        T acc[RT][CT];
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int j = 0; j < CT; ++j) acc[i][j].x = acc[i][j].y = 0;
        constexpr int U = 2, LU = 1;               // steps unrolled
#pragma unroll 1
        for (int k0 = live ? 0 : G; k0 < G; k0 += U) {
            uint32_t o0 = s0;
#pragma unroll
            for (int b = LU; b < K; ++b)
                if ((k0 >> b) & 1) o0 ^= ts[b];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const uint32_t o = o0 ^ ((k & 1) ? ts[0] : 0u) ^ ((k & 2) ? ts[1] : 0u);
                T u[RT], x[CT];
                load_rows(u, Ut + (k0 + k) * G + rg * RT);
#pragma unroll
                for (int j = 0; j < CT; ++j) x[j] = A[o ^ cs[j]];
#pragma unroll
                for (int i = 0; i < RT; ++i)
#pragma unroll
                    for (int j = 0; j < CT; ++j) mac(acc[i][j], u[i], x[j]);
            }
        }
        if constexpr (RG > 1) __syncthreads();       // a column's rows are shared by RG threads
        if (live) {
            uint32_t o0 = s0;
#pragma unroll
            for (int b = LRT; b < K; ++b)
                if (((rg * RT) >> b) & 1) o0 ^= ts[b];
#pragma unroll
            for (int j = 0; j < CT; ++j) {
                if (j >= ncol) continue;
#pragma unroll
                for (int i = 0; i < RT; ++i)
                    A[o0 ^ cs[j] ^ ((i & 1) ? ts[0] : 0u) ^ ((i & 2) ? ts[1] : 0u) ^
                      ((i & 4) ? ts[2] : 0u)] = acc[i][j];
            }
        }
    }
}

template <typename R, int K>                         // two gates at a time (dense_two)
constexpr bool dense_pairs = sizeof(R) == 4 && K == 2;
template <typename R, int K, int RT>
constexpr int dense_ctas() {
    return RT == 1 && !dense_pairs<R, K> ? 3 : sizeof(R) == 4 && (K == 3 || K == 4) ? 3 : 2;
}

// K: the k of every gate in the pass (one code path per kernel: with all of them in one
// the compiler ran out of registers)
template <typename R, int K, int RT, int CT>
__global__ void __launch_bounds__(kThreads, dense_ctas<R, K, RT>())
    k_dense(typename Amp<R>::T *__restrict__ psi, const __grid_constant__ DenseParams P,
            const uint8_t *__restrict__ cbits) {
    using T = typename Amp<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *A = reinterpret_cast<T *>(smem_raw);
    const uint32_t dim = 1u << P.m;
    T *mats = A + dim;
    const int tid = threadIdx.x, lane = tid & 31;
    uint64_t off0 = P.base;                          // the thread's part of every offset
    for (int k = 0; k < 8 && k < P.m; ++k)
        if ((tid >> k) & 1) off0 |= 1ull << P.S[k];
    uint64_t st[5];                                  // strides of local bits 8..12
#pragma unroll
    for (int k = 0; k < 5; ++k) st[k] = 8 + k < P.m ? 1ull << P.S[8 + k] : 0ull;
    const int rounds = dim > kThreads ? (int)(dim / kThreads) : 1;
    const bool live = (uint32_t)tid < dim;
    // every op's matrix (transposed for dense_gate); a CTA runs over several tiles, so this is
    // paid once and the CTAs of an SM drift apart, one loading while the other computes
    constexpr int G = 1 << K;
    for (int o = 0; o < P.nops; ++o) {
        const T *gm = reinterpret_cast<const T *>(P.ops[o].mat);
        T *to = mats + o * (G * G);
        for (int e = tid; e < G * G; e += kThreads) to[dense_pairs<R, K> ? e : (e & (G - 1)) * G + (e >> K)] = gm[e];
    }
    unsigned condok = 0;
    for (int c = 0; c < P.n_conds; ++c) {
        bool ok = true;
        for (int k = 0; k < P.conds[c].n; ++k) ok = ok && cbits[P.conds[c].idx[k]] != 0;
        condok |= (ok ? 1u : 0u) << c;
    }
    for (uint64_t tile = blockIdx.x; tile < P.n_tiles; tile += gridDim.x) {
        T *base = psi + off0;
        {
            const uint64_t v = lane < P.nfix && ((tile >> lane) & 1u) ? 1ull << P.fixed[lane] : 0ull;
            base += ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(v >> 32)) << 32) |
                    __reduce_or_sync(0xffffffffu, (uint32_t)v);
        }
        // a thread loads and stores the same slots, so nothing separates one tile's
        // stores from the next one's loads
        if (live) {
            for (int j0 = 0; j0 < rounds; j0 += 8) {
                T v[8];
                T *p = base + ((j0 & 8) ? st[3] : 0) + ((j0 & 16) ? st[4] : 0);
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (j0 + j < rounds) v[j] = p[((j & 1) ? st[0] : 0) + ((j & 2) ? st[1] : 0) + ((j & 4) ? st[2] : 0)];
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (j0 + j < rounds) A[dense_slot(tid + (j0 + j) * kThreads)] = v[j];
            }
        }
        for (int o = 0; o < P.nops; ++o) {
            const DenseOp &op = P.ops[o];
            if (((uint32_t)tile & op.tmask) != op.tmask) continue;
            if (op.cond != 0xff && !((condok >> op.cond) & 1u)) continue;
            __syncthreads();                         // the tile and matrices, or the previous gate
            if constexpr (dense_pairs<R, K>) {
                dense_two(A, op, mats + o * (G * G), mats + (op.pair ? o + 1 : o) * (G * G));
                if (op.pair) ++o;
            } else {
                dense_gate<R, K, RT, CT>(A, mats + o * (G * G), op);
            }
        }
        __syncthreads();
        if (live) {
            for (int j0 = 0; j0 < rounds; j0 += 8) {
                T *p = base + ((j0 & 8) ? st[3] : 0) + ((j0 & 16) ? st[4] : 0);
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (j0 + j < rounds)
                        p[((j & 1) ? st[0] : 0) + ((j & 2) ? st[1] : 0) + ((j & 4) ? st[2] : 0)] =
                            A[dense_slot(tid + (j0 + j) * kThreads)];
            }
        }
    }
}

template <typename R, int K, int RT, int CT>
cudaError_t dense_k(void *psi, const DenseParams &p, const uint8_t *cbits, int sms, cudaStream_t s) {
    using T = typename Amp<R>::T;
    const size_t sm = (sizeof(T) << p.m) + sizeof(T) * ((size_t)p.nops << (2 * K));
    static SmemLimit limit;
    const cudaError_t e =
        smem_limit(k_dense<R, K, RT, CT>, sizeof(T) * (((size_t)1 << kDenseMaxBits) + kDenseElems), limit);
    if (e != cudaSuccess) return e;
    const uint64_t cap = (uint64_t)sms * dense_ctas<R, K, RT>();
    k_dense<R, K, RT, CT><<<(unsigned)(p.n_tiles < cap ? p.n_tiles : cap), kThreads, sm, s>>>((T *)psi, p, cbits);
    return cudaGetLastError();
}
// 4 x 2 per thread takes 2^11 amplitudes for every thread to have columns, 8 x 4 2^13
template <typename R>
cudaError_t dense_r(void *psi, const DenseParams &p, const uint8_t *cbits, int sms, cudaStream_t s) {
    constexpr bool kF = sizeof(R) == 4;
    const bool big = kF && p.m >= (p.k >= 5 ? 13 : 11);
    switch (p.k) {
        case 2: return dense_k<R, 2, 1, 1>(psi, p, cbits, sms, s);
        case 3: if constexpr (kF) if (big) return dense_k<R, 3, 4, 2>(psi, p, cbits, sms, s);
                return dense_k<R, 3, 1, 1>(psi, p, cbits, sms, s);
        case 4: if constexpr (kF) if (big) return dense_k<R, 4, 4, 2>(psi, p, cbits, sms, s);
                return dense_k<R, 4, 1, 1>(psi, p, cbits, sms, s);
        case 5: if constexpr (kF) if (big) return dense_k<R, 5, 8, 4>(psi, p, cbits, sms, s);
                return dense_k<R, 5, 1, 1>(psi, p, cbits, sms, s);
        default: if constexpr (kF) if (big) return dense_k<R, 6, 8, 4>(psi, p, cbits, sms, s);
                return dense_k<R, 6, 1, 1>(psi, p, cbits, sms, s);
    }
}

}  // namespace

cudaError_t launch_dense(int prec, void *psi, const DenseParams &p, const uint8_t *cbits, int sms, cudaStream_t s) {
    if (p.k < 2 || p.k > kDenseMaxK || p.m < p.k || p.m > kDenseMaxBits || p.nops < 1 || p.nops > kDenseOps ||
        p.nfix > 31 || p.n_tiles > 0x7fffffffull || (p.nops << (2 * p.k)) > kDenseElems)
        return cudaErrorInvalidValue;
    for (int i = 0; i < p.nops; ++i)
        if (p.ops[i].pair && (p.k != 2 || i + 1 >= p.nops)) return cudaErrorInvalidValue;
    return prec == 0 ? dense_r<float>(psi, p, cbits, sms, s) : dense_r<double>(psi, p, cbits, sms, s);
}

}  // namespace qk
