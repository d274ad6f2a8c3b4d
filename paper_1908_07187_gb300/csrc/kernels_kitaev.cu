// K7: one fused stage of Kitaev's one-control-qubit order finding.
//
// The generic stage is H(c); controlled x -> f(x) on the register; the
// semiclassical phase exp(i theta) on c = |1>; H(c); measure c; X(c) if the
// outcome is 1.  When c is |0> at the start (it is reset at the end of every
// stage), with w the amplitudes on c = 0 and v = U w (v(y) = w(f^-1(y))), the
// state just before the measurement is
//     c = 0:  (w + e^{i theta} v) / 2,     c = 1:  (w - e^{i theta} v) / 2,
// so one reduction gives s0 = sum |w + e^{i theta} v|^2 and s1 = sum |w - ...|^2,
// P0 = s0 / (s0 + s1), and after the outcome m and the reset the c = 0 amplitudes
// are (w + (-1)^m e^{i theta} v) / sqrt(s_m).  Two passes over the c = 0 half
// replace six gate passes.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "qk_kernels.cuh"

namespace qk {
namespace {

constexpr int kThreads = 256;

template <typename R> struct Amp;
template <> struct Amp<float> { using T = float2; };
template <> struct Amp<double> { using T = double2; };

template <typename I>
__device__ __forceinline__ I insert_zero(I j, int pos) {
    const I lo = j & (((I)1 << pos) - 1);
    return ((j - lo) << 1) | lo;
}

// index of the amplitude whose register value is f^-1(register value of i)
template <typename I>
__device__ __forceinline__ I source_index(I i, const KitaevArgs &a) {
    const uint32_t y = reg_get<I>(i, a.field, a.rpos, a.w);
    uint32_t x = y;
    if (a.kind != 0) x = a.finv[y];
    else if (y < a.mul.N) x = mul_mod(y, a.mul);
    return reg_put<I>(i, x, a.field, a.rpos, a.w);
}

// the stage's phase factor, formed in FP64 by one warp per block (GB300's FP64 rate is
// low) and shared
__device__ __forceinline__ double2 block_rphase(const KitaevArgs &a, const uint8_t *cbits) {
    __shared__ double2 s_om;
    if (threadIdx.x < 32) {
        const double2 om = warp_rphase(a.rphase_idx, a.n_rphase, cbits);
        if (threadIdx.x == 0) s_om = om;
    }
    __syncthreads();
    return s_om;
}

template <typename R>
__global__ void __launch_bounds__(kThreads) k_kitaev_reduce(const typename Amp<R>::T *__restrict__ psi, KitaevArgs a,
                                                            const uint8_t *cbits, double *partials, Decide dec) {
    __shared__ double sh[kThreads];
    const double2 om = block_rphase(a, cbits);
    const R wr = (R)om.x, wi = (R)om.y;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    // complex64: compensated FP32 sums; complex128: FP64
    FSum g0, g1;
    double d0 = 0.0, d1 = 0.0;
#pragma unroll 4
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < a.n_half; j += stride) {
        const uint64_t i = insert_zero(j, a.cpos);   // control bit 0
        const typename Amp<R>::T w = psi[i], v = psi[source_index(i, a)];
        const R tr = wr * v.x - wi * v.y, ti = wr * v.y + wi * v.x;
        const R pr = w.x + tr, pi = w.y + ti, mr = w.x - tr, mi = w.y - ti;
        if constexpr (sizeof(R) == 4) {
            g0.add(pr * pr + pi * pi);
            g1.add(mr * mr + mi * mi);
        } else {
            d0 += pr * pr + pi * pi;
            d1 += mr * mr + mi * mi;
        }
    }
    if constexpr (sizeof(R) == 4) {
        d0 = g0.value();
        d1 = g1.value();
    }
    const double s0 = block_sum_w0(d0, sh);
    const double s1 = block_sum_w0(d1, sh);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = s0;
        partials[2 * blockIdx.x + 1] = s1;
    }
    last_block_decides(partials, dec);
}

template <typename R>
__global__ void __launch_bounds__(kThreads) k_kitaev_update(const typename Amp<R>::T *__restrict__ psi,
                                                            typename Amp<R>::T *__restrict__ out, KitaevArgs a,
                                                            const uint8_t *cbits, const MeasSlot *slot) {
    // the decision and the phase, converted to the working precision once per block
    __shared__ R s_f[3];
    {
        const double2 om = block_rphase(a, cbits);
        if (threadIdx.x == 0) {
            const double sg = slot->m ? -1.0 : 1.0;
            s_f[0] = (R)slot->scale;
            s_f[1] = (R)(sg * om.x);
            s_f[2] = (R)(sg * om.y);
        }
        __syncthreads();
    }
    const R sc = s_f[0], wr = s_f[1], wi = s_f[2];
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < a.n_half; j += stride) {
        const uint64_t i = insert_zero(j, a.cpos);
        const typename Amp<R>::T w = psi[i], v = psi[source_index(i, a)];
        typename Amp<R>::T o, z;
        o.x = (w.x + wr * v.x - wi * v.y) * sc;
        o.y = (w.y + wr * v.y + wi * v.x) * sc;
        z.x = 0;
        z.y = 0;
        out[i] = o;                         // control back at |0>
        out[i | (1ull << a.cpos)] = z;
    }
}

// The whole stage in one launch for states whose c = 0 half fits the register files:
// each thread loads its amplitudes w and the gathered partners v once, the grid forms
// the sums, the last block to arrive decides (partials added in a fixed order), and
// after a grid barrier every thread updates its amplitudes from registers.  The two
// kernels above read and gather everything twice and form the phase (FP64, about 2 us
// of one thread's latency) in front of their loads; here the loads are in flight
// meanwhile.  A cooperative launch, so all blocks are resident; the barrier's wait has a
// limit, after which the error flag that qk_sync reports is set and the block returns.
// 21 qubits, complex64: 30.4 -> 20 us a stage (the gather moves 32-byte sectors for 8
// of their bytes: 64 MB through L2 a stage).
constexpr int kStageThreads = 512;
constexpr int kStageBlocksPerSM = 2;
constexpr int kStageWaitLimit = 1 << 22;   // polls of about 0.5 us: seconds

__device__ __forceinline__ void fsum_merge(FSum &a, float hi, float lo) {
    const float s = a.hi + hi;
    const float bp = s - a.hi;
    a.lo += lo + ((a.hi - (s - bp)) + (hi - bp));
    a.hi = s;
}

template <typename R, int A>
__global__ void __launch_bounds__(kStageThreads, kStageBlocksPerSM)
    k_kitaev_stage(const typename Amp<R>::T *__restrict__ psi, typename Amp<R>::T *__restrict__ out,
                   const __grid_constant__ KitaevArgs a, const uint8_t *cbits, double *partials, unsigned *bar, Decide dec,
                   int *err) {
    using T = typename Amp<R>::T;
    __shared__ double2 s_om;
    __shared__ double s_part[2][kStageThreads / 32];
    __shared__ unsigned s_gen, s_last;
    __shared__ R s_f[3];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the states that fit have far fewer than 2^32 amplitudes
    const uint32_t n_half = (uint32_t)a.n_half, step = gridDim.x * kStageThreads, j0 = blockIdx.x * kStageThreads + tid;
    T w[A], v[A];
#pragma unroll
    for (int k = 0; k < A; ++k) {
        const uint32_t j = j0 + k * step;
        w[k].x = w[k].y = v[k].x = v[k].y = 0;
        if (j < n_half) {
            const uint32_t i = insert_zero(j, a.cpos);
            w[k] = psi[i];
            v[k] = psi[source_index(i, a)];
        }
    }
    if (warp == 0) {
        const double2 om = warp_rphase(a.rphase_idx, a.n_rphase, cbits);
        if (lane == 0) s_om = om;
    }
    if (tid == 0) {
        s_gen = *(volatile unsigned *)(bar + 1);   // the barrier's generation, before this block arrives
    }
    __syncthreads();
    const R wr = (R)s_om.x, wi = (R)s_om.y;
    FSum g0, g1;
    double d0 = 0.0, d1 = 0.0;
#pragma unroll
    for (int k = 0; k < A; ++k) {
        const R tr = wr * v[k].x - wi * v[k].y, ti = wr * v[k].y + wi * v[k].x;
        const R pr = w[k].x + tr, pi = w[k].y + ti, mr = w[k].x - tr, mi = w[k].y - ti;
        if constexpr (sizeof(R) == 4) {
            g0.add(pr * pr + pi * pi);
            g1.add(mr * mr + mi * mi);
        } else {
            d0 += pr * pr + pi * pi;
            d1 += mr * mr + mi * mi;
        }
    }
    if constexpr (sizeof(R) == 4) {
        // The warp's sums stay float pairs: FP64 additions here take 1.3 of 23 us a stage.
        // Their error (2^-47) is far below that of the FP32 terms: over 2^5 .. 2^21 amplitudes
        // the sums are as far from 64-bit ones as with FP64 additions, to six digits.
        for (int o = 16; o > 0; o >>= 1) {
            fsum_merge(g0, __shfl_down_sync(0xffffffffu, g0.hi, o), __shfl_down_sync(0xffffffffu, g0.lo, o));
            fsum_merge(g1, __shfl_down_sync(0xffffffffu, g1.hi, o), __shfl_down_sync(0xffffffffu, g1.lo, o));
        }
        if (lane == 0) {
            d0 = g0.value();
            d1 = g1.value();
        }
    } else {
        for (int o = 16; o > 0; o >>= 1) {
            d0 += __shfl_down_sync(0xffffffffu, d0, o);
            d1 += __shfl_down_sync(0xffffffffu, d1, o);
        }
    }
    if (lane == 0) {
        s_part[0][warp] = d0;
        s_part[1][warp] = d1;
    }
    __syncthreads();
    if (warp == 0) {
        double s0 = lane < kStageThreads / 32 ? s_part[0][lane] : 0.0;
        double s1 = lane < kStageThreads / 32 ? s_part[1][lane] : 0.0;
        for (int o = kStageThreads / 64; o > 0; o >>= 1) {
            s0 += __shfl_down_sync(0xffffffffu, s0, o);
            s1 += __shfl_down_sync(0xffffffffu, s1, o);
        }
        if (lane == 0) {
            partials[2 * blockIdx.x] = s0;
            partials[2 * blockIdx.x + 1] = s1;
            __threadfence();                       // the partials before the ticket
            s_last = atomicAdd(bar, 1u) == gridDim.x - 1 ? 1u : 0u;
        }
        __syncwarp();
        if (s_last) {
            __threadfence();
            double t0 = 0.0, t1 = 0.0;
            for (int b = lane; b < (int)gridDim.x; b += 32) {
                t0 += __ldcg(&partials[2 * b]);
                t1 += __ldcg(&partials[2 * b + 1]);
            }
            for (int o = 16; o > 0; o >>= 1) {
                t0 += __shfl_down_sync(0xffffffffu, t0, o);
                t1 += __shfl_down_sync(0xffffffffu, t1, o);
            }
            if (lane == 0) {
                const double tot = t0 + t1, p0 = tot > 0.0 ? t0 / tot : 1.0;
                const int m = dec.u >= p0 ? 1 : 0;
                const double pm = m ? t1 : t0;
                volatile MeasSlot *sl = dec.slot;
                sl->p0 = p0;
                sl->m = m;
                sl->scale = pm > 0.0 ? 1.0 / sqrt(pm) : 0.0;
                if (dec.dest >= 0) dec.cbits[dec.dest] = (uint8_t)m;
                *bar = 0;
                __threadfence();                   // the decision before the next generation
                atomicAdd(bar + 1, 1u);
            }
        } else if (lane == 0) {
            int polls = 0;
            while (*(volatile unsigned *)(bar + 1) == s_gen && ++polls < kStageWaitLimit) __nanosleep(64);
            if (polls >= kStageWaitLimit) s_last = 2u;
            __threadfence();
        }
        __syncwarp();
        if (lane == 0 && s_last != 2u) {
            const volatile MeasSlot *sl = dec.slot;
            s_f[0] = (R)sl->scale;
            s_f[1] = sl->m ? (R)-1 : (R)1;
        }
    }
    __syncthreads();
    if (s_last == 2u) {                            // the wait ran out: nothing is written
        if (tid == 0) *err = 1;
        return;
    }
    // formed from v again, in two FMAs onto w: from the rounded product e^{i theta} v the
    // error is that of |v| even where the two nearly cancel
    const R sc = s_f[0], ur = s_f[1] * wr, ui = s_f[1] * wi;
#pragma unroll
    for (int k = 0; k < A; ++k) {
        const uint32_t j = j0 + k * step;
        if (j >= n_half) continue;
        const uint32_t i = insert_zero(j, a.cpos);
        T o, z;
        o.x = (w[k].x + ur * v[k].x - ui * v[k].y) * sc;
        o.y = (w[k].y + ur * v[k].y + ui * v[k].x) * sc;
        z.x = 0;
        z.y = 0;
        if constexpr (sizeof(R) == 4) {
            if (a.cpos == 0) {                     // both values of the control in one store
                *reinterpret_cast<float4 *>(out + i) = make_float4(o.x, o.y, 0.f, 0.f);
                continue;
            }
        }
        out[i] = o;                                // control back at |0>
        out[i | (1u << a.cpos)] = z;
    }
}

inline unsigned grid_for(uint64_t units, int sms) {
    uint64_t b = (units + kThreads - 1) / kThreads;
    const uint64_t cap = (uint64_t)sms * 16;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (unsigned)b;
}

}  // namespace

cudaError_t launch_kitaev_reduce(int prec, const void *psi, const KitaevArgs &a, const uint8_t *cbits,
                                 double *partials, int nblocks, const Decide &d, cudaStream_t s) {
    if (prec == 0)
        k_kitaev_reduce<float><<<nblocks, kThreads, 0, s>>>((const float2 *)psi, a, cbits, partials, d);
    else
        k_kitaev_reduce<double><<<nblocks, kThreads, 0, s>>>((const double2 *)psi, a, cbits, partials, d);
    return cudaGetLastError();
}

cudaError_t launch_kitaev_update(int prec, const void *psi, void *out, const KitaevArgs &a, const uint8_t *cbits,
                                 const MeasSlot *slot, int sms, cudaStream_t s) {
    if (prec == 0)
        k_kitaev_update<float><<<grid_for(a.n_half, sms), kThreads, 0, s>>>((const float2 *)psi, (float2 *)out, a,
                                                                            cbits, slot);
    else
        k_kitaev_update<double><<<grid_for(a.n_half, sms), kThreads, 0, s>>>((const double2 *)psi, (double2 *)out,
                                                                             a, cbits, slot);
    return cudaGetLastError();
}

// amplitudes per thread that the registers hold
static int stage_max_amps(int prec) { return prec == 0 ? 8 : 4; }

bool kitaev_stage_fits(int prec, uint64_t n_half, int sms) {
    return n_half <= (uint64_t)sms * kStageBlocksPerSM * kStageThreads * stage_max_amps(prec);
}

template <typename R, int A>
static cudaError_t stage_launch(const void *psi, void *out, const KitaevArgs &a, const uint8_t *cbits, double *partials,
                                unsigned *bar, const Decide &d, int *err, unsigned grid, cudaStream_t s) {
    using T = typename Amp<R>::T;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kStageThreads);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_kitaev_stage<R, A>, (const T *)psi, (T *)out, a, cbits, partials, bar, d, err);
}

template <typename R>
static cudaError_t stage_r(const void *psi, void *out, const KitaevArgs &a, const uint8_t *cbits, double *partials,
                           unsigned *bar, const Decide &d, int *err, int sms, cudaStream_t s) {
    const uint64_t cap = (uint64_t)sms * kStageBlocksPerSM;
    const uint64_t want = (a.n_half + kStageThreads - 1) / kStageThreads;
    const unsigned grid = (unsigned)(want < cap ? want : cap);
    const uint64_t per = (want + grid - 1) / grid;
    if (per <= 1) return stage_launch<R, 1>(psi, out, a, cbits, partials, bar, d, err, grid, s);
    if (per <= 2) return stage_launch<R, 2>(psi, out, a, cbits, partials, bar, d, err, grid, s);
    if (per <= 4) return stage_launch<R, 4>(psi, out, a, cbits, partials, bar, d, err, grid, s);
    if constexpr (sizeof(R) == 4) return stage_launch<R, 8>(psi, out, a, cbits, partials, bar, d, err, grid, s);
    return cudaErrorInvalidValue;
}

cudaError_t launch_kitaev_stage(int prec, const void *psi, void *out, const KitaevArgs &a, const uint8_t *cbits,
                                double *partials, unsigned *bar, const Decide &d, int *err, int sms, cudaStream_t s) {
    if (!kitaev_stage_fits(prec, a.n_half, sms)) return cudaErrorInvalidValue;
    return prec == 0 ? stage_r<float>(psi, out, a, cbits, partials, bar, d, err, sms, s)
                     : stage_r<double>(psi, out, a, cbits, partials, bar, d, err, sms, s);
}

}  // namespace qk
