// epochs.cuh -- what the epoch loops of the forward model (forward_run.cuh) and of the amoeba
// (polish_run.cuh) share: the staged lightcurve, the decoding of a candidate and the re-solve queue.
#pragma once

#include "forward.cuh"
#include "forward_launch.cuh"

namespace sblm {

// the lightcurve as one thread reads it: staged in shared memory (FP64: t, F, 1/sigma; FP32
// modes: (t_hi, t_lo, F, 1/sigma) as float4) or straight from global memory
struct LCView {
    const double* t;
    const double* flux;
    const double* sigma;
    const double* s_t;
    const double* s_f;
    const double* s_w;
    const float4* s_ep;
};

// Stage n_ep epochs in `smem` (every thread of the block calls this; it ends with a barrier).
// FP32 modes split t = t_hi + t_lo so that t - t0 keeps full precision through a two-sum.
template <int MODE, bool CHI2>
__device__ __forceinline__ LCView stage_lightcurve(unsigned char* smem, const double* __restrict__ t,
                                                   const double* __restrict__ flux,
                                                   const double* __restrict__ sigma, int n_ep) {
    LCView v{t, flux, sigma, nullptr, nullptr, nullptr, nullptr};
    if (MODE == SBLM_FP64) {
        double* s_t = reinterpret_cast<double*>(smem);
        double* s_f = s_t + n_ep;
        double* s_w = s_f + (CHI2 ? n_ep : 0);
        for (int e = threadIdx.x; e < n_ep; e += blockDim.x) {
            s_t[e] = t[e];
            if (CHI2) {
                s_f[e] = flux[e];
                s_w[e] = 1.0 / sigma[e];
            }
        }
        v.s_t = s_t;
        v.s_f = s_f;
        v.s_w = s_w;
    } else {
        float4* s_ep = reinterpret_cast<float4*>(smem);
        for (int e = threadIdx.x; e < n_ep; e += blockDim.x) {
            const double te = t[e];
            const float th = (float)te;
            s_ep[e] = make_float4(th, (float)(te - (double)th), CHI2 ? (float)flux[e] : 0.f,
                                  CHI2 ? (float)(1.0 / sigma[e]) : 0.f);
        }
        v.s_ep = s_ep;
    }
    __syncthreads();
    return v;
}

template <bool FROM_GENES>
__device__ __forceinline__ Cand candidate(const double* __restrict__ src, const Bounds& b, int c) {
    if (!FROM_GENES) return load_cand(src, c);
    // Eq. (EMMA-encoding): a_j = lo_j + (hi_j - lo_j) p_j; gene 5 is log10 q
    const double* p = src + 6 * (size_t)c;
    double a[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) a[j] = b.lo[j] + (b.hi[j] - b.lo[j]) * p[j];
    Cand k;
    k.t0 = a[0];
    k.inv_tE = 1.0 / a[1];
    k.u0 = a[2];
    sincos(a[3], &k.sa, &k.ca);
    k.d = a[4];
    k.q = exp10(a[5]);
    return k;
}

// the general re-solve's Aberth stop rule (relative correction), see solve_epoch
constexpr double kResolveCubic = 1e-6;

// Where MIXED and FP64 work goes. Epochs to re-solve in FP64 are appended to `queue` (slots taken
// with one atomic per warp, so that a later pass re-solves them side by side). An epoch that finds
// the queue full takes the general solver in place; the pass over the queue then sends the queued
// ones to it too, so that an epoch's result does not depend on whether it found a place. Every epoch's chi^2
// term is stored in the candidate's row of the dense term array (the others here, the re-solved ones
// by the re-solve, wherever it runs), and the row is summed afterwards in a fixed order: the chi^2
// does not depend on the order in which the queue filled. `term_row` is the candidate's row
// (epoch e at term_row[e]); null when no chi^2 is wanted.
struct DeferSink {
    Deferred* queue;
    unsigned* queue_count;
    unsigned queue_cap;
};

}  // namespace sblm
