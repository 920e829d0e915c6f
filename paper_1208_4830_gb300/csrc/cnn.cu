// cnn.cu -- the learned proposal: training curves generated by the forward model, binning of
// observed curves, the network's forward and backward passes on the tensor cores (cnn_gemm.cuh),
// AdamW, and seed rows for the EA. Entry points are declared in include/sblm_cnn.h.
//
// Data layout (channels innermost, batch outermost):
//   x   [B][256][2]  FP32 network input
//   h_l [B][L_l][64] BF16 activations after GELU (L = 256, 128, 64, 32), h5 [B][128]
//   z_l              FP32 pre-activations kept for the backward pass (training only)
//   dz_l             BF16 gradients of the pre-activations
//   weights          FP32 master copy; BF16 copies as stored (input gradients) and with every
//                    weight matrix transposed to [fan_out][fan_in] (forward products)
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <vector>

#include "../../include/sblm_cnn.h"
#include "cnn_gemm.cuh"
#include "cnn_launch.cuh"
#include "common.cuh"
#include "forward_launch.cuh"
#include "proposal.cuh"
#include "runtime.cuh"

namespace sblm {
namespace cnn {

constexpr int kBins = 256;
constexpr int kMinKept = 16;
constexpr int kMaxBatch = 4096;
constexpr double kPi = 3.141592653589793;

enum : uint64_t { OP_CNN_INIT = 7, OP_CNN_GEN = 8, OP_CNN_NOISE = 9 };  // seed rows: kOpCnnSample

// layer l: weight [K][N] at kOff[l], bias [N] after it
constexpr int kOffH[7] = {0, 704, 21248, 41792, 62336, 324608, 326156};
constexpr int kKH[6] = {10, 320, 320, 320, 2048, 128};
constexpr int kNH[6] = {64, 64, 64, 64, 128, 12};
static_assert(kOffH[6] == kNParams, "parameter count");
__constant__ int c_off[7] = {0, 704, 21248, 41792, 62336, 324608, 326156};
__constant__ int c_K[6] = {10, 320, 320, 320, 2048, 128};
__constant__ int c_N[6] = {64, 64, 64, 64, 128, 12};

// training prior in window units (natural logs of the range ends written out)
constexpr double kT0Lo = -0.4, kT0Hi = 0.4;
constexpr double kLnTELo = -3.2188758248682006, kLnTEHi = 0.4054651081081644;   // 0.04, 1.5
constexpr double kLnDLo = -1.2039728043259361, kLnDHi = 1.0986122886681098;     // 0.3, 3
constexpr double kLqLo = -4.0, kLqHi = 0.0;
constexpr double kTcLo = -0.8, kTcHi = 0.8;
constexpr double kLnSigLo = -9.210340371976182, kLnSigHi = -2.995732273553991;  // 1e-4, 0.05
constexpr double kDropMax = 0.7, kGapProb = 0.5, kGapMax = 0.4;

// ------------------------------------------------------------------------------------------
// device helpers
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// (r cos a, r sin a) with r = sqrt(-2 ln(1 - u0)), a = 2 pi u1
__device__ __forceinline__ void box_muller(uint64_t x0, uint64_t x1, double* z0, double* z1) {
    const double r = sqrt(-2.0 * log(1.0 - u01(x0)));
    const double a = 2.0 * kPi * u01(x1);
    *z0 = r * cos(a);
    *z1 = r * sin(a);
}

__device__ __forceinline__ int layer_of(int idx) {
    int l = 0;
    while (l < 5 && idx >= c_off[l + 1]) ++l;
    return l;
}

// learning rate of 1-based step t: linear warm-up, cosine decay to 0.1 lr0 at n_steps
__device__ __forceinline__ double lr_at(int64_t t, int n_steps, int warmup, double lr0) {
    const double warm = warmup > 0 ? fmin(1.0, (double)t / warmup) : 1.0;
    const double frac = fmin(1.0, (double)(t - 1) / (double)max(1, n_steps));
    return lr0 * warm * (0.1 + 0.45 * (1.0 + cos(kPi * frac)));
}

// A caustic point: root `pick` (ordered by real, then imaginary part) of the critical quartic
// e^{i phi} z^2 (z - d)^2 - (1 + q) z^2 + 2 d z - d^2 = 0 (det J = 0), mapped to the source plane
// by the lens equation. The roots of the monic form are found by Aberth-Ehrlich iteration in FP32
// (the FP64 pipe is a sixty-fourth of the FP32 one) and finished by Newton steps in FP64.
__device__ cx<double> critical_point(double d, double q, double phi, int pick) {
    using C = cx<double>;
    using Cf = cx<float>;
    const C ce = {cos(phi), -sin(phi)};  // e^{-i phi}
    C a[5];
    a[4] = {1.0, 0.0};
    a[3] = {-2.0 * d, 0.0};
    a[2] = C{d * d, 0.0} - (1.0 + q) * ce;
    a[1] = (2.0 * d) * ce;
    a[0] = (-d * d) * ce;
    Cf af[5];
    for (int k = 0; k < 5; ++k) af[k] = Cf{(float)a[k].re, (float)a[k].im};
    float R = sqrtf(sqrtf(norm2(af[0])));
    if (!(R > 0.f) || !isfinite(R)) R = 1.f;
    Cf zf[4];
    for (int k = 0; k < 4; ++k) {
        const float ang = 0.4f + k * 1.5707963267948966f;
        zf[k] = Cf{R * cosf(ang), R * sinf(ang)};
    }
    // FP32: a root is final at the rounding noise of its Horner evaluation (16 eps sum |a_k| |z|^k)
    // or when its correction is below 1e-6 (1 + |z|)
    bool done[4] = {false, false, false, false};
    for (int it = 0; it < 100; ++it) {
        bool all = true;
        for (int k = 0; k < 4; ++k) {
            if (done[k]) continue;
            Cf p = af[4], dp = {0.f, 0.f};
            const float r = sqrtf(norm2(zf[k]));
            float bound = 1.f;
            for (int deg = 3; deg >= 0; --deg) {
                dp = dp * zf[k] + p;
                p = p * zf[k] + af[deg];
                bound = bound * r + sqrtf(norm2(af[deg]));
            }
            if (sqrtf(norm2(p)) <= 16.f * 0x1.0p-24f * bound) {
                done[k] = true;
                continue;
            }
            const Cf ratio = div(p, dp);
            Cf sum = {0.f, 0.f};
            for (int j = 0; j < 4; ++j)
                if (j != k) sum = sum + inv(zf[k] - zf[j]);
            const Cf w = div(ratio, Cf{1.f, 0.f} - ratio * sum);
            if (finite2(w)) {
                zf[k] = zf[k] - w;
                if (sqrtf(norm2(w)) <= 1e-6f * (1.f + sqrtf(norm2(zf[k])))) done[k] = true;
            }
            all = all && done[k];
        }
        if (all) break;
    }
    // FP64: Newton steps z <- z - p(z) / p'(z) on the same quartic (quadratic convergence from
    // FP32 accuracy), stopped at the FP64 noise level
    C z[4];
    for (int k = 0; k < 4; ++k) {
        z[k] = C{(double)zf[k].re, (double)zf[k].im};
        for (int it = 0; it < 4; ++it) {
            C p = a[4], dp = {0.0, 0.0};
            const double r = sqrt(norm2(z[k]));
            double bound = 1.0;
            for (int deg = 3; deg >= 0; --deg) {
                dp = dp * z[k] + p;
                p = p * z[k] + a[deg];
                bound = bound * r + sqrt(norm2(a[deg]));
            }
            if (sqrt(norm2(p)) <= 16.0 * 0x1.0p-53 * bound) break;
            const C w = div(p, dp);
            if (!finite2(w)) break;
            z[k] = z[k] - w;
        }
    }
    for (int i = 1; i < 4; ++i)
        for (int j = i; j > 0 && (z[j].re < z[j - 1].re || (z[j].re == z[j - 1].re && z[j].im < z[j - 1].im)); --j) {
            const C t = z[j];
            z[j] = z[j - 1];
            z[j - 1] = t;
        }
    const C zc = z[pick], zb = conj(zc);
    return zc - inv(zb) + q * inv(C{d, 0.0} - zb);
}

// 256 values, one per thread, sorted ascending in s (bitonic network)
template <typename T>
__device__ void block_sort256(T* s) {
    const int tid = threadIdx.x;
    for (int k = 2; k <= kBins; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            const int o = tid ^ j;
            if (o > tid) {
                const bool asc = (tid & k) == 0;
                const T a = s[tid], b = s[o];
                if ((a > b) == asc) {
                    s[tid] = b;
                    s[o] = a;
                }
            }
            __syncthreads();
        }
}

// input normalisation of one curve, thread j = bin j: asinh(10 (F / median - 1)) / 3 and the mask
// (T = float for training curves, double for observed ones)
template <typename T>
__device__ float2 normalise_block(T F, bool kept, int n_kept, T* s_v) {
    const int j = threadIdx.x;
    s_v[j] = kept ? F : T(INFINITY);
    __syncthreads();
    block_sort256(s_v);
    T med = T(1);
    if (n_kept > 0) med = (n_kept & 1) ? s_v[n_kept / 2] : T(0.5) * (s_v[n_kept / 2 - 1] + s_v[n_kept / 2]);
    if (!(med > T(0) && isfinite(med))) med = T(1);
    float2 o = make_float2(0.f, 0.f);
    if (kept) o = make_float2((float)(asinh(T(10) * (F / med - T(1))) / T(3)), 1.f);
    return o;
}

// The network input in BF16 as the first convolution's products read it: [B][260][2], two zero positions on
// either side of a sample. Position j of sample i, by thread j of 256.
constexpr int kInputRow = kBins + 4;
__device__ __forceinline__ void store_input(__nv_bfloat16* xb, int i, int j, float2 v) {
    uint32_t* row = reinterpret_cast<uint32_t*>(xb) + (size_t)i * kInputRow;
    row[j + 2] = pack_bf2(v.x, v.y);
    if (j < 4) row[j < 2 ? j : kBins + j] = 0u;
}

// ------------------------------------------------------------------------------------------
// kernels around the network
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kBins) input_kernel(const float* x, __nv_bfloat16* xb) {
    store_input(xb, blockIdx.x, threadIdx.x, reinterpret_cast<const float2*>(x)[(size_t)blockIdx.x * kBins + threadIdx.x]);
}
// ctr[0], ctr[1]: the network's step and the first step of the run; ctr[2]: the generator's step
__global__ void set_counter_kernel(int64_t* ctr, int64_t step, int64_t first) {
    ctr[0] = step;
    ctr[1] = first;
    ctr[2] = step;
}
__global__ void advance_kernel(int64_t* ctr) { ctr[0] += 1; }

__global__ void grid_kernel(double* t) {
    const int j = threadIdx.x;
    t[j] = -1.0 + (2.0 * j + 1.0) / kBins;
}

__global__ void init_kernel(float* w, uint64_t seed) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= kNParams) return;
    const int l = layer_of(idx), r = idx - c_off[l];
    float v = 0.f;
    if (r < c_K[l] * c_N[l]) {
        const u64x4 x = philox4x64((uint64_t)(idx >> 1), OP_CNN_INIT, 0, 0, seed, 0);
        double z0, z1;
        box_muller(x.x[0], x.x[1], &z0, &z1);
        const double z = (idx & 1) ? z1 : z0;
        const double std = l == 5 ? 0.1 * sqrt(1.0 / c_K[l]) : sqrt(2.0 / c_K[l]);
        v = (float)(z * std);
    }
    w[idx] = v;
}

// training sample i of step *ctr: parameters (window units), noise settings, targets
__global__ void gen_kernel(uint64_t seed, const int64_t* ctr, int B, double forced_frac, double* theta, double* aux,
                           float* y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B) return;
    const uint64_t step = (uint64_t)ctr[0];
    double u[16];
    uint64_t pick_word = 0;
    for (int k = 0; k < 4; ++k) {
        const u64x4 r = philox4x64(step, OP_CNN_GEN, (uint64_t)i, (uint64_t)k, seed, 0);
        for (int j = 0; j < 4; ++j) u[4 * k + j] = u01(r.x[j]);
        if (k == 2) pick_word = r.x[0];
    }
    double t0 = kT0Lo + (kT0Hi - kT0Lo) * u[0];
    const double tE = exp(kLnTELo + (kLnTEHi - kLnTELo) * u[1]);
    double u0 = u[2];
    double alpha = 2.0 * kPi * u[3];
    const double d = exp(kLnDLo + (kLnDHi - kLnDLo) * u[4]);
    const double lq = kLqLo + (kLqHi - kLqLo) * u[5];
    const double q = pow(10.0, lq);
    if (u[6] < forced_frac) {
        const double phi = 2.0 * kPi * u[7];
        const int pick = (int)uniform_int(pick_word, 4);
        const cx<double> zc = critical_point(d, q, phi, pick);
        const double ca = cos(alpha), sa = sin(alpha);
        double v0 = zc.re * ca + zc.im * sa;
        double tau = zc.re * sa - zc.im * ca;
        double al = alpha;
        if (v0 < 0.0) {
            al = alpha + kPi;
            if (al >= 2.0 * kPi) al -= 2.0 * kPi;
            v0 = -v0;
            tau = -tau;
        }
        const double tc = kTcLo + (kTcHi - kTcLo) * u[9];
        const double tt = tc - tau * tE;
        if (isfinite(v0) && isfinite(tt)) {  // keep the prior draw if the root iteration failed
            u0 = v0;
            alpha = al;
            t0 = tt;
        }
    }
    const double sig = exp(kLnSigLo + (kLnSigHi - kLnSigLo) * u[10]);
    const double p_drop = kDropMax * u[11];
    const bool gap = u[12] < kGapProb;
    const double g0 = kBins * u[13];
    const double gw = gap ? kGapMax * kBins * u[14] : 0.0;
    double* th = theta + 6 * (size_t)i;
    th[0] = t0;
    th[1] = tE;
    th[2] = u0;
    th[3] = alpha;
    th[4] = d;
    th[5] = q;
    double* ax = aux + 4 * (size_t)i;
    ax[0] = sig;
    ax[1] = p_drop;
    ax[2] = g0;
    ax[3] = gw;
    float* yy = y + 6 * (size_t)i;
    yy[0] = (float)t0;
    yy[1] = (float)log(tE);
    yy[2] = (float)u0;
    yy[3] = (float)(alpha / (2.0 * kPi));
    yy[4] = (float)log(d);
    yy[5] = (float)log10(q);
}

// noise, mask and normalisation of training curve blockIdx.x (thread = bin). The noise and the
// normalisation run in FP32 (the FP64 pipe is slow and the inputs are FP32); the mask decisions
// compare the 53-bit uniforms in FP64.
__global__ void __launch_bounds__(kBins) prep_kernel(const double* A, const double* aux, uint64_t seed,
                                                      const int64_t* ctr, float* x, __nv_bfloat16* xb) {
    __shared__ float s_v[kBins];
    const int i = blockIdx.x, j = threadIdx.x;
    const uint64_t step = (uint64_t)ctr[0];
    const double* ax = aux + 4 * (size_t)i;
    const u64x4 r = philox4x64(step, OP_CNN_NOISE, (uint64_t)i, (uint64_t)(j >> 1), seed, 0);
    const float rr = sqrtf(-2.f * logf((float)(1.0 - u01(r.x[0]))));
    const float ang = 6.283185307179586f * (float)u01(r.x[1]);
    const float z = (j & 1) ? rr * sinf(ang) : rr * cosf(ang);
    const double ud = u01(r.x[2 + (j & 1)]);
    double dj = (double)j - ax[2];
    if (dj < 0.0) dj += kBins;
    bool kept = ud >= ax[1] && !(dj < ax[3]);
    int n = __syncthreads_count(kept);
    if (n < kMinKept) {
        kept = true;
        n = kBins;
    }
    const float F = (float)A[(size_t)i * kBins + j] * (1.f + (float)ax[0] * z);
    const float2 v = normalise_block<float>(F, kept, n, s_v);
    if (x) reinterpret_cast<float2*>(x)[(size_t)i * kBins + j] = v;
    if (xb) store_input(xb, i, j, v);
}

// observed curve blockIdx.x resampled to the bins over its own span (thread = bin)
constexpr int kBinChunk = 1024;
__global__ void __launch_bounds__(kBins) bin_kernel(const double* t, const double* flux, const double* sigma,
                                                     const int64_t* offsets, float* x, double* window) {
    __shared__ double s_v[kBins];
    __shared__ int s_bin[kBinChunk];
    __shared__ double s_w[kBinChunk], s_wf[kBinChunk];
    const int lc = blockIdx.x, j = threadIdx.x;
    const int64_t e0 = offsets[lc];
    const int n = (int)(offsets[lc + 1] - e0);
    double lo = INFINITY, hi = -INFINITY;
    for (int e = j; e < n; e += kBins) {
        lo = fmin(lo, t[e0 + e]);
        hi = fmax(hi, t[e0 + e]);
    }
    s_v[j] = lo;
    __syncthreads();
    for (int o = kBins / 2; o > 0; o >>= 1) {
        if (j < o) s_v[j] = fmin(s_v[j], s_v[j + o]);
        __syncthreads();
    }
    const double tmin = s_v[0];
    __syncthreads();
    s_v[j] = hi;
    __syncthreads();
    for (int o = kBins / 2; o > 0; o >>= 1) {
        if (j < o) s_v[j] = fmax(s_v[j], s_v[j + o]);
        __syncthreads();
    }
    const double tmax = s_v[0];
    __syncthreads();
    double span = tmax - tmin;
    if (!(span > 0.0)) span = 1.0;
    double sw = 0.0, swf = 0.0;
    for (int base = 0; base < n; base += kBinChunk) {
        const int m = min(kBinChunk, n - base);
        for (int e = j; e < m; e += kBins) {
            const double te = t[e0 + base + e], se = sigma[e0 + base + e];
            const int b = (int)floor((te - tmin) / span * kBins);
            s_bin[e] = min(kBins - 1, b);
            const double w = 1.0 / (se * se);
            s_w[e] = w;
            s_wf[e] = __dmul_rn(w, flux[e0 + base + e]);
        }
        __syncthreads();
        for (int e = 0; e < m; ++e)
            if (s_bin[e] == j) {
                sw += s_w[e];
                swf += s_wf[e];
            }
        __syncthreads();
    }
    const bool kept = sw > 0.0;
    const double F = kept ? swf / sw : 0.0;
    const int n_kept = __syncthreads_count(kept);
    reinterpret_cast<float2*>(x)[(size_t)lc * kBins + j] = normalise_block<double>(F, kept, n_kept, s_v);
    if (j == 0) {
        window[2 * lc] = 0.5 * (tmin + tmax);
        window[2 * lc + 1] = 0.5 * span;
    }
}

// Gaussian negative log-likelihood (mean over the batch) and its gradient for the outputs: one
// thread per (sample, target) in FP32, block sums in FP64 written per block, then summed in
// block order by loss_sum_kernel
constexpr int kLossThreads = 256;
__global__ void __launch_bounds__(kLossThreads) loss_terms_kernel(const float* out, const float* y, int B,
                                                                  float* dout, double* part) {
    __shared__ double s[kLossThreads];
    const int idx = blockIdx.x * kLossThreads + threadIdx.x;
    double term = 0.0;
    if (idx < 6 * B) {
        const int b = idx / 6, j = idx - 6 * b;
        const float mu = out[12 * b + j], sv = out[12 * b + 6 + j];
        const float r = y[6 * b + j] - mu, e = expf(-sv);
        term = 0.5 * ((double)(r * r * e) + (double)sv);
        dout[12 * b + j] = -r * e / (float)B;
        dout[12 * b + 6 + j] = 0.5f * (1.f - r * r * e) / (float)B;
    }
    s[threadIdx.x] = term;
    __syncthreads();
    for (int o = kLossThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = s[0];
}

__global__ void loss_sum_kernel(const double* part, int n_part, int B, double* loss, float* hist, const int64_t* ctr) {
    double acc = 0.0;
    for (int k = 0; k < n_part; ++k) acc += part[k];
    const double L = acc / B;
    if (loss) *loss = L;
    if (hist) hist[ctr[0] - ctr[1]] = (float)L;
}

int loss_blocks(int B) { return (6 * B + kLossThreads - 1) / kLossThreads; }

cudaError_t launch_loss(const float* out, const float* y, int B, float* dout, double* part, double* loss, float* hist,
                        const int64_t* ctr, cudaStream_t s) {
    loss_terms_kernel<<<loss_blocks(B), kLossThreads, 0, s>>>(out, y, B, dout, part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    loss_sum_kernel<<<1, 1, 0, s>>>(part, loss_blocks(B), B, loss, hist, ctr);
    return cudaGetLastError();
}

__global__ void cast_kernel(const float* w, __nv_bfloat16* wb, __nv_bfloat16* wbt) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= kNParams) return;
    const int l = layer_of(idx), r = idx - c_off[l], K = c_K[l], N = c_N[l];
    const __nv_bfloat16 v = __float2bfloat16_rn(w[idx]);
    wb[idx] = v;
    if (r < K * N) wbt[c_off[l] + (r % N) * K + r / N] = v;
}

struct PartTab {
    const float* p[6];  // per layer: [splits][(K + 1) N] weight-gradient partials
    int z[6];
};
struct AdamArgs {
    bool on;
    float* m;
    float* v;
    double lr0, b1, b2, eps, wd;
    int n_steps, warmup;
    int64_t t;              // 1-based step
    const double* scalars;  // the step's learning rate and bias corrections, or null: computed from t
};

// the learning rate of 1-based step t and the bias corrections 1 / (1 - beta^t): a cosine and two powers, some
// 400 instructions of the FP64 pipe
__device__ __forceinline__ double adam_scalar(const AdamArgs& ad, int64_t t, int k) {
    if (k == 0) return lr_at(t, ad.n_steps, ad.warmup, ad.lr0);
    return 1.0 / (1.0 - pow(k == 1 ? ad.b1 : ad.b2, (double)t));
}
// the scalars of step ctr[0] + 1, once instead of in every block of the update
__global__ void adam_scalars_kernel(AdamArgs ad, const int64_t* ctr, double* out) {
    if (threadIdx.x < 3) out[threadIdx.x] = adam_scalar(ad, ctr[0] + 1, threadIdx.x);
}

// gradient = sum of the partials in split order (or grad_in); optional AdamW step and BF16 copies
__global__ void update_kernel(PartTab tab, const float* grad_in, float* grad_out, AdamArgs ad, float* w,
                              __nv_bfloat16* wb, __nv_bfloat16* wbt) {
    // the step's learning rate and bias corrections 1 / (1 - beta^t), once per block
    __shared__ double s_sc[3];
    if (ad.on && threadIdx.x < 3)
        s_sc[threadIdx.x] = ad.scalars ? ad.scalars[threadIdx.x] : adam_scalar(ad, ad.t, threadIdx.x);
    __syncthreads();
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= kNParams) return;
    const int l = layer_of(idx), r = idx - c_off[l], K = c_K[l], N = c_N[l];
    float g;
    if (grad_in) {
        g = grad_in[idx];
    } else {
        // partials of split s summed in four interleaved chains (s mod 4), combined in a fixed order:
        // independent loads in flight, the same bits on every call
        const int cnt = (K + 1) * N, z = tab.z[l];
        const float* p = tab.p[l] + r;
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
        int s = 0;
#pragma unroll 4
        for (; s + 4 <= z; s += 4) {
            a0 += p[(size_t)s * cnt];
            a1 += p[(size_t)(s + 1) * cnt];
            a2 += p[(size_t)(s + 2) * cnt];
            a3 += p[(size_t)(s + 3) * cnt];
        }
        for (; s < z; ++s) a0 += p[(size_t)s * cnt];
        g = (a0 + a1) + (a2 + a3);
    }
    if (grad_out) grad_out[idx] = g;
    float wv = w[idx];
    if (ad.on) {
        const double lr = s_sc[0];
        double wd = (double)wv * (1.0 - lr * ad.wd);
        const double m = ad.b1 * (double)ad.m[idx] + (1.0 - ad.b1) * g;
        const double v = ad.b2 * (double)ad.v[idx] + (1.0 - ad.b2) * (double)g * g;
        const double mh = m * s_sc[1];
        const double vh = v * s_sc[2];
        wd = wd - lr * mh / (sqrt(vh) + ad.eps);
        ad.m[idx] = (float)m;
        ad.v[idx] = (float)v;
        wv = (float)wd;
        w[idx] = wv;
    }
    if (wb) {
        const __nv_bfloat16 b = __float2bfloat16_rn(wv);
        wb[idx] = b;
        if (r < K * N) wbt[c_off[l] + (r % N) * K + r / N] = b;
    }
}

// seed row (lc, r) of draw round 0 from the Gaussian outputs of curve lc
__global__ void propose_kernel(const float* out, const double* window, int n_lc, Bounds b, int n_seed, uint64_t seed,
                               double* genes) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)n_lc * n_seed) return;
    const int lc = (int)(idx / n_seed), r = (int)(idx % n_seed);
    proposal_row(out + 12 * (size_t)lc, window[2 * lc], window[2 * lc + 1], b, seed, (uint64_t)lc, (uint64_t)r, 0,
                 genes + 6 * (size_t)idx);
}

// ------------------------------------------------------------------------------------------
// tensor-core epilogues
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ float4 add4(float4 v, const float* b) {
    return make_float4(v.x + b[0], v.y + b[1], v.z + b[2], v.w + b[3]);
}
__device__ __forceinline__ void store_bf4(__nv_bfloat16* p, float a, float b, float c, float d) {
    *reinterpret_cast<uint2*>(p) = make_uint2(pack_bf2(a, b), pack_bf2(c, d));
}
struct EpiAct {  // z = acc + bias; keep z (training) and GELU(z) in BF16
    const float* bias;
    float* z;
    __nv_bfloat16* h;
    int M, N;
    __device__ void operator()(int m, int n, float4 v, int) const {
        if (m >= M || n >= N) return;
        v = add4(v, bias + n);
        const size_t i = (size_t)m * N + n;
        if (z) *reinterpret_cast<float4*>(z + i) = v;
        store_bf4(h + i, gelu(v.x), gelu(v.y), gelu(v.z), gelu(v.w));
    }
};
struct EpiOut {  // network output: acc + bias, FP32
    const float* bias;
    float* out;
    int M, N;
    __device__ void operator()(int m, int n, float4 v, int) const {
        if (m >= M || n >= N) return;
        *reinterpret_cast<float4*>(out + (size_t)m * N + n) = add4(v, bias + n);
    }
};
struct EpiDgrad {  // gradient of the pre-activation: acc * GELU'(z), BF16; row m at m * ld + off
    const float* z;
    __nv_bfloat16* dz;
    int M, N, ld, off;
    __device__ void operator()(int m, int n, float4 v, int) const {
        if (m >= M || n >= N) return;
        const size_t i = (size_t)m * ld + off + n;
        const float4 zz = *reinterpret_cast<const float4*>(z + i);
        store_bf4(dz + i, v.x * gelu_grad(zz.x), v.y * gelu_grad(zz.y), v.z * gelu_grad(zz.z), v.w * gelu_grad(zz.w));
    }
};
struct EpiPart {  // weight-gradient partial of split z
    float* part;
    int M, N;
    __device__ void operator()(int m, int n, float4 v, int z) const {
        if (m >= M || n >= N) return;
        *reinterpret_cast<float4*>(part + ((size_t)z * M + m) * N + n) = v;  // every N is a multiple of 4
    }
};

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------
struct Split {
    int z = 1, ksplit = 0;  // splits of the reduction, and its length in each
};

constexpr int kSplitUnit = 32;

Split split_for(int M, int N, int K, int sms) {
    const int nt = (K + kSplitUnit - 1) / kSplitUnit;
    const int tiles = ((M + BM - 1) / BM) * ((N + BN - 1) / BN);
    int want = std::max(1, (sms + tiles - 1) / tiles);
    want = std::min(want, nt);
    const int tps = (nt + want - 1) / want;
    Split s;
    s.z = (nt + tps - 1) / tps;
    s.ksplit = tps * kSplitUnit;
    return s;
}

template <bool AK, bool BKM, int STAGES, class LA, class LB, class EP>
cudaError_t launch_gemm(const LA& la, const LB& lb, const EP& ep, int M, int N, int K, Split sp, cudaStream_t s) {
    auto kern = gemm_kernel<AK, BKM, STAGES, LA, LB, EP>;
    // opt in to the tile ring (> 48 KB) once per device and instantiation; the first
    // launch of a sequence runs outside any stream capture
    cudaError_t e = raise_smem_limit((const void*)kern, gemm_smem(STAGES));
    if (e != cudaSuccess) return e;
    dim3 grid((M + BM - 1) / BM, (N + BN - 1) / BN, sp.z);
    kern<<<grid, kGemmThreads, gemm_smem(STAGES), s>>>(la, lb, ep, M, N, K, sp.ksplit);
    return cudaGetLastError();
}
template <bool AK, bool BKM, class LA, class LB, class EP>
cudaError_t gemm(const LA& la, const LB& lb, const EP& ep, int M, int N, int K, Split sp, cudaStream_t s) {
    return launch_gemm<AK, BKM, kDeep>(la, lb, ep, M, N, K, sp, s);
}
template <bool AK, bool BKM, int STAGES = kShallow, class LA, class LB, class EP>
cudaError_t gemm1(const LA& la, const LB& lb, const EP& ep, int M, int N, int K, cudaStream_t s) {
    Split sp;
    sp.z = 1;
    sp.ksplit = K;
    return launch_gemm<AK, BKM, STAGES>(la, lb, ep, M, N, K, sp, s);
}

// lay out consecutive 256-byte aligned pieces of one region; with base == nullptr only sizes
struct Carver {
    char* base;
    size_t off = 0;
    template <typename T>
    T* take(size_t count) {
        const size_t o = (off + 255) & ~size_t(255);
        off = o + sizeof(T) * count;
        return base ? reinterpret_cast<T*>(base + o) : nullptr;
    }
};

int sm_count() { return device_sm_count(); }

// one batch's activations, gradients and weight copies
struct Net {
    int B = 0;
    bool train = false;
    __nv_bfloat16* xb = nullptr;  // [B][260][2], carved unless the caller brings its own
    __nv_bfloat16 *wb = nullptr, *wbt = nullptr;
    __nv_bfloat16 *h1, *h2, *h3, *h4, *h5;
    float *z1 = nullptr, *z2 = nullptr, *z3 = nullptr, *z4 = nullptr, *z5 = nullptr;
    float* out = nullptr;
    float* dout = nullptr;
    double* loss_part = nullptr;
    __nv_bfloat16 *dz1 = nullptr, *dz2 = nullptr, *dz3 = nullptr, *dz4 = nullptr, *dz5 = nullptr;
    float* part[6] = {};
    Split sp[6];
};

// wgrad product sizes of layer l: rows K + 1 (bias row), columns N, reduction length
void wgrad_shape(int l, int B, int* M, int* N, int* K) {
    static const int Lo[4] = {256, 128, 64, 32};
    *M = kKH[l] + 1;
    *N = kNH[l];
    *K = l < 4 ? B * Lo[l] : B;
}

Net carve_net(Carver& c, int B, bool train, int sms, bool own_input = true) {
    Net n;
    n.B = B;
    n.train = train;
    n.wb = c.take<__nv_bfloat16>(kNParams);
    n.wbt = c.take<__nv_bfloat16>(kNParams);
    n.xb = own_input ? c.take<__nv_bfloat16>((size_t)B * kInputRow * 2) : nullptr;
    n.h1 = c.take<__nv_bfloat16>((size_t)B * 256 * 64);
    n.h2 = c.take<__nv_bfloat16>((size_t)B * 128 * 64);
    n.h3 = c.take<__nv_bfloat16>((size_t)B * 64 * 64);
    n.h4 = c.take<__nv_bfloat16>((size_t)B * 32 * 64);
    n.h5 = c.take<__nv_bfloat16>((size_t)B * 128);
    n.out = c.take<float>((size_t)B * 12);
    if (train) {
        n.z1 = c.take<float>((size_t)B * 256 * 64);
        n.z2 = c.take<float>((size_t)B * 128 * 64);
        n.z3 = c.take<float>((size_t)B * 64 * 64);
        n.z4 = c.take<float>((size_t)B * 32 * 64);
        n.z5 = c.take<float>((size_t)B * 128);
        n.dout = c.take<float>((size_t)B * 12);
        n.loss_part = c.take<double>((size_t)loss_blocks(B));
        n.dz1 = c.take<__nv_bfloat16>((size_t)B * 256 * 64);
        n.dz2 = c.take<__nv_bfloat16>((size_t)B * 128 * 64);
        n.dz3 = c.take<__nv_bfloat16>((size_t)B * 64 * 64);
        n.dz4 = c.take<__nv_bfloat16>((size_t)B * 32 * 64);
        n.dz5 = c.take<__nv_bfloat16>((size_t)B * 128);
        for (int l = 0; l < 6; ++l) {
            int M, N, K;
            wgrad_shape(l, B, &M, &N, &K);
            n.sp[l] = split_for(M, N, K, sms);
            n.part[l] = c.take<float>((size_t)n.sp[l].z * M * N);
        }
    }
    return n;
}

// The stream that draws training batches beside the network, and its fork and join events: one set per
// device, kept until the process exits; used under the call lock
struct SideStream {
    cudaStream_t stream = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
};

sblm_status side_stream(SideStream** out) {
    static std::map<int, SideStream>* sets = new std::map<int, SideStream>();
    int dev = 0;
    SBLM_CUDA(cudaGetDevice(&dev));
    SideStream& s = (*sets)[dev];
    if (!s.stream) SBLM_CUDA(cudaStreamCreateWithFlags(&s.stream, cudaStreamNonBlocking));
    if (!s.fork) SBLM_CUDA(cudaEventCreateWithFlags(&s.fork, cudaEventDisableTiming));
    if (!s.join) SBLM_CUDA(cudaEventCreateWithFlags(&s.join, cudaEventDisableTiming));
    *out = &s;
    return SBLM_OK;
}

#define CNN_TRY(call)                              \
    do {                                           \
        cudaError_t e_ = (call);                   \
        if (e_ != cudaSuccess) return e_;          \
    } while (0)

// forward pass; z_l kept when the net was laid out for training
cudaError_t net_forward(const Net& n, const float* w, cudaStream_t s) {
    const int B = n.B;
    const __nv_bfloat16* wbt = n.wbt;
    CNN_TRY((gemm1<true, true>(InputCols{n.xb, B}, DenseBFAny{wbt + kOffH[0], 64, 10, 10},
                               EpiAct{w + kOffH[0] + 640, n.z1, n.h1, B * 256, 64}, B * 256, 64, 10, s)));
    CNN_TRY((gemm1<true, true>(Im2col{n.h1, B, 7}, DenseBF{wbt + kOffH[1], 64, 320, 320, false},
                               EpiAct{w + kOffH[1] + 20480, n.z2, n.h2, B * 128, 64}, B * 128, 64, 320, s)));
    CNN_TRY((gemm1<true, true>(Im2col{n.h2, B, 6}, DenseBF{wbt + kOffH[2], 64, 320, 320, false},
                               EpiAct{w + kOffH[2] + 20480, n.z3, n.h3, B * 64, 64}, B * 64, 64, 320, s)));
    CNN_TRY((gemm1<true, true>(Im2col{n.h3, B, 5}, DenseBF{wbt + kOffH[3], 64, 320, 320, false},
                               EpiAct{w + kOffH[3] + 20480, n.z4, n.h4, B * 32, 64}, B * 32, 64, 320, s)));
    CNN_TRY((gemm1<true, true, kDeep>(DenseBF{n.h4, B, 2048, 2048, false}, DenseBF{wbt + kOffH[4], 128, 2048, 2048, false},
                               EpiAct{w + kOffH[4] + 262144, n.z5, n.h5, B, 128}, B, 128, 2048, s)));
    CNN_TRY((gemm1<true, true>(DenseBF{n.h5, B, 128, 128, false}, DenseBF{wbt + kOffH[5], 12, 128, 128, false},
                               EpiOut{w + kOffH[5] + 1536, n.out, B, 12}, B, 12, 128, s)));
    return cudaSuccess;
}

// gradient of the pre-activations z of a stride-2 convolution's input [B][2 Lo][64] from that of its
// output: one product per parity of the input position
cudaError_t conv_input_gradient(const __nv_bfloat16* dz_out, int B, int log_lo, const __nv_bfloat16* w, const float* z,
                                __nv_bfloat16* dz, cudaStream_t s) {
    const int M = B << log_lo;
    CNN_TRY((gemm1<true, true>(ConvGrad<0>{dz_out, B, log_lo}, ConvWT<0>{w}, EpiDgrad{z, dz, M, 64, 128, 0}, M, 64, 192,
                               s)));
    return gemm1<true, true>(ConvGrad<1>{dz_out, B, log_lo}, ConvWT<1>{w}, EpiDgrad{z, dz, M, 64, 128, 64}, M, 64, 128,
                             s);
}

// backward pass from n.dout: weight-gradient partials of every layer
cudaError_t net_backward(const Net& n, cudaStream_t s) {
    const int B = n.B;
    const __nv_bfloat16* wb = n.wb;
    // dense 128 -> 12
    CNN_TRY((gemm<false, false>(DenseBF{n.h5, B, 128, 128, true}, DenseF32{n.dout, B, 12, 12},
                                EpiPart{n.part[5], 129, 12}, 129, 12, B, n.sp[5], s)));
    CNN_TRY((gemm1<true, true>(DenseF32{n.dout, B, 12, 12}, DenseBFAny{wb + kOffH[5], 128, 12, 12},
                               EpiDgrad{n.z5, n.dz5, B, 128, 128, 0}, B, 128, 12, s)));
    // dense 2048 -> 128
    CNN_TRY((gemm<false, false>(DenseBF{n.h4, B, 2048, 2048, true}, DenseBF{n.dz5, B, 128, 128, false},
                                EpiPart{n.part[4], 2049, 128}, 2049, 128, B, n.sp[4], s)));
    CNN_TRY((gemm1<true, true>(DenseBF{n.dz5, B, 128, 128, false}, DenseBF{wb + kOffH[4], 2048, 128, 128, false},
                               EpiDgrad{n.z4, n.dz4, B, 2048, 2048, 0}, B, 2048, 128, s)));
    // conv 4 (64 -> 32 positions)
    CNN_TRY((gemm<false, false>(Im2colT{n.h3, B, 5}, DenseBF{n.dz4, B * 32, 64, 64, false},
                                EpiPart{n.part[3], 321, 64}, 321, 64, B * 32, n.sp[3], s)));
    CNN_TRY(conv_input_gradient(n.dz4, B, 5, wb + kOffH[3], n.z3, n.dz3, s));
    // conv 3 (128 -> 64)
    CNN_TRY((gemm<false, false>(Im2colT{n.h2, B, 6}, DenseBF{n.dz3, B * 64, 64, 64, false},
                                EpiPart{n.part[2], 321, 64}, 321, 64, B * 64, n.sp[2], s)));
    CNN_TRY(conv_input_gradient(n.dz3, B, 6, wb + kOffH[2], n.z2, n.dz2, s));
    // conv 2 (256 -> 128)
    CNN_TRY((gemm<false, false>(Im2colT{n.h1, B, 7}, DenseBF{n.dz2, B * 128, 64, 64, false},
                                EpiPart{n.part[1], 321, 64}, 321, 64, B * 128, n.sp[1], s)));
    CNN_TRY(conv_input_gradient(n.dz2, B, 7, wb + kOffH[1], n.z1, n.dz1, s));
    // conv 1 (input)
    CNN_TRY((gemm<false, false>(InputCols{n.xb, B}, DenseBF{n.dz1, B * 256, 64, 64, false},
                                EpiPart{n.part[0], 11, 64}, 11, 64, B * 256, n.sp[0], s)));
    return cudaSuccess;
}

PartTab part_tab(const Net& n) {
    PartTab t{};
    for (int l = 0; l < 6; ++l) {
        t.p[l] = n.part[l];
        t.z[l] = n.sp[l].z;
    }
    return t;
}

constexpr int kUpdThreads = 256;
constexpr int kUpdBlocks = (kNParams + kUpdThreads - 1) / kUpdThreads;

cudaError_t launch_cast(const float* w, __nv_bfloat16* wb, __nv_bfloat16* wbt, cudaStream_t s) {
    cast_kernel<<<kUpdBlocks, kUpdThreads, 0, s>>>(w, wb, wbt);
    return cudaGetLastError();
}

cudaError_t launch_input(const float* x, const Net& n, cudaStream_t s) {
    input_kernel<<<n.B, kBins, 0, s>>>(x, n.xb);
    return cudaGetLastError();
}

// generator buffers of one training batch
struct Gen {
    double* theta;
    double* aux;
    double* A;
    float* y;
    double* grid;
    void* mixed;
    int64_t* ctr;
};

Gen carve_gen(Carver& c, int B, int precision, bool own_theta) {
    Gen g{};
    g.theta = own_theta ? c.take<double>((size_t)B * 6) : nullptr;
    g.aux = c.take<double>((size_t)B * 4);
    g.A = c.take<double>((size_t)B * kBins);
    g.y = c.take<float>((size_t)B * 6);
    g.grid = c.take<double>(kBins);
    g.mixed = c.take<unsigned char>(mixed_scratch_bytes(precision, B, kBins, false));
    g.ctr = c.take<int64_t>(4);
    return g;
}

// draw a batch at step ctr[2]: parameters, forward model, noise and normalisation
cudaError_t launch_gen(const Gen& g, int B, int precision, double forced_frac, uint64_t seed, float* x, __nv_bfloat16* xb,
                       float* y, cudaStream_t s) {
    // one warp per block: the caustic-aimed samples (an FP64 root iteration each) spread over the SMs
    gen_kernel<<<(B + 31) / 32, 32, 0, s>>>(seed, g.ctr + 2, B, forced_frac, g.theta, g.aux, y);
    CNN_TRY(cudaGetLastError());
    ForwardArgs fa{};
    fa.src = g.theta;
    fa.n_cand = B;
    fa.t = g.grid;
    fa.n_ep = kBins;
    fa.A_out = g.A;
    fa.mode = precision;
    fa.G = choose_group(B, kBins);
    fa.mixed = g.mixed;
    CNN_TRY(launch_forward(fa, s));
    prep_kernel<<<B, kBins, 0, s>>>(g.A, g.aux, seed, g.ctr + 2, x, xb);
    return cudaGetLastError();
}

sblm_status check_train_params(const sblm_cnn_train_params* p) {
    if (!p) return fail(SBLM_EINVAL, "train params are NULL");
    if (p->batch < 1 || p->batch > kMaxBatch) return fail(SBLM_EINVAL, "batch must be in [1, %d]", kMaxBatch);
    if (p->n_steps < 1 || p->warmup < 0) return fail(SBLM_EINVAL, "n_steps must be >= 1 and warmup >= 0");
    if (p->precision < SBLM_FP64 || p->precision > SBLM_FP32) return fail(SBLM_EINVAL, "unknown precision %d", p->precision);
    if (!(p->lr > 0) || !(p->beta1 >= 0 && p->beta1 < 1) || !(p->beta2 >= 0 && p->beta2 < 1) || !(p->eps > 0) ||
        !(p->weight_decay >= 0))
        return fail(SBLM_EINVAL, "optimiser settings out of range");
    if (!(p->forced_frac >= 0 && p->forced_frac <= 1)) return fail(SBLM_EINVAL, "forced_frac must be in [0, 1]");
    return SBLM_OK;
}

AdamArgs adam_args(const sblm_cnn_train_params* p, float* state, int64_t t, const double* scalars) {
    AdamArgs a{};
    a.on = true;
    a.m = state;
    a.v = state + kNParams;
    a.lr0 = p->lr;
    a.b1 = p->beta1;
    a.b2 = p->beta2;
    a.eps = p->eps;
    a.wd = p->weight_decay;
    a.n_steps = p->n_steps;
    a.warmup = p->warmup;
    a.t = t;
    a.scalars = scalars;
    return a;
}

template <typename T>
void put(std::vector<unsigned char>& k, const T& v) {
    const unsigned char* p = reinterpret_cast<const unsigned char*>(&v);
    k.insert(k.end(), p, p + sizeof(T));
}

// ---------------- inference scratch for the seeded batched fit ----------------
InferScratch carve_infer(Carver& c, int n, int n_seed, Net* net) {
    InferScratch sc{};
    sc.x = c.take<float>((size_t)n * 2 * kBins);
    sc.window = c.take<double>((size_t)n * 2);
    sc.genes = c.take<double>((size_t)n * std::max(1, n_seed) * 6);
    Net nn = carve_net(c, n, false, 1);
    sc.wb = nn.wb;
    sc.wbt = nn.wbt;
    sc.act = nn.h1;
    sc.out = nn.out;
    if (net) *net = nn;
    return sc;
}

size_t infer_scratch_bytes(int n, int n_seed) {
    Carver c{nullptr};
    carve_infer(c, n, n_seed, nullptr);
    return c.off;
}

InferScratch infer_scratch_carve(void* base, int n, int n_seed) {
    Carver c{static_cast<char*>(base)};
    return carve_infer(c, n, n_seed, nullptr);
}

cudaError_t launch_seed_rows(const double* t, const double* flux, const double* sigma, const int64_t* offsets,
                             int n_lc, const float* weights, const Bounds& b, int n_seed, uint64_t seed,
                             const InferScratch& sc, cudaStream_t s) {
    // the carve is deterministic: recover the network's pointers from the same base
    Carver c{reinterpret_cast<char*>(sc.x)};
    Net net;
    carve_infer(c, n_lc, n_seed, &net);
    bin_kernel<<<n_lc, kBins, 0, s>>>(t, flux, sigma, offsets, sc.x, sc.window);
    CNN_TRY(cudaGetLastError());
    CNN_TRY(launch_cast(weights, net.wb, net.wbt, s));
    CNN_TRY(launch_input(sc.x, net, s));
    CNN_TRY(net_forward(net, weights, s));
    const long long total = (long long)n_lc * n_seed;
    if (total > 0) {
        propose_kernel<<<(unsigned)((total + 127) / 128), 128, 0, s>>>(net.out, sc.window, n_lc, b, n_seed, seed,
                                                                      sc.genes);
        CNN_TRY(cudaGetLastError());
    }
    return cudaSuccess;
}

// one block whose bounded wait on an mbarrier that nothing arrives on runs out after `polls`
// polls: the give-up path of the tensor-core tiles (flag set, no hang), with no tensor memory or
// MMA involved
__global__ void wait_selftest_kernel(int polls) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar)));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    __syncthreads();
    mbar_wait(smem_u32(&bar), 0u, polls);  // phase 0 never completes
    __syncthreads();
}

sblm_status check_timeout(cudaStream_t s) {
    int flag = 0;
    SBLM_CUDA(cudaMemcpyFromSymbolAsync(&flag, g_tc_timeout, sizeof(int), 0, cudaMemcpyDeviceToHost, s));
    SBLM_CUDA(cudaStreamSynchronize(s));
    if (flag) {
        const int zero = 0;
        SBLM_CUDA(cudaMemcpyToSymbol(g_tc_timeout, &zero, sizeof(int)));
        return fail(SBLM_ETIMEOUT, "a tensor-core tile gave up waiting for its MMAs; results are invalid");
    }
    return SBLM_OK;
}

}  // namespace cnn

sblm_status check_bounds(const sblm_bounds* b, Bounds* out);

}  // namespace sblm

using namespace sblm;
using namespace sblm::cnn;

extern "C" {

void sblm_cnn_train_params_default(sblm_cnn_train_params* p) {
    if (!p) return;
    std::memset(p, 0, sizeof *p);
    p->batch = 256;
    p->n_steps = 4096;
    p->warmup = 200;
    p->precision = SBLM_FP32;
    p->lr = 2e-3;
    p->beta1 = 0.9;
    p->beta2 = 0.999;
    p->eps = 1e-8;
    p->weight_decay = 1e-4;
    p->forced_frac = 0.1;
    p->seed = 0;
}

int32_t sblm_cnn_num_params(void) { return kNParams; }

sblm_status sblm_cnn_selftest_timeout(int32_t polls, void* stream) {
    if (polls < 1 || polls > (1 << 20)) return fail(SBLM_EINVAL, "polls must be in [1, 2^20]");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CallLock lock;
    wait_selftest_kernel<<<1, 64, 0, s>>>(polls);
    SBLM_CUDA(cudaGetLastError());
    return check_timeout(s);
}

sblm_status sblm_cnn_init(float* weights, uint64_t seed, void* stream) {
    if (!weights) return fail(SBLM_EINVAL, "weights is NULL");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CallLock lock;
    Staging st(s);
    int i_w;
    SBLM_TRY(st.arg(weights, sizeof(float) * kNParams, false, true, &i_w));
    SBLM_TRY(st.begin());
    init_kernel<<<kUpdBlocks, kUpdThreads, 0, s>>>(static_cast<float*>(st.dev(i_w)), seed);
    SBLM_CUDA(cudaGetLastError());
    return st.end();
}

sblm_status sblm_cnn_make_batch(uint64_t seed, int64_t step, int32_t batch, double forced_frac, int32_t precision,
                                float* x, float* y, double* theta, void* stream) {
    if (batch < 1 || batch > kMaxBatch) return fail(SBLM_EINVAL, "batch must be in [1, %d]", kMaxBatch);
    if (!(forced_frac >= 0 && forced_frac <= 1)) return fail(SBLM_EINVAL, "forced_frac must be in [0, 1]");
    if (precision < SBLM_FP64 || precision > SBLM_FP32) return fail(SBLM_EINVAL, "unknown precision %d", precision);
    if (!x || !y) return fail(SBLM_EINVAL, "x and y are required");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CallLock lock;
    Staging st(s);
    int i_x, i_y, i_th;
    SBLM_TRY(st.arg(x, sizeof(float) * (size_t)batch * 2 * kBins, false, true, &i_x));
    SBLM_TRY(st.arg(y, sizeof(float) * (size_t)batch * 6, false, true, &i_y));
    SBLM_TRY(st.arg(theta, theta ? sizeof(double) * (size_t)batch * 6 : 0, false, true, &i_th));
    Carver probe{nullptr};
    carve_gen(probe, batch, precision, true);
    const int k = st.scratch(probe.off);
    SBLM_TRY(st.begin());
    Carver c{static_cast<char*>(st.scratch_ptr(k))};
    Gen g = carve_gen(c, batch, precision, true);
    if (theta) g.theta = static_cast<double*>(st.dev(i_th));
    set_counter_kernel<<<1, 1, 0, s>>>(g.ctr, step, step);
    grid_kernel<<<1, kBins, 0, s>>>(g.grid);
    SBLM_CUDA(launch_gen(g, batch, precision, forced_frac, seed, static_cast<float*>(st.dev(i_x)),
                         nullptr, static_cast<float*>(st.dev(i_y)), s));
    return st.end();
}

sblm_status sblm_cnn_bin(const double* t, const double* flux, const double* sigma, const int64_t* offsets,
                         int32_t n_lc, float* x, double* window, void* stream) {
    if (n_lc < 1) return fail(SBLM_EINVAL, "n_lc must be >= 1");
    if (!t || !flux || !sigma || !offsets || !x || !window) return fail(SBLM_EINVAL, "NULL buffer");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CallLock lock;
    std::vector<int64_t> off(n_lc + 1);
    bool od = false;
    SBLM_TRY(is_device_pointer(offsets, &od));
    if (od)
        SBLM_CUDA(cudaMemcpy(off.data(), offsets, sizeof(int64_t) * (n_lc + 1), cudaMemcpyDeviceToHost));
    else
        std::memcpy(off.data(), offsets, sizeof(int64_t) * (n_lc + 1));
    if (off[0] != 0) return fail(SBLM_EINVAL, "offsets[0] must be 0");
    for (int i = 0; i < n_lc; ++i)
        if (off[i + 1] - off[i] < 1) return fail(SBLM_EINVAL, "lightcurve %d has no epochs", i);
    const size_t total = (size_t)off[n_lc];
    Staging st(s);
    int i_t, i_f, i_s, i_o, i_x, i_w;
    SBLM_TRY(st.arg(t, sizeof(double) * total, true, false, &i_t));
    SBLM_TRY(st.arg(flux, sizeof(double) * total, true, false, &i_f));
    SBLM_TRY(st.arg(sigma, sizeof(double) * total, true, false, &i_s));
    SBLM_TRY(st.arg(offsets, sizeof(int64_t) * (n_lc + 1), true, false, &i_o));
    SBLM_TRY(st.arg(x, sizeof(float) * (size_t)n_lc * 2 * kBins, false, true, &i_x));
    SBLM_TRY(st.arg(window, sizeof(double) * 2 * (size_t)n_lc, false, true, &i_w));
    bool d1, d2, d3;
    SBLM_TRY(is_device_pointer(t, &d1));
    SBLM_TRY(is_device_pointer(flux, &d2));
    SBLM_TRY(is_device_pointer(sigma, &d3));
    if (!d1 && !d2 && !d3) SBLM_TRY(check_lightcurve_host(t, flux, sigma, (int)total));
    SBLM_TRY(st.begin());
    bin_kernel<<<n_lc, kBins, 0, s>>>(static_cast<const double*>(st.dev(i_t)), static_cast<const double*>(st.dev(i_f)),
                                      static_cast<const double*>(st.dev(i_s)), static_cast<const int64_t*>(st.dev(i_o)),
                                      static_cast<float*>(st.dev(i_x)), static_cast<double*>(st.dev(i_w)));
    SBLM_CUDA(cudaGetLastError());
    return st.end();
}

sblm_status sblm_cnn_forward(const float* weights, const float* x, int32_t batch, float* out, void* stream) {
    if (batch < 1) return fail(SBLM_EINVAL, "batch must be >= 1");
    if (!weights || !x || !out) return fail(SBLM_EINVAL, "NULL buffer");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CallLock lock;
    Staging st(s);
    int i_w, i_x, i_o;
    SBLM_TRY(st.arg(weights, sizeof(float) * kNParams, true, false, &i_w));
    SBLM_TRY(st.arg(x, sizeof(float) * (size_t)batch * 2 * kBins, true, false, &i_x));
    SBLM_TRY(st.arg(out, sizeof(float) * (size_t)batch * 12, false, true, &i_o));
    Carver probe{nullptr};
    carve_net(probe, batch, false, 1);
    const int k = st.scratch(probe.off);
    SBLM_TRY(st.begin());
    Carver c{static_cast<char*>(st.scratch_ptr(k))};
    Net n = carve_net(c, batch, false, 1);
    const float* w = static_cast<const float*>(st.dev(i_w));
    SBLM_CUDA(launch_cast(w, n.wb, n.wbt, s));
    SBLM_CUDA(launch_input(static_cast<const float*>(st.dev(i_x)), n, s));
    SBLM_CUDA(net_forward(n, w, s));
    SBLM_CUDA(cudaMemcpyAsync(st.dev(i_o), n.out, sizeof(float) * (size_t)batch * 12, cudaMemcpyDeviceToDevice, s));
    SBLM_TRY(check_timeout(s));
    return st.end();
}

sblm_status sblm_cnn_loss_grad(const float* weights, const float* x, const float* y, int32_t batch, double* loss,
                               float* grad, void* stream) {
    if (batch < 1 || batch > kMaxBatch) return fail(SBLM_EINVAL, "batch must be in [1, %d]", kMaxBatch);
    if (!weights || !x || !y || !loss || !grad) return fail(SBLM_EINVAL, "NULL buffer");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CallLock lock;
    Staging st(s);
    int i_w, i_x, i_y, i_l, i_g;
    SBLM_TRY(st.arg(weights, sizeof(float) * kNParams, true, false, &i_w));
    SBLM_TRY(st.arg(x, sizeof(float) * (size_t)batch * 2 * kBins, true, false, &i_x));
    SBLM_TRY(st.arg(y, sizeof(float) * (size_t)batch * 6, true, false, &i_y));
    SBLM_TRY(st.arg(loss, sizeof(double), false, true, &i_l));
    SBLM_TRY(st.arg(grad, sizeof(float) * kNParams, false, true, &i_g));
    const int sms = sm_count();
    Carver probe{nullptr};
    carve_net(probe, batch, true, sms);
    const int k = st.scratch(probe.off);
    SBLM_TRY(st.begin());
    Carver c{static_cast<char*>(st.scratch_ptr(k))};
    Net n = carve_net(c, batch, true, sms);
    float* w = static_cast<float*>(st.dev(i_w));
    SBLM_CUDA(launch_cast(w, n.wb, n.wbt, s));
    SBLM_CUDA(launch_input(static_cast<const float*>(st.dev(i_x)), n, s));
    SBLM_CUDA(net_forward(n, w, s));
    SBLM_CUDA(launch_loss(n.out, static_cast<const float*>(st.dev(i_y)), batch, n.dout, n.loss_part,
                          static_cast<double*>(st.dev(i_l)), nullptr, nullptr, s));
    SBLM_CUDA(net_backward(n, s));
    AdamArgs off{};
    update_kernel<<<kUpdBlocks, kUpdThreads, 0, s>>>(part_tab(n), nullptr, static_cast<float*>(st.dev(i_g)), off, w,
                                                      nullptr, nullptr);
    SBLM_CUDA(cudaGetLastError());
    SBLM_TRY(check_timeout(s));
    return st.end();
}

sblm_status sblm_cnn_adamw(float* weights, float* adam_state, const float* grad, const sblm_cnn_train_params* p,
                           int64_t t, void* stream) {
    SBLM_TRY(check_train_params(p));
    if (t < 1) return fail(SBLM_EINVAL, "t must be >= 1");
    if (!weights || !adam_state || !grad) return fail(SBLM_EINVAL, "NULL buffer");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CallLock lock;
    Staging st(s);
    int i_w, i_a, i_g;
    SBLM_TRY(st.arg(weights, sizeof(float) * kNParams, true, true, &i_w));
    SBLM_TRY(st.arg(adam_state, sizeof(float) * 2 * kNParams, true, true, &i_a));
    SBLM_TRY(st.arg(grad, sizeof(float) * kNParams, true, false, &i_g));
    SBLM_TRY(st.begin());
    update_kernel<<<kUpdBlocks, kUpdThreads, 0, s>>>(
        PartTab{}, static_cast<const float*>(st.dev(i_g)), nullptr,
        adam_args(p, static_cast<float*>(st.dev(i_a)), t, nullptr), static_cast<float*>(st.dev(i_w)), nullptr, nullptr);
    SBLM_CUDA(cudaGetLastError());
    return st.end();
}

sblm_status sblm_cnn_train(float* weights, float* adam_state, const sblm_cnn_train_params* p, int64_t first_step,
                           int32_t n_run, float* loss_history, void* stream) {
    SBLM_TRY(check_train_params(p));
    if (first_step < 0 || n_run < 0) return fail(SBLM_EINVAL, "first_step and n_run must be >= 0");
    if (!weights || !adam_state) return fail(SBLM_EINVAL, "weights and adam_state are required");
    if (n_run == 0) return SBLM_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CallLock lock;
    Staging st(s);
    int i_w, i_a, i_h;
    SBLM_TRY(st.arg(weights, sizeof(float) * kNParams, true, true, &i_w));
    SBLM_TRY(st.arg(adam_state, sizeof(float) * 2 * kNParams, true, true, &i_a));
    SBLM_TRY(st.arg(loss_history, loss_history ? sizeof(float) * (size_t)n_run : 0, false, true, &i_h));
    const int B = p->batch, sms = sm_count();
    const size_t nx = (size_t)B * kInputRow * 2, ny = (size_t)B * 6;
    Carver probe{nullptr};
    carve_net(probe, B, true, sms, false);
    carve_gen(probe, B, p->precision, true);
    probe.take<__nv_bfloat16>(2 * nx);
    probe.take<float>(2 * ny);
    probe.take<double>(3);
    const int k = st.scratch(probe.off);
    SBLM_TRY(st.begin());
    Carver c{static_cast<char*>(st.scratch_ptr(k))};
    Net n = carve_net(c, B, true, sms, false);
    Gen g = carve_gen(c, B, p->precision, true);
    __nv_bfloat16* x = c.take<__nv_bfloat16>(2 * nx);  // two batches: the one in training and the next one
    float* y = c.take<float>(2 * ny);
    double* scalars = c.take<double>(3);
    float* w = static_cast<float*>(st.dev(i_w));
    float* state = static_cast<float*>(st.dev(i_a));
    float* hist = static_cast<float*>(st.dev(i_h));
    SideStream* side = nullptr;
    SBLM_TRY(side_stream(&side));
    set_counter_kernel<<<1, 1, 0, s>>>(g.ctr, first_step, first_step);
    grid_kernel<<<1, kBins, 0, s>>>(g.grid);
    SBLM_CUDA(launch_cast(w, n.wb, n.wbt, s));
    const AdamArgs ad = adam_args(p, state, 0, scalars);
    const PartTab tab = part_tab(n);
    auto generate = [&](cudaStream_t q, int buf) -> cudaError_t {
        CNN_TRY(launch_gen(g, B, p->precision, p->forced_frac, p->seed, nullptr, x + buf * nx, y + buf * ny, q));
        advance_kernel<<<1, 1, 0, q>>>(g.ctr + 2);
        return cudaGetLastError();
    };
    // One step on batch `buf`. The next batch does not depend on the weights: with `more` it is drawn into the
    // other buffer beside the network's products (the generator keeps the FP32 and FP64 pipes busy, the
    // products wait on memory): a step of batch 1024 takes 0.55 ms, 0.64 ms one after the other.
    auto step = [&](cudaStream_t q, int buf, bool more) -> cudaError_t {
        CNN_TRY(cudaEventRecord(side->fork, q));
        CNN_TRY(cudaStreamWaitEvent(side->stream, side->fork, 0));
        adam_scalars_kernel<<<1, 32, 0, side->stream>>>(ad, g.ctr, scalars);
        CNN_TRY(cudaGetLastError());
        if (more) CNN_TRY(generate(side->stream, buf ^ 1));
        CNN_TRY(cudaEventRecord(side->join, side->stream));
        Net nb = n;
        nb.xb = x + buf * nx;
        CNN_TRY(net_forward(nb, w, q));
        CNN_TRY(launch_loss(nb.out, y + buf * ny, B, nb.dout, nb.loss_part, nullptr, hist, g.ctr, q));
        CNN_TRY(net_backward(nb, q));
        CNN_TRY(cudaStreamWaitEvent(q, side->join, 0));
        update_kernel<<<kUpdBlocks, kUpdThreads, 0, q>>>(tab, nullptr, nullptr, ad, w, n.wb, n.wbt);
        CNN_TRY(cudaGetLastError());
        advance_kernel<<<1, 1, 0, q>>>(g.ctr);
        return cudaGetLastError();
    };
    std::vector<unsigned char> key;
    const char tag[] = "cnn_train";
    key.insert(key.end(), tag, tag + sizeof tag);
    put(key, B);
    put(key, p->precision);
    put(key, p->forced_frac);
    put(key, p->seed);
    put(key, p->lr);
    put(key, p->beta1);
    put(key, p->beta2);
    put(key, p->eps);
    put(key, p->weight_decay);
    put(key, p->n_steps);
    put(key, p->warmup);
    put(key, st.scratch_ptr(k));
    put(key, w);
    put(key, state);
    put(key, hist);
    int dev = 0;
    SBLM_CUDA(cudaGetDevice(&dev));
    put(key, dev);
    // two steps (both buffers) per graph while a later step needs the second one's batch, the rest directly
    auto pair = [&](cudaStream_t q) -> cudaError_t {
        CNN_TRY(step(q, 0, true));
        return step(q, 1, true);
    };
    SBLM_CUDA(generate(s, 0));
    int left = n_run;
    for (; left >= 3; left -= 2) SBLM_TRY(run_cached_graph(key, pair, s));
    if (left == 2) SBLM_CUDA(step(s, 0, true));
    SBLM_CUDA(step(s, left == 2 ? 1 : 0, false));
    SBLM_TRY(check_timeout(s));
    return st.end();
}

sblm_status sblm_cnn_propose(const float* out, const double* window, int32_t n_lc, const sblm_bounds* bounds,
                             int32_t n_seed, uint64_t seed, double* genes, void* stream) {
    if (n_lc < 1 || n_seed < 0) return fail(SBLM_EINVAL, "n_lc must be >= 1 and n_seed >= 0");
    if (!out || !window || (n_seed > 0 && !genes)) return fail(SBLM_EINVAL, "NULL buffer");
    Bounds b;
    SBLM_TRY(check_bounds(bounds, &b));
    if (n_seed == 0) return SBLM_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CallLock lock;
    Staging st(s);
    int i_o, i_w, i_g;
    SBLM_TRY(st.arg(out, sizeof(float) * 12 * (size_t)n_lc, true, false, &i_o));
    SBLM_TRY(st.arg(window, sizeof(double) * 2 * (size_t)n_lc, true, false, &i_w));
    SBLM_TRY(st.arg(genes, sizeof(double) * 6 * (size_t)n_lc * n_seed, false, true, &i_g));
    SBLM_TRY(st.begin());
    const long long total = (long long)n_lc * n_seed;
    propose_kernel<<<(unsigned)((total + 127) / 128), 128, 0, s>>>(
        static_cast<const float*>(st.dev(i_o)), static_cast<const double*>(st.dev(i_w)), n_lc, b, n_seed, seed,
        static_cast<double*>(st.dev(i_g)));
    SBLM_CUDA(cudaGetLastError());
    return st.end();
}

}  // extern "C"
