// forward_run.cuh -- one thread's run of consecutive epochs of one candidate: the unit of work
// that the population-wide forward kernel and the persistent batched fitter share.
#pragma once

#include "epochs.cuh"
#include "refine.cuh"

namespace sblm {

// Decode the block's candidates c0 .. c0 + n - 1 (those below n_cand) into shared memory, one thread
// each, and into `out` (when given) for the re-solve; the caller's next barrier publishes them. The
// decode's exp10, sincos and division are about 120 instructions of the FP64 pipe, which takes them
// at the same rate from a warp with one active lane as from a full one, so a block's candidates
// share one or a few warps instead of every warp decoding its own.
template <bool FROM_GENES>
__device__ __forceinline__ void decode_candidates(const double* __restrict__ src, const Bounds& b, int c0, int n,
                                                  int n_cand, Cand* s_cand, Cand* out) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        Cand k{};
        if (c0 + i < n_cand) {
            k = candidate<FROM_GENES>(src, b, c0 + i);
            if (out) out[c0 + i] = k;
        }
        s_cand[i] = k;
    }
}

// General FP64 solve of one epoch, warm-started from its FP32 roots: what resolve_group leaves open.
// Out of line: a lane that must do it in place keeps its state on the stack instead of competing
// with the FP64 solver for registers.
static __device__ __noinline__ double solve_general(const cx<float>* z32, const Cand* kk, double te, uint8_t* flag) {
    cx<double> zz[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) zz[i] = mk<double>(z32[i].re, z32[i].im);
    bool w2 = true;
    const EpochOut<double> o2 = solve_epoch<double>(zeta64(*kk, te), kk->d, kk->q, zz, w2, nullptr, kResolveCubic);
    *flag = o2.flag;
    return o2.A;
}

// An FP64 re-solve's results: magnification and flags when the row pointers are given (MIXED: the
// FP64 bit and the triggers beside the solver's own flags); returns the chi^2 term from the FP64
// flux fe and weight we = 1/sigma.
template <int MODE>
__device__ __forceinline__ double store_resolved(double A, uint8_t flag, uint32_t why, double fe, double we,
                                                 double* A_row, uint8_t* f_row, int e) {
    if (A_row) A_row[e] = A;
    if (f_row) f_row[e] = MODE == SBLM_MIXED ? (uint8_t)(flag | FLAG_FP64 | why) : flag;
    const double r = (fe - A) * we;
    return r * r;
}

// One warp's share of the queued epochs [0, n): groups of five lanes take them six at a time, warp
// `w` of `n_w` starting at epoch 6 w. What the groups leave open is collected, a lane per epoch, and takes
// the general solver when the warp's lanes are nearly all taken, and at the end: FP64 instructions cost the same
// for one lane as for 32, and lenses outside the refined range leave every epoch open. MIXED chi^2 of 4096 x
// 2000 at q < 5e-5, d > 10, d < 0.25: 4.24, 4.75, 15.7 ms with the solver in place on the lanes r = 0, 2.97, 2.66,
// 9.0 to 9.5 ms so; an FP64 batch at q < 1e-4 (152 curves, 128 x 6 generations): 635, 371 ms. `cand(c)` is candidate c, `data(c, e)` the epoch's time, flux and
// 1/sigma, and `store(c, e, A, flag, why, fe, we)` takes the result (one lane per epoch). Every lane
// of the warp calls it.
struct EpochData {
    double t, flux, w;
};
template <class CandFn, class DataFn, class StoreFn>
__device__ __forceinline__ void resolve_queue(const Deferred* __restrict__ queue, unsigned n, unsigned w, unsigned n_w,
                                              CandFn cand, DataFn data, StoreFn store) {
    const int lane = threadIdx.x & 31, grp = lane / kResolveLanes, r = lane - grp * kResolveLanes;
    int pending = 0;    // epochs left open; lane l < pending holds the queue index of one
    unsigned mine = 0;
    for (unsigned first = w * kResolvePerWarp;; first += n_w * kResolvePerWarp) {
        const bool more = first < n;
        if (more) {
            const unsigned i = first + grp;
            const bool valid = grp < kResolvePerWarp && i < n;
            const Deferred& q = queue[valid ? i : first];
            const int c = q.c, e = q.e;
            const Cand k = cand(c);
            const EpochData ed = data(c, e);
            double A;
            const bool done = resolve_group(q.z[r], valid, zeta64(k, ed.t), k.d, k.q, &A);
            if (valid && r == 0 && done) store(c, e, A, (uint8_t)0, q.why, ed.flux, ed.w);
            const unsigned open = __ballot_sync(0xffffffffu, valid && r == 0 && !done);
#pragma unroll
            for (int g = 0; g < kResolvePerWarp; ++g) {
                if (!(open >> (g * kResolveLanes) & 1u)) continue;
                if (lane == pending) mine = first + g;
                ++pending;
            }
        }
        if (more ? pending > 32 - kResolvePerWarp : pending > 0) {
            if (lane < pending) {
                const Deferred& q = queue[mine];
                const Cand k = cand(q.c);
                const EpochData ed = data(q.c, q.e);
                uint8_t flag;
                const double A = solve_general(q.z, &k, ed.t, &flag);
                store(q.c, q.e, A, flag, q.why, ed.flux, ed.w);
            }
            pending = 0;
            __syncwarp();
        }
        if (!more) break;
    }
}

// The same with the general solver, a lane per epoch: lane `first` takes epochs first, first + step, ...
template <class CandFn, class DataFn, class StoreFn>
__device__ __forceinline__ void resolve_queue_lanes(const Deferred* __restrict__ queue, unsigned n, unsigned first,
                                                    unsigned step, CandFn cand, DataFn data, StoreFn store) {
    for (unsigned i = first; i < n; i += step) {
        const Deferred& q = queue[i];
        const Cand k = cand(q.c);
        const EpochData ed = data(q.c, q.e);
        uint8_t flag;
        const double A = solve_general(q.z, &k, ed.t, &flag);
        store(q.c, q.e, A, flag, q.why, ed.flux, ed.w);
    }
}

// The thread's epochs [e0, e1) of candidate k (all lanes of a warp run `seg` iterations so that
// queue slots can be reserved warp-wide). Writes A and flags when the row pointers are given.
// FP32: returns the thread's chi^2 over its epochs, accumulated in FP64 in epoch order. MIXED and
// FP64: writes each epoch's chi^2 term to term_row (CHI2) and returns 0; `c_tag` is the candidate
// index recorded in its queue entries.
// FP64 solves the quintic in FP32 too: its roots tell images from spurious ones unless a trigger
// (refine_trigger, wider than MIXED's) sends the epoch to the re-solve, and the images are refined in
// FP64 (refine_images). 32 epochs of three images cost a warp about 200 FP64 instructions instead of
// some 6000 of an FP64 root iteration over the union of its lanes' sweeps.
template <int MODE, bool CHI2, bool STAGED>
__device__ __forceinline__ double eval_run(const Cand& k, bool valid, int c_tag, int e0, int e1, int seg,
                                           const LCView& lc, double* A_row, uint8_t* f_row, const DeferSink& sink,
                                           double* term_row) {
    double chi = 0.0;
    const float t0h = (float)k.t0, t0l = (float)(k.t0 - (double)t0h);
    const float itE = (float)k.inv_tE, sa = (float)k.sa, ca = (float)k.ca, u0 = (float)k.u0;
    const float d = (float)k.d, q = (float)k.q;
    const unsigned lane = threadIdx.x & 31u;
    const bool refined = MODE == SBLM_FP64 && refine_lens(d, q);
    cx<float> z[5];
    bool warm = false;
    for (int it = 0; it < seg; ++it) {
        const int e = e0 + it;
        const bool act = valid && e < e1;
        bool defer = false;
        uint8_t why = 0;
        if constexpr (MODE == SBLM_FP64) {
            if (act) {
                const double te = STAGED ? lc.s_t[e] : lc.t[e];
                const cx<double> zd = zeta64(k, te);
                const cx<float> zeta = mk<float>((float)zd.re, (float)zd.im);
                Root<float> rp[5];
                unsigned images = 0;
                EpochOut<float> o =
                    solve_epoch<float>(zeta, d, q, z, warm, nullptr, Tol<float>::cubic, rp, &images);
                double A = 0.0;
                defer = refine_trigger(o) || !refined || !refine_source(zeta, d);
                if (!defer) defer = !refine_images(rp, images, zd, k.d, k.q, &A);
                if (!defer) {
                    if (A_row) A_row[e] = A;
                    if (f_row) f_row[e] = 0;
                    if (CHI2) {
                        const double fe = STAGED ? lc.s_f[e] : lc.flux[e];
                        const double we = STAGED ? lc.s_w[e] : 1.0 / lc.sigma[e];
                        const double r = (fe - A) * we;
                        term_row[e] = r * r;
                    }
                }
            }
        } else if (act) {
            float4 ep;
            if (STAGED) {
                ep = lc.s_ep[e];
            } else {
                const double te = lc.t[e];
                const float th = (float)te;
                ep = make_float4(th, (float)(te - (double)th), CHI2 ? (float)lc.flux[e] : 0.f,
                                 CHI2 ? (float)(1.0 / lc.sigma[e]) : 0.f);
            }
            const float tau = diff_ff(ep.x, ep.y, t0h, t0l) * itE;
            const cx<float> zeta = mk<float>(tau * sa + u0 * ca, -tau * ca + u0 * sa);
            EpochOut<float> o = solve_epoch<float>(zeta, d, q, z, warm);
            o.flag = mixed_trigger_flags(o);
            if (MODE == SBLM_MIXED) defer = o.flag != 0;
            why = o.flag;
            if (A_row) A_row[e] = o.A;
            if (f_row) f_row[e] = o.flag;
            if (CHI2 && !defer) {
                const double r = (double)((ep.z - o.A) * ep.w);
                if (MODE == SBLM_MIXED)
                    term_row[e] = r * r;
                else
                    chi += r * r;
            }
        }
        if constexpr (MODE != SBLM_FP32) {
            // one atomic per warp reserves queue slots for the lanes that defer
            const unsigned b = __ballot_sync(0xffffffffu, defer);
            if (b) {
                const int leader = __ffs(b) - 1;
                unsigned base = 0;
                if ((int)lane == leader) base = atomicAdd(sink.queue_count, (unsigned)__popc(b));
                base = __shfl_sync(0xffffffffu, base, leader);
                if (defer) {
                    const unsigned slot = base + (unsigned)__popc(b & ((1u << lane) - 1u));
                    if (slot < sink.queue_cap) {
                        Deferred& qd = sink.queue[slot];
#pragma unroll
                        for (int i = 0; i < 5; ++i) qd.z[i] = z[i];
                        qd.c = c_tag;
                        qd.e = e;
                        qd.why = why;
                    } else {  // queue full: re-solve here, from the FP64 data
                        const double te = lc.t[e];
                        cx<float> zc[5];  // a copy, so that z's address is never taken and z stays in registers
#pragma unroll
                        for (int i = 0; i < 5; ++i) zc[i] = z[i];
                        uint8_t flag;
                        const double A = solve_general(zc, &k, te, &flag);
                        const double fe = CHI2 ? lc.flux[e] : 0.0, we = CHI2 ? 1.0 / lc.sigma[e] : 0.0;
                        const double tm = store_resolved<MODE>(A, flag, why, fe, we, A_row, f_row, e);
                        if (CHI2) term_row[e] = tm;
                    }
                }
            }
        }
    }
    return chi;
}

// MIXED and FP64: sum of a candidate's term row over the lanes of its group of G threads (G a power of two
// <= 32, groups aligned within the warp): lane g adds epochs g, g + G, ... in order, then a fixed
// butterfly combines the lanes; every lane of the group gets the sum. All lanes of the warp call it.
__device__ __forceinline__ double term_row_sum(const double* __restrict__ row, int n_ep, int g, int G, bool valid) {
    double s = 0.0;
    for (int e = g; valid && e < n_ep; e += G) s += row[e];
    for (int off = G / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    return s;
}

}  // namespace sblm
