// polish_run.cuh -- one thread's run of consecutive epochs of one candidate in the amoeba's objective.
// An epoch loop apart from forward_run.cuh's: the compiler fuses the FP32 products here in
// another way at each of the kernel's call sites, and any change of the loop moves MIXED chi^2 by 1e-7,
// which a simplex amplifies. What bounds the amoeba is the chain of one chi^2 after the other; the FP64
// re-solves, each by one thread, were a third of it: 64 curves of 500 epochs, 200 evaluations, 32.0 ms with the
// general solver for each, 25.1 ms with the epoch's roots refined first (resolve_thread). FP64 solves the
// quintic of every epoch in FP64, warm from the previous epoch.
#pragma once

#include "epochs.cuh"
#include "refine.cuh"

namespace sblm {

// FP64 re-solve of one deferred epoch (MIXED), warm-started from its FP32 roots; returns the
// chi^2 term from the FP64 flux fe and weight we = 1/sigma. Out of line: an FP32 lane that must
// do it in place keeps its state on the stack instead of competing with the FP64 solver for
// registers.
static __device__ __noinline__ double resolve_fp64(const cx<float>* z32, uint32_t why, const Cand* kk,
                                                   double te, double fe, double we, double* A_row,
                                                   uint8_t* f_row, int e, bool chi2) {
    const cx<double> zeta = zeta64(*kk, te);
    double A;
    uint8_t flag = 0;
    if (!resolve_thread(z32, zeta, kk->d, kk->q, &A)) {
        cx<double> zz[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) zz[i] = mk<double>(z32[i].re, z32[i].im);
        bool w2 = true;
        const EpochOut<double> o2 = solve_epoch<double>(zeta, kk->d, kk->q, zz, w2, nullptr, kResolveCubic);
        A = o2.A;
        flag = o2.flag;
    }
    if (A_row) A_row[e] = A;
    if (f_row) f_row[e] = (uint8_t)(flag | FLAG_FP64 | why);
    if (!chi2) return 0.0;
    const double r = (fe - A) * we;
    return r * r;
}

// The thread's epochs [e0, e1) of candidate k on the staged lightcurve (all lanes of a warp run `seg`
// iterations so that MIXED can reserve queue slots warp-wide). Writes A when A_row is given.
// FP64 and FP32: returns the thread's chi^2 over its epochs, accumulated in FP64 in epoch order.
// MIXED: writes each epoch's chi^2 term to term_row, or queues the epoch (the queue has room for
// every epoch of the lightcurve), and returns 0. The branch for a full queue, the entry's unused fields
// and resolve_fp64's unused arguments stay: without them the FP32 loop is fused differently.
template <int MODE>
__device__ __forceinline__ double polish_epochs(const Cand& k, int e0, int e1, int seg, const LCView& lc, double* A_row,
                                                const DeferSink& sink, double* term_row) {
    double chi = 0.0;
    if constexpr (MODE == SBLM_FP64) {
        cx<double> z[5];
        bool warm = false;
        for (int e = e0; e < e1; ++e) {
            const double te = lc.s_t[e];
            const EpochOut<double> o = solve_epoch<double>(zeta64(k, te), k.d, k.q, z, warm);
            if (A_row) A_row[e] = o.A;
            const double fe = lc.s_f[e], we = lc.s_w[e];
            const double r = (fe - o.A) * we;
            chi += r * r;
        }
    } else {
        const float t0h = (float)k.t0, t0l = (float)(k.t0 - (double)t0h);
        const float itE = (float)k.inv_tE, sa = (float)k.sa, ca = (float)k.ca, u0 = (float)k.u0;
        const float d = (float)k.d, q = (float)k.q;
        const unsigned lane = threadIdx.x & 31u;
        cx<float> z[5];
        bool warm = false;
        for (int it = 0; it < seg; ++it) {
            const int e = e0 + it;
            bool defer = false;
            uint8_t why = 0;
            if (e < e1) {
                const float4 ep = lc.s_ep[e];
                const float tau = diff_ff(ep.x, ep.y, t0h, t0l) * itE;
                const cx<float> zeta = mk<float>(tau * sa + u0 * ca, -tau * ca + u0 * sa);
                EpochOut<float> o = solve_epoch<float>(zeta, d, q, z, warm);
                o.flag = mixed_trigger_flags(o);
                if (MODE == SBLM_MIXED) defer = o.flag != 0;
                why = o.flag;
                if (A_row) A_row[e] = o.A;
                if (!defer) {
                    const double r = (double)((ep.z - o.A) * ep.w);
                    if (MODE == SBLM_MIXED)
                        term_row[e] = r * r;
                    else
                        chi += r * r;
                }
            }
            if constexpr (MODE == SBLM_MIXED) {
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
                            qd.c = 0;
                            qd.e = e;
                            qd.why = why;
                        } else {  // queue full (its size rules that out)
                            const double te = lc.t[e];
                            const double fe = lc.flux[e], we = 1.0 / lc.sigma[e];
                            cx<float> zc[5];  // a copy, so that z's address is never taken and z stays in registers
#pragma unroll
                            for (int i = 0; i < 5; ++i) zc[i] = z[i];
                            term_row[e] = resolve_fp64(zc, why, &k, te, fe, we, A_row, nullptr, e, true);
                        }
                    }
                }
            }
        }
    }
    return chi;
}

}  // namespace sblm
