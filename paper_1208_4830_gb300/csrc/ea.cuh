// ea.cuh -- device side of the evolutionary algorithm of Appendix A (Rajpaul 2012).
//
// Random numbers: Philox4x64-10 with key (seed, stream id) and counter
// (generation, operator, index, sub-index); see common.cuh for the draw conventions.
// Offspring arithmetic uses explicitly rounded operations (no fused multiply-add) so that the
// same draws give bit-identical genes on every implementation that evaluates the same
// expressions in IEEE double.
#pragma once

#include <cuda_runtime.h>

#include "../../include/sblm.h"
#include "common.cuh"

namespace sblm {

constexpr int kMaxPop = 8192;          // largest N_pop of the single-block ranking
constexpr int kInitIndexBits = 20;     // element index in the low bits of the init sort keys
constexpr double kLnEps = -36.04365338911715;  // ln(2^-52), FP64 machine epsilon
constexpr double kPMutMax = 0.5;

struct EAConst {
    int n_pop, n_par, n_tourn, stag_window, restart_after;
    double p_mut0, stag_rel;
    uint64_t seed, stream;
};

struct EACtrl {
    double p_mut_used;  // jump probability of this generation's offspring
    int restart;        // 1: the next population is a fresh initialisation
    int pad;
};

// Appendix A, "Initialisation": sort key of element e (top 44 bits of a Philox word, index in
// the low bits, so that all keys differ).
__device__ __forceinline__ uint64_t init_key(const EAConst& c, uint64_t gen, uint64_t e) {
    const uint64_t w = philox4x64(gen, OP_INIT_PERM, e, 0, c.seed, c.stream).x[0];
    return ((w >> kInitIndexBits) << kInitIndexBits) | e;
}

// Value of the element whose key has rank `pos`: pairs (2k, 2k+1) of the sorted order get
// X_k and 1 - X_k; an odd leftover gets a plain draw.
__device__ __forceinline__ double init_value(const EAConst& c, uint64_t gen, uint64_t pos, uint64_t m) {
    const uint64_t n_pairs = m / 2;
    const uint64_t k = pos < 2 * n_pairs ? pos / 2 : n_pairs;
    const double x = u01(philox4x64(gen, OP_INIT_U, k, 0, c.seed, c.stream).x[0]);
    return (pos < 2 * n_pairs && (pos & 1)) ? __dsub_rn(1.0, x) : x;
}

// Appendix A, "Selection": parent rank = min of n_tourn uniform draws from {0..N_pop-1}, the draws
// shared by the L lanes of an aligned group (all lanes of the warp call it). The integer draw is
// monotonic in the word's top 32 bits, so their minimum gives the smallest draw.
template <int L>
__device__ __forceinline__ int tournament(const EAConst& c, uint64_t gen, uint64_t slot, int lane) {
    uint32_t best = 0xffffffffu;
    for (int b = lane; 4 * b < c.n_tourn; b += L) {
        const u64x4 w = philox4x64(gen, OP_SELECT, slot, (uint64_t)b, c.seed, c.stream);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (4 * b + j < c.n_tourn) best = min(best, (uint32_t)(w.x[j] >> 32));
    }
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
    return (int)uniform_int((uint64_t)best << 32, (uint32_t)c.n_pop);
}

// the draw u01(x) < p as an integer comparison: (x >> 11) < ceil(p 2^53)
__device__ __forceinline__ uint64_t jump_threshold(double p_mut) { return (uint64_t)ceil(p_mut * 0x1.0p53); }

// v clamped to [0, 1] by its bits (NaN and -0 become 0, as fmin(fmax(v, 0), 1) gives)
__device__ __forceinline__ double clamp_unit(double v) {
    const long long b = __double_as_longlong(v);
    if (b < 0 || b > 0x7ff0000000000000ll) return 0.0;
    return b > 0x3ff0000000000000ll ? 1.0 : v;
}

// Appendix A, "Creep and jump mutation" of gene j of population row `row`. The FP64 pipe takes a warp
// instruction per 64 cycles and bounds the offspring kernel with the draws, so both creep directions
// share their operations, and the clamp and the jump test run on the integer pipe.
__device__ __forceinline__ double mutate_gene(const EAConst& c, uint64_t gen, uint64_t row, uint64_t j, double p,
                                              uint64_t p_jump) {
    const u64x4 w = philox4x64(gen, OP_MUT, row, j, c.seed, c.stream);
    const double X = exp(__dmul_rn(kLnEps, u01(w.x[0])));
    const bool up = top_bit(w.x[1]);
    const double step = __dmul_rn(up ? __dsub_rn(1.0, p) : p, X);
    const double v = __dadd_rn(p, up ? step : -step);
    return (w.x[2] >> 11) < p_jump ? u01(w.x[3]) : clamp_unit(v);
}

// Appendix A, "Stagnation checks", applied by one thread after the ranking of generation t.
// Returns 1 when the next population must be re-initialised.
__device__ __forceinline__ int stagnation_update(sblm_ea_state& s, const EAConst& c, double best) {
    const int W = c.stag_window;
    if (s.n_hist == W + 1) {
        for (int i = 0; i < W; ++i) s.hist[i] = s.hist[i + 1];
        s.n_hist = W;
    }
    s.hist[s.n_hist++] = best;
    bool stagnant = false;
    if (s.n_hist == W + 1) {
        const double old = s.hist[0];
        stagnant = isfinite(old) && (__dsub_rn(old, best) <= __dmul_rn(c.stag_rel, old));
    }
    const double p_min = 1.0 / (double)(c.n_pop * c.n_par);
    if (stagnant) {
        s.p_mut = fmin(__dmul_rn(s.p_mut, 1.5), kPMutMax);
        s.stag_run += 1;
    } else {
        s.p_mut = fmax(__dmul_rn(s.p_mut, 0.5), p_min);
        s.stag_run = 0;
    }
    if (s.stag_run >= c.restart_after) {
        s.p_mut = c.p_mut0;
        s.n_hist = 0;
        s.stag_run = 0;
        s.n_restarts += 1;
        return 1;
    }
    return 0;
}

// ---------------------------------------------------------------------------------------------
// Block-level building blocks, shared by the single-population kernels and the persistent
// batched fitter. Every thread of the calling block must call them (they hold barriers).
// ---------------------------------------------------------------------------------------------

// fitness as an unsigned integer in the same order (NaN as +inf, -0 as 0), and back
__device__ __forceinline__ uint64_t order_key(double v) {
    uint64_t b = (uint64_t)__double_as_longlong(v);
    if ((b << 1) > 0xffe0000000000000ull) b = 0x7ff0000000000000ull;
    if ((b << 1) == 0) b = 0;
    return (b >> 63) ? ~b : b | 0x8000000000000000ull;
}
__device__ __forceinline__ double order_value(uint64_t k) {
    return __longlong_as_double((long long)((k >> 63) ? k & 0x7fffffffffffffffull : ~k));
}
__device__ __forceinline__ bool pair_less(uint64_t ka, int ia, uint64_t kb, int ib) {
    return ka < kb || (ka == kb && ia < ib);
}

// Ascending bitonic sort of n = E T (key, index) pairs by the block's first T threads (T a power of two,
// 32 <= T <= blockDim.x), thread t holding elements t E .. t E + E - 1. Strides below E stay in
// registers, strides below 32 E are warp shuffles, and only the longer ones go through shared memory
// (bkey, bidx: n each, element e of thread t at e T + t, so consecutive threads touch consecutive
// words). Every thread of the block calls it. Keys are integers: a comparison of doubles would run on
// the FP64 pipe. Ranking 32 populations of 4096 (a block each): 175 us with every stage on doubles in
// shared memory behind a barrier (78 stages), 41 us with 15 such stages on integers.
template <int E>
__device__ __forceinline__ void block_sort(uint64_t (&key)[E], int (&idx)[E], int T, uint64_t* bkey, int* bidx) {
    const int t = threadIdx.x, n = E * T;
    for (int k = 2; k <= n; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= 32 * E) {
                const int x = j / E;
                if (t < T) {
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        bkey[e * T + t] = key[e];
                        bidx[e * T + t] = idx[e];
                    }
                }
                __syncthreads();
                if (t < T) {
                    const bool low = !(t & x);
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const uint64_t ok = bkey[e * T + (t ^ x)];
                        const int oi = bidx[e * T + (t ^ x)];
                        const bool up = ((t * E + e) & k) == 0;
                        if (pair_less(ok, oi, key[e], idx[e]) == (up == low)) {
                            key[e] = ok;
                            idx[e] = oi;
                        }
                    }
                }
                __syncthreads();
            } else if (j >= E) {
                if (t < T) {  // whole warps
                    const int x = j / E;
                    const bool low = !(t & x);
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const uint64_t ok = __shfl_xor_sync(0xffffffffu, key[e], x);
                        const int oi = __shfl_xor_sync(0xffffffffu, idx[e], x);
                        const bool up = ((t * E + e) & k) == 0;
                        if (pair_less(ok, oi, key[e], idx[e]) == (up == low)) {
                            key[e] = ok;
                            idx[e] = oi;
                        }
                    }
                }
            } else {
#pragma unroll
                for (int jj = E / 2; jj > 0; jj >>= 1) {
                    if (jj != j) continue;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        if (e & jj) continue;
                        const bool up = ((t * E + e) & k) == 0;
                        if (pair_less(key[e + jj], idx[e + jj], key[e], idx[e]) == up) {
                            const uint64_t tk = key[e];
                            key[e] = key[e + jj];
                            key[e + jj] = tk;
                            const int ti = idx[e];
                            idx[e] = idx[e + jj];
                            idx[e + jj] = ti;
                        }
                    }
                }
            }
        }
    }
}

template <int E>
__device__ __forceinline__ void block_rank_regs(const double* chi2, int n_pop, int n2, int T, double* skey, int* sidx) {
    uint64_t key[E];
    int idx[E];
    const int t = threadIdx.x;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = t * E + e;
        const bool in = t < T && i < n_pop;
        key[e] = in ? order_key(chi2[i]) : ~0ull;
        idx[e] = in ? i : 0x7fffffff;
    }
    block_sort<E>(key, idx, T, reinterpret_cast<uint64_t*>(skey), sidx);
    if (t < T) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = t * E + e;
            if (i < n2) {
                skey[i] = i < n_pop ? order_value(key[e]) : INFINITY;
                sidx[i] = idx[e];
            }
        }
    }
    __syncthreads();
}

// (fitness, row) pairs of the population in shared memory, NaN as +inf, padded to n2 (a power
// of two) with (+inf, INT_MAX), sorted ascending (ties by row): skey and sidx hold n2 entries
__device__ __forceinline__ void block_rank(const double* __restrict__ chi2, int n_pop, int n2, double* skey,
                                           int* sidx) {
    // threads in use: the largest power of two that gives each at least one element
    int T = 32;
    while (2 * T <= (int)blockDim.x && 2 * T <= n2) T <<= 1;
    switch (max(1, n2 / T)) {
        case 1: return block_rank_regs<1>(chi2, n_pop, n2, T, skey, sidx);
        case 2: return block_rank_regs<2>(chi2, n_pop, n2, T, skey, sidx);
        case 4: return block_rank_regs<4>(chi2, n_pop, n2, T, skey, sidx);
        case 8: return block_rank_regs<8>(chi2, n_pop, n2, T, skey, sidx);
    }
    // more than eight elements per thread (small blocks of the batched fitter): all in shared memory
    uint64_t* bkey = reinterpret_cast<uint64_t*>(skey);
    for (int i = threadIdx.x; i < n2; i += blockDim.x) {
        bkey[i] = i < n_pop ? order_key(chi2[i]) : ~0ull;
        sidx[i] = i < n_pop ? i : 0x7fffffff;
    }
    __syncthreads();
    for (int k = 2; k <= n2; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < n2; i += blockDim.x) {
                const int l = i ^ j;
                if (l > i && pair_less(bkey[l], sidx[l], bkey[i], sidx[i]) == ((i & k) == 0)) {
                    const uint64_t tk = bkey[i];
                    bkey[i] = bkey[l];
                    bkey[l] = tk;
                    const int ti = sidx[i];
                    sidx[i] = sidx[l];
                    sidx[l] = ti;
                }
            }
            __syncthreads();
        }
    }
    for (int i = threadIdx.x; i < n2; i += blockDim.x) skey[i] = i < n_pop ? order_value(bkey[i]) : INFINITY;
    __syncthreads();
}

// One thread's bookkeeping after the ranking of generation `gen`: archive of the best ever,
// stagnation check. Returns 1 when the next population is a fresh initialisation; *p_used is the
// jump probability of this generation's offspring.
__device__ __forceinline__ int block_bookkeeping(const EAConst& c, int gen, double best, const double* best_row,
                                                 sblm_ea_state& s, bool produce, double* p_used) {
    if (best < s.best_chi2) {
        s.best_chi2 = best;
        for (int j = 0; j < c.n_par; ++j) s.best_genes[j] = best_row[j];
    }
    *p_used = s.p_mut;
    const int restart = produce ? stagnation_update(s, c, best) : 0;
    s.generation = gen + 1;
    return restart;
}

// Reproductive pairing k of generation `gen` (Appendix A, "Selection", "Reproduction",
// "Creep and jump mutation") by the L lanes of an aligned group (lane 0 .. L - 1; all lanes of the
// warp call it, `valid` false beyond the last pairing): two tournament parents from the ranked
// population (order[r] is the row of rank r), the weighting-matrix mode and diagonal,
// Eq. (rep1)/(rep2), then creep and jump of both children into rows 1 + 2k and 2 + 2k of P_next (the
// second dropped past N_pop). The lanes share the tournaments' draws and the genes.
template <int L>
__device__ __forceinline__ void offspring_pair(const EAConst& c, int gen, const double* __restrict__ P,
                                               const int* __restrict__ order, double p_mut, int k, int lane,
                                               bool valid, double* __restrict__ P_next) {
    const int n_par = c.n_par;
    const uint64_t g = (uint64_t)gen;
    const int ra = tournament<L>(c, g, 2 * (uint64_t)k, lane);
    const int rb = tournament<L>(c, g, 2 * (uint64_t)k + 1, lane);
    if (!valid) return;
    const double* pa = P + (size_t)order[ra] * n_par;
    const double* pb = P + (size_t)order[rb] * n_par;
    const uint32_t mode = uniform_int(philox4x64(g, OP_MODE, (uint64_t)k, 0, c.seed, c.stream).x[0], 3u);
    const uint64_t p_jump = jump_threshold(p_mut);
    const int row1 = 1 + 2 * k, row2 = 2 + 2 * k;
    for (int j = lane; j < n_par; j += L) {
        const uint64_t w = philox4x64(g, OP_F, (uint64_t)k, (uint64_t)j, c.seed, c.stream).x[0];
        const double f = mode == 0 ? u01(w) : (mode == 1 ? (double)top_bit(w) : 1.0);
        const double omf = __dsub_rn(1.0, f);
        const double a = pa[j], b = pb[j];
        const double c1 = __dadd_rn(__dmul_rn(a, f), __dmul_rn(b, omf));
        const double c2 = __dadd_rn(__dmul_rn(b, f), __dmul_rn(a, omf));
        P_next[(size_t)row1 * n_par + j] = mutate_gene(c, g, (uint64_t)row1, (uint64_t)j, c1, p_jump);
        if (row2 < c.n_pop)
            P_next[(size_t)row2 * n_par + j] = mutate_gene(c, g, (uint64_t)row2, (uint64_t)j, c2, p_jump);
    }
}

// Elements first + tid + k * step (k = 0, 1, ... while below m) of the initialisation of
// generation `gen`: each element's key is ranked against all m keys (read in tiles of `tile_n`
// through the shared array `tile`), and the rank gives its pairing and value. The trip counts are
// uniform over the block.
__device__ __forceinline__ void block_init_values(const EAConst& c, int gen, const uint64_t* __restrict__ keys,
                                                  int m, double* __restrict__ P, int first, int step,
                                                  uint64_t* tile, int tile_n) {
    for (int base = first; base < m; base += step) {
        const int e = base + threadIdx.x;
        const uint64_t mine = e < m ? keys[e] : 0;
        uint32_t pos = 0;
        for (int t0 = 0; t0 < m; t0 += tile_n) {
            const int n = min(tile_n, m - t0);
            __syncthreads();
            for (int i = threadIdx.x; i < n; i += blockDim.x) tile[i] = keys[t0 + i];
            __syncthreads();
            if (e < m)
                for (int i = 0; i < n; ++i) pos += tile[i] < mine;
        }
        if (e < m) P[e] = init_value(c, (uint64_t)gen, pos, (uint64_t)m);
        if (step >= m) break;
    }
}

__device__ __forceinline__ void state_reset(const EAConst& c, sblm_ea_state& s) {
    s.p_mut = c.p_mut0;
    s.best_chi2 = INFINITY;
    for (int i = 0; i <= SBLM_MAX_WINDOW; ++i) s.hist[i] = 0.0;
    s.n_hist = 0;
    s.stag_run = 0;
    s.n_restarts = 0;
    s.generation = 0;
    for (int j = 0; j < SBLM_MAX_NPAR; ++j) s.best_genes[j] = NAN;
}

}  // namespace sblm
