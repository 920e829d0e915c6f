// cnn_gemm.cuh -- the proposal network's dense contractions on the 5th-generation tensor cores.
//
// One tile kernel computes C[M, N] = sum_k A(m, k) B(k, n) with BF16 operands and FP32
// accumulators held in tensor memory: tcgen05.mma (kind::f16, M = 128, N = 64, K = 16 per
// instruction) issued by one thread, operands read by the tensor core from shared memory through
// matrix descriptors, results brought back with tcgen05.ld for the epilogue. Loader functors map
// (row, column) of an operand to 8 consecutive BF16 values along its contiguous dimension, so the
// convolution's im2col and its adjoint are never materialised: the loader gathers the rows
// straight from the activations. K-major operands serve the forward and input-gradient products,
// MN-major operands (the instruction descriptor's MN-major bit) the weight-gradient products,
// reductions over batch x position split over K with one FP32 partial per split so the reduction
// order is fixed.
//
// Tiles are rows of 128 bytes (64 values along the contiguous dimension: K-major a row of M or N with 64
// k, MN-major a k with 64 of M or N) in the 128-byte swizzle: 16-byte chunk c of row r at chunk
// c ^ (r & 7). Eight lanes copy one row, so a warp touches four whole 128-byte lines: 40 bytes a clock and
// SM, against 16 for the 16-byte core-matrix columns of the no-swizzle layout, whose gather took one
// lane a clock and bounded every product (770 cycles per 12 KB, with tcgen05.mma at 160 cycles). The
// products of a training step of batch 1024 took 0.61 ms so (K-steps of 32 behind block-wide barriers,
// two tiles ahead through registers, integer divisions in the loaders), 0.32 ms now.
//
// The warps have roles, so that no K-step holds a block-wide barrier: warps 0-7 fill a ring of K-tiles
// (cp.async, zero fill outside the operand, arriving on the stage's `full` barrier when it lands), one
// thread of warp 8 waits for a full stage, makes it visible to the tensor core and issues its
// MMAs, and tcgen05.commit arrives on the stage's `empty` barrier. Warps 0-7 then run the epilogue.
// Positions per sample are powers of two, so rows split by shifts.
// Every wait is bounded; a wait that gives up sets g_tc_timeout, which the host reads after the call.
// After a give-up the thread leaves its loop (the waits that depend on it run out as well), the block
// takes one decision (__syncthreads_and) before the epilogue, skips it, and waits for the MMAs already
// issued (one more commit on a drain barrier) before it frees its tensor memory.
// The accumulators leave tensor memory through a shared-memory staging tile, so that half a warp's
// epilogue covers one whole 64-column row (coalesced). Epilogue functors receive four adjacent columns
// (m, n .. n + 3) per call.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

namespace sblm {
namespace cnn {

constexpr int BM = 128, BN = 64, BK = 64;
constexpr int kProducers = 256;    // warps 0-7 fill the ring and run the epilogue: warp w reads
                                   // accumulator rows 32 (w % 4) .. + 31, columns 32 (w / 4) .. + 31
constexpr int kGemmThreads = 288;  // warp 8 issues the MMAs
// K-tiles in the ring: three leave room for three blocks per SM, which overlap one another's
// epilogues; eight keep enough copies in flight where a product has one block per SM and many K-steps
// (weight gradients, the wide dense layer)
constexpr int kShallow = 3, kDeep = 8;
constexpr uint32_t kTileA = BM * BK * 2, kTileB = BN * BK * 2;
constexpr int kEpiLd = BN + 4;  // padded row of the accumulator staging tile (floats)
// dynamic shared memory: the ring (the epilogue's staging tile reuses it) and room to align it to 1 KB
constexpr size_t gemm_smem(int stages) { return (size_t)stages * (kTileA + kTileB) + 1024; }
static_assert(gemm_smem(kShallow) - 1024 >= sizeof(float) * BM * kEpiLd, "the staging tile fits the ring");
constexpr uint32_t kTmemCols = 64;                                 // FP32 accumulator columns (= BN)
constexpr int kWaitLimit = 1 << 24;

__device__ int g_tc_timeout;

__device__ __forceinline__ uint32_t pack_bf2(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ uint4 pack8(const float* v) {
    return make_uint4(pack_bf2(v[0], v[1]), pack_bf2(v[2], v[3]), pack_bf2(v[4], v[5]), pack_bf2(v[6], v[7]));
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// shared-memory matrix descriptor, 128-byte swizzle: start address, leading-dimension byte offset
// (MN-major: between blocks of 64 along M or N; not used K-major), stride-dimension byte offset (between
// groups of 8 rows), descriptor version 1, swizzle mode 2
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// instruction descriptor of kind::f16: FP32 accumulator (bits 4-5), BF16 A and B (bits 7-9,
// 10-12), A and B MN-major flags (bits 15, 16), N / 8 at bits 17-22, M / 16 at bits 24-28
__host__ __device__ constexpr uint32_t idesc_f16(bool a_mn, bool b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
           ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity, int limit = kWaitLimit) {
    for (int it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(addr), "r"(parity)
            : "memory");
        if (done) return true;
    }
    atomicExch(&g_tc_timeout, 1);
    return false;
}

// 16 bytes global -> shared, asynchronous; a null source fills with zeros
__device__ __forceinline__ void copy16(uint32_t dst, const void* src, const void* any) {
    const int n = src ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src ? src : any), "r"(n) : "memory");
}

__device__ __forceinline__ void copy4(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

struct InputCols;

// One tile of ROWS (M or N) x BK into the stage's tile at s, `kc` (a multiple of 16) of its BK along K in
// use. K-major: row r of ROWS at 128 r. MN-major: for each block of 64 along M or N, row k at 128 k.
// Loaders of aligned BF16 data give addresses (asynchronous copies), the others values.
template <bool KMAJ, int ROWS, class L>
__device__ __forceinline__ void tile_load(const L& ld, int mn0, int k0, int kc, unsigned char* s) {
    if constexpr (std::is_same<L, InputCols>::value) {
        // rows of ten values, five 4-byte copies each; the rest of the tile was written once (input_tile_init)
        constexpr int rows = KMAJ ? ROWS : BK;
        for (int v = threadIdx.x; v < 5 * rows; v += kProducers) {
            const int r = v / 5, e = v - 5 * r;
            const void* src = ld.src((KMAJ ? mn0 : k0) + r, e);
            if (src && (KMAJ || r < kc))
                copy4(smem_u32(s) + 128u * (uint32_t)r + 16u * (uint32_t)((e >> 2) ^ (r & 7)) + 4u * (uint32_t)(e & 3), src);
        }
        return;
    }
    constexpr int per = ROWS * BK / 8 / kProducers;
#pragma unroll
    for (int i = 0; i < per; ++i) {
        const int v = threadIdx.x + i * kProducers, r = v >> 3, c = v & 7;
        const uint32_t at = 128u * (uint32_t)r + 16u * (uint32_t)(c ^ (r & 7));
        const int row = KMAJ ? mn0 + r : k0 + r % BK;
        const int col = KMAJ ? k0 + 8 * c : mn0 + 64 * (r / BK) + 8 * c;
        if (KMAJ ? 8 * c >= kc : r % BK >= kc) continue;
        if constexpr (std::is_same<L, InputCols>::value) {
        } else if constexpr (L::kAsync) {
            copy16(smem_u32(s) + at, ld.src(row, col), ld.base());
        } else {
            *reinterpret_cast<uint4*>(s + at) = ld(row, col);
        }
    }
}

// matrix descriptor of the 16-k slice ks of a tile: K-major, 32 bytes along the swizzled rows; MN-major, 16
// rows down
template <bool KMAJ>
__device__ __forceinline__ uint64_t tile_desc(uint32_t base, int ks) {
    if (KMAJ) return smem_desc(base + (uint32_t)ks * 32, 16, 1024);
    return smem_desc(base + (uint32_t)ks * 2048, BK * 128, 1024);
}

__device__ __forceinline__ void mbar_init(uint64_t* b, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count));
}
__device__ __forceinline__ void commit_mmas(uint64_t* b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(b)));
}

// C[M, N] (+ epilogue) over k in [z * ksplit, (z + 1) * ksplit) of split z = blockIdx.z (ksplit a multiple of
// 32 when there are several)
template <bool AK, bool BKM, int kStages, class LA, class LB, class EP>
__global__ void __launch_bounds__(kGemmThreads) gemm_kernel(LA la, LB lb, EP ep, int M, int N, int K, int ksplit) {
    extern __shared__ unsigned char dsmem[];
    __shared__ __align__(8) uint64_t full[kStages], empty[kStages];
    __shared__ __align__(8) uint64_t mbar_drain;  // completes once every MMA issued has
    __shared__ uint32_t s_tmem;
    constexpr uint32_t kStage = kTileA + kTileB;
    unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)dsmem + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
    const int k_begin = blockIdx.z * ksplit, k_end = min(K, k_begin + ksplit);

    if constexpr (std::is_same<LA, InputCols>::value) {
        // the tile outside the copied values: zeros, and in the weight gradient the bias row's ones (column 10)
        for (int v = tid; v < kStages * (int)(kTileA / 16); v += kGemmThreads) {
            const int st = v / (kTileA / 16), i = v % (kTileA / 16), r = i >> 3, c = (i & 7) ^ (r & 7);
            reinterpret_cast<uint4*>(base + st * kStage)[i] =
                make_uint4(0u, !AK && r < BK && c == 1 ? 0x3f80u : 0u, 0u, 0u);
        }
    }
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], kProducers);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&mbar_drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = s_tmem;

    bool ok = true;
    if (tid < kProducers) {
        int st = 0;
        uint32_t par = 1;  // the first pass over the ring finds every stage empty
        for (int k = k_begin; k < k_end; k += BK) {
            if (k - k_begin >= kStages * BK && !mbar_wait(smem_u32(&empty[st]), par)) {
                ok = false;
                break;
            }
            unsigned char* s = base + st * kStage;
            const int kc = min(BK, (k_end - k + 15) & ~15);
            tile_load<AK, BM>(la, m0, k, kc, s);
            tile_load<BKM, BN>(lb, n0, k, kc, s + kTileA);
            if constexpr (LA::kAsync && LB::kAsync) {
                asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&full[st])) : "memory");
            } else {  // plain stores among them: landed and fenced before the arrival
                asm volatile("cp.async.wait_all;" ::: "memory");
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&full[st])) : "memory");
            }
            if (++st == kStages) {
                st = 0;
                par ^= 1u;
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (tid == kProducers) {
        int st = 0;
        uint32_t par = 0;
        for (int k = k_begin; k < k_end; k += BK) {
            if (!mbar_wait(smem_u32(&full[st]), par)) {
                ok = false;
                break;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t a0 = smem_u32(base + st * kStage), b0 = a0 + kTileA;
            const int n_ks = (min(BK, k_end - k) + 15) / 16;
            for (int ks = 0; ks < n_ks; ++ks) {
                const uint64_t ad = tile_desc<AK>(a0, ks);
                const uint64_t bd = tile_desc<BKM>(b0, ks);
                const uint32_t acc = (k > k_begin || ks > 0) ? 1u : 0u;
                asm volatile(
                    "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                    " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                    "l"(ad), "l"(bd), "r"(idesc_f16(!AK, !BKM)), "r"(acc));
            }
            commit_mmas(&empty[st]);
            if (++st == kStages) {
                st = 0;
                par ^= 1u;
            }
        }
        commit_mmas(&mbar_drain);  // tracks every MMA issued, also after a give-up
        ok = mbar_wait(smem_u32(&mbar_drain), 0u) && ok;
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    ok = __syncthreads_and(ok) != 0;
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (ok && k_end > k_begin && tid < kProducers) {
        float* sE = reinterpret_cast<float*>(base);  // the tile ring is free: every MMA has completed
        const int q = warp & 3, half = warp >> 2;
#pragma unroll
        for (int h = 0; h < 32; h += 16) {
            uint32_t r[16];
            const int col = half * 32 + h;
            const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)col;
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                "[%16];"
                : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                  "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                  "=r"(r[15])
                : "r"(taddr));
            asm volatile("tcgen05.wait::ld.sync.aligned;");
            uint4* row = reinterpret_cast<uint4*>(sE + (q * 32 + lane) * kEpiLd + col);
#pragma unroll
            for (int j = 0; j < 4; ++j) row[j] = make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kProducers) : "memory");  // the epilogue's warps
        // half a warp covers one row's 16 column quads
#pragma unroll 4
        for (int p = tid; p < BM * (BN / 4); p += kProducers) {
            const int rr = p / (BN / 4), pc = p % (BN / 4);
            ep(m0 + rr, n0 + 4 * pc, *reinterpret_cast<const float4*>(sE + rr * kEpiLd + 4 * pc), blockIdx.z);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

// ------------------------------------------------------------------------------------------
// loaders: the 8 values at stored (row, col .. col + 7), zero outside the operand: their address
// (src; kAsync) or the values (operator())
// ------------------------------------------------------------------------------------------

// a one and seven zeros: the vector that holds the bias row's ones in a weight-gradient operand
__device__ uint4 g_ones8 = {0x3f80u, 0u, 0u, 0u};

// dense BF16 matrix [rows][ld] whose rows start on 16-byte boundaries (ld and cols multiples of 8); with
// `ones`, column `cols` reads as 1 on valid rows
struct DenseBF {
    static constexpr bool kAsync = true;
    const __nv_bfloat16* p;
    int rows, cols, ld;
    bool ones;
    __device__ const void* base() const { return p; }
    __device__ const void* src(int r, int c) const {
        if (r >= rows || c > cols || (c == cols && !ones)) return nullptr;
        return c == cols ? static_cast<const void*>(&g_ones8) : p + (size_t)r * ld + c;
    }
};

// dense BF16 matrix [rows][ld] of any alignment
struct DenseBFAny {
    static constexpr bool kAsync = false;
    const __nv_bfloat16* p;
    int rows, cols, ld;
    __device__ uint4 operator()(int r, int c) const {
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int e = c + i;
            v[i] = (r < rows && e < cols) ? __bfloat162float(p[(size_t)r * ld + e]) : 0.f;
        }
        return pack8(v);
    }
};

// dense FP32 matrix [rows][ld], rounded to BF16 on load
struct DenseF32 {
    static constexpr bool kAsync = false;
    const float* p;
    int rows, cols, ld;
    __device__ uint4 operator()(int r, int c) const {
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int e = c + i;
            v[i] = (r < rows && e < cols) ? p[(size_t)r * ld + e] : 0.f;
        }
        return pack8(v);
    }
};

// im2col of a [B][2 Lo][64] BF16 activation for a kernel-5, pad-2 convolution of stride 2, Lo = 2^log_lo:
// row m = b * Lo + l, column k = kk * 64 + c -> h[b][2 l + kk - 2][c]   (K-major A)
struct Im2col {
    static constexpr bool kAsync = true;
    const __nv_bfloat16* h;
    int B, log_lo;
    __device__ const void* base() const { return h; }
    __device__ const void* src(int m, int k) const {
        const int b = m >> log_lo, l = m & ((1 << log_lo) - 1);
        const int i = 2 * l + (k >> 6) - 2;
        if (b >= B || k >= 5 * 64 || i < 0 || i >= (2 << log_lo)) return nullptr;
        return h + (((size_t)b << (log_lo + 1)) + i) * 64 + (k & 63);
    }
};

// the same gather stored MN-major for the weight gradient: row = b * Lo + l, column m = kk * 64 + c,
// and column 320 reads as 1 (the bias row of the gradient)
struct Im2colT {
    static constexpr bool kAsync = true;
    const __nv_bfloat16* h;
    int B, log_lo;
    __device__ const void* base() const { return h; }
    __device__ const void* src(int r, int m) const {
        const int b = r >> log_lo, l = r & ((1 << log_lo) - 1);
        if (b >= B || m > 5 * 64) return nullptr;
        if (m == 5 * 64) return &g_ones8;
        const int i = 2 * l + (m >> 6) - 2;
        if (i < 0 || i >= (2 << log_lo)) return nullptr;
        return h + (((size_t)b << (log_lo + 1)) + i) * 64 + (m & 63);
    }
};

// im2col of the network input for the first (stride-1) convolution, from its BF16 copy with two zero
// positions on either side of a sample, xb [B][260][2]: row b * 256 + l holds the ten values from position
// l on, column kk * 2 + c. K-major A of the forward product; MN-major A of the weight gradient, where
// column 10 reads as 1 (the bias row). src: the pair of values at tap e.
struct InputCols {
    static constexpr bool kAsync = true;
    const __nv_bfloat16* xb;
    int B;
    __device__ const void* src(int m, int e) const {
        return (m >> 8) < B ? xb + ((size_t)(m >> 8) * 260 + (m & 255) + e) * 2 : nullptr;
    }
};

// The input gradient of such a convolution from its output gradient dz [B][Lo][64], Lo = 2^log_lo: the
// input positions 2 p + PAR of a sample get dz[p + 1 - j] through tap kk = 2 j + PAR, j = 0 .. 2 (PAR 0) or
// 0 .. 1 (PAR 1), so each parity is a product over its own taps and no zeros are multiplied:
// row m = b * Lo + p, column k = j * 64 + o   (K-major A)
template <int PAR>
struct ConvGrad {
    static constexpr bool kAsync = true;
    const __nv_bfloat16* dz;
    int B, log_lo;
    __device__ const void* base() const { return dz; }
    __device__ const void* src(int m, int k) const {
        const int b = m >> log_lo, l = (m & ((1 << log_lo) - 1)) + 1 - (k >> 6);
        if (b >= B || k >= (3 - PAR) * 64 || l < 0 || l >= (1 << log_lo)) return nullptr;
        return dz + (((size_t)b << log_lo) + l) * 64 + (k & 63);
    }
};

// a convolution weight W [(kk * 64 + c)][o] read as the K-major B of that product:
// stored row n = c, column k = j * 64 + o, kk = 2 j + PAR
template <int PAR>
struct ConvWT {
    static constexpr bool kAsync = true;
    const __nv_bfloat16* w;
    __device__ const void* base() const { return w; }
    __device__ const void* src(int n, int k) const {
        if (n >= 64 || k >= (3 - PAR) * 64) return nullptr;
        return w + ((size_t)(2 * (k >> 6) + PAR) * 64 + n) * 64 + (k & 63);
    }
};

}  // namespace cnn
}  // namespace sblm
