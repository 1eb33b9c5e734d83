// mlp_gemm.cu -- BF16 GEMM on the 5th-generation tensor cores (tcgen05),
// for the dense layers of the MLP energy surrogate.
//
// C (FP32) = A . B with BF16 operands stored row-major in one of three forms:
//   NT  A[M x K], B[N x K]: the contraction index is contiguous in both;
//   NN  A[M x K], B[K x N]: products with the transpose of a weight;
//   TN  A[K x M], B[K x N]: weight gradients, contracted over the samples.
// The tensor core reads either order from shared memory, so no operand is
// ever transposed in memory.  Persistent kernel, one CTA per SM, in clusters
// of two CTAs that compute the 128 x BN output tiles of two adjacent row
// blocks in the same column block, so that the BN x 64 B tile of each k-step
// is read from L2 once per cluster instead of once per CTA.  Ten warps with
// fixed roles:
//   * warp 0 streams the CTA's 128 x 64 tile of A and its half
//     of the shared B tile with TMA (cp.async.bulk.tensor, 128-byte swizzle,
//     out-of-range rows and columns zero-filled), the B half multicast into
//     both CTAs' stage, into a ring of kStages shared-memory stages, each
//     completing a transaction-count mbarrier; a stage is refilled once the
//     products of both CTAs have read it;
//   * warp 1 issues four tcgen05.mma (M 128, N BN, K 16) per operand
//     tile into one of two FP32 accumulators of BN tensor-memory columns,
//     frees each stage in both CTAs with a multicast tcgen05.commit, and
//     commits the accumulator when a tile's last product is issued;
//   * warps 2..9 drain a finished accumulator with tcgen05.ld (warp w reads
//     tensor-memory lanes 32 (w mod 4) ..), apply the bias and the layer's
//     output transform, store through shared memory, and hand the
//     accumulator back -- so the epilogue of one tile runs while the tensor
//     core works on the next.
//
// A k-step is bound by what one thread issues, not by the copies: the stage
// holds two k-tiles where the ring is deep enough, the abort flag is read only
// in the slow part of a wait, slot and parity are counters, and the warps walk
// the ring as a whole with an elected lane issuing, which spares the issue
// loops over lanes that a single-lane branch costs (per 64 of K at BN = 64:
// 0.41 us before, 0.15 now; 512 x 8192 x 64: 59.5 -> 28.8 us; 65536 x 512 x
// 2776 at BN = 256: 178 -> 169 us, and 150 with the stores below, 1.24 PFLOP/s).
//
// Every wait on an mbarrier is bounded: after kWaitLimit polls the waiting
// role records PAMD_ETIMEOUT and raises a shared abort flag, the others stop
// at their next wait, the CTA waits (bounded) for its own copies and products
// in flight, meets its partner at a cluster barrier (so that neither leaves
// while the other may still write to it), frees its tensor memory and returns.
// A partner that timed out stops feeding the other, whose own bounded waits
// then run out as well.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <mutex>

#include "pamd_internal.h"

namespace pamd {

namespace {

constexpr int kBM = 128;
constexpr int kBK = 64;   // contraction depth of one operand tile (128 bytes of BF16)
// warp 0: TMA producer, warp 1: MMA issuer, warps 2..9: epilogue (two warps
// per tensor-memory lane quarter, each taking one half of the tile's columns)
constexpr int kEpiWarps = 8, kThreads = 64 + 32 * kEpiWarps, kEpiThreads = 32 * kEpiWarps;
constexpr int kTileA = kBM * kBK * 2;  // 16 KiB
constexpr int kRingBytes = 192 * 1024;
constexpr int kEpiStage = 4096;  // shared memory of one epilogue warp, after the ring
constexpr uint32_t kWaitLimit = 1u << 22;

// Per tile width BN: bytes of a B tile and a stage [A A | B B], stages of the
// ring (192 KiB), tensor-memory columns (two accumulators).
template <int BN>
struct Tile {
    static constexpr int kSub = BN == 256 ? 1 : 2;  // operand tiles per ring stage
    static constexpr int kTileB = BN * kBK * 2;
    static constexpr int kStageBytes = kSub * (kTileA + kTileB);
    static constexpr int kStages = kRingBytes / kStageBytes;  // 4, 3, 4 for BN = 256, 128, 64
    static constexpr int kTmemCols = 2 * BN;
};

// instruction descriptor of tcgen05.mma.kind::f16: D FP32 (bits 4-5 = 1),
// A BF16 (bits 7-9 = 1), B BF16 (bits 10-12 = 1), bits 15 and 16: A and B
// stored with the row index of the product contiguous, not the contraction
// index; N >> 3 at bits 17-22, M >> 4 at bits 24-28
template <int BN, int MODE>
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (MODE == kGemmTN ? 1u << 15 : 0u) |
                            (MODE != kGemmNT ? 1u << 16 : 0u) | ((uint32_t)(BN >> 3) << 17) |
                            ((uint32_t)(kBM >> 4) << 24);

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor: K-major operand in the 128-byte swizzle
// layout, 8-row groups 1024 bytes apart (stride byte offset), descriptor
// version 1 (bits 46-47), swizzle mode 2 = 128 B (bits 61-63).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// The same for an operand stored [k][row]: groups of 64 rows of the
// product are 128 bytes wide and kBK k-rows (8 KiB) long, one after another
// (leading byte offset), groups of 8 k-rows 1024 bytes apart (stride).
__device__ __forceinline__ uint64_t sw128_desc_tn(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)(kBK * 128 >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait (polls, then polls with a short sleep); false on timeout, or
// when another role has raised the abort flag.  The flag is read only in the
// slow part: the producer and the issuer are single threads, and 30 cycles of
// a shared-memory read in each of their steps were a quarter of a k-step.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const volatile int* abort_flag = nullptr) {
    for (uint32_t i = 0; i < kWaitLimit; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if (i >= 1024) {
            if (abort_flag && *abort_flag) return false;
            __nanosleep(64);
        }
    }
    return false;
}

// the same by all lanes of a warp, with one result
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, const volatile int* abort_flag) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag));
}

// true in one lane of a converged warp, the same one on each call
__device__ __forceinline__ bool elect_one() {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok));
    return ok != 0;
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

// TMA: tile of a 2-D tensor map at element coordinates (x = column, y = row)
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// TMA load multicast to the CTAs of the cluster in `mask`: the tile lands at
// the same shared-memory offset in each and completes each one's mbarrier at
// the same offset
__device__ __forceinline__ void tma_load_2d_mc(uint32_t dst, const CUtensorMap* map, int x, int y,
                                               uint32_t bar, uint16_t mask) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        ".multicast::cluster [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar), "h"(mask)
        : "memory");
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                     : "memory");
}

// arrive on the mbarrier at this offset in every CTA of `mask` once the
// products issued so far are done
__device__ __forceinline__ void mma_commit_mc(uint32_t bar, uint16_t mask) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            bar),
        "h"(mask)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// 32 columns of FP32 accumulator for this thread's row (TMEM lane)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}


__device__ __forceinline__ float sigmoid(float z) { return __fdividef(1.0f, 1.0f + __expf(-z)); }

// the first n of 32 consecutive values of one row
__device__ __forceinline__ void store_row32(float* dst, const float (&v)[32], int n) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
        if (j < n) dst[j] = v[j];
}

__device__ __forceinline__ void store_row32_bf16(__nv_bfloat16* dst, const float (&v)[32], int n) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
        if (j < n) dst[j] = __float2bfloat16(v[j]);
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// 32 rows x 32 columns of a warp through its 4 KiB of shared memory, so that
// global memory sees whole 128- (FP32) or 64-byte (BF16) row pieces instead of
// 16 bytes in each of 32 rows.  The 16-byte slots of a row are swizzled: writes
// by row and reads across rows are both free of bank conflicts.  65536 x 2776 x
// 512 with FP32 results: 331 -> 182 us, 65536 x 512 x 512: 64 -> 43 us.
__device__ __forceinline__ uint4* slot_f32(unsigned char* st, int r, int q) {
    return reinterpret_cast<uint4*>(st + r * 128 + ((q ^ (r & 7)) << 4));
}
__device__ __forceinline__ uint4* slot_b16(unsigned char* st, int r, int q) {
    return reinterpret_cast<uint4*>(st + r * 64 + ((q ^ ((r >> 1) & 3)) << 4));
}

// dst: row 0 of the warp's 32, column 0 of the 32; rows of them exist
__device__ __forceinline__ void store_block_f32(float* dst, int ld, int rows, const float (&v)[32], unsigned char* st) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 8; ++q)
        *reinterpret_cast<float4*>(slot_f32(st, lane, q)) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    __syncwarp();
#pragma unroll
    for (int it = 0; it < 8; ++it) {
        const int r = 4 * it + (lane >> 3);
        const uint4 w = *slot_f32(st, r, lane & 7);
        if (r < rows) *reinterpret_cast<uint4*>(dst + (size_t)r * ld + 4 * (lane & 7)) = w;
    }
}

__device__ __forceinline__ void store_block_bf16(__nv_bfloat16* dst, int ld, int rows, const float (&v)[32], unsigned char* st) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t w[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(v[8 * q + 2 * t], v[8 * q + 2 * t + 1]);
            w[t] = *reinterpret_cast<const uint32_t*>(&h);
        }
        *slot_b16(st, lane, q) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    __syncwarp();
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int r = 8 * it + (lane >> 2);
        const uint4 w = *slot_b16(st, r, lane & 3);
        if (r < rows) *reinterpret_cast<uint4*>(dst + (size_t)r * ld + 8 * (lane & 3)) = w;
    }
}

// v *= the same block of src
__device__ __forceinline__ void mul_block_f32(const float* src, int ld, int rows, float (&v)[32], unsigned char* st) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
#pragma unroll
    for (int it = 0; it < 8; ++it) {
        const int r = 4 * it + (lane >> 3);
        if (r < rows) *slot_f32(st, r, lane & 7) = *reinterpret_cast<const uint4*>(src + (size_t)r * ld + 4 * (lane & 7));
    }
    __syncwarp();
    if (lane < rows) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float4 t = *reinterpret_cast<const float4*>(slot_f32(st, lane, q));
            v[4 * q] *= t.x;
            v[4 * q + 1] *= t.y;
            v[4 * q + 2] *= t.z;
            v[4 * q + 3] *= t.w;
        }
    }
}

// Epilogue of `chunks` x 32 columns of a tile: accumulator columns of this
// warp's 32 tensor-memory lanes (rows row0 + lane); taddr and n0 point at the
// first column, st at the warp's shared memory.  Full, aligned blocks of 32
// columns go to memory through it; the rest element by element.
__device__ __forceinline__ void epilogue_tile(const GemmArgs& g, uint32_t taddr, int row0, int n0, int chunks,
                                              unsigned char* st) {
    const int row = row0 + (threadIdx.x & 31), rows = g.M - row0;
    const bool row_ok = row < g.M;
    float head = 0.0f;
    __nv_bfloat16* Cb = static_cast<__nv_bfloat16*>(g.Cb);
    const bool vf = (g.vec_ok & 1) != 0, vb = (g.vec_ok & 2) != 0;
#pragma unroll 1
    for (int cc = 0; cc < chunks; ++cc) {
        float v[32];
        tmem_ld32(taddr + (uint32_t)(cc * 32), v);
        const int col0 = n0 + cc * 32;
        const int n = min(32, g.N - col0);
        if (rows <= 0 || n <= 0) continue;
        const bool bf = vf && n == 32, bb = vb && n == 32;
        const int ns = row_ok ? n : 0;  // of the element-wise forms
        if (g.bias) {
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] += (j < n) ? g.bias[col0 + j] : 0.0f;
        }
        const size_t o = (size_t)row * g.ldc + col0, o0 = (size_t)row0 * g.ldc + col0;
        if (g.C) {
            if (bf) store_block_f32(g.C + o0, g.ldc, rows, v, st);
            else store_row32(g.C + o, v, ns);
        }
        if (g.epi == kEpiSilu || g.epi == kEpiHead) {
            float ds[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const float sg = sigmoid(v[j]);
                ds[j] = sg * (1.0f + v[j] * (1.0f - sg));
                v[j] *= sg;  // silu
            }
            if (g.Cs) {
                if (bf) store_block_f32(g.Cs + o0, g.ldc, rows, ds, st);
                else store_row32(g.Cs + o, ds, ns);
            }
            if (g.epi == kEpiHead) {
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const float w = (j < n) ? g.vec[col0 + j] : 0.0f;
                    head = fmaf(w, v[j], head);
                    v[j] = w * ds[j];
                }
            }
        } else if (g.epi == kEpiMul) {
            if (bf) {
                mul_block_f32(g.mul + o0, g.ldc, rows, v, st);
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] *= (j < ns) ? g.mul[o + j] : 0.0f;
            }
        }
        if (Cb) {
            if (bb) store_block_bf16(Cb + (size_t)row0 * g.ldcb + col0, g.ldcb, rows, v, st);
            else store_row32_bf16(Cb + (size_t)row * g.ldcb + col0, v, ns);
        }
    }
    // one partial sum of the head per 128 columns; a tile of 128 columns that
    // is the last one writes the zero of the missing other half as well
    if (g.epi == kEpiHead && row_ok) {
        const int np = gemm_head_parts(g.N), at = n0 / 128;
        g.part[(size_t)row * np + at] = head;
        if (at + 1 < np && n0 + 128 >= g.N && chunks * 32 == 128 && at % 2 == 0) g.part[(size_t)row * np + at + 1] = 0.0f;
    }
}

template <int BN, int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    gemm_bf16_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                     const __grid_constant__ GemmArgs g) {
    constexpr int kSub = Tile<BN>::kSub;
    constexpr int kBN = BN, kStages = Tile<BN>::kStages, kStageBytes = Tile<BN>::kStageBytes, kTileB = Tile<BN>::kTileB;
    constexpr uint32_t kTmemCols = Tile<BN>::kTmemCols;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long full_bar[kStages], empty_bar[kStages];
    __shared__ __align__(8) unsigned long long accf_bar[2], acce_bar[2], done_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort, s_issued, s_consumed;
    // 1024-byte aligned stages: [A0 | B0 | A1 | B1 | ...]
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int tid = threadIdx.x, warp = tid >> 5;
    // The two CTAs of a cluster take row blocks 2p and 2p + 1 of the same
    // column block: each loads its A tile and half of the shared B tile,
    // multicast to both.
    const int MT = (g.M + kBM - 1) / kBM, NT = (g.N + kBN - 1) / kBN;
    const int tiles = ((MT + 1) / 2) * NT;  // tile pairs
    const int KT = (g.K + kBK - 1) / kBK, KB = (KT + kSub - 1) / kSub;  // operand tiles and stages of a product
    const int crank = (int)cluster_rank();
    const int cid = blockIdx.x >> 1, ncl = gridDim.x >> 1;

    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_slot)),
                     "r"((uint32_t)kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int st = 0; st < kStages; ++st) {
            mbar_init(smem_u32(&full_bar[st]), 1);
            mbar_init(smem_u32(&empty_bar[st]), 2);  // both CTAs' products have read it
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(smem_u32(&accf_bar[q]), 1);
            mbar_init(smem_u32(&acce_bar[q]), kEpiThreads);
        }
        mbar_init(smem_u32(&done_bar), 1);
        s_abort = 0;
        s_issued = 0;
        s_consumed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    cluster_sync();  // the peer's barriers exist before any multicast reaches them
    const uint32_t tmem = tmem_slot;
    volatile int* abort_flag = &s_abort;

    if (warp == 0) {
        {  // TMA producer: the warp walks the ring, one lane issues
            uint32_t gk = 0, st = 0, ph = 0;  // stages so far, ring slot, its use number's parity
            bool stop = false;
            for (int t = cid; t < tiles && !stop; t += ncl) {
                // A box of an odd last row block's missing partner, or a B box
                // past column N, would lie wholly outside its matrix: read a
                // valid box instead (its products land in rows / columns the
                // epilogue drops)
                const int n0 = (t % NT) * kBN;
                const int m0 = min((2 * (t / NT) + crank) * kBM, (MT - 1) * kBM);
                for (int kb = 0; kb < KB; ++kb, ++gk) {
                    if (gk >= (uint32_t)kStages && !mbar_wait_warp(smem_u32(&empty_bar[st]), ph ^ 1u, abort_flag)) {
                        *abort_flag = 1;
                        stop = true;
                        break;
                    }
                    const uint32_t fb = smem_u32(&full_bar[st]);
                    const uint32_t sa = base + st * (uint32_t)kStageBytes, sb = sa + kSub * kTileA;
                    const int subs = min(kSub, KT - kb * kSub);
                    if (elect_one()) {
                        mbar_expect_tx(fb, (uint32_t)(subs * (kTileA + kTileB)));
#pragma unroll
                        for (int u = 0; u < kSub; ++u) {
                            if (u >= subs) break;
                            const uint32_t ta = sa + u * kTileA, tb = sb + u * kTileB;
                            const int k0 = (kb * kSub + u) * kBK;
                            if (MODE == kGemmTN) {  // A: boxes of 64 rows of the product x 64 k-rows
#pragma unroll
                                for (int q = 0; q < kBM / 64; ++q) {
                                    const int x = m0 + 64 * q;
                                    tma_load_2d(ta + q * kBK * 128, &tmA, x < g.M ? x : m0, k0, fb);
                                }
                            } else {
                                tma_load_2d(ta, &tmA, k0, m0, fb);
                            }
                            if (MODE != kGemmNT) {
                                // B: boxes of 64 columns x 32 k-rows, half the k-rows from
                                // each CTA.  The last tile may have no rows for the
                                // second one: it reads the first one's (A is zero there)
                                const int y = k0 + crank * (kBK / 2);
#pragma unroll
                                for (int q = 0; q < BN / 64; ++q) {
                                    const int x = n0 + 64 * q;
                                    tma_load_2d_mc(tb + q * kBK * 128 + crank * (kBK / 2) * 128, &tmB, x < g.N ? x : n0,
                                                   y < g.K ? y : k0, fb, (uint16_t)0x3);
                                }
                            } else {
                                const int yb = (n0 + crank * (kBN / 2) < g.N) ? n0 + crank * (kBN / 2) : n0;
                                tma_load_2d_mc(tb + crank * (kTileB / 2), &tmB, k0, yb, fb, (uint16_t)0x3);
                            }
                        }
                    }
                    __syncwarp();
                    if (++st == (uint32_t)kStages) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
            }
            s_issued = (int)gk;
            // the peer's last releases of this CTA's stages land before it exits
            for (uint32_t u = gk > (uint32_t)kStages ? gk - kStages : 0; u < gk; ++u)
                if (!mbar_wait_warp(smem_u32(&empty_bar[u % kStages]), (u / kStages) & 1u, abort_flag)) {
                    *abort_flag = 1;
                    break;
                }
        }
    } else if (warp == 1) {
        {  // MMA issuer, likewise
            uint32_t gk = 0, st = 0, ph = 0;
            int i = 0;
            bool stop = false;
            for (int t = cid; t < tiles && !stop; t += ncl, ++i) {
                const int acc = i & 1;
                if (i >= 2 && !mbar_wait_warp(smem_u32(&acce_bar[acc]), (uint32_t)((i / 2 - 1) & 1), abort_flag)) {
                    *abort_flag = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t td = tmem + (uint32_t)(acc * kBN);
                for (int kb = 0; kb < KB; ++kb, ++gk) {
                    if (!mbar_wait_warp(smem_u32(&full_bar[st]), ph, abort_flag)) {
                        *abort_flag = 1;
                        stop = true;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = base + st * (uint32_t)kStageBytes, sb = sa + kSub * kTileA;
                    const int subs = min(kSub, KT - kb * kSub);
                    if (elect_one()) {
#pragma unroll
                        for (int u = 0; u < kSub; ++u) {
                            if (u >= subs) break;
                            const uint32_t ta = sa + u * kTileA, tb = sb + u * kTileB;
                            const uint64_t da = MODE == kGemmTN ? sw128_desc_tn(ta) : sw128_desc(ta);
                            const uint64_t db = MODE != kGemmNT ? sw128_desc_tn(tb) : sw128_desc(tb);
                            // 16 of the contraction further: 32 bytes along a row, or 16 rows
#pragma unroll
                            for (int k = 0; k < kBK / 16; ++k)
                                mma_bf16(td, da + (uint64_t)(k * (MODE == kGemmTN ? 16 * 128 : 32) >> 4),
                                         db + (uint64_t)(k * (MODE != kGemmNT ? 16 * 128 : 32) >> 4), kIdesc<BN, MODE>,
                                         (kb > 0 || u > 0 || k > 0) ? 1u : 0u);
                        }
                        mma_commit_mc(smem_u32(&empty_bar[st]), (uint16_t)0x3);
                    }
                    __syncwarp();
                    if (++st == (uint32_t)kStages) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
                if (!stop && elect_one()) mma_commit(smem_u32(&accf_bar[acc]));
                __syncwarp();
            }
            s_consumed = (int)gk;
            // tracks every product issued before it, also on the abort path
            if (elect_one()) mma_commit(smem_u32(&done_bar));
        }
    } else {  // epilogue warps 2..9
        const int q = warp & 3;  // tensor-memory lane quarter this warp may access
        const int half = (warp - 2) >> 2;
        unsigned char* stage = smem_raw + (base - smem_u32(smem_raw)) + kRingBytes + (warp - 2) * kEpiStage;
        int i = 0;
        for (int t = cid; t < tiles; t += ncl, ++i) {
            const int acc = i & 1;
            if (!mbar_wait_warp(smem_u32(&accf_bar[acc]), (uint32_t)((i / 2) & 1), abort_flag)) {
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            const int m0 = (2 * (t / NT) + crank) * kBM, nt = t % NT;
            const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * kBN);
            // the head's partial sums run over 128 columns: with a tile that
            // narrow one warp per quarter takes them all
            if (BN == 128 && g.epi == kEpiHead) {
                if (half == 0) epilogue_tile(g, taddr, m0 + q * 32, nt * kBN, BN / 32, stage);
            } else {
                epilogue_tile(g, taddr + (uint32_t)(half * (kBN / 2)), m0 + q * 32, nt * kBN + half * (kBN / 2),
                              BN / 64, stage);
            }
            tc_fence_before();
            mbar_arrive(smem_u32(&acce_bar[acc]));
        }
    }
    __syncwarp();
    __syncthreads();
    if (tid == 0) {
        if (*abort_flag) {
            atomicCAS(g.status, 0, PAMD_ETIMEOUT);
            // copies issued but never consumed must land before the CTA exits
            for (int gk = s_consumed; gk < s_issued; ++gk)
                mbar_wait(smem_u32(&full_bar[gk % kStages]), (uint32_t)((gk / kStages) & 1));
        }
        mbar_wait(smem_u32(&done_bar), 0u);  // products in flight
    }
    tc_fence_before();
    __syncthreads();
    // neither CTA leaves while the other may still write its shared memory or
    // arrive on its barriers
    cluster_sync();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"((uint32_t)kTmemCols)
                     : "memory");
}

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// Tensor map of a row-major BF16 matrix [rows][ld] read in box_rows x 64-column
// boxes with the 128-byte swizzle; columns >= cols and rows >= rows read as 0.
bool encode_operand(CUtensorMap* map, const void* ptr, int rows, int cols, int ld, int box_rows) {
    const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// True when p is device memory of device dev (not host, pinned host, managed
// or another GPU's memory).
bool on_device(const void* p, int dev) {
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice && a.device == dev;
}

constexpr int kMaxDevices = 64;

using GemmKernel = void (*)(const CUtensorMap, const CUtensorMap, const GemmArgs);
constexpr size_t kGemmSmem = kRingBytes + kEpiWarps * kEpiStage + 1024;

template <int MODE>
GemmKernel gemm_kernel_of(int bn) {
    return bn == 256 ? gemm_bf16_kernel<256, MODE> : bn == 128 ? gemm_bf16_kernel<128, MODE> : gemm_bf16_kernel<64, MODE>;
}
GemmKernel gemm_kernel(int bn, int mode) {
    return mode == kGemmNT ? gemm_kernel_of<kGemmNT>(bn) : mode == kGemmTN ? gemm_kernel_of<kGemmTN>(bn)
                                                                           : gemm_kernel_of<kGemmNN>(bn);
}

// Kernel attributes and resident cluster count, once per device.
cudaError_t gemm_setup(int dev, int* max_clusters_out) {
    const size_t smem = kGemmSmem;
    static std::once_flag once[kMaxDevices];
    static cudaError_t attr[kMaxDevices];
    static int max_clusters[kMaxDevices];
    std::call_once(once[dev], [&] {
        cudaError_t e = cudaSuccess;
        for (int bn = 64; bn <= 256 && e == cudaSuccess; bn *= 2)
            for (int mode = kGemmNT; mode <= kGemmNN && e == cudaSuccess; ++mode)
                e = cudaFuncSetAttribute((const void*)gemm_kernel(bn, mode), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
        // persistent grid: as many two-CTA clusters as can be resident at once
        // (an SM left without a partner in its GPC hosts none)
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(2, 1, 1);
        cfg.blockDim = dim3(kThreads, 1, 1);
        cfg.dynamicSmemBytes = smem;
        int mc = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&mc, gemm_kernel(256, kGemmNT), &cfg);
        if (e == cudaSuccess && mc < 1) e = cudaErrorInvalidConfiguration;
        attr[dev] = e;
        max_clusters[dev] = mc;
    });
    if (max_clusters_out) *max_clusters_out = max_clusters[dev];
    return attr[dev];
}

cudaError_t gemm_prepare_device() {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    return gemm_setup(dev, nullptr);
}

// Tile pairs (two row blocks of one column block) of a product.
long long gemm_tiles(const GemmArgs& g, int bn) {
    return (long long)((g.M + 2 * kBM - 1) / (2 * kBM)) * ((g.N + bn - 1) / bn);
}

// Tile width: the narrowest of 64, 128 and 256 columns whose tile pairs still
// fit the resident clusters in one wave, else 256.  One wave of narrow tiles
// has shorter steps and uses more SMs; past one wave the wide tile reads
// least per product.  Measured with BN = 64 / 128 / 256, us (NT, FP32 result):
//   N 512,  K 2776: M 2048 16.5 / 18.6 / 24.6, 4096 28.8 / 19.9 / 24.7,
//                   8192 53 / 34.9 / 25.4, 65536 346 / 229 / 169;
//   N 512,  K 512:  M 2048 8.3 / 10.3 / 12.4, 8192 14.5 / 12.5 / 12.4;
//   N 2776, K 512:  M 256 8.3 / 10.3 / 12.4, 512 10.4 / 10.3 / 12.4
// (before the stores through shared memory, which the wide tiles gain from).
// The head sums over 128 columns in one thread: not below that.
int tile_width(const GemmArgs& g, int max_clusters) {
    int bn = 256;
    while (bn > (g.epi == kEpiHead ? 128 : 64) && gemm_tiles(g, bn / 2) <= max_clusters) bn /= 2;
    return bn;
}

cudaError_t launch_gemm_bf16(const GemmArgs& ga, cudaStream_t s) {
    if (ga.M <= 0 || ga.N <= 0 || ga.K <= 0 || (ga.K & 7) || (ga.lda & 7) || (ga.ldb & 7) ||
        (reinterpret_cast<uintptr_t>(ga.A) & 15) || (reinterpret_cast<uintptr_t>(ga.B) & 15))
        return cudaErrorInvalidValue;
    int dev = 0;
    cudaError_t de = cudaGetDevice(&dev);
    if (de != cudaSuccess) return de;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    // The B tile is multicast by TMA into both CTAs of a cluster: the tensor
    // maps must cover this GPU's own memory only.
    if (!on_device(ga.A, dev) || !on_device(ga.B, dev)) return cudaErrorInvalidValue;
    int max_clusters = 0;
    const cudaError_t se = gemm_setup(dev, &max_clusters);
    if (se != cudaSuccess) return se;
    const int bn = tile_width(ga, max_clusters);
    CUtensorMap tmA, tmB;
    const bool mapped = (ga.mode == kGemmTN ? encode_operand(&tmA, ga.A, ga.K, ga.M, ga.lda, kBK)
                                            : encode_operand(&tmA, ga.A, ga.M, ga.K, ga.lda, kBM)) &&
                        (ga.mode == kGemmNT ? encode_operand(&tmB, ga.B, ga.N, ga.K, ga.ldb, bn / 2)
                                            : encode_operand(&tmB, ga.B, ga.K, ga.N, ga.ldb, kBK / 2));
    if (!mapped) return cudaErrorInvalidValue;
    GemmArgs g = ga;
    auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    const bool f_ok = (g.ldc % 4 == 0) && al16(g.C) && al16(g.Cs) && al16(g.mul);
    const bool b_ok = (g.ldcb % 8 == 0) && al16(g.Cb);
    g.vec_ok = (f_ok ? 1 : 0) | (b_ok ? 2 : 0);
    // one cluster per pair of row blocks and column block, at most max_clusters
    const long long tiles = gemm_tiles(ga, bn);
    const int grid = 2 * (int)(tiles < max_clusters ? tiles : max_clusters);
    gemm_kernel(bn, ga.mode)<<<grid, kThreads, kGemmSmem, s>>>(tmA, tmB, g);
    return cudaGetLastError();
}

}  // namespace pamd

using namespace pamd;

namespace {

int gemm_entry(const void* A, const void* B, float* C, int32_t M, int32_t N, int32_t K, int32_t lda,
               int32_t ldb, int32_t ldc, int32_t reps, void* stream, float* ms_out) {
    if (!A || !B || !C || M < 1 || N < 1 || K < 1 || (K & 7) || (lda & 7) || (ldb & 7) ||
        lda < K || ldb < K || ldc < N || (reinterpret_cast<uintptr_t>(A) & 15) ||
        (reinterpret_cast<uintptr_t>(B) & 15) || reps < 1 || reps > 1000) {
        set_last_error("pamd_gemm_bf16: null pointer, or sizes / leading dimensions invalid "
                       "(K, lda, ldb multiples of 8; A, B 16-byte aligned; reps 1..1000)");
        return PAMD_EINVAL;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        set_last_error("pamd_gemm_bf16: no usable current device");
        return PAMD_ECUDA;
    }
    if (!on_device(A, dev) || !on_device(B, dev)) {
        set_last_error("pamd_gemm_bf16: A and B must be device memory of the current device");
        return PAMD_EINVAL;
    }
    // one status word per device, allocated on that device's first call
    static std::mutex mu;
    static int* status_of[kMaxDevices] = {};
    int* status = nullptr;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!status_of[dev] && cudaMalloc(&status_of[dev], sizeof(int)) != cudaSuccess) {
            status_of[dev] = nullptr;
            cudaGetLastError();
            set_last_error("pamd_gemm_bf16: status word");
            return PAMD_ENOMEM;
        }
        status = status_of[dev];
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    GemmArgs g{};
    g.A = A;
    g.B = B;
    g.C = C;
    g.M = M;
    g.N = N;
    g.K = K;
    g.lda = lda;
    g.ldb = ldb;
    g.ldc = ldc;
    g.epi = kEpiStore;
    g.status = status;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    cudaError_t e = cudaMemsetAsync(status, 0, sizeof(int), s);
    if (e == cudaSuccess && ms_out) e = cudaEventCreate(&ev[0]);
    if (e == cudaSuccess && ms_out) e = cudaEventCreate(&ev[1]);
    if (e == cudaSuccess && ms_out) e = cudaEventRecord(ev[0], s);
    for (int r = 0; r < reps && e == cudaSuccess; ++r) e = launch_gemm_bf16(g, s);
    if (e == cudaSuccess && ms_out) e = cudaEventRecord(ev[1], s);
    int st = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&st, status, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess && ms_out) {
        float ms = 0.0f;
        e = cudaEventElapsedTime(&ms, ev[0], ev[1]);
        *ms_out = ms / (float)reps;
    }
    for (cudaEvent_t x : ev)
        if (x) cudaEventDestroy(x);
    if (e != cudaSuccess) {
        set_last_error(std::string("pamd_gemm_bf16: ") + cudaGetErrorString(e));
        return PAMD_ECUDA;
    }
    if (st) {
        set_last_error("pamd_gemm_bf16: tensor-core pipeline timed out");
        return st;
    }
    return PAMD_OK;
}

}  // namespace

extern "C" int pamd_gemm_bf16(const void* A, const void* B, float* C, int32_t M, int32_t N,
                              int32_t K, int32_t lda, int32_t ldb, int32_t ldc, void* stream) {
    return gemm_entry(A, B, C, M, N, K, lda, ldb, ldc, 1, stream, nullptr);
}

extern "C" int pamd_gemm_bf16_time(const void* A, const void* B, float* C, int32_t M, int32_t N,
                                   int32_t K, int32_t lda, int32_t ldb, int32_t ldc, int32_t reps,
                                   void* stream, float* ms_out) {
    if (!ms_out) {
        set_last_error("pamd_gemm_bf16_time: null ms_out");
        return PAMD_EINVAL;
    }
    return gemm_entry(A, B, C, M, N, K, lda, ldb, ldc, reps, stream, ms_out);
}
