// Learned proposal network on the 5th-generation tensor cores (sm_103a).
//
// A 4-layer MLP of width 256 (input 32 features padded to 64, output 160
// padded to 256) maps a problem summary to a mixture over the normalised
// arrival time and to 16 space-time waypoints (the learned sampling branch of
// the method's GPU form). Weights are BF16 copies of FP32 master weights; every
// product accumulates in FP32.
//
// GEMM: D[M x N] = A[M x K] . B[N x K]^T, BF16 operands in the canonical
// no-swizzle tile order of the tensor cores (core matrices of 8 rows x 16
// bytes), FP32 accumulation in TMEM. Every BF16 matrix [R][K] (activations,
// their gradients, weights) is stored once, tiled: element (r, k) sits at
//   (((k / BW) * (R / 8) + r / 8) * (BW / 8) + (k % BW) / 8) * 64 + (r % 8) * 8 + k % 8
// with column blocks of BW = 128 (BW = 64 for the 64-wide input): the BW / 8
// core matrices of one 8-row group and one column block are consecutive, then
// the row groups, then the column blocks. So a 128-row x BW stage is one
// contiguous block for a K-major operand (the forward products and the input
// gradients, K = features), and the 64 rows of one column block are one
// contiguous block for an MN-major operand (the weight gradients, K = batch,
// which read the same activations without a transposed copy). Stages move
// into shared memory by bulk asynchronous copies (cp.async.bulk, completion
// on an mbarrier); one elected thread issues tcgen05.mma (kind::f16, M = 128,
// K = 16 per instruction) and tcgen05.commit releases a stage when its MMAs
// have read it; warps read the accumulator back with tcgen05.ld (warp w owns
// TMEM lanes 32 (w % 4) .. + 31 = tile rows) into a fused epilogue.
// Two kernels: chains of products over K <= 256 (all four forward layers: bias
// + ReLU, or bias with FP32 stores for the output layer; the three input
// gradients: ReLU mask and bias-gradient partials) keep a tile's activations in
// shared memory from product to product, one launch a chain (k_chain); the
// weight gradients (K = batch) run split-K with FP32 partials (k_gemm_wgrad).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "stp.h"
#include "stp_internal.cuh"

namespace stp {
namespace mlp {

constexpr int kIn = 32, kInP = 64, kHid = 256, kOut = 160, kOutP = 256;
constexpr int kMix = 8, kWp = 16, kWpDim = 8, kTgt = 130;
// Weight-gradient products: eight warps (warp w reads TMEM lane quadrant
// w % 4 and columns [(w / 4) N/2, (w / 4 + 1) N/2) in the epilogue), 64-wide
// K stages through a four-stage pipeline, one CTA per SM.
constexpr int kTileM = 128, kStageK = 64, kThreads = 256, kWStages = 4;
constexpr float kSMin = -7.f, kSMax = 2.f;
// Bias gradients: every 32 batch rows (a warp of an input-gradient epilogue,
// or a CTA of the loss kernel) write the column sums of their rows as one
// partial [256]; Adam adds the partials in a fixed order.

enum Mode { kHidden = 0, kOutput = 1, kBackward = 2, kWGrad = 3 };  // products, for the byte counts

// Tiled index (layout above) with column blocks of 1 << lbw (lbw 6 or 7).
__host__ __device__ inline size_t tixb(int r, int k, int R, int lbw) {
    const int cpb = 1 << (lbw - 3);  // core matrices per 8-row group and block
    return ((((size_t)(k >> lbw) * (size_t)(R >> 3) + (size_t)(r >> 3)) * (size_t)cpb +
             (size_t)((k >> 3) & (cpb - 1)))
            << 6) +
           (size_t)((r & 7) << 3) + (size_t)(k & 7);
}
__host__ __device__ constexpr int lbw_of(int K) { return K >= 128 ? 7 : 6; }
constexpr int kActLbw = 7;  // the 256-wide activations and gradients

// ---------------------------------------------------------------------------
// tcgen05 / TMEM helpers (inline PTX).
// ---------------------------------------------------------------------------
// Shared-memory matrix descriptor: start address, leading-dimension byte
// offset (between core matrices adjacent along K), stride-dimension byte
// offset (between core matrices adjacent along M or N), descriptor version 1,
// no swizzle. A K-major core matrix holds 8 rows (M or N) of 16 bytes of K;
// an MN-major one holds 8 rows of K of 16 bytes of M or N.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}
// Instruction descriptor, kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// The same with A and B MN-major (bit 15: A, bit 16: B).
__host__ __device__ constexpr uint32_t idesc_bf16_mn(int M, int N) {
    return idesc_bf16(M, N) | (1u << 15) | (1u << 16);
}
__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(da), "l"(db), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

struct GemmArgs {   // one layer's weight gradient
    const __nv_bfloat16* A;  // output gradient, tiled [RA][256] (M = its columns)
    int RA;                  // batch rows (multiple of 128)
    const __nv_bfloat16* B;  // layer input, tiled [RA][N] (N = its columns)
    int KT;                  // 64-row K stages (batch) in total
    int kt_per_split;        // split-K (blockIdx.z): stages [z*kps, min(KT, (z+1)*kps))
    float* out_f;            // FP32 partials [splits][m_valid][ld_f]
    int ld_f;
    int m_valid;             // rows written
    int* err;
};

struct WGradArgs {
    GemmArgs layer[3];  // blockIdx.y
};

// Column sums over the 32 lanes of 16 per-lane values by recursive halving:
// at offset o each lane keeps the half of its columns selected by its lane
// bit and adds its partner's copy of them, so lane l ends with the sum of
// column l & 15 over all 32 lanes (16 shuffles instead of 80).
__device__ __forceinline__ float warp_colsum16(float (&v)[16]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 8, n = 8; o >= 1; o >>= 1, n >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (i < n) {
                const float send = up ? v[i] : v[i + n];
                const float keep = up ? v[i + n] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 16);
}

// Split-K: a launch is one wave, one CTA per SM. More splits than that cost a
// second wave and a second 256 KB of partials per CTA, written here and read by
// Adam (layers 2-4 at 65,536 rows, 152 SMs: 66 splits 59 us, 25 splits 38 us,
// and 200 MB of operands at the copy rate are 30 us). One thread copies, another
// issues the MMAs: a single one waits for each stage's MMAs before it queues the
// next.
//
// Weight gradient dW = dT^T . X: M = 128 output features of tile blockIdx.x
// (column block of dT), N = the layer's input features, K = the batch rows of
// split blockIdx.z. Both operands are MN-major: a stage is 64 batch rows, so an A tile is one
// contiguous 16 KB piece of dT's column block and B one piece of 8 row groups
// per column block of X (one MMA of N = BW per tile, block and K step). The
// dynamic shared memory ends with a guard region so that every
// descriptor-addressed read stays inside the allocation.
template <int N, int LBWB>
__host__ __device__ constexpr int wgrad_smem_bytes() {
    return 1024 + kWStages * (kTileM * kStageK * 2 + N * kStageK * 2) + 21 * 2048 + 256 - (1 << LBWB) * kStageK * 2;
}
template <int N, int LBWB>
__global__ void __launch_bounds__(kThreads, 1) k_gemm_wgrad(const __grid_constant__ WGradArgs all) {
    const GemmArgs& g = all.layer[blockIdx.y];
    constexpr int kStages = kWStages;
    constexpr int kBW = 1 << LBWB;                      // B column block
    constexpr int kNB = N / kBW;                        // B blocks (MMAs per K step and tile)
    constexpr uint32_t kABytes = kTileM * kStageK * 2;  // 16 KB
    constexpr uint32_t kBBlk = kBW * kStageK * 2;
    constexpr uint32_t kBBytes = kNB * kBBlk;
    constexpr uint32_t kTmemCols = N < 32 ? 32 : N;
    constexpr uint32_t kIdesc = idesc_bf16_mn(kTileM, kBW);
    constexpr uint32_t kALbo = 16 * 128, kBLbo = (kBW / 8) * 128;  // one 8-row group of a column block
    static_assert(N % kBW == 0, "whole column blocks");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[kStages], empty[kStages], done;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int fail_sh;

    unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sA = smem;
    unsigned char* sB = smem + kStages * kABytes;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int z = blockIdx.z;
    const int kt0 = z * g.kt_per_split;
    const int kt1 = min(g.KT, kt0 + g.kt_per_split);
    const int nk = kt1 > kt0 ? kt1 - kt0 : 0;

    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        fail_sh = 0;
    }
    if (warp == 0) tmem_alloc(&tmem_base_sh, kTmemCols);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = tmem_base_sh;

    if (tid == 32 && nk > 0) {
        const size_t rg = (size_t)(g.RA >> 3);
        int it = 0;
        for (; it < nk; ++it) {
            const int s = it % kStages;
            if (it >= kStages && !mbar_wait(&empty[s], ((it / kStages) - 1) & 1)) {
                fail_sh = 1;
                if (g.err) atomicOr(g.err, kErrTimeout);
                break;
            }
            const size_t kg = (size_t)(kt0 + it) * (kStageK / 8);  // first 8-row group of the stage
            mbar_expect_tx(&full[s], kABytes + kBBytes);
            bulk_g2s(sA + s * kABytes, g.A + (((size_t)blockIdx.x * rg + kg) * 16) * 64, kABytes, &full[s]);
#pragma unroll
            for (int nb = 0; nb < kNB; ++nb)
                bulk_g2s(sB + s * kBBytes + nb * kBBlk, g.B + (((size_t)nb * rg + kg) * (kBW / 8)) * 64, kBBlk, &full[s]);
        }
        // The last copy into each stage has landed before the CTA may exit.
        for (int s = 0; s < kStages && s < it; ++s) {
            const int j = s + ((it - 1 - s) / kStages) * kStages;
            mbar_wait(&full[s], (j / kStages) & 1);
        }
    } else if (tid == 0 && nk > 0) {
        bool ok = true;
        for (int j = 0; j < nk && ok; ++j) {
            const int s = j % kStages;
            ok = mbar_wait(&full[s], (j / kStages) & 1);
            if (!ok) break;
            fence_after_sync();
            const uint32_t a0 = smem_u32(sA + s * kABytes), b0 = smem_u32(sB + s * kBBytes);
#pragma unroll
            for (int ks = 0; ks < kStageK / 16; ++ks) {
                // K step of 16 batch rows = two 8-row groups.
                const uint64_t da = smem_desc(a0 + ks * 2 * kALbo, kALbo, 128);
#pragma unroll
                for (int nb = 0; nb < kNB; ++nb) {
                    const uint64_t db = smem_desc(b0 + nb * kBBlk + ks * 2 * kBLbo, kBLbo, 128);
                    mma_bf16(tmem + (uint32_t)(nb * kBW), da, db, kIdesc, (j > 0 || ks > 0) ? 1u : 0u);
                }
            }
            mma_commit(&empty[s]);
        }
        // Always close with a commit so that `done` tracks every issued MMA.
        mma_commit(&done);
        if (!ok) {
            fail_sh = 1;
            if (g.err) atomicOr(g.err, kErrTimeout);
        }
    }
    __syncthreads();
    bool have = nk > 0;
    if (have) {
        if (!mbar_wait(&done, 0)) {
            if (lane == 0 && g.err) atomicOr(g.err, kErrTimeout);
            fail_sh = 1;
        }
    }
    fence_after_sync();
    __syncthreads();
    if (fail_sh) have = false;

    // Epilogue: thread (warp, lane) owns row 32 (warp % 4) + lane of the
    // tile and half of the columns; FP32 partial rows of split z.
    const int quad = warp & 3;
    const int cb = (warp >> 2) * (N / 2), ce = cb + N / 2;
    const int r = (int)blockIdx.x * kTileM + 32 * quad + lane;
    const uint32_t trow = tmem + ((uint32_t)(32 * quad) << 16);
#pragma unroll 1
    for (int c0 = cb; c0 < ce; c0 += 16) {
        float v[16];
        if (have) tmem_ld16(trow + (uint32_t)c0, v);
        else {
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = 0.f;
        }
        if (r < g.m_valid) {
            float4* o = reinterpret_cast<float4*>(g.out_f + ((size_t)z * g.m_valid + r) * g.ld_f + c0);
#pragma unroll
            for (int q = 0; q < 4; ++q) o[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        }
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

// ---------------------------------------------------------------------------
// Chains of products over a tile's rows, one launch each: the forward pass
// (input packing, three hidden layers, the output layer) and the input
// gradients of the backward pass (three products).
//
// Persistent, one CTA per SM. A CTA carries two 128-row tiles at a time, slot 0
// and 1, through every layer: a tile's activations stay in one 64 KB buffer of
// shared memory between the layers (128 x 256 BF16 in the tiled order; a layer's
// result overwrites its operand once all its MMAs are done), only the weights
// stream, 32 KB stages (column block kb of the operand, rows of output half h)
// from L2 through a ring. The products run slot 0 layer l, slot 1 layer l, slot 0
// layer l + 1, ..., so one slot's epilogue overlaps the other's products: a
// single tile is a chain of product, epilogue, product in which the tensor
// cores idle half of the time (5,200 cycles a layer measured against 2,048 of
// MMAs; bulk copies deliver 82 bytes a cycle and SM, 2.5 times what is needed).
//
// Warps 0-7 run slot 0's epilogues and 8-15 slot 1's (warp w of a slot: TMEM
// lanes 32 (w % 4) .. + 31 = tile rows, every other 16-column chunk from w / 4),
// warp 16 lane 0 issues the copies, lanes 0 of warps 17 and 18 the MMAs of output
// half 0 and 1 (one thread alone leaves gaps between its parts; both pass every
// stage). Half of a tile's operand is announced at a time, so that the next
// product starts on column block 0 while the epilogue is at block 1. Where the
// activations (or their gradients) are needed later they leave the buffers by
// bulk copies, 32 KB contiguous each, while the next layer runs. Every wait is
// bounded; a role whose wait runs out sets the error flag, the others stop
// working (the epilogue warps keep meeting at their barriers), and the CTA
// drains its copies and frees its TMEM.
//
// Measured, us with events: forward at 65,536 rows 40 (four launches with the
// weights resident and the activations through memory: 50), at 128 rows 18 (28);
// input gradients at 65,536 rows 56. Bound at 65,536 rows by shared memory: 448 KB
// a tile and layer (operands of N = 128 MMAs, weight stages, epilogue) at 128
// bytes a cycle are 3,500 cycles, and each slot's product and epilogue alternate
// at about 3,500 cycles each.
// ---------------------------------------------------------------------------
constexpr int kEpiWarps = 8, kEpiThreads = 32 * kEpiWarps;  // of a slot
constexpr int kChainThreads = 2 * kEpiThreads + 3 * 32;
constexpr int kChainRing = 3;                      // weight stages
constexpr uint32_t kBlk = kTileM * 128 * 2;        // one 128 x 128 block: 32 KB
constexpr int kOutPad = 32 + 4;                    // output staging: 32 columns at a time, padded row
constexpr int kChainSmem = 1024 + (4 + kChainRing) * (int)kBlk;

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Generic-proxy writes of shared memory before asynchronous reads of it.
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, unsigned bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void epi_sync(int slot) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + slot), "n"(kEpiThreads) : "memory");
}
// 16 accumulator columns without waiting for them (tmem_wait).
__device__ __forceinline__ void tmem_ld16_async(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// Keeps the uses of loaded columns behind tmem_wait.
__device__ __forceinline__ void tmem_use(uint32_t (&r)[16]) {
    asm volatile(""
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15]));
}

struct ChainArgs {
    int tiles, RA, B;          // 128-row tiles, padded rows (128 tiles), rows of the batch
    const __nv_bfloat16* W[4]; // weight operands, tiled [256][K] (layer order of the chain)
    const float* bias[4];      // forward
    const float* X;            // forward: features [B][32], 16-byte aligned
    __nv_bfloat16* xt;         // forward with stores: packed features, tiled [RA][64]
    const __nv_bfloat16* A0;   // backward: gradient of the outputs, tiled [RA][256]
    const __nv_bfloat16* act[3];  // backward: forward activation whose sign masks product l
    __nv_bfloat16* out[3];     // tiled [RA][256] results of products 0..2
    float* bpart[3];           // backward: bias-gradient partials [RA / 32][256]
    float* Y;                  // forward: outputs [B][160], 16-byte aligned
    int* err;
};

// BACK: the input gradients; else the forward pass, storing the activations if STORE.
template <bool BACK, bool STORE>
__global__ void __launch_bounds__(kChainThreads, 1) k_chain(const __grid_constant__ ChainArgs g) {
    constexpr int kL = BACK ? 3 : 4;  // products per tile
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t wfull[kChainRing], wempty[kChainRing];
    __shared__ __align__(8) uint64_t afull[2][2];  // column block kb of slot j's operand written (its accumulator columns read)
    __shared__ __align__(8) uint64_t dfull[2];  // accumulator of slot j complete
    __shared__ __align__(8) uint64_t done;
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int abort_sh;
    unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sW = smem + 4 * kBlk;  // the slots' buffers (two blocks each), then the ring
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int s = 0; s < kChainRing; ++s) {
            mbar_init(&wfull[s], 1);
            mbar_init(&wempty[s], 2);  // both issuers pass every stage, so neither can mistake its phase
        }
        for (int j = 0; j < 2; ++j) {
            for (int kb = 0; kb < 2; ++kb) mbar_init(&afull[j][kb], kEpiWarps);
            mbar_init(&dfull[j], 2);
        }
        mbar_init(&done, 2);
        abort_sh = 0;
    }
    if (warp == 0) tmem_alloc(&tmem_base_sh, 512);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = tmem_base_sh;
    auto fail = [&]() {
        abort_sh = 1;
        if (g.err) atomicOr(g.err, kErrTimeout);
    };
    auto half_rows = [](int l) { return !BACK && l == 3 ? kOut / 2 : 128; };
    auto kblocks = [](int l) { return !BACK && l == 0 ? 1 : 2; };
    const size_t rgA = (size_t)(g.RA >> 3);
    // Tiles of the CTA: pair p holds tiles c + 2 p grid (slot 0) and c + (2 p + 1) grid.
    const int step = (int)gridDim.x;

    if (warp == 2 * kEpiWarps) {
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            // One stage of `bytes` from src.
            auto stage = [&](const void* src, uint32_t bytes) {
                const int s = it % kChainRing;
                if (ok && it >= kChainRing && !mbar_wait(&wempty[s], ((it / kChainRing) - 1) & 1)) {
                    fail();
                    ok = false;
                }
                if (!ok || abort_sh) {
                    ok = false;
                    return;
                }
                mbar_expect_tx(&wfull[s], bytes);
                bulk_g2s(sW + s * kBlk, src, bytes, &wfull[s]);
                ++it;
            };
            for (int t0 = blockIdx.x; ok && t0 < g.tiles; t0 += 2 * step) {
                for (int l = 0; ok && l < kL; ++l) {
                    const int rows = half_rows(l), bw = !BACK && l == 0 ? 64 : 128;
                    for (int j = 0; ok && j < 2; ++j) {
                        const int t = t0 + j * step;
                        if (t >= g.tiles) break;
                        for (int kb = 0; ok && kb < kblocks(l); ++kb) {
                            // Backward, first product: its operand A streams too.
                            if (BACK && l == 0)
                                stage(g.A0 + (((size_t)kb * rgA + (size_t)t * (kTileM >> 3)) * 16) * 64, kBlk);
                            for (int h = 0; h < 2; ++h)
                                stage(g.W[l] + (((size_t)kb * 32 + (size_t)h * (rows >> 3)) * (bw / 8)) * 64,
                                      (uint32_t)(rows * bw * 2));
                        }
                    }
                }
            }
            // The last copy issued into each stage has landed before the CTA may exit.
            for (int s = 0; s < kChainRing && s < it; ++s) {
                const int j = s + ((it - 1 - s) / kChainRing) * kChainRing;
                mbar_wait(&wfull[s], (j / kChainRing) & 1);
            }
        }
    } else if (warp > 2 * kEpiWarps) {
        if (lane == 0) {
            const int h = warp - 2 * kEpiWarps - 1;  // output half
            int it = 0;                              // ring stages
            unsigned an[2] = {0, 0};                 // operands of each slot
            bool ok = true;
            auto wait = [&](uint64_t* bar, unsigned parity) {
                if (ok && !mbar_wait(bar, parity)) {
                    fail();
                    ok = false;
                }
            };
            for (int t0 = blockIdx.x; ok && !abort_sh && t0 < g.tiles; t0 += 2 * step) {
                for (int l = 0; ok && l < kL; ++l) {
                    const int rows = half_rows(l);
                    const uint32_t idesc = rows == 128 ? idesc_bf16(kTileM, 128) : idesc_bf16(kTileM, kOut / 2);
                    const uint32_t sbo = !BACK && l == 0 ? 1024u : 2048u;
                    for (int j = 0; ok && j < 2; ++j) {
                        if (t0 + j * step >= g.tiles) break;
                        const uint32_t dst = tmem + (uint32_t)(256 * j + 128 * h);
                        for (int kb = 0; ok && kb < kblocks(l); ++kb) {
                            // The operand's block is in place (the first product of the
                            // backward chain: the accumulator is free), and for output half 1
                            // its accumulator, which the epilogue reads with block 1.
                            wait(&afull[j][kb], an[j] & 1);
                            if (kb == 0 && (h == 1 || kblocks(l) == 1)) wait(&afull[j][1], an[j] & 1);
                            uint32_t a0 = smem_u32(smem + (2 * j + kb) * kBlk);
                            int as = -1;
                            if (BACK && l == 0) {
                                as = it % kChainRing;
                                wait(&wfull[as], (it / kChainRing) & 1);
                                a0 = smem_u32(sW + as * kBlk);
                                ++it;
                            }
                            // This half's stage is the h-th of the two; the other is only passed.
                            for (int hh = 0; ok && hh < 2; ++hh, ++it) {
                                const int s = it % kChainRing;
                                wait(&wfull[s], (it / kChainRing) & 1);
                                if (!ok) break;
                                if (hh != h) {
                                    mbar_arrive(&wempty[s]);
                                    continue;
                                }
                                fence_after_sync();
                                const uint64_t da = smem_desc(a0, 128, sbo), db = smem_desc(smem_u32(sW + s * kBlk), 128, sbo);
                                // A K step is 256 bytes on: 16 in the descriptors' address units.
                                // Two steps for the 32 features of the 64-wide input block and for
                                // the 32 outputs of the output gradient's second block.
                                mma_bf16(dst, da, db, idesc, kb > 0 ? 1u : 0u);
                                mma_bf16(dst, da + 16, db + 16, idesc, 1u);
                                if (!(!BACK && l == 0) && !(BACK && l == 0 && kb == 1)) {
#pragma unroll
                                    for (int ks = 2; ks < 8; ++ks) mma_bf16(dst, da + 16 * ks, db + 16 * ks, idesc, 1u);
                                }
                                mma_commit(&wempty[s]);
                            }
                            if (!ok) break;
                            if (as >= 0) mma_commit(&wempty[as]);
                            if (kb == kblocks(l) - 1) mma_commit(&dfull[j]);
                        }
                        ++an[j];
                    }
                }
            }
            // Every MMA has completed before the TMEM is freed.
            mma_commit(&done);
            if (!mbar_wait(&done, 0)) fail();
        }
    } else {
        const int slot = warp / kEpiWarps, w = warp % kEpiWarps, stid = tid % kEpiThreads;
        const int quad = w & 3, hw = w >> 2;
        const int row = 32 * quad + lane;  // of the tile
        unsigned char* blk = smem + 2 * slot * kBlk;
        const uint32_t trow = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(256 * slot);
        bool ok = true;
        unsigned uses = 0;  // products of the slot
        // The accumulator is complete. A warp whose wait runs out keeps meeting the
        // others at the barriers.
        auto wait_acc = [&]() {
            const bool good = ok && !abort_sh && mbar_wait(&dfull[slot], uses & 1);
            if (ok && !__all_sync(0xffffffffu, good)) {
                if (lane == 0) fail();
                ok = false;
            }
            ++uses;
        };
        // Features of a tile: thread i of the slot holds pieces i, i + 256, ... of its
        // [128][64] block (zero padded), loaded ahead.
        constexpr int kPieces = kTileM * (kInP / 8) / kEpiThreads;
        uint4 xin[kPieces];
        auto load_x = [&](int t) {
            if constexpr (!BACK) {
#pragma unroll
                for (int q = 0; q < kPieces; ++q) {
                    const int i = stid + q * kEpiThreads;
                    const int n = t * kTileM + 8 * (i >> 6) + (i & 7), c = (i >> 3) & 7;
                    float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u;
                    if (t < g.tiles && n < g.B && 8 * c < kIn) {
                        const float4* src = reinterpret_cast<const float4*>(g.X + (size_t)n * kIn + 8 * c);
                        u = __ldg(src);
                        v = __ldg(src + 1);
                    }
                    __align__(16) __nv_bfloat162 b[4] = {__floats2bfloat162_rn(u.x, u.y), __floats2bfloat162_rn(u.z, u.w),
                                                         __floats2bfloat162_rn(v.x, v.y), __floats2bfloat162_rn(v.z, v.w)};
                    xin[q] = *reinterpret_cast<const uint4*>(b);
                }
            }
        };
        auto pack_x = [&](int t) {
            if constexpr (!BACK) {
#pragma unroll
                for (int q = 0; q < kPieces; ++q)
                    *reinterpret_cast<uint4*>(blk + (size_t)(stid + q * kEpiThreads) * 16) = xin[q];
                fence_async_smem();
                if (STORE) {
                    epi_sync(slot);
                    if (stid == 0) {
                        bulk_s2g(g.xt + (size_t)t * kTileM * kInP, blk, kTileM * kInP * 2);
                        bulk_commit();
                    }
                }
            }
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&afull[slot][0]);
                mbar_arrive(&afull[slot][1]);
            }
        };
        int t = (int)blockIdx.x + slot * step;
        load_x(t);
        if (t < g.tiles) pack_x(t);
        for (; t < g.tiles; t += 2 * step) {
#pragma unroll 1
            for (int l = 0; l < kL; ++l) {
                if (BACK || l < 3) {
                    // Two chunks of 16 columns at a time; the mask or the biases of the next pair
                    // are loaded before the current one is stored (a load on demand from L2 made a
                    // pair 900 cycles).
                    uint4 pa[BACK ? 2 : 1][2];
                    float4 bias[BACK ? 1 : 2][4];
                    auto ahead = [&](int pr) {
#pragma unroll
                        for (int ci = 0; ci < 2; ++ci) {
                            const int c = 16 * (hw + 2 * (2 * pr + ci));  // column
                            if constexpr (BACK) {
#pragma unroll
                                for (int hh = 0; hh < 2; ++hh)
                                    pa[ci][hh] = *reinterpret_cast<const uint4*>(
                                        g.act[l] + tixb(t * kTileM + row, c + 8 * hh, g.RA, kActLbw));
                            } else {
#pragma unroll
                                for (int q = 0; q < 4; ++q)
                                    bias[ci][q] = __ldg(reinterpret_cast<const float4*>(g.bias[l] + c) + q);
                            }
                        }
                    };
                    ahead(0);
                    // The copies out of the buffer have read it.
                    if (STORE && stid == 0) bulk_wait_read<0>();
                    if (STORE) epi_sync(slot);
                    wait_acc();
                    if (ok) fence_after_sync();
#pragma unroll 1
                    for (int pr = 0; pr < 4; ++pr) {
                        if (ok) {
                            uint32_t v[2][16];
#pragma unroll
                            for (int ci = 0; ci < 2; ++ci)
                                tmem_ld16_async(trow + (uint32_t)(16 * (hw + 2 * (2 * pr + ci))), v[ci]);
                            tmem_wait();
#pragma unroll
                            for (int ci = 0; ci < 2; ++ci) tmem_use(v[ci]);
                            float x[2][16];
#pragma unroll
                            for (int ci = 0; ci < 2; ++ci) {
#pragma unroll
                                for (int q = 0; q < 16; ++q) x[ci][q] = __uint_as_float(v[ci][q]);
                                if constexpr (BACK) {
#pragma unroll
                                    for (int hh = 0; hh < 2; ++hh) {
                                        __align__(16) __nv_bfloat16 a[8];
                                        *reinterpret_cast<uint4*>(a) = pa[ci][hh];
#pragma unroll
                                        for (int q = 0; q < 8; ++q)
                                            if (!(__bfloat162float(a[q]) > 0.f)) x[ci][8 * hh + q] = 0.f;
                                    }
                                } else {
#pragma unroll
                                    for (int q = 0; q < 4; ++q) {
                                        const float4 b = bias[ci][q];
                                        x[ci][4 * q] = fmaxf(x[ci][4 * q] + b.x, 0.f);
                                        x[ci][4 * q + 1] = fmaxf(x[ci][4 * q + 1] + b.y, 0.f);
                                        x[ci][4 * q + 2] = fmaxf(x[ci][4 * q + 2] + b.z, 0.f);
                                        x[ci][4 * q + 3] = fmaxf(x[ci][4 * q + 3] + b.w, 0.f);
                                    }
                                }
                            }
                            if (pr < 3) ahead(pr + 1);
#pragma unroll
                            for (int ci = 0; ci < 2; ++ci) {
                                const int c = 16 * (hw + 2 * (2 * pr + ci));
                                unsigned char* dst = blk + (c >> 7) * kBlk + (row >> 3) * 2048 + ((c & 127) >> 3) * 128 +
                                                     (row & 7) * 16;
#pragma unroll
                                for (int hh = 0; hh < 2; ++hh) {
                                    __align__(16) __nv_bfloat162 b[4];
#pragma unroll
                                    for (int q = 0; q < 4; ++q)
                                        b[q] = __floats2bfloat162_rn(x[ci][8 * hh + 2 * q], x[ci][8 * hh + 2 * q + 1]);
                                    *reinterpret_cast<uint4*>(dst + 128 * hh) = *reinterpret_cast<const uint4*>(b);
                                }
                                if constexpr (BACK) {
                                    // Bias-gradient partial of these 32 rows, each element by one warp.
                                    const float cs = warp_colsum16(x[ci]);
                                    if (lane < 16) g.bpart[l][(size_t)(t * 4 + quad) * 256 + c + lane] = cs;
                                }
                            }
                        }
                        if (pr & 1) {
                            // Half of the next product's operand, its first block or its second (the
                            // backward chain's last result only leaves: its arrivals free the
                            // accumulator for the next tile).
                            fence_before_sync();
                            fence_async_smem();
                            __syncwarp();
                            if (lane == 0 && (!BACK || l < kL - 1 || t + 2 * step < g.tiles)) mbar_arrive(&afull[slot][pr >> 1]);
                        }
                    }
                    if (STORE) {
                        epi_sync(slot);
                        if (stid == 0) {
                            for (int kb = 0; kb < 2; ++kb)
                                bulk_s2g(g.out[l] + (((size_t)kb * rgA + (size_t)t * (kTileM >> 3)) * 16) * 64,
                                         blk + kb * kBlk, kBlk);
                            bulk_commit();
                        }
                    }
                } else {
                    // Output layer: warps 0-3 of the slot take half 0, warps 4-7 half 1 (80
                    // columns each: 32, 32 and 16), staged in the slot's buffer (its operand is
                    // done with). The biases join on the way out, where a lane keeps its columns.
                    float4 bias[3];
#pragma unroll
                    for (int q = 0; q < 3; ++q)
                        bias[q] = __ldg(reinterpret_cast<const float4*>(g.bias[l] + (kOut / 2) * hw + 32 * q) +
                                        (q < 2 ? lane & 7 : lane & 3));
                    load_x(t + 2 * step);
                    if (STORE && stid == 0) bulk_wait_read<0>();
                    if (STORE) epi_sync(slot);
                    wait_acc();
                    if (ok) {
                        fence_after_sync();
                        float* so = reinterpret_cast<float*>(blk) + w * 32 * kOutPad;
                        const int r0 = t * kTileM + 32 * quad;
                        auto part = [&](auto first, auto count) {
                            constexpr int c0 = decltype(first)::value, cn = decltype(count)::value;  // chunks of 16
                            uint32_t v[cn][16];
#pragma unroll
                            for (int c = 0; c < cn; ++c)
                                tmem_ld16_async(trow + (uint32_t)(128 * hw + 16 * (c0 + c)), v[c]);
                            tmem_wait();
#pragma unroll
                            for (int c = 0; c < cn; ++c) {
                                tmem_use(v[c]);
#pragma unroll
                                for (int q = 0; q < 4; ++q)
                                    *reinterpret_cast<uint4*>(so + lane * kOutPad + 16 * c + 4 * q) =
                                        make_uint4(v[c][4 * q], v[c][4 * q + 1], v[c][4 * q + 2], v[c][4 * q + 3]);
                            }
                            __syncwarp();
                            // 4 cn lanes write the 64 cn contiguous bytes of a row.
                            constexpr int kRows = 32 / (4 * cn);
                            const int rr = lane / (4 * cn), cc = lane % (4 * cn);
                            const float4 b = bias[c0 / 2];
                            float* y = g.Y + (size_t)(r0 + rr) * kOut + (kOut / 2) * hw + 16 * c0 + 4 * cc;
#pragma unroll
                            for (int i = 0; i < 32 / kRows; ++i) {
                                const float4 u = *reinterpret_cast<const float4*>(so + (rr + kRows * i) * kOutPad + 4 * cc);
                                if (r0 + rr + kRows * i < g.B)
                                    *reinterpret_cast<float4*>(y + (size_t)(kRows * i) * kOut) =
                                        make_float4(u.x + b.x, u.y + b.y, u.z + b.z, u.w + b.w);
                            }
                            __syncwarp();
                        };
                        part(std::integral_constant<int, 0>(), std::integral_constant<int, 2>());
                        part(std::integral_constant<int, 2>(), std::integral_constant<int, 2>());
                        part(std::integral_constant<int, 4>(), std::integral_constant<int, 1>());
                        fence_before_sync();
                    }
                    // The next tile's features take the buffer once every warp is done.
                    epi_sync(slot);
                    if (t + 2 * step < g.tiles) pack_x(t + 2 * step);
                }
            }
        }
        if (STORE && stid == 0) bulk_wait_all();
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------------------
// Elementwise kernels.
// ---------------------------------------------------------------------------
// Per-sample loss (mixture NLL of tau + masked waypoint MSE) and dL/dy / B.
// A CTA takes 32 consecutive rows (one bias-gradient partial): their network
// outputs and targets are staged in shared memory by coalesced 16-byte loads
// (the 32 target rows are one contiguous block), four threads share a row
// (mixture components p and p + 4, waypoint elements p, p + 4, ...; the row's
// reductions are shuffles within the four lanes), the gradient overwrites
// the staged outputs, and the CTA then writes its BF16 tiles with consecutive
// threads on consecutive 16-byte pieces, the 256 column sums of its rows, and
// the sum of its row losses.
constexpr int kLossRows = 32, kLossThreads = 128;
constexpr int kLossYS = kOut + 4;                 // staged row stride (floats)
constexpr int kOutUsed = 3 * kMix + kWp * kWpDim;  // 152 network outputs in use
static_assert(kLossThreads == 4 * kLossRows, "four threads per row");
static_assert(kMix == 8 && kWpDim == 8 && (kWp * kWpDim) % 4 == 0, "components and elements split over four lanes");
static_assert((kLossRows * kTgt) % 4 == 0 && (kLossYS * 4) % 16 == 0, "16-byte staging");

__global__ void __launch_bounds__(kLossThreads) k_loss(const float* __restrict__ Y, const float* __restrict__ T,
                                                       int B, float* bpart, __nv_bfloat16* dyt, int Bp,
                                                       double* loss) {
    __shared__ __align__(16) float sy[kLossRows * kLossYS];
    __shared__ __align__(16) float st[kLossRows * kTgt];
    const int tid = threadIdx.x;
    const int n0 = blockIdx.x * kLossRows;
    const int nrow = max(0, min(kLossRows, B - n0));  // rows of this CTA inside the batch
    constexpr int kYv = kOut / 4;                     // float4 per output row
    constexpr int kTv = kLossRows * kTgt / 4;         // float4 of a full target block
    if (nrow == kLossRows) {
        // Row n0 of the targets starts at byte 520 n0, a multiple of 16 (n0 % 32 == 0).
        float4 yv[kLossRows * kYv / kLossThreads];
        float4 tv[(kTv + kLossThreads - 1) / kLossThreads];
        const float4* t4 = reinterpret_cast<const float4*>(T + (size_t)n0 * kTgt);
#pragma unroll
        for (int q = 0; q < kLossRows * kYv / kLossThreads; ++q) {
            const int i = tid + q * kLossThreads, r = i / kYv, c = i % kYv;
            yv[q] = __ldg(reinterpret_cast<const float4*>(Y + (size_t)(n0 + r) * kOut) + c);
        }
#pragma unroll
        for (int q = 0; q < (kTv + kLossThreads - 1) / kLossThreads; ++q) {
            const int i = tid + q * kLossThreads;
            if (i < kTv) tv[q] = __ldg(t4 + i);
        }
#pragma unroll
        for (int q = 0; q < kLossRows * kYv / kLossThreads; ++q) {
            const int i = tid + q * kLossThreads, r = i / kYv, c = i % kYv;
            *reinterpret_cast<float4*>(sy + r * kLossYS + 4 * c) = yv[q];
        }
#pragma unroll
        for (int q = 0; q < (kTv + kLossThreads - 1) / kLossThreads; ++q) {
            const int i = tid + q * kLossThreads;
            if (i < kTv) reinterpret_cast<float4*>(st)[i] = tv[q];
        }
    } else if (nrow > 0) {  // the batch's last, partial CTA
        for (int i = tid; i < nrow * kYv; i += kLossThreads) {
            const int r = i / kYv, c = i % kYv;
            *reinterpret_cast<float4*>(sy + r * kLossYS + 4 * c) =
                __ldg(reinterpret_cast<const float4*>(Y + (size_t)(n0 + r) * kOut) + c);
        }
        for (int i = tid; i < nrow * kTgt; i += kLossThreads) st[i] = __ldg(T + (size_t)n0 * kTgt + i);
    }
    __syncthreads();

    // Every lane runs the row arithmetic (the shuffles need the whole warp);
    // rows past the batch read zeros and write nothing.
    const int r = tid >> 2, p = tid & 3;
    const bool valid = r < nrow;
    float* y = sy + r * kLossYS;
    const float* t = st + r * kTgt;
    const float invB = 1.f / (float)B;
    const float tau = valid ? t[0] : 0.f;
    const int dof = valid ? (int)t[kTgt - 1] : 0;
    // Mixture over tau: this thread's components p and p + 4.
    float a[2], l[2], z[2], sig[2], sr[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int k = p + 4 * h;
        a[h] = valid ? y[k] : 0.f;
        sr[h] = valid ? y[2 * kMix + k] : 0.f;
        const float mu = valid ? y[kMix + k] : 0.f;
        const float s = fminf(fmaxf(sr[h], kSMin), kSMax);
        sig[h] = expf(s);
        z[h] = (tau - mu) / sig[h];
        l[h] = -0.5f * z[h] * z[h] - s - 0.91893853320467274f;  // log N(tau; mu, sig)
    }
    float amax = fmaxf(a[0], a[1]);
    amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
    amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));
    float asum = expf(a[0] - amax) + expf(a[1] - amax);
    asum += __shfl_xor_sync(0xffffffffu, asum, 1);
    asum += __shfl_xor_sync(0xffffffffu, asum, 2);
    const float lse_a = amax + logf(asum);
#pragma unroll
    for (int h = 0; h < 2; ++h) l[h] += a[h] - lse_a;
    float lmax = fmaxf(l[0], l[1]);
    lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, 1));
    lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, 2));
    float lsum = expf(l[0] - lmax) + expf(l[1] - lmax);
    lsum += __shfl_xor_sync(0xffffffffu, lsum, 1);
    lsum += __shfl_xor_sync(0xffffffffu, lsum, 2);
    const float lse_l = lmax + logf(lsum);
    // Waypoints: element e = 4 m + p (waypoint e / 8, coordinate e % 8);
    // the coordinates in use are the arm's dof joints and the time.
    const float cnt = (float)(kWp * (dof + 1));
    const float gscale = 2.f * invB / cnt;  // d(mse / cnt) / B per unit error
    float mse = 0.f;
    if (valid) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = p + 4 * h;
            const float gam = expf(l[h] - lse_l);
            const float pi = expf(a[h] - lse_a);
            y[k] = (pi - gam) * invB;
            y[kMix + k] = -gam * z[h] / sig[h] * invB;
            y[2 * kMix + k] = (sr[h] >= kSMin && sr[h] <= kSMax) ? gam * (1.f - z[h] * z[h]) * invB : 0.f;
        }
#pragma unroll 8
        for (int m = 0; m < kWp * kWpDim / 4; ++m) {
            const int e = 4 * m + p, j = e & (kWpDim - 1);
            const int o = 3 * kMix + e;
            float g = 0.f;
            if (j < dof || j == kWpDim - 1) {
                const float d = y[o] - t[1 + e];
                mse += d * d;
                g = d * gscale;
            }
            y[o] = g;
        }
    }
    mse += __shfl_xor_sync(0xffffffffu, mse, 1);
    mse += __shfl_xor_sync(0xffffffffu, mse, 2);
    // The rows' losses, summed in double (lanes 0, 4, ... hold one row each).
    double row = valid && p == 0 ? (double)(-lse_l + mse / cnt) : 0.0;
#pragma unroll
    for (int o = 16; o >= 4; o >>= 1) row += __shfl_xor_sync(0xffffffffu, row, o);
    __shared__ double sloss[kLossThreads / 32];
    if ((tid & 31) == 0) sloss[tid >> 5] = row;
    __syncthreads();
    if (tid == 0) {
        double sum = 0.0;
        for (int w = 0; w < kLossThreads / 32; ++w) sum += sloss[w];
        loss[blockIdx.x] = sum;
    }

    // dL/dy as BF16 tiles: piece c = (s, core matrix cm, row i) holds columns
    // 128 (s & 1) + 8 cm .. + 7 of row 8 (s >> 1) + i; the 128 pieces of one
    // (s, cm) range are 2 KB of contiguous memory.
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        const int c = tid + s * kLossThreads;
        const int i = c & 7, cm = (c >> 3) & 15;
        const int rr = 8 * (s >> 1) + i, k0 = 128 * (s & 1) + 8 * cm;
        float v[8];
        if (rr < nrow && k0 < kOutUsed) {
            const float4 u0 = *reinterpret_cast<const float4*>(sy + rr * kLossYS + k0);
            const float4 u1 = *reinterpret_cast<const float4*>(sy + rr * kLossYS + k0 + 4);
            v[0] = u0.x; v[1] = u0.y; v[2] = u0.z; v[3] = u0.w;
            v[4] = u1.x; v[5] = u1.y; v[6] = u1.z; v[7] = u1.w;
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = 0.f;
        }
        __align__(16) __nv_bfloat16 b[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) b[q] = __float2bfloat16_rn(v[q]);
        *reinterpret_cast<uint4*>(dyt + tixb(n0 + rr, k0, Bp, kActLbw)) = *reinterpret_cast<const uint4*>(b);
    }
    // Bias-gradient partial of these 32 rows (row n0 / 32 of the partials,
    // as the input-gradient products write theirs; rows added in order, no
    // atomics, so the sums are the same on every run).
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int col = tid + h * kLossThreads;
        float sum = 0.f;
        if (col < kOutUsed)
            for (int rr = 0; rr < nrow; ++rr) sum += sy[rr * kLossYS + col];
        bpart[(size_t)blockIdx.x * kOutP + col] = sum;
    }
}

struct AdamArgs {
    float* w;                 // FP32 master [rows][cols] row-major (or bias [rows])
    float* m;
    float* v;
    const float* gpart;       // gradient partials [nparts][rows][cols]
    int nparts;
    int rows, cols;
    int rows_used;            // rows beyond stay zero
    __nv_bfloat16* wt;        // tiled [rows][cols] (weights only)
    __nv_bfloat16* wtT;       // tiled [cols][rows] (weights only)
    float* gout;              // optional: summed gradient [rows][cols]
    float lr, b1, b2, eps, c1, c2;  // c1 = 1 - b1^t, c2 = 1 - b2^t
    int update;               // 0: only sum gradients (and refresh BF16 copies)
};

// Element i of a parameter tensor: store the summed gradient (optional),
// take the Adam step, refresh the BF16 operand copies.
__device__ __forceinline__ void adam_apply(const AdamArgs& a, int i, float gsum) {
    const int r = i / a.cols, c = i % a.cols;
    if (r >= a.rows_used) gsum = 0.f;
    if (a.gout) a.gout[i] = gsum;
    float w = a.w[i];
    if (a.update && r < a.rows_used) {
        const float m = a.b1 * a.m[i] + (1.f - a.b1) * gsum;
        const float v = a.b2 * a.v[i] + (1.f - a.b2) * gsum * gsum;
        a.m[i] = m;
        a.v[i] = v;
        w -= a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
        a.w[i] = w;
    }
    if (a.wt) {
        const __nv_bfloat16 b = __float2bfloat16_rn(w);
        a.wt[tixb(r, c, a.rows, lbw_of(a.cols))] = b;
        a.wtT[tixb(c, r, a.cols, lbw_of(a.rows))] = b;
    }
}

// Every parameter tensor of one Adam step in one launch. Blocks
// [0, wblk[4]) take 1,024 weight elements each: a thread sums the split-K
// partials of four consecutive elements in split order, eight 16-byte loads in
// flight. The remaining blocks take 16 bias elements each: 64 row lanes sum
// the per-32-row partials (lane k: rows k, k + 64, ...) and the lanes' sums
// are added in lane order. Fixed orders throughout, so every run gives the
// same sums.
// The last block (a training step's) adds the loss kernel's partial sums in a
// fixed order and leaves the batch loss and the error flag together, so that
// one read-back ends the step.
struct MlpResult {
    float loss;
    int err;
};
struct AdamAll {
    AdamArgs t[8];  // weights of layer l at 2 l, its bias at 2 l + 1
    int wblk[5];    // weight blocks before layer l
    int bblk[5];    // bias blocks before layer l
    const double* loss;  // partial sums [nloss] or nullptr: no last block
    int nloss;
    double inv_b;
    const int* err;
    MlpResult* result;
};
constexpr int kAdamThreads = 256, kAdamWElems = 4 * kAdamThreads, kAdamBElems = 16, kAdamLanes = 64;
static_assert(kAdamLanes * (kAdamBElems / 4) == kAdamThreads, "bias block shape");

__global__ void __launch_bounds__(kAdamThreads) k_adam_all(const __grid_constant__ AdamAll A) {
    __shared__ float part[kAdamLanes][kAdamBElems + 1];
    int b = blockIdx.x;
    if (b < A.wblk[4]) {
        int l = 0;
        while (l < 3 && b >= A.wblk[l + 1]) ++l;
        const AdamArgs& a = A.t[2 * l];
        const int n = a.rows * a.cols;
        const int i0 = (b - A.wblk[l]) * kAdamWElems + 4 * (int)threadIdx.x;
        if (i0 >= n) return;
        float g[4] = {0.f, 0.f, 0.f, 0.f};
        if (a.gpart) {
            const float4* src = reinterpret_cast<const float4*>(a.gpart + i0);
            const size_t stride = (size_t)n / 4;
            int p = 0;
            for (; p + 8 <= a.nparts; p += 8) {
                float4 v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) v[q] = src[(size_t)(p + q) * stride];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    g[0] += v[q].x;
                    g[1] += v[q].y;
                    g[2] += v[q].z;
                    g[3] += v[q].w;
                }
            }
            for (; p < a.nparts; ++p) {
                const float4 v = src[(size_t)p * stride];
                g[0] += v.x;
                g[1] += v.y;
                g[2] += v.z;
                g[3] += v.w;
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) adam_apply(a, i0 + q, g[q]);
        return;
    }
    b -= A.wblk[4];
    if (b >= A.bblk[4]) {
        __shared__ double sl[kAdamThreads];
        double sum = 0.0;
        for (int i = threadIdx.x; i < A.nloss; i += kAdamThreads) sum += A.loss[i];
        sl[threadIdx.x] = sum;
        __syncthreads();
        for (int o = kAdamThreads / 2; o > 0; o >>= 1) {
            if ((int)threadIdx.x < o) sl[threadIdx.x] += sl[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            A.result->loss = (float)(sl[0] * A.inv_b);
            A.result->err = *A.err;
        }
        return;
    }
    int l = 0;
    while (l < 3 && b >= A.bblk[l + 1]) ++l;
    const AdamArgs& a = A.t[2 * l + 1];
    const int n = a.rows;  // a bias: rows x 1
    const int c0 = (b - A.bblk[l]) * kAdamBElems;
    const int quad = threadIdx.x & 3, lane = threadIdx.x >> 2;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    if (a.gpart && c0 + 4 * quad < n) {
        const float* src = a.gpart + c0 + 4 * quad;
#pragma unroll 8
        for (int p = lane; p < a.nparts; p += kAdamLanes) {
            const float4 v = *reinterpret_cast<const float4*>(src + (size_t)p * n);
            s[0] += v.x;
            s[1] += v.y;
            s[2] += v.z;
            s[3] += v.w;
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) part[lane][4 * quad + q] = s[q];
    __syncthreads();
    const int e = threadIdx.x;
    if (e < kAdamBElems && c0 + e < n) {
        float g = 0.f;
        for (int k = 0; k < kAdamLanes; ++k) g += part[k][e];
        adam_apply(a, c0 + e, g);
    }
}

}  // namespace mlp
}  // namespace stp

// ---------------------------------------------------------------------------
// Host side and C ABI.
// ---------------------------------------------------------------------------
using namespace stp;
using namespace stp::mlp;

namespace {
// Logical parameter layout (W1 [256][32], b1, W2 [256][256], b2, W3, b3,
// W4 [160][256], b4 [160]) against the padded device tensors.
struct Layer {
    int out, in, out_used, in_used;  // padded / logical
};
constexpr Layer kLayers[4] = {{kHid, kInP, kHid, kIn}, {kHid, kHid, kHid, kHid}, {kHid, kHid, kHid, kHid},
                              {kOutP, kHid, kOut, kHid}};
}  // namespace

struct stp_mlp {
    int max_batch = 0, Bp_max = 0;
    cudaStream_t stream = nullptr;
    char* arena = nullptr;
    size_t arena_bytes = 0;
    // parameters
    float* w[4]{};
    float* b[4]{};
    float *mw[4]{}, *vw[4]{}, *mb[4]{}, *vb[4]{};
    __nv_bfloat16 *wt[4]{}, *wtT[4]{};
    // activations and their gradients (BF16, tiled), FP32 buffers
    __nv_bfloat16* xt = nullptr;
    __nv_bfloat16* ht[3]{};
    __nv_bfloat16* dt[4]{};  // gradient wrt layer outputs (dt[3] = dY)
    float* y = nullptr;       // [Bp][160]
    float* wpart = nullptr;   // weight-gradient partials
    float* bpart = nullptr;   // bias-gradient partials [4][Bp/32][256]
    float* gsum = nullptr;    // summed gradients (gradients API)
    double* loss = nullptr;   // partial loss sums [Bp / 32]
    MlpResult* result = nullptr;
    float* X = nullptr;       // staged inputs [max_batch][32]
    float* T = nullptr;       // staged targets [max_batch][130]
    int* err = nullptr;
    size_t param_floats = 0, moment_floats = 0, grad_floats = 0;  // of the arena's parameter, moment and gradient blocks
    int nsm = 0;              // SMs of the device (persistent product grid)
    int step = 0;
    bool profiling = false;
    // Profiling intervals: 0 forward chain, 1 backward pass, 2 whole training
    // step (event pairs 2i, 2i + 1), read once the stream has been synchronised.
    cudaEvent_t ev[6]{};
    bool ev_pending[3]{};
    double ev_flops[3]{}, ev_bytes[3]{};
    double gemm_ms = 0, gemm_flops = 0, gemm_bytes = 0;
    double step_ms = 0;
    int steps = 0;
    std::string last_error;
};

namespace {
thread_local std::string g_mlp_err;

stp_status fail(stp_mlp* m, stp_status st, const std::string& msg) {
    if (m) m->last_error = msg;
    g_mlp_err = msg;
    return st;
}
#define MLP_CUDA(m, call)                                                               \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess) return fail((m), STP_ERR_CUDA, cudaGetErrorString(e_)); \
    } while (0)

// Split-K of the weight-gradient products: at most kSplitMax splits (the
// partial buffers), at least four K stages each, and one wave of CTAs a launch.
constexpr int kSplitMax = 80;

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

template <int N, int LBWB>
cudaError_t launch_wgrad(const WGradArgs& g, int layers, int splits, cudaStream_t st) {
    constexpr int smem = wgrad_smem_bytes<N, LBWB>();
    static SmemAttr attr;
    cudaError_t e = ensure_smem((const void*)k_gemm_wgrad<N, LBWB>, attr, smem);
    if (e != cudaSuccess) return e;
    k_gemm_wgrad<N, LBWB><<<dim3(kOutP / kTileM, layers, splits), kThreads, smem, st>>>(g);
    return cudaGetLastError();
}

template <bool BACK, bool STORE>
cudaError_t launch_chain(const ChainArgs& g, int nsm, cudaStream_t st) {
    static SmemAttr attr;
    cudaError_t e = ensure_smem((const void*)k_chain<BACK, STORE>, attr, kChainSmem);
    if (e != cudaSuccess) return e;
    k_chain<BACK, STORE><<<std::min(g.tiles, nsm), kChainThreads, kChainSmem, st>>>(g);
    return cudaGetLastError();
}

// Bias-gradient partials per layer: one row per 32 batch rows (written by the
// input-gradient products, and for the last layer by the loss kernel).
size_t bpart_stride(int Bp_max) { return (size_t)(Bp_max / 32) * kOutP; }

// Algorithmic HBM bytes of one product of a training step at batch B over the
// layer's logical shape (in x out, no padding): every operand read once,
// every output written once in one layout (BF16 activations and input
// gradients, FP32 network outputs and weight gradients); the input-gradient
// product also reads the forward activation for the ReLU mask. The padding and
// the split-K partials are this design's choices and are not counted.
double alg_bytes(int B, int in, int out, int mode) {
    const double b = B, i = in, o = out;
    if (mode == kHidden) return 2 * b * i + 2 * i * o + 2 * b * o;
    if (mode == kOutput) return 2 * b * i + 2 * i * o + 4 * b * o;
    if (mode == kWGrad) return 2 * b * o + 2 * b * i + 4 * i * o;
    return 2 * b * o + 2 * i * o + 2 * b * i + 2 * b * i;  // kBackward
}

// Event interval `slot` on the main stream (no host synchronisation inside
// a call: the intervals are read by collect_profile after the stream sync).
void interval_start(stp_mlp* m, int slot) {
    if (m->profiling) cudaEventRecord(m->ev[2 * slot], m->stream);
}
void interval_stop(stp_mlp* m, int slot, double flops, double bytes) {
    if (!m->profiling) return;
    cudaEventRecord(m->ev[2 * slot + 1], m->stream);
    m->ev_pending[slot] = true;
    m->ev_flops[slot] = flops;
    m->ev_bytes[slot] = bytes;
}
void collect_profile(stp_mlp* m) {
    for (int slot = 0; slot < 3; ++slot) {
        if (!m->ev_pending[slot]) continue;
        m->ev_pending[slot] = false;
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, m->ev[2 * slot], m->ev[2 * slot + 1]) != cudaSuccess) continue;
        if (slot == 2) {
            m->step_ms += ms;
            ++m->steps;
        } else {
            m->gemm_ms += ms;
            m->gemm_flops += m->ev_flops[slot];
            m->gemm_bytes += m->ev_bytes[slot];
        }
    }
}

// X: device features [B][32], Y: device outputs [B][160], both 16-byte aligned.
// train: also the packed features and the activations, for the backward pass.
stp_status forward_impl(stp_mlp* m, int B, const float* X, float* Y, bool train) {
    const int Bp = (B + kTileM - 1) / kTileM * kTileM;
    double chain_flops = 0.0, chain_bytes = 0.0;
    ChainArgs g{};
    g.tiles = Bp / kTileM;
    g.RA = Bp;
    g.B = B;
    g.X = X;
    g.xt = m->xt;
    g.Y = Y;
    g.err = m->err;
    for (int l = 0; l < 4; ++l) {
        const Layer& L = kLayers[l];
        chain_flops += 2.0 * B * L.in_used * L.out_used;
        chain_bytes += alg_bytes(B, L.in_used, L.out_used, l < 3 ? kHidden : kOutput);
        g.W[l] = m->wt[l];
        g.bias[l] = m->b[l];
        if (l < 3) g.out[l] = m->ht[l];
    }
    interval_start(m, 0);
    MLP_CUDA(m, train ? (launch_chain<false, true>(g, m->nsm, m->stream))
                      : (launch_chain<false, false>(g, m->nsm, m->stream)));
    interval_stop(m, 0, chain_flops, chain_bytes);
    return STP_OK;
}

// Backward from dY (already in dt[3], its bias partials written by
// the loss kernel) to every parameter's gradient partials.
stp_status backward_impl(stp_mlp* m, int B, int (&nwpart)[4], int* nbpart) {
    const int Bp = (B + kTileM - 1) / kTileM * kTileM;
    cudaStream_t st = m->stream;
    const int KTb = Bp / kStageK;
    // One wave of CTAs a launch (one per SM): layers x kOutP / kTileM row tiles x splits.
    auto stages = [&](int layers) {
        const int target = std::max(1, std::min({kSplitMax, m->nsm / (layers * (kOutP / kTileM)), KTb / 4}));
        return (KTb + target - 1) / target;
    };
    const int kps[4] = {stages(1), stages(3), stages(3), stages(3)};
    for (int l = 0; l < 4; ++l) nwpart[l] = (KTb + kps[l] - 1) / kps[l];  // every split non-empty
    *nbpart = Bp / 32;
    double chain_flops = 0.0, chain_bytes = 0.0;
    for (int l = 3; l >= 0; --l) {
        chain_flops += 2.0 * B * kLayers[l].in_used * kLayers[l].out_used;
        chain_bytes += alg_bytes(B, kLayers[l].in_used, kLayers[l].out_used, kWGrad);
        if (l > 0) {
            chain_flops += 2.0 * B * kLayers[l].in_used * kLayers[l].out_used;
            chain_bytes += alg_bytes(B, kLayers[l].in_used, kLayers[l].out_used, kBackward);
        }
    }
    interval_start(m, 1);
    // Input gradients: product l of the chain is dH_{2-l} = (dT_{3-l} . W_{3-l}) * relu'(h_{2-l}).
    ChainArgs c{};
    c.tiles = Bp / kTileM;
    c.RA = Bp;
    c.B = B;
    c.A0 = m->dt[3];
    c.err = m->err;
    for (int l = 0; l < 3; ++l) {
        c.W[l] = m->wtT[3 - l];
        c.act[l] = m->ht[2 - l];
        c.out[l] = m->dt[2 - l];
        c.bpart[l] = m->bpart + (size_t)(2 - l) * bpart_stride(m->Bp_max);
    }
    MLP_CUDA(m, (launch_chain<true, true>(c, m->nsm, st)));
    // Weight gradients: dW_l = dT_l^T . act_{l-1}   (M = out, N = in, K = batch);
    // layers 2-4 in one launch.
    auto args = [&](int l) {
        GemmArgs g{};
        g.A = m->dt[l];
        g.RA = Bp;
        g.B = (l == 0) ? m->xt : m->ht[l - 1];
        g.KT = KTb;
        g.kt_per_split = kps[l];
        g.out_f = m->wpart + (size_t)l * kSplitMax * kOutP * kHid;
        g.ld_f = kLayers[l].in;
        g.m_valid = kLayers[l].out;
        g.err = m->err;
        return g;
    };
    WGradArgs wide{}, first{};
    for (int l = 0; l < 3; ++l) wide.layer[l] = args(3 - l);
    first.layer[0] = args(0);
    MLP_CUDA(m, (launch_wgrad<kHid, kActLbw>(wide, 3, nwpart[1], st)));
    MLP_CUDA(m, (launch_wgrad<kInP, lbw_of(kInP)>(first, 1, nwpart[0], st)));
    interval_stop(m, 1, chain_flops, chain_bytes);
    return STP_OK;
}

// B > 0: also the batch loss of the loss kernel's partial sums.
stp_status adam_impl(stp_mlp* m, const int (&nwpart)[4], int nbpart, float lr, bool update, bool keep_grads, int B = 0) {
    if (update) ++m->step;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = update ? 1.f - powf(b1, (float)m->step) : 1.f;
    const float c2 = update ? 1.f - powf(b2, (float)m->step) : 1.f;
    float* gout = m->gsum;
    AdamAll A{};
    for (int l = 0; l < 4; ++l) {
        const Layer& L = kLayers[l];
        AdamArgs a{};
        a.w = m->w[l];
        a.m = m->mw[l];
        a.v = m->vw[l];
        a.gpart = m->wpart + (size_t)l * kSplitMax * kOutP * kHid;
        a.nparts = nwpart[l];
        a.rows = L.out;
        a.cols = L.in;
        a.rows_used = L.out_used;
        a.wt = m->wt[l];
        a.wtT = m->wtT[l];
        a.gout = keep_grads ? gout : nullptr;
        a.lr = lr;
        a.b1 = b1;
        a.b2 = b2;
        a.eps = 1e-8f;
        a.c1 = c1;
        a.c2 = c2;
        a.update = update ? 1 : 0;
        const int n = L.out * L.in;
        gout += n;
        AdamArgs bb = a;
        bb.w = m->b[l];
        bb.m = m->mb[l];
        bb.v = m->vb[l];
        // bias partials are [chunk][256]: element e of chunk p at p * 256 + e
        bb.gpart = m->bpart + (size_t)l * bpart_stride(m->Bp_max);
        bb.nparts = nbpart;
        bb.rows = L.out;
        bb.cols = 1;
        bb.wt = nullptr;
        bb.wtT = nullptr;
        bb.gout = keep_grads ? gout : nullptr;
        gout += L.out;
        A.t[2 * l] = a;
        A.t[2 * l + 1] = bb;
        A.wblk[l + 1] = A.wblk[l] + (n + kAdamWElems - 1) / kAdamWElems;
        A.bblk[l + 1] = A.bblk[l] + (L.out + kAdamBElems - 1) / kAdamBElems;
    }
    if (B > 0) {
        A.loss = m->loss;
        A.nloss = ((B + kTileM - 1) / kTileM * kTileM) / kLossRows;
        A.inv_b = 1.0 / B;
        A.err = m->err;
        A.result = m->result;
    }
    k_adam_all<<<A.wblk[4] + A.bblk[4] + (B > 0 ? 1 : 0), kAdamThreads, 0, m->stream>>>(A);
    MLP_CUDA(m, cudaGetLastError());
    return STP_OK;
}

// Device address of n floats of an input: the caller's own where it is this
// GPU's memory on a 16-byte boundary, else a copy in dst.
stp_status stage_in(stp_mlp* m, float* dst, const float* src, size_t n, int flags, const float** used) {
    *used = dst;
    if ((flags & STP_MLP_DEVICE) && ((uintptr_t)src & 15) == 0 && !other_gpu(src)) {
        *used = src;
        return STP_OK;
    }
    MLP_CUDA(m, cudaMemcpyAsync(dst, src, n * sizeof(float),
                                (flags & STP_MLP_DEVICE) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                                m->stream));
    return STP_OK;
}

stp_status timeout_fail(stp_mlp* m) {
    cudaMemsetAsync(m->err, 0, sizeof(int), m->stream);
    return fail(m, STP_ERR_TIMEOUT, "tensor-core pipeline wait exceeded its limit");
}

stp_status check_err(stp_mlp* m) {
    int e = 0;
    MLP_CUDA(m, cudaMemcpyAsync(&e, m->err, sizeof(int), cudaMemcpyDeviceToHost, m->stream));
    MLP_CUDA(m, cudaStreamSynchronize(m->stream));
    collect_profile(m);
    return e ? timeout_fail(m) : STP_OK;
}

// End of a training step: its loss and error flag in one read-back.
stp_status read_result(stp_mlp* m, float* loss) {
    MlpResult r{};
    MLP_CUDA(m, cudaMemcpyAsync(&r, m->result, sizeof(r), cudaMemcpyDeviceToHost, m->stream));
    MLP_CUDA(m, cudaStreamSynchronize(m->stream));
    collect_profile(m);
    if (r.err) return timeout_fail(m);
    if (loss) *loss = r.loss;
    return STP_OK;
}

// Parameters (or the summed gradients) in the logical layout, by one copy.
stp_status read_tensors(stp_mlp* m, float* out, bool grads) {
    std::vector<float> h(grads ? m->grad_floats : m->param_floats);
    MLP_CUDA(m, cudaMemcpyAsync(h.data(), grads ? m->gsum : m->w[0], h.size() * 4, cudaMemcpyDeviceToHost, m->stream));
    MLP_CUDA(m, cudaStreamSynchronize(m->stream));
    const float* g = h.data();
    for (int l = 0; l < 4; ++l) {
        const Layer& L = kLayers[l];
        const float* W = grads ? g : h.data() + (m->w[l] - m->w[0]);
        const float* b = grads ? g + (size_t)L.out * L.in : h.data() + (m->b[l] - m->w[0]);
        for (int r = 0; r < L.out_used; ++r, out += L.in_used)
            std::memcpy(out, W + (size_t)r * L.in, (size_t)L.in_used * 4);
        std::memcpy(out, b, (size_t)L.out_used * 4);
        out += L.out_used;
        g += (size_t)L.out * L.in + L.out;
    }
    return STP_OK;
}

// Logical parameter count and offsets.
size_t nparam() {
    size_t n = 0;
    for (const Layer& L : kLayers) n += (size_t)L.out_used * L.in_used + L.out_used;
    return n;
}
}  // namespace

extern "C" {

stp_status stp_mlp_create(int max_batch, stp_mlp** out) {
    if (nparam() != (size_t)STP_MLP_NPARAM) return fail(nullptr, STP_ERR_INVALID, "parameter layout mismatch");
    if (!out) return fail(nullptr, STP_ERR_INVALID, "out is NULL");
    *out = nullptr;
    if (max_batch <= 0 || max_batch > STP_MLP_MAX_BATCH) return fail(nullptr, STP_ERR_INVALID, "max_batch out of range");
    stp_mlp* m = new (std::nothrow) stp_mlp();
    if (!m) return fail(nullptr, STP_ERR_CAPACITY, "host allocation failed");
    m->max_batch = max_batch;
    const int Bp = (max_batch + kTileM - 1) / kTileM * kTileM;
    m->Bp_max = Bp;
    {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&m->nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || m->nsm < 2) {
            delete m;
            return fail(nullptr, STP_ERR_CUDA, "device query failed");
        }
    }
    // arena layout
    std::vector<std::pair<void**, size_t>> parts;
    auto weights = [](int l) { return (size_t)kLayers[l].out * kLayers[l].in * 4; };
    auto biases = [](int l) { return (size_t)kLayers[l].out * 4; };
    for (int l = 0; l < 4; ++l) parts.push_back({(void**)&m->w[l], weights(l)});
    for (int l = 0; l < 4; ++l) parts.push_back({(void**)&m->b[l], biases(l)});
    for (int l = 0; l < 4; ++l) parts.push_back({(void**)&m->mw[l], weights(l)});
    for (int l = 0; l < 4; ++l) parts.push_back({(void**)&m->vw[l], weights(l)});
    for (int l = 0; l < 4; ++l) parts.push_back({(void**)&m->mb[l], biases(l)});
    for (int l = 0; l < 4; ++l) parts.push_back({(void**)&m->vb[l], biases(l)});
    for (int l = 0; l < 4; ++l) {
        parts.push_back({(void**)&m->wt[l], weights(l) / 2});
        parts.push_back({(void**)&m->wtT[l], weights(l) / 2});
        m->grad_floats += (weights(l) + biases(l)) / 4;
    }
    parts.push_back({(void**)&m->xt, (size_t)Bp * kInP * 2});
    for (int l = 0; l < 3; ++l) {
        parts.push_back({(void**)&m->ht[l], (size_t)Bp * kHid * 2});
    }
    for (int l = 0; l < 4; ++l) {
        parts.push_back({(void**)&m->dt[l], (size_t)Bp * kOutP * 2});
    }
    parts.push_back({(void**)&m->y, (size_t)Bp * kOut * 4});
    parts.push_back({(void**)&m->wpart, (size_t)4 * kSplitMax * kOutP * kHid * 4});
    parts.push_back({(void**)&m->bpart, (size_t)4 * bpart_stride(Bp) * 4});
    parts.push_back({(void**)&m->gsum, (size_t)4 * (kOutP * kHid + kOutP) * 4});
    parts.push_back({(void**)&m->loss, (size_t)(Bp / kLossRows) * 8});
    parts.push_back({(void**)&m->result, sizeof(MlpResult)});
    parts.push_back({(void**)&m->X, (size_t)max_batch * kIn * 4});
    parts.push_back({(void**)&m->T, (size_t)max_batch * kTgt * 4});
    parts.push_back({(void**)&m->err, 256});
    size_t total = 0;
    for (auto& p : parts) total += up256(p.second);
    if (cudaMalloc(&m->arena, total) != cudaSuccess) {
        delete m;
        return fail(nullptr, STP_ERR_CUDA, "device allocation failed");
    }
    m->arena_bytes = total;
    size_t off = 0;
    for (auto& p : parts) {
        *p.first = m->arena + off;
        off += up256(p.second);
    }
    m->param_floats = (size_t)(m->mw[0] - m->w[0]);
    m->moment_floats = (size_t)(reinterpret_cast<float*>(m->wt[0]) - m->mw[0]);
    bool events_ok = true;
    for (cudaEvent_t& e : m->ev) events_ok = events_ok && cudaEventCreate(&e) == cudaSuccess;
    if (cudaMemset(m->arena, 0, total) != cudaSuccess || !events_ok) {
        stp_mlp_free(m);
        return fail(nullptr, STP_ERR_CUDA, "device initialisation failed");
    }
    *out = m;
    return STP_OK;
}

void stp_mlp_free(stp_mlp* m) {
    if (!m) return;
    if (m->stream) cudaStreamSynchronize(m->stream);
    else cudaDeviceSynchronize();
    cudaFree(m->arena);
    for (cudaEvent_t e : m->ev)
        if (e) cudaEventDestroy(e);
    delete m;
}

stp_status stp_mlp_set_stream(stp_mlp* m, void* stream) {
    if (!m) return fail(nullptr, STP_ERR_INVALID, "mlp is NULL");
    m->stream = (cudaStream_t)stream;
    return STP_OK;
}

stp_status stp_mlp_set_params(stp_mlp* m, const float* params) {
    if (!m || !params) return fail(m, STP_ERR_INVALID, "NULL argument");
    // Parameters and moments sit next to each other in the arena: one copy in
    // the padded layout, one clear.
    std::vector<float> h(m->param_floats, 0.f);
    const float* p = params;
    for (int l = 0; l < 4; ++l) {
        const Layer& L = kLayers[l];
        float* W = h.data() + (m->w[l] - m->w[0]);
        float* b = h.data() + (m->b[l] - m->w[0]);
        for (int r = 0; r < L.out_used; ++r, p += L.in_used) std::memcpy(W + (size_t)r * L.in, p, (size_t)L.in_used * 4);
        std::memcpy(b, p, (size_t)L.out_used * 4);
        p += L.out_used;
    }
    MLP_CUDA(m, cudaMemcpyAsync(m->w[0], h.data(), h.size() * 4, cudaMemcpyHostToDevice, m->stream));
    MLP_CUDA(m, cudaMemsetAsync(m->mw[0], 0, (size_t)m->moment_floats * 4, m->stream));
    m->step = 0;
    // refresh the BF16 operand copies (no update)
    stp_status s = adam_impl(m, {}, 0, 0.f, false, false);
    if (s != STP_OK) return s;
    MLP_CUDA(m, cudaStreamSynchronize(m->stream));
    return STP_OK;
}

stp_status stp_mlp_get_params(stp_mlp* m, float* params) {
    if (!m || !params) return fail(m, STP_ERR_INVALID, "NULL argument");
    return read_tensors(m, params, false);
}

stp_status stp_mlp_forward(stp_mlp* m, int B, const float* X, float* Y, int flags) {
    if (!m || !X || !Y) return fail(m, STP_ERR_INVALID, "NULL argument");
    if (B <= 0 || B > m->max_batch) return fail(m, STP_ERR_INVALID, "batch out of range");
    const float* Xd = nullptr;
    stp_status s = stage_in(m, m->X, X, (size_t)B * kIn, flags, &Xd);
    if (s != STP_OK) return s;
    // The output layer writes the caller's buffer where that is this GPU's memory
    // on a 16-byte boundary and not also the input (a tile's outputs would
    // overwrite features that another has not read).
    const bool direct = (flags & STP_MLP_DEVICE) && ((uintptr_t)Y & 15) == 0 &&
                        !ranges_meet(Xd, (size_t)B * kIn * 4, Y, (size_t)B * kOut * 4) && !other_gpu(Y);
    if ((s = forward_impl(m, B, Xd, direct ? Y : m->y, false)) != STP_OK) return s;
    if (!direct)
        MLP_CUDA(m, cudaMemcpyAsync(Y, m->y, (size_t)B * kOut * 4,
                                    (flags & STP_MLP_DEVICE) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                                    m->stream));
    return check_err(m);
}

static stp_status loss_grad(stp_mlp* m, int B, const float* X, const float* T, int flags, int (&nw)[4], int* nb) {
    if (!m || !X || !T) return fail(m, STP_ERR_INVALID, "NULL argument");
    if (B <= 0 || B > m->max_batch) return fail(m, STP_ERR_INVALID, "batch out of range");
    const float *Xd = nullptr, *Td = nullptr;
    stp_status s = stage_in(m, m->X, X, (size_t)B * kIn, flags, &Xd);
    if (s != STP_OK) return s;
    if ((s = stage_in(m, m->T, T, (size_t)B * kTgt, flags, &Td)) != STP_OK) return s;
    interval_start(m, 2);  // the training step's device work, inputs staged
    if ((s = forward_impl(m, B, Xd, m->y, true)) != STP_OK) return s;
    const int Bp = (B + kTileM - 1) / kTileM * kTileM;
    k_loss<<<Bp / kLossRows, kLossThreads, 0, m->stream>>>(
        m->y, Td, B, m->bpart + (size_t)3 * bpart_stride(m->Bp_max), m->dt[3], Bp, m->loss);
    MLP_CUDA(m, cudaGetLastError());
    return backward_impl(m, B, nw, nb);
}

stp_status stp_mlp_gradients(stp_mlp* m, int B, const float* X, const float* T, float* loss, float* grads,
                             int flags) {
    int nw[4] = {}, nb = 0;
    stp_status s = loss_grad(m, B, X, T, flags, nw, &nb);
    if (s != STP_OK) return s;
    if ((s = adam_impl(m, nw, nb, 0.f, false, true, B)) != STP_OK) return s;
    interval_stop(m, 2, 0.0, 0.0);
    if ((s = read_result(m, loss)) != STP_OK) return s;
    return grads ? read_tensors(m, grads, true) : STP_OK;
}

stp_status stp_mlp_train_step(stp_mlp* m, int B, const float* X, const float* T, float lr, float* loss, int flags) {
    if (!(lr >= 0.f)) return fail(m, STP_ERR_INVALID, "learning rate must be >= 0");
    int nw[4] = {}, nb = 0;
    stp_status s = loss_grad(m, B, X, T, flags, nw, &nb);
    if (s != STP_OK) return s;
    if ((s = adam_impl(m, nw, nb, lr, true, false, B)) != STP_OK) return s;
    interval_stop(m, 2, 0.0, 0.0);
    return read_result(m, loss);
}

stp_status stp_mlp_set_profiling(stp_mlp* m, int on) {
    if (!m) return fail(nullptr, STP_ERR_INVALID, "mlp is NULL");
    m->profiling = on != 0;
    m->gemm_ms = 0;
    m->gemm_flops = 0;
    m->gemm_bytes = 0;
    m->step_ms = 0;
    m->steps = 0;
    for (bool& p : m->ev_pending) p = false;
    return STP_OK;
}

stp_status stp_mlp_profile(stp_mlp* m, double* gemm_ms, double* gemm_flops, double* gemm_bytes) {
    if (!m) return fail(nullptr, STP_ERR_INVALID, "mlp is NULL");
    if (gemm_ms) *gemm_ms = m->gemm_ms;
    if (gemm_flops) *gemm_flops = m->gemm_flops;
    if (gemm_bytes) *gemm_bytes = m->gemm_bytes;
    m->gemm_bytes = 0;
    m->gemm_ms = 0;
    m->gemm_flops = 0;
    return STP_OK;
}
stp_status stp_mlp_profile_step(stp_mlp* m, double* step_ms, int* steps) {
    if (!m) return fail(nullptr, STP_ERR_INVALID, "mlp is NULL");
    if (step_ms) *step_ms = m->step_ms;
    if (steps) *steps = m->steps;
    m->step_ms = 0;
    m->steps = 0;
    return STP_OK;
}

const char* stp_mlp_last_error(const stp_mlp* m) { return m ? m->last_error.c_str() : g_mlp_err.c_str(); }

}  // extern "C"
