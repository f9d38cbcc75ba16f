// The step after the feedback: the gradient of the round's loss with respect to the weights of the
// draft model's (linear) output layer,
//     dW[v,j] = sum_r g[r,v] * x[r,j]          dW = g^T X,   g [R,V] (gradient w.r.t. the draft logits,
//                                               Sec. 3.1), X [R,d] (hidden states), R = B*k positions,
// a dense contraction over the positions of the round: the one place on this path where the
// tensor cores apply.  sm_100a: operands by TMA (cp.async.bulk.tensor) into 128-byte-swizzled
// shared memory, tcgen05.mma (bf16 x bf16 -> fp32) with the accumulator in tensor memory,
// tcgen05.ld and TMA stores for the epilogue.
//
// Both operands have the contracted index r as their slow index in memory, so both are "MN-major"
// operands of the instruction: a tile of g is [64 positions][128 vocabulary entries] with the
// vocabulary entries contiguous, a tile of X is [64 positions][128 features] likewise.
//
// A pair of blocks (a cluster of two, one block per SM) shares an output tile of 256 x 256 (cta_group::2):
// block r holds rows 128 r .. 128 r + 127 of the tile, brings their part of g and columns
// 128 r .. 128 r + 127 of X, and each tensor core reads the other half of X from its neighbour's shared
// memory.  Persistent over the tiles; the features run fastest, so the pairs that work at the same time
// share a few tiles of g (each read from HBM once) and all of X (which stays in L2).  Warp roles of a block:
//   warp 0      producer: one thread issues the TMA loads of the block's share of a stage (4 boxes of 64 x 64
//               bf16); they complete on the barrier of the pair's first block
//   warp 1      in the pair's first block one thread issues the MMAs (4 of K = 16 per stage) and the commits,
//               which free the stage in both blocks
//   from warp 2 epilogue: tensor memory -> registers -> 32 x 32 boxes in shared memory -> global memory by TMA
//               stores, which clip at the ends of dW, while the MMAs of the next tile fill the other half of
//               tensor memory.
// What bounds it: for many positions the board's power (1536 positions, 128 256 x 4096: 1240 us = 1.3 PFLOP/s for 20 calls
// on a cool board, 1450 = 1.12 after seconds of it, of 1.64 and 1.39 measured with cuBLAS);
// operands enter an SM at 64 bytes a clock.  One block per tile of 128 x 256 (cta_group::1) needs 96, 27 TB/s of
// L2 at full rate, and took 1377 us.  For few positions the writing of dW, which wants more boxes under way than
// loads (GemmShape): 256 positions 470 us (4.5 TB/s out), with four epilogue warps 512; 128 positions 397 and 413
// (one block per tile: 562 and 549).
// Every wait is bounded; a wait that gives up sets an error word, and the block frees its tensor
// memory and returns.  No multicast of loads.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sd_kernels.cuh"

namespace sdv {

constexpr int kGemmBM = 256;                 // vocabulary entries per tile (rows of dW), half of them in each block
constexpr int kGemmBN = 256;                 // features per tile (columns of dW); each block brings half of them
constexpr int kGemmBK = 64;                  // positions per stage
constexpr int kGemmChunk = 64;               // entries of a 128-byte swizzled row (bf16)
constexpr int kGemmChunkBytes = kGemmBK * kGemmChunk * 2;            // one TMA box: 8 KiB
constexpr int kGemmChunks = 128 / kGemmChunk;                        // boxes of an operand's half tile
constexpr int kGemmABytes = kGemmChunks * kGemmChunkBytes;           // 16 KiB
constexpr int kGemmStageBytes = 2 * kGemmABytes;                     // a block's share of a stage: 32 KiB
constexpr int kGemmTmemCols = 512;           // two accumulators of 128 lanes x 256 fp32 columns
constexpr int kGemmBox = 32;                 // rows and columns of a box of the result
constexpr int kGemmBoxBytes = kGemmBox * kGemmBox * 4;
constexpr int kGemmBoxes = 2;                // boxes per epilogue warp: one leaves while the next is filled
// The two shapes of the kernel (both fill the shared memory of a block).  Few positions: eight epilogue warps, two to
// a quarter of the tensor-memory lanes; many: six stages.  us, six stages / eight warps, calls back to back on a warm board:
//     128 256 x 4096   128 positions 413 / 397, 256 512 / 470, 384 564 / 583, 512 654 / 723, 1536 from cold 1240 / 1317
//     128 256 x 1024   256 152 / 137, 384 161 / 153, 512 167 / 186      151 936 x 2048   256 322 / 289, 384 360 / 368, 512 407 / 433
//      32 000 x 4096   256 160 / 122, 384 146 / 140, 512 158 / 174       32 000 x 1024   256 47 / 48, 384 51 / 47, 768 54 / 60
// So they meet near 384 positions, whatever the other two sizes.
template <bool FEW> struct GemmShape {
    static constexpr int kStages = FEW ? 5 : 6;
    static constexpr int kEpilogueWarps = FEW ? 8 : 4;
    static constexpr int kThreads = (2 + kEpilogueWarps) * 32;
    static constexpr int kColumns = kGemmBN * 4 / kEpilogueWarps;        // of the accumulator, per epilogue warp
    static constexpr int kSmem = kStages * kGemmStageBytes + kEpilogueWarps * kGemmBoxes * kGemmBoxBytes + 1024 /* alignment */ + 256 /* barriers */;
    static_assert(kSmem <= 227 * 1024, "stages and staging do not fit the shared memory of a block");
};
constexpr int kGemmFewPositions = 384;
constexpr long long kGemmLeaveCycles = 2000000ll;     // about a millisecond
constexpr long long kGemmWaitCycles = 4000000000ll;   // about two seconds

struct GemmParams {
    int R, V, d;
    uint32_t* error;         // set when a bounded wait gave up
};

// ---- PTX wrappers --------------------------------------------------------------------------
// One box into this block's shared memory; its bytes count on `bar` (a shared::cluster address), which may be
// the other block's of the pair.
__device__ __forceinline__ void tma_load_2d_pair(void* dst_smem, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
            smem_u32(dst_smem)),
        "l"(map), "r"(bar), "r"(x), "r"(y)
        : "memory");
}
// One box of the result out of shared memory; what lies outside the matrix is not written.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int x, int y, const void* src_smem) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(map), "r"(smem_u32(src_smem)),
                 "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// All but the last `N` boxes of this thread have been read (READ) or written out.
template <int N, bool READ> __device__ __forceinline__ void tma_store_wait() {
    if constexpr (READ) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
    else                asm volatile("cp.async.bulk.wait_group %0;" ::"n"(N) : "memory");
}
// The address of `p` (of this block) in block `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_address(const void* p, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void tmem_alloc(uint32_t* slot_in_smem, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot_in_smem)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// D[tmem] (+)= A[smem] * B[smem] of the pair, each block with its half of the rows; accumulate = 0 overwrites D.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// The barrier gets one arrival in each block of the pair when every MMA issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
                     smem_u32(bar)),
                 "h"((uint16_t)3)
                 : "memory");
}
// 32 lanes x 32 consecutive fp32 columns of tensor memory: thread i of the warp gets lane i.
__device__ __forceinline__ void tmem_ld_32x32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]),
          "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]),
          "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory operand descriptor of an MN-major tile in the 128-byte swizzle: rows of 64 bf16
// along M (or N), 128 bytes apart along K, eight of them to a swizzle atom.  lbo: bytes from one
// group of 64 entries along M/N to the next; sbo: bytes from one group of 8 positions along K to
// the next.  (Bits 0-13 address >> 4, 16-29 lbo >> 4, 32-45 sbo >> 4, 46-47 version 1, 61-63 swizzle 128 B = 2.)
__device__ __forceinline__ uint64_t umma_desc_mn_sw128(uint32_t smem_addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((smem_addr & 0x3ffffu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           (1ull << 46) | (2ull << 61);
}
// Instruction descriptor: fp32 accumulator, bf16 x bf16, both operands MN-major, M x N.
__host__ __device__ constexpr uint32_t umma_idesc_bf16_mn(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Bounded wait on a barrier of this block by one thread; false (and the error word set) when it gives up.
__device__ __forceinline__ bool gemm_wait(uint64_t* bar, uint32_t parity, volatile int* abort, uint32_t* error) {
    long long t0 = 0;
    for (uint32_t it = 0;; ++it) {
        if (mbar_try_wait_cluster(bar, parity)) return true;
        if ((it & 255u) == 255u) {
            if (*abort) return false;
            const long long now = clock64();
            if (t0 == 0) t0 = now;
            else if (now - t0 > kGemmWaitCycles) break;
        }
    }
    *abort = 1;
    atomicExch(error, 1u);
    return false;
}

template <bool FEW> struct GemmShared {
    static constexpr int kGemmStages = GemmShape<FEW>::kStages;
    uint64_t full[kGemmStages];      // stage filled by both blocks' TMA    (first block: 1 arrival + bytes)
    uint64_t empty[kGemmStages];     // stage read by the MMAs              (1: commit)
    uint64_t acc_full[2];            // accumulator complete                (1: commit)
    uint64_t acc_empty[2];           // accumulator read by the epilogues   (first block: one per epilogue warp of the pair)
    uint32_t tmem_base;
    int abort;
};

template <bool FEW>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GemmShape<FEW>::kThreads, 1)
sd_lmhead_kernel(const __grid_constant__ CUtensorMap map_g, const __grid_constant__ CUtensorMap map_x,
                 const __grid_constant__ CUtensorMap map_out, const GemmParams P) {
    using Shape = GemmShape<FEW>;
    constexpr int kGemmStages = Shape::kStages;
    extern __shared__ unsigned char gemm_smem_raw[];
    // (the same offsets in both blocks: the MMAs take them from one block's descriptors)
    unsigned char* smem = gemm_smem_raw + ((1024u - (smem_u32(gemm_smem_raw) & 1023u)) & 1023u);
    unsigned char* boxes = smem + kGemmStages * kGemmStageBytes;
    GemmShared<FEW>& sh = *reinterpret_cast<GemmShared<FEW>*>(boxes + Shape::kEpilogueWarps * kGemmBoxes * kGemmBoxBytes);
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    volatile int* abort = &sh.abort;

    const int tiles_m = (P.V + kGemmBM - 1) / kGemmBM, tiles_n = (P.d + kGemmBN - 1) / kGemmBN;
    const long long tiles = (long long)tiles_m * tiles_n;
    const int kblocks = (P.R + kGemmBK - 1) / kGemmBK;
    const long long first = blockIdx.x >> 1, step = gridDim.x >> 1;

    if (tid == 0) {
        for (int s = 0; s < kGemmStages; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(&sh.acc_full[a], 1); mbar_init(&sh.acc_empty[a], 2 * Shape::kEpilogueWarps); }
        sh.abort = 0;
        fence_barrier_init();
        fence_proxy_async();
    }
    if (warp == 1) tmem_alloc(&sh.tmem_base, kGemmTmemCols);     // the whole warp; the same warp frees it
    tc_fence_before();
    __syncthreads();
    cluster.sync();                            // both blocks' barriers stand before anything arrives on them
    tc_fence_after();
    const uint32_t tmem = sh.tmem_base;

    if (warp == 0) {
        // ---- producer
        if (lane == 0) {
            int stage = 0;
            uint32_t par = 1;                  // parity of the stage's previous use on empty[]
            long long n = 0;                   // stages issued so far
            bool ok = true;
            for (long long tile = first; tile < tiles && ok; tile += step) {
                const int m0 = (int)(tile / tiles_n) * kGemmBM + rank * 128, n0 = (int)(tile % tiles_n) * kGemmBN + rank * 128;
                for (int kb = 0; kb < kblocks; ++kb) {
                    if (n >= kGemmStages && !gemm_wait(&sh.empty[stage], par, abort, P.error)) { ok = false; break; }
                    unsigned char* a = smem + (size_t)stage * kGemmStageBytes;
                    unsigned char* b = a + kGemmABytes;
                    // the first block's barrier counts the bytes of both (boxes out of range count in full); the
                    // neighbour's may arrive before it is armed: the phase cannot end without this arrival
                    if (rank == 0) mbar_expect_tx(&sh.full[stage], 2u * (uint32_t)kGemmStageBytes);
                    const uint32_t bar = cluster_address(&sh.full[stage], 0);
                    const int r0 = kb * kGemmBK;
#pragma unroll
                    for (int c = 0; c < kGemmChunks; ++c)
                        tma_load_2d_pair(a + c * kGemmChunkBytes, &map_g, m0 + c * kGemmChunk, r0, bar);
#pragma unroll
                    for (int c = 0; c < kGemmChunks; ++c)
                        tma_load_2d_pair(b + c * kGemmChunkBytes, &map_x, n0 + c * kGemmChunk, r0, bar);
                    ++n;
                    if (++stage == kGemmStages) { stage = 0; par ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ---- MMA issuer of the pair
        if (lane == 0 && rank == 0) {
            constexpr uint32_t idesc = umma_idesc_bf16_mn(kGemmBM, kGemmBN);
            int stage = 0;
            uint32_t par = 0;
            long long it = 0;                  // tiles of this pair so far
            bool ok = true;
            for (long long tile = first; tile < tiles && ok; tile += step, ++it) {
                const int acc = (int)(it & 1);
                // the epilogues must have read this accumulator's previous tile
                if (it >= 2 && !gemm_wait(&sh.acc_empty[acc], (uint32_t)((it >> 1) - 1) & 1u, abort, P.error)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem + (uint32_t)acc * kGemmBN;
                for (int kb = 0; kb < kblocks; ++kb) {
                    if (!gemm_wait(&sh.full[stage], par, abort, P.error)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t a = smem_u32(smem + (size_t)stage * kGemmStageBytes);
                    const uint32_t b = a + kGemmABytes;
#pragma unroll
                    for (int k4 = 0; k4 < kGemmBK / 16; ++k4) {
                        // 16 positions further: 16 rows of 128 bytes
                        const uint64_t da = umma_desc_mn_sw128(a + k4 * 16 * 128, kGemmChunkBytes, 1024);
                        const uint64_t db = umma_desc_mn_sw128(b + k4 * 16 * 128, kGemmChunkBytes, 1024);
                        umma_bf16(d_tmem, da, db, idesc, (kb | k4) != 0 ? 1u : 0u);
                    }
                    umma_commit(&sh.empty[stage]);          // the stage is free once these MMAs have read it
                    if (++stage == kGemmStages) { stage = 0; par ^= 1u; }
                }
                if (ok) umma_commit(&sh.acc_full[acc]);
            }
        }
    } else {
        // ---- epilogue: warp w reads the tensor-memory lanes 32*(w%4) .. +31 (rows of this block's half)
        const int q = warp & 3, c0 = ((warp - 2) >> 2) * (Shape::kColumns / kGemmBox);
        unsigned char* const mine = boxes + (size_t)(warp - 2) * kGemmBoxes * kGemmBoxBytes;
        long long it = 0;
        int box = 0;
        bool ok = true;
        for (long long tile = first; tile < tiles && ok; tile += step, ++it) {
            const int acc = (int)(it & 1);
            const int m0 = (int)(tile / tiles_n) * kGemmBM + rank * 128, n0 = (int)(tile % tiles_n) * kGemmBN;
            int got = 1;
            if (lane == 0) got = gemm_wait(&sh.acc_full[acc], (uint32_t)(it >> 1) & 1u, abort, P.error) ? 1 : 0;
            got = __shfl_sync(0xffffffffu, got, 0);
            if (!got) { ok = false; break; }
            tc_fence_after();
            const int vbase = m0 + q * 32;               // first row of this warp's 32
#pragma unroll 1
            for (int c = c0; c < c0 + Shape::kColumns / kGemmBox; ++c) {
                uint32_t r[32];
                tmem_ld_32x32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * kGemmBN + c * kGemmBox), r);
                tmem_ld_wait();
                // the box that left from here two boxes ago has been read
                if (lane == 0) tma_store_wait<kGemmBoxes - 1, true>();
                __syncwarp();
                // lane = row of the box, 128 bytes; 16-byte pieces in the order of the 128-byte swizzle
                unsigned char* const stg = mine + box * kGemmBoxBytes;
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    *reinterpret_cast<uint4*>(stg + lane * 128 + ((e ^ (lane & 7)) << 4)) =
                        make_uint4(r[4 * e], r[4 * e + 1], r[4 * e + 2], r[4 * e + 3]);
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) {
                    if (vbase < P.V && n0 + c * kGemmBox < P.d) tma_store_2d(&map_out, n0 + c * kGemmBox, vbase, stg);
                    tma_store_commit();
                }
                box = box + 1 == kGemmBoxes ? 0 : box + 1;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(&sh.acc_empty[acc], 0);
        }
        if (lane == 0) tma_store_wait<0, false>();
    }
    __syncwarp();

    // leaving early: loads and MMAs in flight, whose barriers may be the neighbour's, have landed before either
    // block goes away
    tc_fence_before();
    __syncthreads();
    if (*abort) {
        const long long t0 = clock64();
        while (clock64() - t0 < kGemmLeaveCycles) {}
    }
    cluster.sync();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, kGemmTmemCols);
}

}  // namespace sdv
