// Tensor-core (tcgen05 / TMEM / TMA) instructions and conventions shared by the kernels that run on them.
#pragma once
#include <cuda.h>
#include <stdint.h>

#include "mbar.cuh"

namespace exmoe {

constexpr int BM = 128;            // weight rows per tile
constexpr int B_SBO = 1024;        // token operand: 128-byte swizzle, 8-row atoms of 1024 B
constexpr int N_MAPS = 16;         // tensor maps per operand: boxes of 16, 32, ..., 256 rows

struct Tile { int key, before, nrows, row0; };     // a run of grouped rows of one expert: key, weight of the tiles before it, rows, first row of the plan
// What a tile costs per weight tile, for the split of the work over the CTAs of the streaming tensor-core kernels: a block of 128 x 128
// takes 617 / 524 cycles (gate/up / down) with 16 rows, 597 / 704 with 32, 795 / 840 with 48, 773 / 989 with 64.
__host__ __device__ __forceinline__ int tile_weight(int nrows) { return 6 + (nrows + 15) / 16; }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit_at(uint32_t bar) {       // barrier by its shared-memory address
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// K order of the kernels whose weights are in tensor memory: position, inside its 64, of element w.  A lane (q, c) holds the codes
// of k = 8 c .. 8 c + 7 of every 32, and tcgen05.st.16x128b gives it every fourth cell (a cell is a pair of elements): inside every
// 32 the pairs (c, s) are stored as (s, c).  A sum over k does not care, as long as both operands agree.
__host__ __device__ __forceinline__ int k_position(int w) { return (w & 33) | ((w & 6) << 2) | ((w & 24) >> 2); }

// shared-memory matrix descriptor of the tokens, K-major, version 1 (sm_100)
__device__ __forceinline__ uint64_t make_desc_b(uint32_t saddr) {            // 128-byte swizzle
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3fff);
    d |= (uint64_t)1 << 16;                                                  // leading offset unused with swizzle
    d |= (uint64_t)((B_SBO >> 4) & 0x3fff) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}
// instruction descriptor: D fp32, A/B BF16, both K-major, M = 128, N = n
__device__ __forceinline__ uint32_t make_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

}  // namespace exmoe
