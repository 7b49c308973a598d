// Streaming tensor-core kernels: the two grouped W4A16 GEMMs of a wave (Section 3.4, Eq. 2) for some dozens of rows per
// expert, where the bound is the stream of packed bytes and the tensor cores are fed straight from it.
//
// As in the large-row kernels the weights are the UMMA A operand (128 rows = 8 panels) and the tokens the B operand, but
//   - A is the CODES, (u - 8) x 2^-10 as BF16 (exact, 11 instructions per eight codes against 19 with the scale multiplied in),
//     in TENSOR MEMORY: written by tcgen05.st.16x128b, which hands a lane the cells of its fragment-ordered codes;
//   - every 128-wide block gets an accumulator of its own, and the drain warps add scale x accumulator to binary32 sums in
//     registers: the weights are not rounded to BF16;
//   - the packed bytes come through a ring of bulk copies, 135 KB deep, in copies of two blocks (eight copies of one block per A
//     block took the issuing warp 480 cycles, more than HBM needs for the block).
// With A in shared memory a 128 x 128 block costs 256 cycles of stores and 256 of operand reads of the 128 B per clock that the
// shared memory moves, next to the tokens' 100 to 200; with A in tensor memory the weights touch it once, as packed bytes.  A block
// takes 617 / 524 cycles (gate/up / down) with 16 rows against 893 / 851 in the other tensor-core kernels, 773 / 989 against
// 972 / 1003 with 64; HBM would deliver one every 377.  Bound: instructions, 1,700 of a warp per block, 0.62 issued per cycle and
// scheduler (43 % of them on the ALU pipe, 28 % on the FMA pipe); the split leaves the compiler 72 registers: it spills 12 bytes
// (gate/up) and 36 (down).  OLMoE-shaped layer, uniform routing / Zipf 0.5: 100 tokens 94 -> 78 /
// 102 -> 82 us, 128 tokens 95 -> 82 / 103 -> 84.
// Built and no faster: eight conversion warps of two panels, sixteen of one; a barrier per A block, accumulator and token slot
// (1,800 cycles per 128 of K); barrier waits with a suspend hint (+3 %) or in tight loops (+4 %); 16x256b stores (+2 %).
//
// Work: unit = (token tile of up to 64 rows, 128 weight rows); every CTA (one per SM) takes a contiguous share of the units of equal
// weight.  A step is two units that share a token tile (the tokens are fetched once for both), or one where the share or the tile ends.
// Per 128 of K a step has one or two products (A block x tokens); product i belongs to drain set i.
//
// Warps:  0       issues the MMAs (8 x K16 per product) and the commits
//         1       token producer: tensor-map loads, two boxes of 64 columns per 128 of K
//         2, 3    weight producers: eight bulk copies of 2112 bytes (two blocks of a panel each) per 256 of K and A block
//         4-11    drain sets 0 and 1, four warps each (TMEM lane quarter = warp % 4): 64 columns of binary32 sums per lane,
//                 then SwiGLU -> BF16 activations, or routing weight -> pair buffer
//         12-27   conversion: two groups of eight, alternate 128s of K
// TMEM (512 columns): two stages of two A blocks (64 columns each: 128 codes of a row, two per cell) and two accumulators (64).
//
// K order: inside every 64 of K the cells of a lane's codes belong to a permuted k; the token matrices are written in the
// same order (k_position), the grouped copy by its kernel, the activations by the gate/up epilogue.
//
// Every wait is bounded: on expiry the CTA raises EXMOE_ERR_TIMEOUT, all roles leave their loops, the producers wait (bounded)
// for their copies in flight, TMEM is freed.
#include <algorithm>

#include "common.cuh"
#include "frag.cuh"
#include "mbar.cuh"
#include "tc.cuh"

namespace exmoe {

namespace {

constexpr int kConvWarps = 16, kDrainWarps = 8;
constexpr int kThreads = 32 * (4 + kDrainWarps + kConvWarps);
constexpr int kListed = 128;                       // tiles of the list that a CTA keeps in shared memory
constexpr int kSetRows = 64;                       // token rows of a product
constexpr int kStageCols = 256, kACols = 64;       // TMEM: a stage's two A blocks, then its two accumulators
constexpr int kBSlots = 5, kBHalf = kSetRows * 128, kBSlotBytes = 2 * kBHalf;
constexpr int kWStages = 4, kWPanel = 2 * kBlockBytes, kWSub = 8 * kWPanel, kWStageBytes = 2 * kWSub;
constexpr size_t kSmemBytes = (size_t)kBSlots * kBSlotBytes + (size_t)kWStages * kWStageBytes + 1024 + 512 + kListed * 16;
static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");
// registers per thread after the split; the shares come out of the launch's own
constexpr int kRegsMisc = 40, kRegsDrain = 120, kRegsConv = 56;
constexpr int kRegsSplit = 128 * kRegsMisc + 32 * kDrainWarps * kRegsDrain + 32 * kConvWarps * kRegsConv;
static_assert(kRegsSplit <= 65536 / kThreads / 8 * 8 * kThreads, "more than a launch can bring");

struct TcStreamArgs {
    const uint8_t* slots;
    size_t slot_stride;
    const int32_t* perm;
    const Tile* tiles;
    const int32_t* n_tiles;    // device: tiles of the list, their weight
    int tile_cap;              // tiles that the list has room for
    int num_slots, H, I;
    int* status;
};

__device__ __forceinline__ void tc_mma_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// 16 lanes x 32 columns: lane (q, c) gives, for i = 0..7, column 4i + c: r[2i] = row q, r[2i+1] = row q + 8
__device__ __forceinline__ void tc_st_16x128b_x8(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile("tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                   "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
                 : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&r)[32]) {           // 16 columns into r[0..15]
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
// the loads are complete; the registers pass through, so that nothing that reads them moves in front of the wait
__device__ __forceinline__ void tc_wait_ld_of(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                   "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]),
                   "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]),
                   "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :: "memory");
}
__device__ __forceinline__ void tc_wait_ld_of16(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                   "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :: "memory");
}
// two binary32 fused multiply-adds: acc += s * (lo, hi)
__device__ __forceinline__ void fma2(float2& acc, float s, uint32_t lo, uint32_t hi) {
    asm("{\n\t.reg .b64 d, m, v;\n\t"
        "mov.b64 d, {%0, %1};\n\tmov.b64 m, {%2, %2};\n\tmov.b64 v, {%3, %4};\n\t"
        "fma.rn.f32x2 d, m, v, d;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "+f"(acc.x), "+f"(acc.y) : "f"(s), "r"(lo), "r"(hi));
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void expect_tx_at(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_load_at(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
// eight codes of one word -> (q, q') x 2^-10 pairs as BF16, K order.  A block's sum of 128 products is then no larger than its
// largest activation, whatever the codes are, so that what the scaled sum can hold the accumulator can hold too; the drain's scales
// give the 2^10 back.  (Codes as integers overflowed from activations of 3e35 on.)
constexpr float kCodeUnit = 1024.f;
__device__ __forceinline__ void codes_bf16(uint32_t w, uint32_t (&out)[4]) {
    uint32_t bias = 0x3e083e08u;                                   // BF16 136 x 2^-10 twice
    const __nv_bfloat162 b2 = *reinterpret_cast<__nv_bfloat162*>(&bias);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        uint32_t v;
        asm("lop3.b32 %0, %1, 0x000f000f, 0x3e003e00, 0xea;" : "=r"(v) : "r"(w >> (4 * s)));   // (128+u, 128+u') x 2^-10
        const __nv_bfloat162 q2 = __hsub2(*reinterpret_cast<__nv_bfloat162*>(&v), b2);         // exact: integers of 2^-10
        out[s] = *reinterpret_cast<const uint32_t*>(&q2);
    }
}

// Tile t of the list, past L1: the list's memory is another call's before this one.
__device__ __forceinline__ Tile listed_tile(const Tile* tiles, const int4* listed, int t) {
    const int4 v = t < kListed ? listed[t] : load_behind_wait_cg(reinterpret_cast<const int4*>(tiles) + t);
    return Tile{v.x, v.y, v.z, v.w};
}

// The steps of a CTA's share of the units, in order.  Walked by every role that needs to know a step's tile.
struct Steps {
    const Tile* tiles;
    const int4* listed;
    int left, mt_count, t, mt;                     // units left, weight tiles per token tile, current ones
    Tile cur;
    int n_a, m;                                    // this step: A blocks per 128 of K, first weight tile
    __device__ __forceinline__ void init(const Tile* tl, const int4* first, const int4 share, int mtc) {
        tiles = tl;
        listed = first;
        t = share.x;
        mt = share.y;
        left = share.z;
        mt_count = mtc;
        if (left > 0) cur = listed_tile(tiles, listed, t);
    }
    __device__ __forceinline__ bool step() {       // false: the share is done
        if (left <= 0) return false;
        if (mt == mt_count) {
            mt = 0;
            ++t;
            cur = listed_tile(tiles, listed, t);
        }
        m = mt;
        n_a = left >= 2 && mt + 1 < mt_count ? 2 : 1;
        mt += n_a;
        left -= n_a;
        return true;
    }
};

template <bool GATEUP>
__global__ void __launch_bounds__(kThreads, 1)
tc_stream_kernel(const TcStreamArgs a, const CUtensorMap* __restrict__ maps, __nv_bfloat16* __restrict__ act_out,
                 const float* __restrict__ topk_w, float* __restrict__ y_out) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);   // swizzled boxes need 1 KB alignment
    unsigned char* sB = smem;
    unsigned char* sW = smem + kBSlots * kBSlotBytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sW + kWStages * kWStageBytes);
    uint64_t* w_full = bars;                       // [kWStages] weight bytes
    uint64_t* w_empty = w_full + kWStages;
    uint64_t* b_full = w_empty + kWStages;         // [kBSlots] token boxes
    uint64_t* b_empty = b_full + kBSlots;
    uint64_t* full = b_empty + kBSlots;            // [2] the stage's A blocks are written, its accumulators have been read
    uint64_t* done = full + 2;                     // [2] the stage's MMAs are complete
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int4* s_share = reinterpret_cast<int4*>(tmem_slot + 4);            // first token tile, its first weight tile, units, token tiles
    int4* s_tiles = s_share + 1;                                       // [kListed] the list's first tiles

    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const int K = GATEUP ? a.H : a.I, KB = K / kGroup;
    const int MT = (GATEUP ? 2 * a.I : a.H) / BM;
    if (tid == 0) {
        for (int s = 0; s < kWStages; ++s) { mbar_init(&w_full[s], 2); mbar_init(&w_empty[s], kConvWarps); }
        for (int s = 0; s < kBSlots; ++s) { mbar_init(&b_full[s], 1); mbar_init(&b_empty[s], 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(&full[s], kConvWarps / 2 + kDrainWarps); mbar_init(&done[s], 1); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // The gate/up kernel needs the tile list.  The down kernel is a programmatic dependent of the gate/up kernel of the same
    // wave, whose CTAs are past this wait when it starts: only its tokens (and what its epilogue writes) wait.
    if (GATEUP) grid_dependency_wait();
    grid_launch_dependents();
    if (warp == 0) {
        // This CTA's share: the units whose middle lies in its part of the total weight.  Equal numbers of units left the CTAs of
        // experts with many rows 28 % behind the mean (128 tokens, Zipf 0.5: 93 k cycles against 73 k).  The list's first 128 tiles are
        // requested together with its length.
        int4 tl[kListed / 32];
#pragma unroll
        for (int j = 0; j < kListed / 32; ++j)
            tl[j] = 32 * j + lane < a.tile_cap ? load_behind_wait_cg(reinterpret_cast<const int4*>(a.tiles) + 32 * j + lane) : make_int4(0, 0, 0, 0);
        const int n = load_behind_wait_cg(a.n_tiles);
        const long long total = (long long)load_behind_wait_cg(a.n_tiles + 1) * MT;
#pragma unroll
        for (int j = 0; j < kListed / 32; ++j) s_tiles[32 * j + lane] = tl[j];
        __syncwarp();
        int at[2][2] = {{0, 0}, {0, 0}};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const long long edge = total * ((int)blockIdx.x + i) / gridDim.x;
            int count = 0;                             // tiles that begin at or before the edge
#pragma unroll
            for (int j = 0; j < kListed / 32; ++j)
                count += __popc(__ballot_sync(0xffffffffu, 32 * j + lane < n && (long long)tl[j].y * MT <= edge));
            for (int base = kListed; base < n; base += 32)
                count += __popc(__ballot_sync(0xffffffffu, base + lane < n && (long long)load_behind_wait_cg(&a.tiles[base + lane].before) * MT <= edge));
            if (count > 0) {
                const Tile v = listed_tile(a.tiles, s_tiles, count - 1);
                const int w = tile_weight(v.nrows);
                const long long in = edge - (long long)v.before * MT;
                at[i][0] = count - 1;
                at[i][1] = (int)min((long long)MT, (2 * in + w - 1) / (2 * w));        // units of the tile whose middle is before the edge
            }
        }
        if (lane == 0) *s_share = make_int4(at[0][0], at[0][1], (at[1][0] - at[0][0]) * MT + at[1][1] - at[0][1], n);
    }
    __syncthreads();
    const size_t mat_off = GATEUP ? 0 : matrix_bytes(2 * a.I, a.H);
    const uint32_t w_full_a = smem_u32(w_full), w_empty_a = smem_u32(w_empty), b_full_a = smem_u32(b_full), b_empty_a = smem_u32(b_empty),
                   full_a = smem_u32(full), done_a = smem_u32(done);
    auto matrix_of = [&](int key) { return a.slots + (size_t)(key < a.num_slots ? key : key % a.num_slots) * a.slot_stride + mat_off; };

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsMisc));
        Steps st;
        st.init(a.tiles, s_tiles, *s_share, MT);
        if (warp == 0) {
            // ---------------------------------------------------------- MMA issuer
            // One wait, one group of MMAs and two commits per 128 of K.  With a barrier and a commit of its own for every A block,
            // accumulator and token slot this warp took 1,800 cycles for two products of 80.
            int bs = 0, sg = 0;
            uint32_t bph = 0, ph = 0;
            const uint32_t tm = warp_uniform(tmem);
            const uint64_t db0 = make_desc_b(smem_u32(sB));
            bool ok = true;
            auto product = [&](uint32_t d_tmem, uint32_t a_tmem, uint64_t db, uint32_t idesc) {
#pragma unroll
                for (int j = 0; j < 8; ++j)            // K16 step: A 8 columns on, B 32 bytes on inside its 64-column box
                    tc_mma_ta(d_tmem, a_tmem + 8 * j, db + (uint64_t)(((j >> 2) * kBHalf + (j & 3) * 32) >> 4), idesc, j ? 1u : 0u);
            };
            while (ok && st.step()) {
                const bool two = st.n_a == 2;
                const uint32_t idesc = warp_uniform(make_idesc((st.cur.nrows + 15) & ~15));
                for (int kb = 0; kb < KB; ++kb) {
                    const uint64_t db = db0 + (uint64_t)(bs * (kBSlotBytes >> 4));
                    const uint32_t ta = tm + sg * kStageCols, td = ta + 2 * kACols;
                    ok = mbar_wait_warp(b_full_a + 8 * bs, bph, abort_flag, a.status) && mbar_wait_warp(full_a + 8 * sg, ph, abort_flag, a.status);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        product(td, ta, db, idesc);
                        if (two) product(td + kSetRows, ta + kACols, db, idesc);
                        tc_commit_at(done_a + 8 * sg);
                        tc_commit_at(b_empty_a + 8 * bs);
                    }
                    __syncwarp();
                    if (++bs == kBSlots) { bs = 0; bph ^= 1; }
                    sg ^= 1;
                    if (!sg) ph ^= 1;
                }
            }
        } else if (warp == 1) {
            // ---------------------------------------------------------- token producer
            if (!GATEUP) grid_dependency_wait();       // the gate/up kernel's activations are complete and visible
            int s = 0, n = 0;
            uint32_t ph = 1;
            bool ok = true;
            while (ok && st.step()) {
                const int box = (st.cur.nrows + 15) >> 4;
                const CUtensorMap* map = maps + box - 1;
                for (int kb = 0; kb < KB; ++kb) {
                    ok = mbar_wait_warp(b_empty_a + 8 * s, ph, abort_flag, a.status);
                    if (!ok) break;
                    if (elect_one()) {
                        const uint32_t dst = smem_u32(sB) + s * kBSlotBytes, bar = b_full_a + 8 * s;
                        expect_tx_at(bar, (uint32_t)box * 16 * 256);
                        tma_load_at(dst, map, kb * kGroup, st.cur.row0, bar);
                        tma_load_at(dst + kBHalf, map, kb * kGroup + 64, st.cur.row0, bar);
                    }
                    __syncwarp();
                    ++n;
                    if (++s == kBSlots) { s = 0; ph ^= 1; }
                }
            }
            if (*abort_flag)                           // boxes in flight land before the shared memory is given up
                for (int j = max(0, n - kBSlots); j < n; ++j) {
                    const long long t0 = clock64();
                    while (!mbar_try_at(b_full_a + 8 * (j % kBSlots), (j / kBSlots) & 1) && clock64() - t0 < kWaitBudget) {}
                }
        } else {
            // ---------------------------------------------------------- weight producers: warp 2 the first A block, warp 3 the second
            const int sub = warp - 2;
            int s = 0, n = 0;
            uint32_t ph = 1;
            bool ok = true;
            const size_t panel_bytes = (size_t)KB * kBlockBytes;
            while (ok && st.step()) {
                const uint8_t* src = reinterpret_cast<const uint8_t*>(warp_uniform(reinterpret_cast<unsigned long long>(matrix_of(st.cur.key) + (size_t)(st.m + sub) * 8 * panel_bytes)));
                for (int kb = 0; kb < KB; kb += 2, src += kWPanel) {
                    ok = mbar_wait_warp(w_empty_a + 8 * s, ph, abort_flag, a.status);
                    if (!ok) break;
                    const uint32_t bar = w_full_a + 8 * s, bytes = kb + 1 < KB ? kWPanel : kBlockBytes;
                    if (elect_one()) {
                        if (sub < st.n_a) {
                            expect_tx_at(bar, 8 * bytes);
                            const uint32_t to = smem_u32(sW) + s * kWStageBytes + sub * kWSub;
#pragma unroll
                            for (int p = 0; p < 8; ++p) bulk_load(to + p * kWPanel, src + p * panel_bytes, bytes, bar);
                        } else {
                            mbar_arrive_at(bar);
                        }
                    }
                    __syncwarp();
                    ++n;
                    if (++s == kWStages) { s = 0; ph ^= 1; }
                }
            }
            if (*abort_flag)                           // copies in flight land before the shared memory is given up
                for (int j = max(0, n - kWStages); j < n; ++j) {
                    const long long t0 = clock64();
                    while (!mbar_try_at(w_full_a + 8 * (j % kWStages), (j / kWStages) & 1) && clock64() - t0 < kWaitBudget) {}
                }
        }
    } else if (warp < 12) {
        // -------------------------------------------------------------- drain
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsDrain));
        const int set = (warp - 4) >> 2, e = warp & 3;
        const uint32_t tm = tmem + 2 * kACols + kSetRows * set + ((uint32_t)(32 * e) << 16);
        const int rr = lane & 15, scale_at = kCodeBytes + 2 * (2 * (rr & 7) + (rr >> 3));      // this lane's row of its panel
        Steps st;
        st.init(a.tiles, s_tiles, *s_share, MT);
        int sg = 0;
        uint32_t ph = 0;
        bool ok = true;
        if (elect_one()) {                             // both stages' accumulators are free
            mbar_arrive_at(full_a);
            mbar_arrive_at(full_a + 8);
        }
        __syncwarp();
        while (ok && st.step()) {
            if (set && st.n_a == 1) { // nothing for the second set: it only passes the stages on
                for (int kb = 0; kb < KB; ++kb) {
                    ok = mbar_wait_warp(done_a + 8 * sg, ph, abort_flag, a.status);
                    if (!ok) break;
                    if (elect_one()) mbar_arrive_at(full_a + 8 * sg);
                    __syncwarp();
                    sg ^= 1;
                    if (!sg) ph ^= 1;
                }
                continue;
            }
            const int mt = st.m + set, ncols = st.cur.nrows, row0 = st.cur.row0;
            const uint8_t* sp = matrix_of(st.cur.key) + ((size_t)mt * 8 + 2 * e + (lane >> 4)) * KB * kBlockBytes + scale_at;
            constexpr int AHEAD = 4;                   // scales in flight
            unsigned short sc[AHEAD];
#pragma unroll
            for (int i = 0; i < AHEAD; ++i) sc[i] = i < KB ? __ldg(reinterpret_cast<const unsigned short*>(sp + (size_t)i * kBlockBytes)) : 0;
            float2 acc[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] = make_float2(0.f, 0.f);
            for (int kb0 = 0; kb0 < KB && ok; kb0 += AHEAD) {
#pragma unroll
                for (int u = 0; u < AHEAD; ++u) {
                    const int kb = kb0 + u;
                    if (kb >= KB) break;
                    const float s = __half2float(__ushort_as_half(sc[u])) * kCodeUnit;     // exact
                    if (kb + AHEAD < KB) sc[u] = __ldg(reinterpret_cast<const unsigned short*>(sp + (size_t)(kb + AHEAD) * kBlockBytes));
                    ok = mbar_wait_warp(done_a + 8 * sg, ph, abort_flag, a.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t td = tm + sg * kStageCols;
                    uint32_t v[32];
                    if (ncols <= 16) {
                        tc_ld16(td, v);
                        tc_wait_ld_of16(v);
                    } else {
                        tc_ld32(td, v);
                        tc_wait_ld_of(v);
                    }
                    if (ncols > 32) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) fma2(acc[i], s, v[2 * i], v[2 * i + 1]);
                        tc_ld32(td + 32, v);
                        tc_wait_ld_of(v);
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (elect_one()) mbar_arrive_at(full_a + 8 * sg);
                    sg ^= 1;
                    if (!sg) ph ^= 1;
                    if (ncols > 32) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) fma2(acc[16 + i], s, v[2 * i], v[2 * i + 1]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 8; ++i) fma2(acc[i], s, v[2 * i], v[2 * i + 1]);
                        if (ncols > 16)
#pragma unroll
                            for (int i = 8; i < 16; ++i) fma2(acc[i], s, v[2 * i], v[2 * i + 1]);
                    }
                }
            }
            if (!ok) break;
            if (!GATEUP) {
#pragma unroll
                for (int ch = 0; ch < 2; ++ch) {
                    if (32 * ch >= ncols) break;
                    int pair = 0;
                    float w = 0.f;
                    if (32 * ch + lane < ncols) {
                        pair = a.perm[row0 + 32 * ch + lane];
                        w = topk_w[pair];
                    }
                    const int h = mt * BM + 32 * e + lane;
#pragma unroll
                    for (int j = 0; j < 32; ++j) {     // lane j holds pair and weight of its column
                        const int pj = __shfl_sync(0xffffffffu, pair, j);
                        const float wj = __shfl_sync(0xffffffffu, w, j);
                        const float val = j & 1 ? acc[16 * ch + j / 2].y : acc[16 * ch + j / 2].x;
                        if (32 * ch + j < ncols) y_out[(size_t)pj * a.H + h] = wj * val;
                    }
                }
            } else {
                // lanes 0-15: gate rows, lanes 16-31: up rows of the same 16 intermediates
                const int interm = (mt * 4 + e) * 16 + (lane & 15);
                const int pos = (interm & ~63) | k_position(interm & 63);
#pragma unroll
                for (int ch = 0; ch < 2; ++ch) {
                    if (32 * ch >= ncols) break;
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float lo = j & 1 ? acc[16 * ch + j / 2].y : acc[16 * ch + j / 2].x;
                        const float hi = j & 1 ? acc[16 * ch + 8 + j / 2].y : acc[16 * ch + 8 + j / 2].x;
                        const float recv = __shfl_xor_sync(0xffffffffu, (lane < 16) ? hi : lo, 16);
                        const int n = 32 * ch + ((lane < 16) ? j : j + 16);
                        const float g = (lane < 16) ? lo : recv;
                        const float up = (lane < 16) ? recv : hi;
                        if (n < ncols) act_out[(size_t)(row0 + n) * a.I + pos] = __float2bfloat16_rn(__fdividef(g, 1.f + __expf(-g)) * up);
                    }
                }
            }
        }
    } else {
        // -------------------------------------------------------------- conversion
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsConv));
        // Two groups of eight warps take alternate 128s of K, group i those of TMEM stage i.  In a group, two sets of four: where a
        // step has two A blocks, set i converts block i; where it has one, set i converts its i-th 64 columns.  A warp serves the two
        // panels of its TMEM lane quarter.
        const int e = warp & 3, grp = (warp - 12) >> 3, set = ((warp - 12) >> 2) & 1;
        Steps st;
        st.init(a.tiles, s_tiles, *s_share, MT);
        const uint32_t src0 = smem_u32(sW) + 2 * e * kWPanel + lane * 16;
        const uint32_t dst0 = tmem + grp * kStageCols + ((uint32_t)(32 * e) << 16);
        int ws = 0, sg = 0;
        uint32_t wph = 0, ph = 1;
        bool ok = true;
        auto half = [&](uint32_t at, uint32_t (&r)[16]) {          // 64 of K of the panel: 16 rows x 32 cells
            uint32_t wx, wy, wz, ww, x[4];
            asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(wx), "=r"(wy), "=r"(wz), "=r"(ww) : "r"(at) : "memory");
            codes_bf16(wx, x);                                     // row q, k = 8 c ..
            r[0] = x[0]; r[2] = x[1]; r[4] = x[2]; r[6] = x[3];
            codes_bf16(wy, x);                                     // row q + 8, the same k
            r[1] = x[0]; r[3] = x[1]; r[5] = x[2]; r[7] = x[3];
            codes_bf16(wz, x);                                     // row q, k = 32 + 8 c ..
            r[8] = x[0]; r[10] = x[1]; r[12] = x[2]; r[14] = x[3];
            codes_bf16(ww, x);
            r[9] = x[0]; r[11] = x[1]; r[13] = x[2]; r[15] = x[3];
        };
        while (ok && st.step()) {
            const bool two = st.n_a == 2;
            const uint32_t srcs = src0 + (two ? set * kWSub : set * 512), dsts = dst0 + (two ? set * kACols : set * (kACols / 2));
            for (int kb = 0; kb < KB; ++kb) {
                if (!(kb & 1)) ok = mbar_wait_warp(w_full_a + 8 * ws, wph, abort_flag, a.status);
                if (!ok) break;
                const bool last = (kb & 1) || kb + 1 == KB;
                if (sg == grp) {
                    const uint32_t src = srcs + ws * kWStageBytes + (kb & 1) * kBlockBytes;
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        uint32_t r0[16], r1[16];
                        half(src + p * kWPanel, r0);
                        if (two) half(src + p * kWPanel + 512, r1);
                        if (p == 0) {
                            ok = mbar_wait_warp(done_a + 8 * grp, ph, abort_flag, a.status);
                            if (!ok) break;
                            tc_fence_after();
                        } else if (last) {
                            __syncwarp();
                            if (elect_one()) mbar_arrive_at(w_empty_a + 8 * ws);
                        }
                        tc_st_16x128b_x8(dsts + ((uint32_t)(16 * p) << 16), r0);
                        if (two) tc_st_16x128b_x8(dsts + ((uint32_t)(16 * p) << 16) + kACols / 2, r1);
                    }
                    if (!ok) break;
                    tc_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (elect_one()) mbar_arrive_at(full_a + 8 * grp);
                    ph ^= 1;
                } else if (last) {
                    __syncwarp();
                    if (elect_one()) mbar_arrive_at(w_empty_a + 8 * ws);
                }
                if (last && ++ws == kWStages) { ws = 0; wph ^= 1; }
                sg ^= 1;
            }
        }
    }

    // ---------------------------------------------------------------------- teardown (all roles, abort or not)
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

template <bool GATEUP>
bool tc_stream_kernel_runs() {
    static SmemOnce once;
    cudaFuncAttributes at{};
    // the warpgroups' shares come out of the registers that the launch brings: fewer, and the split would wait for good
    return allow_smem(tc_stream_kernel<GATEUP>, (int)kSmemBytes, once) && cudaFuncGetAttributes(&at, tc_stream_kernel<GATEUP>) == cudaSuccess &&
           at.numRegs * kThreads >= kRegsSplit;
}

template <bool GATEUP>
bool launch_tc_stream(const TcStreamArgs& a, const CUtensorMap* maps, __nv_bfloat16* act, const float* topk_w, float* y, cudaStream_t st) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        sms = 148;
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(sms);
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = kSmemBytes;
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
#ifdef EXMOE_DISABLE_PDL
    lc.numAttrs = 0;
#endif
    if (cudaLaunchKernelEx(&lc, tc_stream_kernel<GATEUP>, a, maps, act, topk_w, y) != cudaSuccess) return false;
    count_launch();
    return true;
}

}  // namespace

bool tc_stream_runs() {
    const bool runs = tc_stream_kernel_runs<true>() && tc_stream_kernel_runs<false>();
    if (!runs) cudaGetLastError();
    return runs;
}

bool launch_tc_stream_wave(const GemmArgs& g, const Tile* tiles, int tile_cap, const int32_t* n_tiles, int* status, const PrefillMaps* maps, __nv_bfloat16* act,
                           const float* topk_w, float* y, bool gateup, bool down, cudaStream_t st) {
    TcStreamArgs a{};
    a.slots = g.slots;
    a.slot_stride = g.slot_stride;
    a.perm = g.perm;
    a.tiles = tiles;
    a.n_tiles = n_tiles;
    a.tile_cap = tile_cap;
    a.num_slots = g.num_slots;
    a.H = g.H;
    a.I = g.I;
    a.status = status;
    const CUtensorMap* mx = reinterpret_cast<const CUtensorMap*>(maps->dev);
    return (!gateup || launch_tc_stream<true>(a, mx, act, nullptr, nullptr, st)) &&
           (!down || launch_tc_stream<false>(a, mx + N_MAPS, nullptr, topk_w, y, st));
}

}  // namespace exmoe
