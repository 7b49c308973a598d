// Streaming grouped W4A16 kernels for the middle regime (a few to a few dozen rows per expert): the two
// grouped expert GEMMs of a wave (Section 3.4, Eq. 2) as HBM-bound streams over the packed expert bytes,
// with the memory system decoupled from the arithmetic.
//
// The work of a wave is cut into units: (active group = expert, pass over up to eight of the group's rows,
// tile of PP panels; gate/up: PP gate+up panel pairs).  A tile is ONE contiguous range of the packed
// expert image.  Units are ordered group-major, then pass, then tile, and every persistent CTA (one per
// SM) takes an equal contiguous share, so that the load is balanced by arithmetic, not by expert, and a
// CTA's consecutive units share their activation rows.  A group with more rows than one pass holds
// re-reads its tiles once per pass (they come from L2).  Roles by warp:
//   warps 0-15  two consumer groups of eight warps that take alternate units: read the tile's packed bytes from shared
//               memory (the image is already in MMA fragment order), turn every word into FP16 operands (one shift, four
//               ANDs: see frag.cuh), mma.sync against the pass's rows, scale per 128-wide block in binary32; the K-split
//               partials cross shared memory once and the group's warps finish the tile (fixed summation order; SwiGLU
//               or routing weight; store).  When a unit starts a new (group, pass), all sixteen warps fetch its rows
//               (gathered through the plan's permutation for gate/up), convert them and store them.
//   warp 16     weight producer: one cp.async.bulk per unit into a ring of stages, completion counted in
//               bytes on the stage's mbarrier; runs as many stages ahead as the ring is deep.
// Bound: HBM for the gate/up kernel, 6.2 TB/s (96 % of the measured copy rate) per further expert, plus 7.5 us per launch
// that do not depend on the number of experts (plan, rows, first and last unit).  The down kernel's units take 2,000 cycles
// where HBM would take 1,470.  With BF16 operands (128 + u: three shifts and four lop3 a word, a second copy of the block
// corrections per group) the consumers were the bound: layer 53.2 -> 48.2 us at 16 tokens, 89.2 -> 77.6 at 64.
// Built and slower at 16 tokens: codes and split activations as e4m3 (mma.sync on e4m3 runs as conversions to FP16 and two
// FP16 MMAs here), 67 us; sixteen independent warps with their blocks in registers, no ring and no exchange per
// unit, 62 us (a warp's loads share a few scoreboards: waiting for the oldest block waits for the newest as well).
// The down kernel is a programmatic dependent of the gate/up kernel: its weight ring fills while the
// gate/up kernel drains; the consumers wait for the dependency before they fetch rows.
// Every mbarrier wait is bounded: on expiry the CTA raises EXMOE_ERR_TIMEOUT, all roles leave their
// loops and the producers wait (bounded) for their copies in flight before the CTA exits.
#include "common.cuh"
#include "frag.cuh"
#include "mbar.cuh"

#include <algorithm>
#include <type_traits>

namespace exmoe {

namespace {

constexpr int kGroupWarps = 8;                       // warps of one consumer group
constexpr int kGroupThreads = 32 * kGroupWarps;
constexpr int kGroups = 2;                           // consumer groups, alternate units (a third one: no change)
constexpr int kConsumerWarps = kGroups * kGroupWarps;
constexpr int kStreamThreads = 32 * (kConsumerWarps + 1);
constexpr int kMaxStages = 8;
constexpr int kPassRows = 8;                         // rows of one pass: the columns of one MMA tile (sixteen: slower at every size)
constexpr size_t kSmemLimit = 227 * 1024;
constexpr int kScanChunks = 4;                       // chunks of 32 groups whose plan entries the scan keeps in registers
constexpr int kMetaGroups = 64;                      // most groups one CTA's share of the units can touch (see stream_geometry)

// one lane waits, the whole warp learns the outcome (the producers' control flow stays warp-uniform)
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status) {
    int ok = 1;
    if ((threadIdx.x & 31) == 0) ok = mbar_wait(bar, parity, abort_flag, status) ? 1 : 0;
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}
// untiled bulk copy global -> shared (both 16-byte aligned, size a multiple of 16), no multicast
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void group_sync(int grp) {              // named barrier of one consumer group
    asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(kGroupThreads) : "memory");
}

// The gate/up producer starts when the first rows have been requested: behind a full ring of weight requests from every SM
// (20 MB) they came 2,000 cycles later, and no unit can start without them (44.6 -> 43.7 us per layer at 16 tokens).
__device__ __forceinline__ void rows_requested() { asm volatile("bar.arrive 9, %0;" ::"n"(kStreamThreads) : "memory"); }
__device__ __forceinline__ void wait_rows_requested() { asm volatile("bar.sync 9, %0;" ::"n"(kStreamThreads) : "memory"); }
__device__ __forceinline__ void rows_sync() {                      // all consumers
    asm volatile("bar.sync 8, %0;" ::"n"(32 * kConsumerWarps) : "memory");
}

struct StreamGeom {
    int PP, KS, tiles, n_stages, n_xbuf;
    uint32_t stage_bytes, x_stride;
    size_t off_x, off_part, off_cst, off_row, off_bar, total;
};

constexpr size_t kBarBytes = 2 * kMaxStages * 8 + 64;                 // mbarriers, abort flag, unit range
constexpr int kInlineKeys = kStreamOwnPlanKeys;
constexpr size_t kCtrlBytes = kBarBytes + (size_t)kMetaGroups * 16    // + plan entries of the CTA's groups
                              + (size_t)kStreamOwnPlanPairs * 4 + kInlineKeys * 4 + kConsumerWarps * 8 * 4;

#ifndef EXMOE_STREAM_PP
#define EXMOE_STREAM_PP 0                                              // 0: choose; 1/2/4/8: force where feasible (timing experiments)
#endif

// Tile shape and shared-memory budget for one matrix kind.  The eight warps of a consumer group are PP panels x
// (gate | up) x KS ranges of K (ranges differ by one block where KS does not divide it, and are empty where K has fewer).
// Preference: a ring of at least four stages, then two row buffers over one, then the larger tile.
__host__ bool stream_geometry(int K, int NR, int NM, int R, StreamGeom* out) {
    const int KB = K / kGroup;
    const size_t x_stride = (size_t)K * 2 + 64;                        // bytes of one row; + 64: conflict-free 16-byte fragment loads
    long best = -1;
    for (int NX = 2; NX >= 1; --NX)
        for (int PP = 8 / NM; PP >= 1; PP >>= 1) {
            const int KS = 8 / (PP * NM);
            if (NR % (kPanelRows * PP)) continue;
            if (EXMOE_STREAM_PP && PP != EXMOE_STREAM_PP) continue;
            const size_t stage = (size_t)NM * PP * KB * kBlockBytes;
            if (stage > 96 * 1024) continue;
            const size_t xs = (size_t)NX * R * x_stride;
            const size_t part = (size_t)kGroups * 2 * kGroupWarps * (R / 8) * 128 * 4;
            const size_t cst = (size_t)NX * KB * R * 8;
            const size_t fixed = xs + part + cst + (size_t)NX * R * 8 + kCtrlBytes + 256;
            if (fixed + 2 * stage > kSmemLimit) continue;
            int S = (int)((kSmemLimit - fixed) / stage);
            if (S > kMaxStages) S = kMaxStages;
            const long score = (S >= 4 ? 2 : S == 3 ? 1 : 0) * 1000 + NX * 100 + PP;
            if (score <= best) continue;
            best = score;
            StreamGeom g{};
            g.PP = PP; g.KS = KS; g.tiles = NR / (kPanelRows * PP); g.n_stages = S; g.n_xbuf = NX;
            g.stage_bytes = (uint32_t)stage; g.x_stride = (uint32_t)x_stride;
            g.off_x = (size_t)S * stage;
            g.off_part = g.off_x + xs;
            g.off_cst = g.off_part + part;
            g.off_row = g.off_cst + cst;
            g.off_bar = (g.off_row + (size_t)NX * R * 8 + 63) & ~(size_t)63;
            g.total = g.off_bar + kCtrlBytes;
            *out = g;
        }
    return best >= 0;
}

// OLMoE's two matrices have instantiations with their geometry as literals (d_model 2048: 16 blocks, one panel pair per tile, K in
// four ranges; d_ff 1024: 8 blocks, four panels per tile, K in two ranges)
inline bool literal_geometry(bool gateup, int K, const StreamGeom& g) { return gateup ? K / kGroup == 16 && g.PP == 1 : K / kGroup == 8 && g.PP == 4; }

struct StreamArgs {
    GemmArgs a;
    const __nv_bfloat16* x_src;     // gate/up: hidden [T, H]; down: activations [pairs, I] in grouped row order
    __nv_bfloat16* act_out;         // gate/up result
    const float* topk_w;
    float* y_out;                   // down result x routing weight, [pairs, H] in pair order
    int* status;
    int PP, KS, n_stages, n_xbuf;
    uint32_t stage_bytes, x_stride;
    uint32_t off_x, off_part, off_cst, off_row, off_bar;
};

// position of a unit inside the CTA's share: index into the cached plan entries, pass, tile
struct Cursor {
    int gi, pass, tile;
    __device__ __forceinline__ void advance(int tiles, int passes) {
        if (++tile == tiles) {
            tile = 0;
            if (++pass == passes) {
                pass = 0;
                ++gi;
            }
        }
    }
};

// KBc, PPc: blocks along K and panels per tile as COMPILE-TIME constants (0 = taken from the
// arguments).  With run-time values about a third of the executed instructions were address arithmetic, predicates and
// loop control around the conversion and the MMAs; the shapes that matter (OLMoE's two matrices) get their own
// instantiations with the block loop unrolled and every stride a literal, all others run the generic one.
template <bool GATEUP, int KBc = 0, int PPc = 0>
__global__ void __launch_bounds__(kStreamThreads, 1)
stream_gemm_kernel(const StreamArgs p) {
    constexpr int NM = GATEUP ? 2 : 1;                                // matrices per tile
    constexpr int R = kPassRows;
    extern __shared__ __align__(128) unsigned char smem[];
    const GemmArgs& a = p.a;
    constexpr bool FIXED = KBc > 0;
    const int NR = GATEUP ? a.I : a.H;
    const int KB = FIXED ? KBc : (GATEUP ? a.H : a.I) / kGroup, K = KB * kGroup;
    const int PP = FIXED ? PPc : p.PP, KS = FIXED ? 8 / (PPc * NM) : p.KS;
    const uint32_t x_stride = FIXED ? (uint32_t)(KBc * kGroup * 2 + 64) : p.x_stride;
    const uint32_t stage_bytes = FIXED ? (uint32_t)(NM * PPc * KBc * kBlockBytes) : p.stage_bytes;
    const int tiles = NR / (kPanelRows * PP);
    const int S = p.n_stages, NX = p.n_xbuf;
    unsigned char* wst = smem;
    unsigned char* xs = smem + p.off_x;                                // [NX][R][x_stride]
    float* part = reinterpret_cast<float*>(smem + p.off_part);
    float2* cst = reinterpret_cast<float2*>(smem + p.off_cst);         // [NX][KB][R]
    int2* rowinfo = reinterpret_cast<int2*>(smem + p.off_row);         // [NX][R] down: (pair, routing weight)
    uint64_t* w_full = reinterpret_cast<uint64_t*>(smem + p.off_bar);
    uint64_t* w_empty = w_full + kMaxStages;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(w_empty + kMaxStages);
    int* s_range = const_cast<int*>(abort_flag) + 4;                   // [0] first unit, [1] end, [2] its pass, [3] its tile
    int4* meta_w = reinterpret_cast<int4*>(smem + p.off_bar + kBarBytes);             // (slot, rows, first row, first unit)
    const int4* meta = meta_w;
    int* s_key = reinterpret_cast<int*>(meta_w + kMetaGroups);         // [pairs] plan formed here: key of every pair
    int* s_cnt = s_key + kStreamOwnPlanPairs;                              // [kInlineKeys] pairs per key
    int* s_rows = s_cnt + kInlineKeys;                                 // [consumer warps][8] pairs of a pass's rows
    // With every expert resident (key = expert id) and a few hundred pairs, every CTA forms the plan by itself from the ids:
    // no grouping kernel before this one (2.5 us, and a launch), one L2 round trip before the first weight copy.
    const bool own_plan = a.ids != nullptr;

    const int tid = threadIdx.x, lane = tid & 31, warp = warp_uniform(tid >> 5);
    if (tid == 32) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&w_full[s], 1);
            mbar_init(&w_empty[s], kConsumerWarps);                    // both groups: see the consumer loop
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (own_plan && tid < kInlineKeys) s_cnt[tid] = 0;
#ifndef EXMOE_STREAM_NO_ENTRY_PDL
    // The gate/up kernel is itself launched as a programmatic dependent (of the grouping kernel when that runs
    // just before it, else of whatever does): its CTAs are placed and their barriers initialised while the ids or the plan
    // are still being written; they are read only after this wait.  The down kernel reads the ids and the plan without
    // waiting: it starts when every gate/up CTA is past its own wait.
    if (GATEUP) grid_dependency_wait();
#endif
    if (own_plan) {
        constexpr int PT = (kStreamOwnPlanPairs + kStreamThreads - 1) / kStreamThreads;
        int id[PT];
#pragma unroll
        for (int i = 0; i < PT; ++i) {
            const int pr = tid + i * kStreamThreads;
            id[i] = pr < a.n_pairs ? a.ids[pr] : -1;
        }
        __syncthreads();
        bool bad = false;
#pragma unroll
        for (int i = 0; i < PT; ++i) {
            const int pr = tid + i * kStreamThreads;
            if (pr >= a.n_pairs) continue;
            const bool valid = id[i] >= 0 && id[i] < a.num_slots;      // every expert has its slot: num_slots is their number (the key space, direct_keys, may be larger)
            s_key[pr] = valid ? id[i] : -1;
            if (valid) atomicAdd(&s_cnt[id[i]], 1);
            bad |= !valid;
            if (GATEUP && blockIdx.x == 0) a.keep_ids[pr] = id[i];     // the plan can be materialised from these on request
        }
        if (GATEUP && blockIdx.x == 0 && bad) atomicExch(p.status, EXMOE_ERR_BAD_EXPERT_ID);
        __syncthreads();
        if (warp == 0) {
            // rows and passes before each key in one scan: passes << 16 | rows
            constexpr int CH = kInlineKeys / 32;
            int rows[CH], incl[CH];
#pragma unroll
            for (int j = 0; j < CH; ++j) {
                rows[j] = s_cnt[32 * j + lane];
                incl[j] = ((rows[j] + R - 1) / R) << 16 | rows[j];
            }
#pragma unroll
            for (int m = 1; m < 32; m <<= 1)
#pragma unroll
                for (int j = 0; j < CH; ++j) {
                    const int v = __shfl_up_sync(0xffffffffu, incl[j], m);
                    if (lane >= m) incl[j] += v;
                }
            int before[CH + 1];
            before[0] = 0;
#pragma unroll
            for (int j = 0; j < CH; ++j) before[j + 1] = before[j] + __shfl_sync(0xffffffffu, incl[j], 31);
            const int U = (before[CH] >> 16) * tiles, share = U / (int)gridDim.x, longer = U - share * (int)gridDim.x;
            int u0 = share * (int)blockIdx.x + min((int)blockIdx.x, longer);       // the first CTAs take one more
            int u1 = u0 + share + ((int)blockIdx.x < longer ? 1 : 0);
            int found = 0;
#pragma unroll
            for (int j = 0; j < CH; ++j) {
                const int passes = (rows[j] + R - 1) / R, excl = before[j] + incl[j] - (passes << 16 | rows[j]);
                const int ustart = (excl >> 16) * tiles, uend = ustart + passes * tiles;
                const bool overlap = passes > 0 && ustart < u1 && uend > u0;
                const unsigned ballot = __ballot_sync(0xffffffffu, overlap);
                const int idx = found + __popc(ballot & ((1u << lane) - 1u));
                if (overlap && idx < kMetaGroups) meta_w[idx] = make_int4(32 * j + lane, rows[j], excl & 0xffff, ustart);
                found += __popc(ballot);
            }
            if (found > kMetaGroups) {
                if (lane == 0) atomicExch(p.status, EXMOE_ERR_STATE);
                u1 = u0;
            }
            if (lane == 0) {
                s_range[0] = u0;
                s_range[1] = u1;
            }
            __syncwarp();
            if (lane == 0 && u0 < u1) {
                const int off = u0 - meta[0].w, pass = off / tiles;
                s_range[2] = pass;
                s_range[3] = off - pass * tiles;
            }
        }
    } else if (warp == 0) {
        // This CTA's share of the wave's units, and the plan entries of the groups it touches (usually one or
        // two).  The plan entries of up to 32 * kScanChunks active groups are fetched in one go and kept in
        // registers for both steps (count the units; find the overlapping groups); beyond that they are re-read.
        // With every expert resident the keys are the expert ids and the wave is the whole call: counts and offsets are
        // then read by key at once (empty keys are empty groups), one round trip to L2 instead of three dependent ones
        // (wave_start, then group_keys, then counts / offsets) before the first weight copy can be issued.
        const bool direct = a.direct_keys > 0 && a.direct_keys <= 32 * kScanChunks;
        const int g0 = direct ? 0 : a.wave_start[0], n_groups = direct ? a.direct_keys : a.wave_start[1] - g0;
        int rkey[kScanChunks], rrows[kScanChunks], rrow0[kScanChunks];
#pragma unroll
        for (int j = 0; j < kScanChunks; ++j) {
            rkey[j] = 0;
            if (32 * j + lane < n_groups) rkey[j] = direct ? 32 * j + lane : a.group_keys[g0 + 32 * j + lane];
        }
#pragma unroll
        for (int j = 0; j < kScanChunks; ++j) {
            rrows[j] = rrow0[j] = 0;
            if (32 * j + lane < n_groups) {
                rrows[j] = a.counts[rkey[j]];
                rrow0[j] = a.offsets[rkey[j]];
            }
        }
        // group filter (miss fetch overlapped with compute): a launch takes only the groups whose expert was resident
        // (1) or only those that were fetched for this wave (2); the others count as empty
        const int filter = a.key_miss ? a.group_filter : 0;
#pragma unroll
        for (int j = 0; j < kScanChunks; ++j)
            if (filter && 32 * j + lane < n_groups && (a.key_miss[rkey[j]] != 0) != (filter == 2)) rrows[j] = 0;
        auto entry = [&](int chunk, int& key, int& rows, int& row0) {
            key = rows = row0 = 0;
            bool have = false;
#pragma unroll
            for (int j = 0; j < kScanChunks; ++j)
                if (chunk == j) {
                    key = rkey[j];
                    rows = rrows[j];
                    row0 = rrow0[j];
                    have = true;
                }
            if (!have && 32 * chunk + lane < n_groups) {
                key = a.group_keys[g0 + 32 * chunk + lane];
                rows = a.counts[key];
                row0 = a.offsets[key];
                if (filter && (a.key_miss[key] != 0) != (filter == 2)) rows = 0;
            }
        };
        int total = 0;
        for (int chunk = 0; 32 * chunk < n_groups; ++chunk) {
            int key, rows, row0;
            entry(chunk, key, rows, row0);
            int passes = (rows + R - 1) / R;
#pragma unroll
            for (int m = 16; m >= 1; m >>= 1) passes += __shfl_xor_sync(0xffffffffu, passes, m);
            total += passes;
        }
        const int U = total * tiles, share = U / (int)gridDim.x, longer = U - share * (int)gridDim.x;    // the first CTAs take one more
        int u0 = share * (int)blockIdx.x + min((int)blockIdx.x, longer);
        int u1 = u0 + share + ((int)blockIdx.x < longer ? 1 : 0);
        int run = 0, found = 0;
        for (int chunk = 0; 32 * chunk < n_groups && u0 < u1; ++chunk) {
            int key, rows, row0;
            entry(chunk, key, rows, row0);
            const int passes = (rows + R - 1) / R;
            int incl = passes;
#pragma unroll
            for (int m = 1; m < 32; m <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, m);
                if (lane >= m) incl += v;
            }
            const int ustart = (run + incl - passes) * tiles, uend = ustart + passes * tiles;
            const bool overlap = passes > 0 && ustart < u1 && uend > u0;
            const unsigned ballot = __ballot_sync(0xffffffffu, overlap);
            if (overlap) {
                const int idx = found + __popc(ballot & ((1u << lane) - 1u));
                if (idx < kMetaGroups) meta_w[idx] = make_int4(key % a.num_slots, rows, row0, ustart);   // .x = slot of the group
            }
            found += __popc(ballot);
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (found > kMetaGroups) {                     // cannot happen for the sizes this path is chosen for; never index past the table
            if (lane == 0) atomicExch(p.status, EXMOE_ERR_STATE);
            u1 = u0;
        }
        if (lane == 0) {
            s_range[0] = u0;
            s_range[1] = u1;
        }
        __syncwarp();
        if (lane == 0 && u0 < u1) {
            const int off = u0 - meta[0].w, pass = off / tiles;
            s_range[2] = pass;
            s_range[3] = off - pass * tiles;
        }
    }
    __syncthreads();
    grid_launch_dependents();                          // gate/up: the down kernel may start filling its weight ring; down: the
                                                       // combine kernel may be placed (it waits for this grid before it reads)
    const int u0 = s_range[0], u1 = s_range[1];
    const size_t mat_off = GATEUP ? 0 : matrix_bytes(2 * a.I, a.H);
    Cursor cur{0, s_range[2], s_range[3]};

    if (warp == kConsumerWarps) {
        // ---------------------------------------------------------------- weight producer
        // ring position and phase are carried along: no division in any per-unit path of this kernel (a runtime
        // integer division costs some 25 instructions, several of them on the quarter-rate conversion pipe)
        int n = 0, s = 0;
        uint32_t ph = 1;                               // parity of the stage's previous phase
        for (int u = u0; u < u1; ++u, ++n) {
            if (GATEUP && n == 0) wait_rows_requested();
            if (n >= S && !warp_wait(&w_empty[s], ph, abort_flag, p.status)) break;
            const int4 gm = meta[cur.gi];
            if (lane == 0) {
                const uint8_t* src = a.slots + (size_t)gm.x * a.slot_stride + mat_off + (size_t)cur.tile * stage_bytes;
                mbar_expect_tx(&w_full[s], stage_bytes);
                bulk_load(wst + (size_t)s * stage_bytes, src, stage_bytes, &w_full[s]);
            }
            __syncwarp();
            cur.advance(tiles, (gm.y + R - 1) / R);
            if (++s == S) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (*abort_flag && lane == 0) {                // copies in flight land before the shared memory is given up
            for (int j = (n > S ? n - S : 0); j < n; ++j) {
                const long long t0 = clock64();
                while (!mbar_try(&w_full[j % S], (j / S) & 1) && clock64() - t0 < kWaitBudget) {}
            }
        }
    } else {
        // ---------------------------------------------------------------- consumers
        const int grp = warp / kGroupWarps, cw = warp % kGroupWarps;
        const int q = lane >> 2, c = lane & 3;
        const int ks = cw % KS, mw = (cw / KS) % NM, pp = cw / (KS * NM);    // K range, matrix, panel
        const int kb_lo = ks * KB / KS, kb_hi = (ks + 1) * KB / KS;
        const uint32_t w_full_a = smem_u32(w_full), w_empty_a = smem_u32(w_empty);
        // partials of one unit: [pp][matrix][ks][word][lane], one buffer per group and unit parity
        constexpr int part_words = kGroupWarps * 128;
        float* partg = part + (size_t)grp * 2 * part_words;
        const int panel_local = NM * pp + mw;
        // this lane's places: packed words and scales of the warp's first block, row q, constants of rows 2c, 2c + 1
        const unsigned char* w_lane = wst + ((size_t)panel_local * KB + kb_lo) * kBlockBytes + lane * 16;
        const unsigned char* s_lane = wst + ((size_t)panel_local * KB + kb_lo) * kBlockBytes + kCodeBytes + q * 4;
        const unsigned char* x_lane = xs + (size_t)q * x_stride + (kb_lo * kGroup + 8 * c) * 2;
        const float2* c_lane = cst + (size_t)kb_lo * R + 2 * c;
        // fetching rows: item = (row, block), 16 lanes each
        const int hw = warp * 2 + (lane >> 4), l16 = lane & 15;
        int mine_cnt = 0;
        int s = -1, xb = 0;                            // weight stage and row buffer of the current unit
        uint32_t w_ph = 1;                             // the stage's barrier parity (flipped when the index wraps to 0)
        bool dep = false;
        // Both groups walk ALL units in order and observe every phase of every full barrier, also for units the other group
        // computes on, and release each stage only then: a parity wait is only valid for a waiter that is at most one phase
        // behind.  A failed (expired or aborted) wait never changes the control flow: the named barriers below need
        // all warps, so the thread runs on over whatever the buffers hold, stores nothing, and every later wait
        // returns at once because the abort flag is up.
        bool ok = true;
        for (int u = u0, n = 0; u < u1; ++u, ++n) {
            const int4 gm = meta[cur.gi];
            const int m_rows = gm.y, row0 = gm.z, tile = cur.tile, pass0 = cur.pass * R;
            const bool fresh = (u == u0 || tile == 0);
            cur.advance(tiles, (m_rows + R - 1) / R);
            const int rows_here = min(R, m_rows - pass0);
            if (++s == S) s = 0;
            if (s == 0) w_ph ^= 1u;
            if (fresh) {
                if (NX == 2) xb ^= 1;
                else rows_sync();                      // everybody is done with the rows in the only buffer
                if (!GATEUP && !dep) {
                    grid_dependency_wait();            // the gate/up kernel's activations are complete and visible
                    dep = true;
                }
                // With two buffers the one written here was last read two passes ago, and every warp has been past that
                // since the previous pass's barrier.
                unsigned char* xw = xs + (size_t)xb * R * x_stride + l16 * 16;
                float2* cwr = cst + (size_t)xb * KB * R;
                int* rows_w = s_rows + warp * 8;
                if (own_plan && (GATEUP || warp == 0)) {               // this warp's own list of the pass's pairs, in pair order
                    int seen = -pass0;
                    for (int p0 = 0; p0 < a.n_pairs && seen < rows_here; p0 += 32) {
                        const bool hit = p0 + lane < a.n_pairs && s_key[p0 + lane] == gm.x;
                        const unsigned b = __ballot_sync(0xffffffffu, hit);
                        const int rank = seen + __popc(b & ((1u << lane) - 1u));
                        if (hit && rank >= 0 && rank < rows_here) rows_w[rank] = p0 + lane;
                        seen += __popc(b);
                    }
                    __syncwarp();
                }
                int pair = 0;
                float weight = 0.f;
                if (!GATEUP && warp == 0 && lane < rows_here) {
                    pair = own_plan ? rows_w[lane] : a.perm[row0 + pass0 + lane];
                    weight = p.topk_w[pair];
                }
                const int items = rows_here * KB;
                constexpr int FL = 4;                  // items in flight per half-warp
                if (GATEUP && u == u0 && hw - (lane >> 4) >= items) rows_requested();
                for (int it0 = hw; it0 - (lane >> 4) < items; it0 += 2 * kConsumerWarps * FL) {
                    uint4 raw[FL];
#pragma unroll
                    for (int f = 0; f < FL; ++f) {
                        const int it = it0 + 2 * kConsumerWarps * f;
                        raw[f] = make_uint4(0, 0, 0, 0);
                        if (it < items) {
                            const int r = it / KB, row = row0 + pass0 + r;
                            const size_t src = GATEUP ? (size_t)((own_plan ? rows_w[r] : a.perm[row]) / a.top_k) : (size_t)row;
                            raw[f] = reinterpret_cast<const uint4*>(p.x_src + src * K + (it % KB) * kGroup)[l16];
                        }
                    }
                    if (GATEUP && u == u0 && it0 == hw) rows_requested();
#pragma unroll
                    for (int f = 0; f < FL; ++f) {
                        const int it = it0 + 2 * kConsumerWarps * f;
                        if (it - (lane >> 4) >= items) break;          // the same for the whole warp
                        float2 k2;
                        const uint4 x = f16_block(raw[f], k2);
                        if (it < items) {
                            const int r = it / KB, kb = it % KB;
                            *reinterpret_cast<uint4*>(xw + (size_t)r * x_stride + kb * kGroup * 2) = x;
                            if (l16 == 0) cwr[kb * R + r] = k2;
                        }
                    }
                }
                if (!GATEUP && warp == 0 && lane < rows_here) rowinfo[xb * R + lane] = make_int2(pair, __float_as_int(weight));
                rows_sync();
            }
            ok = mbar_wait_warp(w_full_a + 8 * s, w_ph, abort_flag, p.status) && ok;
            if (n % kGroups != grp) {                      // the other group's unit: nothing of this warp reads it
                if (elect_one()) mbar_arrive_at(w_empty_a + 8 * s);
                continue;
            }
            const unsigned char* w0 = w_lane + (size_t)s * stage_bytes;
            const unsigned char* s0 = s_lane + (size_t)s * stage_bytes;
            const unsigned char* x0 = x_lane + (size_t)xb * R * x_stride;
            const float2* c0 = c_lane + (size_t)xb * KB * R;
            float* pb = partg + (mine_cnt & 1) * part_words;
            ++mine_cnt;
            // the unit's blocks (columns of rows that the pass does not have hold whatever the buffer does: columns are
            // independent and theirs are never stored)
            float tot[4] = {0.f, 0.f, 0.f, 0.f};
            [[maybe_unused]] const int nb = kb_hi - kb_lo;
            [[maybe_unused]] constexpr int NBc = FIXED ? KBc / (8 / ((PPc > 0 ? PPc : 1) * NM)) : 1;
            auto block = [&](int b) {
                const uint4 w[2] = {*reinterpret_cast<const uint4*>(w0 + b * kBlockBytes),
                                    *reinterpret_cast<const uint4*>(w0 + b * kBlockBytes + 512)};
                const uint32_t sv = *reinterpret_cast<const uint32_t*>(s0 + b * kBlockBytes);
                float d[2][4];                                         // two chains
#pragma unroll
                for (int i = 0; i < 4; ++i) d[0][i] = d[1][i] = 0.f;
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int set = 0; set < 2; ++set) {
                        const CodeFrag cf(set ? w[h].z : w[h].x, set ? w[h].w : w[h].y);
                        const uint4 x = *reinterpret_cast<const uint4*>(x0 + (b * kGroup + 64 * h + 32 * set) * 2);
                        cf.first(d[set], x);
                        cf.second(d[set], x);
                    }
                const float2 sc = scales16(sv);
                const float4 k4 = *reinterpret_cast<const float4*>(c0 + b * R);            // rows 2 c and 2 c + 1
                tot[0] = fmaf(sc.x, fmaf(d[0][0] + d[1][0], k4.x, k4.y), tot[0]);
                tot[1] = fmaf(sc.x, fmaf(d[0][1] + d[1][1], k4.z, k4.w), tot[1]);
                tot[2] = fmaf(sc.y, fmaf(d[0][2] + d[1][2], k4.x, k4.y), tot[2]);
                tot[3] = fmaf(sc.y, fmaf(d[0][3] + d[1][3], k4.z, k4.w), tot[3]);
            };
            if constexpr (FIXED) {
#pragma unroll
                for (int b = 0; b < NBc; ++b) block(b);
            } else {
#pragma unroll 2
                for (int b = 0; b < nb; ++b) block(b);
            }
            __syncwarp();
            if (elect_one()) mbar_arrive_at(w_empty_a + 8 * s);        // this warp is done with the weight stage
            // Partials cross shared memory once (buffer alternates with the group's units, so one barrier per unit
            // is enough); then the warps finish the slices (panel, word): the sum over the K ranges in ascending
            // order, SwiGLU or routing weight, store.
            float* pw = pb + (size_t)((pp * NM + mw) * KS + ks) * 128 + lane;
#pragma unroll
            for (int i = 0; i < 4; ++i) pw[i * 32] = tot[i];
            group_sync(grp);
            const int slices = PP * 4;
#pragma unroll(FIXED ? (PPc > 1 ? PPc / 2 : 1) : 1)
            for (int sl = cw; sl < slices; sl += kGroupWarps) {
                const int spp = FIXED && PPc == 1 ? 0 : sl / 4, ji = sl - spp * 4;
                float v[NM];
#pragma unroll
                for (int mg = 0; mg < NM; ++mg) {
                    const float* pr = pb + (size_t)((spp * NM + mg) * KS) * 128 + ji * 32 + lane;
                    float sum = pr[0];
                    for (int k2 = 1; k2 < KS; ++k2) sum += pr[k2 * 128];
                    v[mg] = sum;
                }
                const int rr = 2 * c + (ji & 1);                       // row of the pass
                if (rr >= rows_here || !ok) continue;
                const int orow = (tile * PP + spp) * kPanelRows + q + 8 * (ji >> 1);
                if (GATEUP) {
                    const float gv = v[0], uv = v[NM - 1];
                    p.act_out[(size_t)(row0 + pass0 + rr) * a.I + orow] = __float2bfloat16_rn(gv / (1.f + __expf(-gv)) * uv);
                } else {
                    const int2 ri = rowinfo[xb * R + rr];
                    p.y_out[(size_t)ri.x * a.H + orow] = __int_as_float(ri.y) * v[0];
                }
            }
        }
    }
}

template <bool GATEUP>
bool launch_stream_cfg(const GemmArgs& a, const __nv_bfloat16* x, __nv_bfloat16* act, const float* w, float* y, int* status,
                       int max_groups, bool dependent, cudaStream_t st) {
    constexpr int NM = GATEUP ? 2 : 1;
    StreamGeom g;
    if (!stream_geometry(GATEUP ? a.H : a.I, GATEUP ? a.I : a.H, NM, kPassRows, &g)) return false;
    void (*kern)(const StreamArgs) = stream_gemm_kernel<GATEUP>;
    int variant = 0;
#ifndef EXMOE_STREAM_GENERIC_ONLY
    if (literal_geometry(GATEUP, GATEUP ? a.H : a.I, g)) {
        kern = stream_gemm_kernel<GATEUP, GATEUP ? 16 : 8, GATEUP ? 1 : 4>;
        variant = 1;
    }
#endif
    static SmemOnce smem_once[2];
    allow_smem(kern, (int)kSmemLimit, smem_once[variant]);
    int sms = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        sms = 148;
    StreamArgs p{};
    p.a = a;
    p.x_src = x;
    p.act_out = act;
    p.topk_w = w;
    p.y_out = y;
    p.status = status;
    p.PP = g.PP;
    p.KS = g.KS;
    p.n_stages = g.n_stages;
    p.n_xbuf = g.n_xbuf;
    p.stage_bytes = g.stage_bytes;
    p.x_stride = g.x_stride;
    p.off_x = (uint32_t)g.off_x;
    p.off_part = (uint32_t)g.off_part;
    p.off_cst = (uint32_t)g.off_cst;
    p.off_row = (uint32_t)g.off_row;
    p.off_bar = (uint32_t)g.off_bar;
    const long long units = (long long)max_groups * g.tiles;          // the wave's units when every group takes one pass
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3((unsigned)(units < sms ? (units < 1 ? 1 : units) : sms));
    lc.blockDim = dim3(kStreamThreads);
    lc.dynamicSmemBytes = g.total;
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = dependent ? 1 : 0;
#ifdef EXMOE_DISABLE_PDL
    lc.numAttrs = 0;
#endif
    cudaLaunchKernelEx(&lc, kern, p);
    count_launch();
    return true;
}

}  // namespace

int stream_max_pairs(const exmoe_shape& s) {
    StreamGeom gu, dn;
    if (!stream_geometry(s.d_model, s.d_ff, 2, kPassRows, &gu) || !stream_geometry(s.d_ff, s.d_model, 1, kPassRows, &dn)) return 0;
    const bool even = (s.d_model / kGroup) % gu.KS == 0 && (s.d_ff / kGroup) % dn.KS == 0;
    int sms = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        sms = 148;
    const int tiles = s.num_experts * std::max(2 * s.d_ff, s.d_model) / 128;
    const int rows = tiles <= sms ? kStreamMaxRowsFew : kStreamMaxRows;
    int pairs = even ? kStreamMaxPairs : kStreamMaxPairsUneven;
    if (literal_geometry(true, s.d_model, gu) && literal_geometry(false, s.d_ff, dn) && s.num_experts <= kStreamMaxExpertsLiteral)
        pairs = std::max(pairs, kStreamMaxRowsLiteral * s.num_experts - 1);
    return std::min(pairs, rows * s.num_experts);
}

// One wave on the streaming kernels: passes of eight rows of a group.
bool launch_stream_wave(const GemmArgs& a, const __nv_bfloat16* hidden, __nv_bfloat16* act, const float* topk_w, float* y,
                        int* status, int max_groups, bool gateup, bool down, cudaStream_t st) {
    bool ok = true;
#ifndef EXMOE_STREAM_NO_ENTRY_PDL
    const bool entry_dependent = true;
#else
    const bool entry_dependent = false;
#endif
    if (gateup) ok = launch_stream_cfg<true>(a, hidden, act, topk_w, y, status, max_groups, entry_dependent, st);
    // a programmatic dependent only when the gate/up kernel of the same wave was launched just before it
    if (down && ok) ok = launch_stream_cfg<false>(a, act, act, topk_w, y, status, max_groups, gateup, st);
    return ok;
}

}  // namespace exmoe
