// Shared declarations of the exmoe CUDA library (sm_100a only).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <stddef.h>
#include "../../include/exmoe.h"

namespace exmoe {

// ---- packed layout (Eq. 3 / Eq. 4): 16-row panels x 128-wide blocks of 1056 bytes -------------
constexpr int kGroup = 128;          // scale group along K
constexpr int kPanelRows = 16;       // rows per panel (one m16 MMA tile)
constexpr int kBlockBytes = 1056;    // 1024 code bytes + 16 FP16 scales
constexpr int kCodeBytes = 1024;

// bytes of a packed [rows, K] matrix
__host__ __device__ inline size_t matrix_bytes(int rows, int K) {
    return (size_t)(rows / kPanelRows) * (K / kGroup) * kBlockBytes;
}

// ---- plan buffers shared by the resolution, grouping and GEMM kernels ------------------------
// header words
enum { HDR_N_ACTIVE = 0, HDR_N_WAVES = 1, HDR_N_MISSES = 2, HDR_BAD_ID = 3, HDR_N_GROUPS = 4, HDR_N_VALID = 5,
       HDR_WORDS = 8 };

struct PlanPtrs {
    int32_t* header;        // [HDR_WORDS]
    int32_t* wave_of;       // [E]
    int32_t* slot_of;       // [E]
    int32_t* misses;        // [3*E] (expert, slot, wave)
    int32_t* key_miss;      // [n_keys] 1 where the group (wave, slot) holds an expert that missed in this call
    int n_keys;
    int32_t* counts;        // [n_keys]
    int32_t* offsets;       // [n_keys + 1]
    int32_t* group_keys;    // [n_keys] active keys, ascending
    int32_t* wave_start;    // [max_waves + 1] index into group_keys
    int32_t* perm;          // [max_pairs]
    int32_t* chunk_table;   // [n_keys][chunks] scratch of the chunked grouping (may be null)
    size_t chunk_table_words;
    int32_t* chunk_done;    // arrival counter of the chunked grouping (zero between calls)
};

struct LayerState {         // Section 3.3 state of one layer, device memory
    int32_t* expert_slot;   // [E]
    int32_t* slot_expert;   // [C]
    uint64_t* slot_stamp;   // [C]
    uint64_t* tick;         // [1]
    uint64_t* stats;        // [6] lookups, hits, misses, waves, h2d_bytes, forwards
};

struct GemmArgs {
    const uint8_t* slots;       // slot memory of the layer
    size_t slot_stride;         // bytes per slot
    const int32_t* counts;
    const int32_t* offsets;
    const int32_t* group_keys;
    const int32_t* wave_start;  // already offset to the wave: [0] first group, [1] end
    const int32_t* perm;
    const int32_t* key_miss;    // [n_keys] (see PlanPtrs); may be null
    int group_filter;           // 0 all groups of the wave; 1 only groups whose expert was resident; 2 only the missed ones
    int direct_keys;            // > 0: every key 0 .. direct_keys-1 is a (possibly empty) group of the call's only wave
                                // (all experts resident, key = expert id): kernels may read counts / offsets by key at
                                // once instead of going through wave_start and group_keys first.  The size of the key
                                // space: more than the number of experts where wave_cap is below num_slots
    // Streaming kernels, all experts resident: the ids of the call (null: read the plan).  Every CTA then groups them itself.
    const int32_t* ids;
    int n_pairs;
    int32_t* keep_ids;          // copy of the ids, from which the plan can be materialised on request
    int num_slots;              // C (key % C = slot)
    int top_k;
    int H, I;
};

// One wave of the small-problem path (decode): the GEMM kernels rebuild the grouping themselves.
struct SmallWave {
    const int32_t* ids;         // [n_pairs] top-k ids
    const int32_t* wave_of;     // null when C = E (slot = expert id, single wave)
    const int32_t* slot_of;
    int n_pairs, E, wave;
    PlanPtrs plan;              // published for the test hooks
    int* status;
    int* arrive;                // [T * H/16] zero-initialised arrival counters of the fused combine
    const __nv_bfloat16* hidden;
    __nv_bfloat16* act;
    const float* topk_w;
    float* y;
    __nv_bfloat16* out;
    int max_rows, max_groups;
    bool pairwise;              // T*k <= kPairMaxPairs and a single wave: per-pair gate/up, by-token down
    int32_t* saved_ids;         // [kPairMaxPairs]
};
constexpr int kPairMaxPairs = 32;
#ifndef EXMOE_SMALL_MAX_PAIRS
#define EXMOE_SMALL_MAX_PAIRS 24
#endif
constexpr int kSmallMaxPairs = EXMOE_SMALL_MAX_PAIRS;
constexpr int kSmallMaxSlots = 1024;

// launch accounting (exmoe_launch_count)
void count_launch(int n = 1);

// Raise a kernel's dynamic shared-memory limit once per device (function attributes are per device; the cache of
// "already done" is the caller's static SmemOnce, one per kernel instantiation).
struct SmemOnce { unsigned long long mask = 0; };
template <typename F>
inline bool allow_smem(F kern, int bytes, SmemOnce& once) {
    int dev = 0;
    const bool known = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64;
    if (known && ((once.mask >> dev) & 1ull)) return true;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
    if (known) once.mask |= 1ull << dev;
    return true;
}

// ---- kernel launchers (defined in the .cu files) ------------------------------------------------
int* pack_flag_word();      // a device word for one exmoe_pack call's non-finite flag (no allocation)
int launch_pack(const exmoe_shape& s, int n_experts, const void* wg, const void* wu, const void* wd, void* out,
                int* d_flag, cudaStream_t st);
void launch_resolve(const exmoe_shape& s, int C, int Cw, size_t bytes_per_expert, const int32_t* ids, int n_pairs,
                    LayerState state, PlanPtrs plan, int* d_status, cudaStream_t st);
// Device-initiated miss path: one kernel copies wave `wave`'s missed experts from the mapped host bank into their slots.
void launch_fetch_misses(const PlanPtrs& plan, int wave, const uint8_t* bank_dev, uint8_t* slots, size_t bpe, int E, int C,
                         cudaStream_t st, bool small_grid = false, bool follows_resolve = true);
void launch_group(const exmoe_shape& s, int C, int n_keys, int max_waves, bool identity, const int32_t* ids,
                  int n_pairs, PlanPtrs plan, int* d_status, cudaStream_t st);
// Streaming kernels (bulk-copy weight ring in shared memory) above kSmallMaxPairs pairs, up to 640.  Their time grows with the
// eight-row passes over the experts' weights, that of the tensor-core kernels with the experts that have rows, and the
// host knows neither.  Up to twelve rows per expert they would win beyond 640 pairs where the routing is uniform (64 experts
// of 2048 x 1024, top-8, 81 tokens: 82 against 97 us per layer) and lose where it is skewed (Zipf of strength 1.5: 74 against
// 63; 128 experts of 896 x 2048, 427 tokens: 124 against 48).
constexpr int kStreamMaxPairs = 640;
// ... and up to twelve rows per expert of at most 64 where both matrices run with their geometry as literals (d_model 2048,
// d_ff 1024): the kernels are faster there. 64 experts, top-8, 81 and 94 tokens: uniform routing 0.84 and 0.93 of the
// tensor-core kernels' time, Zipf 1.0 1.03 and 1.00, Zipf 1.5 1.17 and 1.28; and the weights are not rounded to BF16.
constexpr int kStreamMaxRowsLiteral = 12, kStreamMaxExpertsLiteral = 64;
// ... and up to 14 rows per expert on average, or 28 where the tensor-core kernels would leave SMs idle (the 128-row weight
// tiles of all experts are no more than the SMs). Against the tensor-core kernels at 12 / 14 / 20 / 24 rows per expert, uniform
// routing: 32 experts of 1024 x 512 0.94 / 0.95 / 1.21 / 1.28 of their time, 24 of 1536 x 768 0.99 / 1.11 / 1.34 / 1.52; with
// fewer tiles than SMs 16 of 512 x 256 0.64 / 0.91 / 0.97 / 0.99 (32 rows: 1.28), 8 of 256 x 128 0.65 / 0.92 / 0.98 / 1.02.
constexpr int kStreamMaxRows = 14, kStreamMaxRowsFew = 28;
// ... and up to 192 pairs where the eight warps of a consumer group cannot share K evenly (7, 9, 11, 13, 15 ... blocks): a group's
// time is its longest range's. 48 experts of 2048 x 1920, 480 pairs, Zipf 1.5: 1.36 of the tensor-core kernels' time;
// an offloaded cache of 16 of 48 experts of 1024 x 1664, top-1, no misses: 200 pairs 1.2, 341 pairs 1.3, 500 pairs 1.5.
constexpr int kStreamMaxPairsUneven = 192;
constexpr int kStreamOwnPlanKeys = 128, kStreamOwnPlanPairs = 640;        // most experts and pairs that the streaming kernels group themselves
int stream_max_pairs(const exmoe_shape& s);      // most pairs of a call that the streaming kernels take; 0: not this shape
[[nodiscard]] bool launch_stream_wave(const GemmArgs& a, const __nv_bfloat16* hidden, __nv_bfloat16* act, const float* topk_w, float* y,
                        int* status, int max_groups, bool gateup, bool down, cudaStream_t st);
void launch_small_wave(const GemmArgs& a, const SmallWave& w, cudaStream_t st, bool gateup, bool down);
// the per-pair kernels on HOST inputs that travel as kernel parameters; false (nothing queued) where that does not apply
[[nodiscard]] bool launch_pair_inline(const GemmArgs& a, const SmallWave& w, const void* hidden, const int32_t* ids, const float* weights, cudaStream_t st);
bool pair_path_fits(int H, int I, int top_k);                           // shared memory of the per-pair kernels within limits
bool small_path_fits(int H, int I, int num_slots, int n_pairs);         // ... of the in-CTA-grouping kernels
size_t prefill_scratch_bytes(int max_pairs, int num_experts);
// CUtensorMap objects of the grouped hidden rows and of the activations, in device memory: per matrix a family of 16
// maps whose boxes hold 16, 32, ..., 256 rows (a tile's box holds exactly the rows its MMAs read); x family, then act
constexpr size_t kPrefillMapBytes = 2 * 16 * 128;
struct PrefillMaps { unsigned char* dev; };
int prefill_setup(PrefillMaps* maps, const __nv_bfloat16* xg, const __nv_bfloat16* act, int max_pairs, int H, int I);
struct Tile;
// one wave on the streaming tensor-core kernels (token matrices in their K order); false: not launched
[[nodiscard]] bool launch_tc_stream_wave(const GemmArgs& g, const Tile* tiles, int tile_cap, const int32_t* n_tiles, int* status, const PrefillMaps* maps, __nv_bfloat16* act,
                           const float* topk_w, float* y, bool gateup, bool down, cudaStream_t st);
void launch_wait_selftest(int* status, long long budget_cycles, int* result, cudaStream_t st);
// Grouping and grouped copy of the hidden rows in one launch, for calls within these limits.  Its CTAs each count all pairs
// in shared memory: measured at 64 experts it wins up to 8192 pairs, at 16384 the separate kernels are 3 us faster.
constexpr int kPlanGatherPairs = 8192, kPlanGatherKeys = 1024;
void launch_plan_gather(const exmoe_shape& s, int C, int n_keys, int max_waves, bool identity, const __nv_bfloat16* hidden,
                        const int32_t* ids, int n_pairs, PlanPtrs plan, int* status, __nv_bfloat16* xg, bool single_wave,
                        void* scratch, int tile_rows, bool k_order, cudaStream_t st);
// grouped copy of the hidden rows; when `single_wave` is given its CTA 0 also builds that wave's tile list in `scratch`
void launch_gather_rows(const __nv_bfloat16* hidden, const int32_t* perm, const int32_t* n_valid, int n_pairs, int top_k,
                        int H, __nv_bfloat16* xg, const GemmArgs* single_wave, const int32_t* wave_start, void* scratch,
                        int tile_rows, bool k_order, cudaStream_t st);
// which: bit 0 = gate/up GEMM + SwiGLU, bit 1 = down GEMM x routing weight, bit 2 = (re)build the wave's tile list
// kind: the 64-row, eight-stage kernel shape (a few dozen rows per expert), the 256-row, four-stage one, or the streaming kernels
// false: not launched
[[nodiscard]] bool launch_prefill_wave(const GemmArgs& g, const int32_t* wave_start, void* scratch, int* status, const PrefillMaps* maps,
                         __nv_bfloat16* act, const float* topk_w, float* y, int which, int kind, int tile_rows, cudaStream_t st);
enum { TC_SMALL_N = EXMOE_TENSOR_ROWS64, TC_LARGE = EXMOE_TENSOR_ROWS256, TC_STREAM = EXMOE_TENSOR_STREAM };     // kind of a tensor-core call
// Whether this device can run the streaming tensor-core kernels.  Asked when a cache is created: a call's rows are copied in
// these kernels' own K order, so the choice cannot be taken back where they are launched.
bool tc_stream_runs();
// The streaming tensor-core kernels: beyond the streaming kernels' range up to 24 rows per expert, for layers whose gate/up
// matrices come to 100 blocks of 128 x 128 per SM and whose K is at least 2048 (their launches take 2.5 us longer to their first MMA than
// the other tensor-core kernels, which smaller layers and few active experts do not earn back).  Up to 1024 pairs, where the others
// have tiles of 64 rows too and convert a hot expert's weights as often; beyond, where these take up to 256 rows per conversion, up to
// 144 tokens (an expert has no more rows than that).  Of the other kernels' time, routing uniform / Zipf 0.5 / 1.0 / 1.25 / 1.5, means
// of four routings:
//   64 experts of 2048 x 1024, top-8: 100 tokens 0.82 / 0.81 / 0.87 / 0.89 / 1.02    128: 0.87 / 0.81 / 0.91 / 0.93 / 0.94    144: 0.86 / 0.87 / 0.92 / 0.98 / 1.00
//                                     160: 0.87 / 0.88 / 0.94 / 0.99 / 1.02 (not taken)   192: 0.86 / 0.88 / 0.91 / 1.02 / 1.03 (not taken)   top-6, 192 tokens: 1.10 at Zipf 1.5 (not taken)
//   60 of 2048 x 1408, top-4: 170 tokens 0.78 / 0.83 / 0.86 / 0.93 / 0.92    256: 0.83 / 0.82 / 0.88 / 0.91 / 0.98    300: 0.83 / 0.85 / 0.92 / - / 1.17 (not taken)
//   96 of 4096 x 512, top-2: 400 tokens 0.79 / 0.84 / 0.95 / 0.87 / 1.04    1150: 0.85 / 0.89 / 1.01 / - / 1.19 (not taken)
//   48 of 2304 x 1536, top-2: 500 tokens 0.84 / 0.82 / 0.89 / 0.94 / 0.93    570: 0.83 / 0.89 / 0.98 / - / 1.27 (not taken)
//   Not taken for their size: 96 of 1024 x 1408, top-2, 500 tokens 0.80 / 0.90 / - / - / 1.13; 40 of 896 x 1152, top-5, 150 1.02 / 0.96 / - / - / 1.16; 16 of 512 x 256,
//   top-4, 200 1.33 / 1.27 / - / - / 1.29.
// By the layer's experts, not the cache's slots: a call's bits do not depend on these.
constexpr int kTcStreamMaxRows = 24, kTcStreamMaxTokens = 144, kTcStreamMinBlocksPerSm = 100, kTcStreamMinModel = 2048;
bool tc_stream_takes(const exmoe_shape& s, int n_pairs);
int prefill_tile_rows(const exmoe_shape& s, int n_pairs, int experts_per_wave, int kind);     // most grouped rows per tile
#ifndef EXMOE_PREFILL_SMALL_N_MAX_PAIRS
#define EXMOE_PREFILL_SMALL_N_MAX_PAIRS 1024
#endif
constexpr int kPrefillSmallNMaxPairs = EXMOE_PREFILL_SMALL_N_MAX_PAIRS;
void launch_combine(const float* y, const int32_t* ids, int E, int T, int k, int H, __nv_bfloat16* out,
                    cudaStream_t st);

}  // namespace exmoe
