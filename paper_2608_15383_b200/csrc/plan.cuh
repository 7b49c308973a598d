// Device code shared by the kernels that group the pairs of a call by (wave, slot).
#pragma once
#include "common.cuh"

namespace exmoe {

// ------------------------------------------------------------------------------------------------
// Grouping.  key(pair p) = wave_of[e]*C + slot_of[e]  (identity mode, C = E: key = e).
// Pairs with an invalid id are left out.  perm = pair indices ordered by key, ties by ascending p.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int pair_key(int id, int E, int C, bool identity, const int32_t* wave_of,
                                        const int32_t* slot_of) {
    if (id < 0 || id >= E) return -1;
    if (identity) return id;
    return wave_of[id] * C + slot_of[id];
}

// warp 0: exclusive scan of counts, list of active keys, first group of every wave, header
__device__ __forceinline__ void scan_keys_warp0(const int32_t* cnt, int n_keys, int C, int max_waves, PlanPtrs plan,
                                                int32_t* off_out, bool identity, int n_active_hint) {
    const int lane = threadIdx.x;
    const unsigned lt = (1u << lane) - 1u;
    int running = 0, ng = 0;
    for (int base = 0; base < n_keys; base += 32) {
        const int kx = base + lane;
        const int v = kx < n_keys ? cnt[kx] : 0;
        int incl = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        if (kx < n_keys) {
            off_out[kx] = running + incl - v;
            plan.counts[kx] = v;
            plan.offsets[kx] = running + incl - v;
        }
        const unsigned b = __ballot_sync(0xffffffffu, v > 0);
        if (v > 0) plan.group_keys[ng + __popc(b & lt)] = kx;
        ng += __popc(b);
        running += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
    __threadfence_block();
    if (lane == 0) {
        plan.offsets[n_keys] = running;
        off_out[n_keys] = running;
        plan.header[HDR_N_GROUPS] = ng;
        plan.header[HDR_N_VALID] = running;
        if (identity) {                                   // no resolution kernel ran: fill its header words
            plan.header[HDR_N_ACTIVE] = ng;
            plan.header[HDR_N_WAVES] = ng ? 1 : 0;
            plan.header[HDR_N_MISSES] = 0;
        }
    }
    __syncwarp();
    for (int w = lane; w <= max_waves; w += 32) {          // wave_start[w] = #active keys below w*C
        int c = 0;
        if (w * C >= n_keys) c = ng;                       // a single wave: nothing to read back
        else
            for (int g = 0; g < (w ? ng : 0); ++g) c += (plan.group_keys[g] < w * C);
        plan.wave_start[w] = c;
    }
}

}  // namespace exmoe
