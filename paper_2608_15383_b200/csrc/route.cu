// Fused router (Eq. 1 of the paper, Section 3.1): z_t = W_r h_t (+ optional per-expert bias), softmax over all
// E experts, the k largest (ties to the lower expert id), mixture weights = the selected probabilities, not
// renormalised (Section 3.4).  It produces exmoe_moe_forward's `topk_ids` / `topk_weights` on the device, so a
// whole stack step can be captured in one CUDA graph without host-side routing.
//
// What bounds it: at decode sizes latency, at prefill sizes the binary32 FMA pipe and the L2 reads of the router
// matrix (E x H BF16, 256 KB for OLMoE).  So the experts of a group of tokens are spread over a CLUSTER of CTAs: with
// eight CTAs of eight warps and 64 experts every warp owns one expert, its whole 4 KB row in flight at once, instead
// of one SM pulling the 256 KB by itself (one CTA per token took 13.8 us at T = 1, weights cold, and 190 us at
// T = 8192, where every token re-read the matrix from L2).  From a few dozen tokens on a cluster takes several tokens
// per read of the matrix.  The arithmetic of a logit is the same in both forms, bit for bit (lane-strided chunks of
// eight products in ascending order, then a shuffle tree).  Above that the logits are a GEMM and run on the tensor
// cores (route_mma_kernel), with every decision that their rounding could turn repeated in that same arithmetic, so
// the choice of experts does not depend on the batch size.
// The logits travel through the cluster's shared memory to the CTA that owns the token, which does the softmax (expf,
// binary32) and the choice of the k largest, equal probabilities ordered by ascending id.
#include <cooperative_groups.h>

#include "common.cuh"
#include "frag.cuh"

namespace exmoe {

namespace {

namespace cg = cooperative_groups;

constexpr int kRouteThreads = 256;
constexpr int kRouteSmemMax = 200 * 1024;
constexpr int kRouteFewTokens = 48;       // several tokens per cluster from here on
constexpr int kRouteTokenTokens = 192;    // one CTA per token, few experts, from here on
constexpr int kRouteMmaTokens = 193;      // tensor cores from here on,
constexpr int kRouteMmaTokensShort = 224; // ... from here on up to 64 experts of d_model below 640
constexpr int kRouteWideTokens = 1152;    // ... with 32 instead of 16 experts per CTA
constexpr int kRouteWarps = kRouteThreads / 32;

__device__ __forceinline__ void unpack8(const uint4& a, float (&x)[8]) {
    const uint32_t r[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        x[2 * i] = __uint_as_float(r[i] << 16);
        x[2 * i + 1] = __uint_as_float(r[i] & 0xffff0000u);
    }
}
__device__ __forceinline__ float dot8(const float (&w)[8], const float (&x)[8]) {
    float d = 0.f;
#pragma unroll
    for (int n = 0; n < 8; ++n) d = fmaf(w[n], x[n], d);
    return d;
}
__device__ __forceinline__ float warp_sum(float s) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
    return s;
}

// Softmax over the E logits in `prob` (this CTA's shared memory) and the k largest, by one warp.
__device__ __forceinline__ void softmax_topk(float* prob, int E, int k, int lane, int32_t* __restrict__ ids_out,
                                             float* __restrict__ w_out) {
    float mx = -INFINITY;
    for (int e = lane; e < E; e += 32) mx = fmaxf(mx, prob[e]);
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, m));
    float sum = 0.f;
    for (int e = lane; e < E; e += 32) {
        const float v = expf(prob[e] - mx);
        prob[e] = v;
        sum += v;
    }
    sum = warp_sum(sum);
    __syncwarp();
    const float inv = 1.f / sum;
    // Arg-max over the experts not yet taken.  Probabilities are non-negative, so their bit patterns order as they do:
    // key = bits + 2, 1 for a NaN (chosen last), 0 for a taken expert; equal keys go to the lower id.
    for (int j = 0; j < k; ++j) {
        uint32_t best = 0;
        int best_e = 0x7fffffff;
        for (int e = lane; e < E; e += 32) {
            const float v = prob[e];
            const uint32_t key = v >= 0.f ? __float_as_uint(v) + 2u : v < 0.f ? 0u : 1u;
            if (key > best) {                                          // ascending e: the first maximum wins
                best = key;
                best_e = e;
            }
        }
        const uint32_t top = __reduce_max_sync(0xffffffffu, best);
        const int e = __reduce_min_sync(0xffffffffu, best == top ? best_e : 0x7fffffff);
        if (lane == 0) {
            ids_out[j] = e;
            w_out[j] = prob[e] * inv;
            prob[e] = -2.f;
        }
        __syncwarp();
    }
}

// The same by a whole CTA, for one token: the rounds of the arg-max (120 cycles each) are replaced by counting, for every
// expert, the experts that come before it (four threads per expert).  `pv`: E more floats of shared memory.  The counting
// takes time by E * E, the rounds by k: equal at about 160 experts for eight choices (one token, d_model 2048, rounds against
// counting: 64 experts 5.1 / 3.9 us, 128: 6.1 / 5.8, 192: 7.6 / 8.0, 256: 8.2 / 10.3; 4096 experts, d_model 1024: 58 / 755).
constexpr bool choose_by_counting(int E, int k) { return (long long)E * E <= 3200ll * k; }
static_assert(choose_by_counting(64, 8) && choose_by_counting(128, 8) && choose_by_counting(8, 2) && choose_by_counting(256, 64));
static_assert(!choose_by_counting(192, 8) && !choose_by_counting(256, 8) && !choose_by_counting(4096, 8));
__device__ __forceinline__ void softmax_topk_cta(float* prob, float* pv, int E, int k, int32_t* __restrict__ ids_out,
                                                 float* __restrict__ w_out) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float mx = -INFINITY;
    for (int e = lane; e < E; e += 32) mx = fmaxf(mx, prob[e]);
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, m));
    float sum = 0.f;                                                       // every warp for itself, in the same order
    for (int e = lane; e < E; e += 32) {
        const float v = expf(prob[e] - mx);
        if (warp == 0) pv[e] = v;
        sum += v;
    }
    sum = warp_sum(sum);
    __syncthreads();
    if (!(sum < INFINITY)) {                                               // a NaN among the logits
        if (warp == 0) softmax_topk(prob, E, k, lane, ids_out, w_out);
        return;
    }
    const float inv = 1.f / sum;
    for (int e0 = 0; e0 < E; e0 += kRouteThreads / 4) {
        const int e = e0 + (tid >> 2);
        const float v = e < E ? pv[e] : 0.f;
        int before = 0;
        for (int j = tid & 3; j < E; j += 4) {
            const float o = pv[j];
            before += o > v || (o == v && j < e);
        }
        before += __shfl_xor_sync(0xffffffffu, before, 1);
        before += __shfl_xor_sync(0xffffffffu, before, 2);
        if ((tid & 3) == 0 && e < E && before < k) {
            ids_out[before] = e;
            w_out[before] = v * inv;
        }
    }
}

// CL: CTAs per cluster; TB: tokens per cluster; COUNT: the choice by counting.
// Shared memory: the cluster's TB hidden rows (every CTA keeps all of them), then the logits of the ceil(TB / CL) tokens
// this CTA owns (token i belongs to rank i % CL).
template <int CL, int TB, bool COUNT>
__global__ void __launch_bounds__(kRouteThreads)
route_kernel(const __nv_bfloat16* hidden, const __nv_bfloat16* __restrict__ w_router,
             const float* __restrict__ bias, int T, int H, int E, int k, int32_t* __restrict__ ids_out,
             float* __restrict__ w_out) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint4* xs = reinterpret_cast<uint4*>(smem);                            // [TB][H / 8]
    float* prob = reinterpret_cast<float*>(smem + (size_t)TB * H * 2);     // [ceil(TB / CL)][E]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = blockIdx.x % CL, t0 = (blockIdx.x / CL) * TB;
    const int n_tok = min(TB, T - t0);
    const int chunks = H / 8;
    // A programmatic dependent of whatever precedes it in the stream: nothing is read before that has completed; and the
    // kernel after it may be placed at once (it waits for this one in the same way).
    grid_dependency_wait();
    grid_launch_dependents();
    constexpr int JB = 8;                                                  // chunks of an expert in flight
    const int gw = rank * kRouteWarps + warp;
    uint4 raw[JB];
    auto fetch = [&](int e, int j0) {
#pragma unroll
        for (int j = 0; j < JB; ++j) {
            const int i = lane + 32 * (j0 + j);
            raw[j] = make_uint4(0, 0, 0, 0);
            if (i < chunks && e < E) raw[j] = reinterpret_cast<const uint4*>(w_router + (size_t)e * H)[i];
        }
    };
    fetch(gw, 0);                                                    // in flight while the hidden rows are staged
    {
        const uint4* xrow = reinterpret_cast<const uint4*>(hidden + (size_t)t0 * H);
        for (int i = tid; i < n_tok * chunks; i += kRouteThreads) xs[i] = xrow[i];
        for (int i = n_tok * chunks + tid; i < TB * chunks; i += kRouteThreads) xs[i] = make_uint4(0, 0, 0, 0);
    }
    cg::cluster_group cluster = cg::this_cluster();
    __syncthreads();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // every CTA runs: its memory may be written
    const int nj = (chunks + 31) / 32;
    bool joined = false;
    for (int e0 = gw; e0 < E; e0 += CL * kRouteWarps) {
        float acc[TB];
#pragma unroll
        for (int t = 0; t < TB; ++t) acc[t] = 0.f;
        for (int j0 = 0; j0 < nj; j0 += JB) {
            if (j0 > 0 || e0 != gw) fetch(e0, j0);
#pragma unroll
            for (int j = 0; j < JB; ++j) {
                if (j0 + j >= nj) break;
                const int i = lane + 32 * (j0 + j);
                float w[8];
                unpack8(raw[j], w);
#pragma unroll
                for (int t = 0; t < TB; ++t) {
                    float x[8];
                    unpack8(i < chunks ? xs[t * chunks + i] : make_uint4(0, 0, 0, 0), x);
                    acc[t] += dot8(w, x);
                }
            }
        }
        if (!joined) {                                                     // before the first store into another CTA's memory
            asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
            joined = true;
        }
        const float b = bias ? bias[e0] : 0.f;
#pragma unroll
        for (int t = 0; t < TB; ++t) {
            const float sum = warp_sum(acc[t]);
            if (lane == 0 && t < n_tok) {
                float* dst = cluster.map_shared_rank(prob, t % CL);
                dst[(t / CL) * E + e0] = sum + b;
            }
        }
    }
    if (!joined) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    cluster.sync();
    static_assert(TB <= CL, "a CTA owns at most one token");
    if constexpr (COUNT) {
        if (rank < n_tok) softmax_topk_cta(prob, prob + E, E, k, ids_out + (size_t)(t0 + rank) * k, w_out + (size_t)(t0 + rank) * k);
    } else {
        if (rank < n_tok && warp == 0) softmax_topk(prob, E, k, lane, ids_out + (size_t)(t0 + rank) * k, w_out + (size_t)(t0 + rank) * k);
    }
}

// One CTA per token, no cluster and nothing held ahead in registers: many CTAs per SM.  For calls with more tokens than
// there is room for clusters and so few experts that reading the matrix again for every token costs little.  Same arithmetic.
__global__ void __launch_bounds__(kRouteThreads)
route_token_kernel(const __nv_bfloat16* hidden, const __nv_bfloat16* __restrict__ w_router,
                   const float* __restrict__ bias, int T, int H, int E, int k, int32_t* __restrict__ ids_out,
                   float* __restrict__ w_out) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint4* xs = reinterpret_cast<uint4*>(smem);                            // [H / 8]
    float* prob = reinterpret_cast<float*>(smem + (size_t)H * 2);          // [E]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, chunks = H / 8;
    grid_dependency_wait();
    const uint4* xrow = reinterpret_cast<const uint4*>(hidden + (size_t)blockIdx.x * H);
    for (int i = tid; i < chunks; i += kRouteThreads) xs[i] = xrow[i];
    __syncthreads();
    for (int e = warp; e < E; e += kRouteWarps) {
        const uint4* wrow = reinterpret_cast<const uint4*>(w_router + (size_t)e * H);
        float s = 0.f;
        for (int i = lane; i < chunks; i += 32) {
            const uint4 wv = wrow[i], xv = xs[i];
            const uint32_t wr[4] = {wv.x, wv.y, wv.z, wv.w}, xr[4] = {xv.x, xv.y, xv.z, xv.w};
            float d = 0.f;                                                 // dot8 without the sixteen unpacked values
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                d = fmaf(__uint_as_float(wr[n] << 16), __uint_as_float(xr[n] << 16), d);
                d = fmaf(__uint_as_float(wr[n] & 0xffff0000u), __uint_as_float(xr[n] & 0xffff0000u), d);
            }
            s += d;
        }
        s = warp_sum(s);
        if (lane == 0) prob[e] = s + (bias ? bias[e] : 0.f);
    }
    // not earlier: CTAs of the next kernel that wait in their places keep this kernel's from spreading evenly
    grid_launch_dependents();
    __syncthreads();
    if (warp == 0) softmax_topk(prob, E, k, lane, ids_out + (size_t)blockIdx.x * k, w_out + (size_t)blockIdx.x * k);
}

// every form is a programmatic dependent of the kernel before it in the stream (it waits for it before it reads anything)
template <typename F>
int launch_dependent(F kern, int ctas, int cluster, size_t smem, const exmoe_shape& s, const __nv_bfloat16* hidden,
                     const __nv_bfloat16* w, const float* bias, int T, int32_t* ids, float* wts, cudaStream_t st) {
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3((unsigned)ctas);
    lc.blockDim = dim3(kRouteThreads);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = cluster > 1 ? 2 : 1;
#ifdef EXMOE_DISABLE_PDL
    lc.attrs = attr + 1;
    --lc.numAttrs;
#endif
    if (cudaLaunchKernelEx(&lc, kern, hidden, w, bias, T, s.d_model, s.num_experts, s.top_k, ids, wts) != cudaSuccess) {
        cudaGetLastError();
        return EXMOE_ERR_CUDA;
    }
    count_launch();
    return EXMOE_OK;
}

template <int CL, int TB>
int launch_route(const exmoe_shape& s, const __nv_bfloat16* hidden, const __nv_bfloat16* w, const float* bias, int T,
                 int32_t* ids, float* wts, cudaStream_t st) {
    const size_t smem = (size_t)TB * s.d_model * 2 + 2 * (size_t)s.num_experts * 4;
    static SmemOnce once[2];
    const bool count = choose_by_counting(s.num_experts, s.top_k);
    const auto kern = count ? route_kernel<CL, TB, true> : route_kernel<CL, TB, false>;
    if (!allow_smem(kern, kRouteSmemMax + 4096 * 4, once[count])) return EXMOE_ERR_CUDA;
    return launch_dependent(kern, (T + TB - 1) / TB * CL, CL, smem, s, hidden, w, bias, T, ids, wts, st);
}

int launch_route_token(const exmoe_shape& s, const __nv_bfloat16* hidden, const __nv_bfloat16* w, const float* bias, int T,
                       int32_t* ids, float* wts, cudaStream_t st) {
    static SmemOnce once;
    if (!allow_smem(route_token_kernel, kRouteSmemMax, once)) return EXMOE_ERR_CUDA;
    return launch_dependent(route_token_kernel, T, 1, (size_t)s.d_model * 2 + (size_t)s.num_experts * 4, s, hidden, w, bias, T, ids, wts, st);
}

// ---- many tokens: the logits as a tensor-core GEMM -------------------------------------------------------------
// A CTA takes 16 tokens; its eight warps split K (32-wide steps, round robin) and their partial logits meet in shared
// memory.  Operands come straight from L2 in 16-byte loads: a lane's eight consecutive k serve two m16n8k16 steps of both
// operands, the permutation of K inside the step being the same on both sides.  Batches of a few hundred tokens are
// latency again: a cluster of four CTAs then splits the experts (16 of them each, four steps of loads in flight per warp);
// where these no longer find room on the chip at once (two CTAs per SM), two CTAs share the 16 tokens, half of the experts
// each, and read every row half as often (1024 tokens: 11.8 against 12.4 us, 1184: 16.2 against 13.9, 4096: 33 against 24).
// An MMA truncates: every product to 2^-25 of the largest one's (and the accumulator's) binade, the result to 24 bits (both
// measured).  So each starts from zero and its 16 products are added in binary32, to two running sums, which meet with
// the other warps' in a tree: against 64 bits the logits are off by 1.7e-9 |x| |w| in the root mean square at d_model 2048
// (the binary32 form 1.65e-9; all the MMAs of a warp in one accumulator 5.2e-9, and up to 3e-6 for rows with their largest
// values in front), the probabilities by no more than the binary32 form's.
// The experts are an integer decision, and the one made by the binary32 form above is kept: where two of a token's k + 1
// largest logits are closer than the two forms can be apart, those experts' logits are recomputed in the binary32 form
// and the choice is made on these.  With S = sum |x_i w_i| <= |x| |w|: the MMAs lose less than 15 / 4 + 1 units of 2^-23 of
// their products, together under 2^-20 S; every logit passes H / 512 + 6 additions here and 8 + H / 256 + 5 in the
// binary32 form, each off by 2^-24 S at most; |x| and |w| come out of BF16 sums of H / 64 terms, short of the true ones
// by (1 - 2^-9)^(H / 128) at most, both together by 1 / 1.14.
constexpr int kMmaMaxExperts = 128;
constexpr float kExpSubnormal = 85.f, kExpZero = 106.f;    // expf(-x): normal below the first (2^-126 is e^-87.3), 0 above the second (2^-150: e^-104)
constexpr int kMmaMaxModel = 4096;                    // |x|^2 and |w|^2 are summed in BF16 over H / 64 terms per lane
__device__ __forceinline__ float route_bound(int H) { return 1.14f * (0x1p-20f + (float)(21 + 3 * H / 512) * 0x1p-24f); }

// Binary32 logit of one expert, by one warp.
__device__ __noinline__ float logit_again(const __nv_bfloat16* x, const __nv_bfloat16* __restrict__ w, int H, int lane) {
    const uint4 *xr = reinterpret_cast<const uint4*>(x), *wr = reinterpret_cast<const uint4*>(w);
    float s = 0.f;
    for (int j0 = 0; j0 < H / 8; j0 += 256) {
        uint4 wv[8], xv[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (j0 + 32 * j + lane < H / 8) {
                wv[j] = wr[j0 + 32 * j + lane];
                xv[j] = xr[j0 + 32 * j + lane];
            }
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (j0 + 32 * j + lane < H / 8) {
                float wf[8], xf[8];
                unpack8(wv[j], wf);
                unpack8(xv[j], xf);
                s += dot8(wf, xf);
            }
    }
    return warp_sum(s);
}
// softmax_topk for at most kMmaMaxExperts experts and 32 choices: the same arithmetic and order, keys in registers, one store at the end
// (2.4 -> 1.0 us in a call's tail).
__device__ __forceinline__ void softmax_topk_few(const float* z, int E, int k, int lane, int32_t* __restrict__ ids, float* __restrict__ wts) {
    constexpr int PER = kMmaMaxExperts / 32;
    float mx = -INFINITY, v[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i)
        if (lane + 32 * i < E) mx = fmaxf(mx, z[lane + 32 * i]);
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, m));
    float sum = 0.f;
    uint32_t key[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        key[i] = 0;
        v[i] = 0.f;
        if (lane + 32 * i < E) {
            v[i] = expf(z[lane + 32 * i] - mx);
            key[i] = v[i] >= 0.f ? __float_as_uint(v[i]) + 2u : 1u;        // 1: a NaN, chosen last
            sum += v[i];
        }
    }
    const float inv = 1.f / warp_sum(sum);
    int mine = 0;
    float weight = 0.f;
    for (int j = 0; j < k; ++j) {
        uint32_t best = 0;
        int at = 0;
        float p = 0.f;
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (key[i] > best) {                                           // ascending experts: the first maximum wins
                best = key[i];
                at = i;
                p = v[i];
            }
        const uint32_t top = __reduce_max_sync(0xffffffffu, best);
        const int e = (int)__reduce_min_sync(0xffffffffu, best == top ? (unsigned)(lane + 32 * at) : 0x7fffffffu);
        p = __shfl_sync(0xffffffffu, p, e & 31);
        if (j == lane) {
            mine = e;
            weight = p * inv;
        }
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (lane + 32 * i == e) key[i] = 0;
    }
    if (lane < k) {
        ids[lane] = mine;
        wts[lane] = weight;
    }
}

// One token's choice from its tensor-core logits, by one warp: the k + 1 largest in order; where two of them are within
// `slack`, both are recomputed (at the cut everything that could displace the k-th) and the choice is made again.  A lane
// holds the logits of experts lane, lane + 32, ... as order-preserving integers.  What is to be recomputed is left in `todo` (a bit
// per expert) for the whole CTA, and true returned.
// The other forms order binary32 PROBABILITIES, equal ones by id, and so does the choice made again.  Two logits may share a
// probability where they differ: closer than expf resolves (its argument z - max is rounded to 2^-24 of itself, the
// result to a few units of 2^-23), or far enough below the largest that their probabilities are subnormal or zero.  So
// the first enters `near`, and a choice that reaches the second is made again in any case, with those logits recomputed
// whose probability is subnormal; the exponential of anything below them is zero in every form.
__device__ __forceinline__ bool choose(const float* z, float slack, int E, int k, int lane, uint32_t* todo, int32_t* __restrict__ ids,
                                       float* __restrict__ wts) {
    constexpr int PER = kMmaMaxExperts / 32;
    uint32_t key[PER];                                                     // 0: no expert, or taken
    bool odd = !(slack < INFINITY);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int e = lane + 32 * i;
        key[i] = 0;
        if (e < E) {
            const float v = z[e];
            odd |= !(v < INFINITY);                                        // a NaN or +infinity (-infinity: a masked expert)
            const uint32_t b = __float_as_uint(v);
            key[i] = b & 0x80000000u ? ~b : b | 0x80000000u;
        }
    }
    odd = __any_sync(0xffffffffu, odd);
    unsigned again = 0;
    float prev = INFINITY, top_v = 0.f;
    bool deep = false;
    int prev_e = 0, first_e = 0, mine = 0;                                              // mine, lane j: the j-th choice (k <= 32)
    for (int j = 0; j <= k && j < E && !odd; ++j) {
        uint32_t best = 0;
        int be = 0x7fffffff;
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (key[i] > best) {
                best = key[i];
                be = lane + 32 * i;
            }
        const uint32_t top = __reduce_max_sync(0xffffffffu, best);
        const int e = __reduce_min_sync(0xffffffffu, best == top ? be : 0x7fffffff);
        const float v = __uint_as_float(top & 0x80000000u ? top & 0x7fffffffu : ~top);
        if (j == 0) {
            top_v = v;
            first_e = e;
            odd = v == -INFINITY;                                          // every expert masked: NaN probabilities
        } else if (prev < top_v - kExpSubnormal + 2.f * slack) {           // another one follows: both may be subnormal or zero
            deep = true;
        }
        const float near = slack + 2.4e-7f * (fabsf(prev) + fabsf(v) + (top_v - v)) + 1e-6f;
        if (j > 0 && v > -INFINITY && prev - v <= near) {
            if (lane == (prev_e & 31)) again |= 1u << (prev_e >> 5);
            if (lane == (e & 31)) again |= 1u << (e >> 5);
            if (j == k)                                                    // the rest of the k-th's neighbourhood
#pragma unroll
                for (int i = 0; i < PER; ++i)
                    if (key[i] && z[lane + 32 * i] >= prev - near) again |= 1u << i;
        }
        if (j == lane && j < k) mine = e;
        prev = v;
        prev_e = e;
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (lane + 32 * i == e) key[i] = 0;
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int e = lane + 32 * i;
        if (odd) again |= 1u << i;
        if (deep && e < E && z[e] < top_v - kExpSubnormal + 2.f * slack && z[e] > top_v - kExpZero - 2.f * slack) again |= 1u << i;
        if (e >= E) again &= ~(1u << i);
    }
    if (deep || __any_sync(0xffffffffu, again != 0)) {
        if (lane == (first_e & 31)) again |= 1u << (first_e >> 5);         // the maximum, from which expf's arguments are measured
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const unsigned b = __ballot_sync(0xffffffffu, (again >> i) & 1u);
            if (lane == 0) todo[i] = b;
        }
        return true;
    }
    const float mx = __shfl_sync(0xffffffffu, z[mine], 0);
    float sum = 0.f;
    for (int e = lane; e < E; e += 32) sum += expf(z[e] - mx);
    sum = warp_sum(sum);
    if (lane < k) {
        ids[lane] = mine;
        wts[lane] = expf(z[mine] - mx) / sum;
    }
    return false;
}

// 16 tokens per CTA; NT: 8-expert tiles per CTA; CL: CTAs per cluster (CL * NT = 8: 64 experts per pass); U: steps of loads in
// flight (even: they alternate between the two running sums).  Two CTAs share an SM.
template <int NT, int CL, int U>
__global__ void __launch_bounds__(kRouteThreads, 2)
route_mma_kernel(const __nv_bfloat16* hidden, const __nv_bfloat16* __restrict__ w_router,
                 const float* __restrict__ bias, int T, int H, int E, int k, int32_t* __restrict__ ids_out,
                 float* __restrict__ w_out) {
    constexpr int TM = 16, EC = 8 * NT, EB = CL * EC;                       // experts of a CTA / of the cluster per pass
    static_assert(U % 2 == 0, "the two running sums");
    constexpr int TOK = TM / CL;                                           // tokens whose choice this CTA makes
    extern __shared__ __align__(16) unsigned char smem[];
    float* part = reinterpret_cast<float*>(smem);                          // [warp][TM][EC + 1]
    float* logit = part + kRouteWarps * TM * (EC + 1);                     // [TOK][kMmaMaxExperts] token i of the cluster: rank i % CL
    float* xn = logit + TOK * kMmaMaxExperts;                              // [warp][TM] partial |x|^2
    float* wn = xn + kRouteWarps * TM;                                     // [warp][EC] partial |w|^2
    float* wmax_of = wn + kRouteWarps * EC;                                // [CL][2] largest |w|^2 of each CTA's experts
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int q = lane >> 2, c = lane & 3;
    const int rank = blockIdx.x % CL, t0 = (blockIdx.x / CL) * TM, n_tok = min(TM, T - t0);
    const int steps = H / 32;
    cg::cluster_group cluster = cg::this_cluster();
    grid_dependency_wait();
    grid_launch_dependents();
    if (CL > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // every CTA runs: its memory may be written
    const __nv_bfloat162 zero2(__float2bfloat16(0.f), __float2bfloat16(0.f));
    const uint4* xrow[2];
    __nv_bfloat162 xsq[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {                                          // rows beyond the last token repeat it
        xrow[r] = reinterpret_cast<const uint4*>(hidden + (size_t)(t0 + min(8 * r + q, n_tok - 1)) * H) + c;
        xsq[r] = zero2;
    }
    auto square = [](__nv_bfloat162& sum, const uint4& v) {
        const uint32_t r[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const __nv_bfloat162 p = *reinterpret_cast<const __nv_bfloat162*>(&r[i]);
            sum = __hfma2(p, p, sum);
        }
    };
    auto quad_sum = [](const __nv_bfloat162& v) {
        float s = __low2float(v) + __high2float(v);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        return s + __shfl_xor_sync(0xffffffffu, s, 2);
    };
    float wtop = 0.f;
    for (int p0 = 0; p0 < E; p0 += EB) {
        const int e0 = p0 + rank * EC;
        float acc[2][NT][4];                                           // two running sums
        __nv_bfloat162 wsq[NT];
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            wsq[n] = zero2;
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[0][n][i] = acc[1][n][i] = 0.f;
        }
        const uint4* wrow = reinterpret_cast<const uint4*>(w_router) + (size_t)(e0 + q) * (H / 8) + c;
        const size_t wstep = (size_t)H;                                    // eight expert rows, in 16-byte chunks
        for (int s0 = warp; s0 < steps; s0 += U * kRouteWarps) {
            uint4 a[U][2], b[U][NT];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int s = s0 + u * kRouteWarps;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    a[u][r] = make_uint4(0, 0, 0, 0);
                    if (s < steps) a[u][r] = xrow[r][4 * s];
                }
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    b[u][n] = make_uint4(0, 0, 0, 0);
                    if (s < steps && e0 + 8 * n + q < E) b[u][n] = wrow[n * wstep + 4 * s];
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    const uint4 &lo = a[u][0], &hi = a[u][1];
                    float d[2][4] = {};
                    mma_m16n8k16(d[0], lo.x, hi.x, lo.y, hi.y, b[u][n].x, b[u][n].y);
                    mma_m16n8k16(d[1], lo.z, hi.z, lo.w, hi.w, b[u][n].z, b[u][n].w);
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[u & 1][n][i] += d[0][i] + d[1][i];
                }
#pragma unroll
                for (int n = 0; n < NT; ++n) square(wsq[n], b[u][n]);
                if (p0 == 0)
#pragma unroll
                    for (int r = 0; r < 2; ++r) square(xsq[r], a[u][r]);
            }
        }
        float* mine = part + warp * TM * (EC + 1);
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) mine[(q + 8 * (i >> 1)) * (EC + 1) + 8 * n + 2 * c + (i & 1)] = acc[0][n][i] + acc[1][n][i];
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const float v = quad_sum(wsq[n]);
            if (c == 0) wn[warp * EC + 8 * n + q] = v;
        }
        if (p0 == 0)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const float v = quad_sum(xsq[r]);
                if (c == 0) xn[warp * TM + 8 * r + q] = v;
            }
        __syncthreads();
        if (CL > 1 && p0 == 0) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        for (int i = tid; i < TM * EC; i += kRouteThreads) {
            const int t = i / EC, e = i % EC;
            float p[kRouteWarps];
#pragma unroll
            for (int w = 0; w < kRouteWarps; ++w) p[w] = part[(w * TM + t) * (EC + 1) + e];
            static_assert(kRouteWarps == 8, "the tree of the partial sums");
            const float v = ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
            if (e0 + e < E) {
                float* dst = CL == 1 ? logit : cluster.map_shared_rank(logit, t % CL);
                dst[(t / CL) * kMmaMaxExperts + e0 + e] = v + (bias ? bias[e0 + e] : 0.f);
            }
        }
        if (tid < EC) {
            float v = 0.f;
            for (int w = 0; w < kRouteWarps; ++w) v += wn[w * EC + tid];
            wtop = fmaxf(wtop, v);
        }
        __syncthreads();
    }
    static_assert(EC <= 64, "threads 0 .. EC - 1 are the first two warps");
    if (warp < 2) {
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) wtop = fmaxf(wtop, __shfl_xor_sync(0xffffffffu, wtop, m));
        if (lane < CL) (CL == 1 ? wmax_of : cluster.map_shared_rank(wmax_of, lane))[2 * rank + warp] = wtop;
    }
    if (CL > 1) cluster.sync(); else __syncthreads();
    float wmax = 0.f;
#pragma unroll
    for (int r = 0; r < 2 * CL; ++r) wmax = fmaxf(wmax, wmax_of[r]);
    static_assert(TOK <= 32, "a bit per token");
    __shared__ uint32_t todo[TOK][kMmaMaxExperts / 32];
    unsigned again = 0;                                                    // this warp's tokens that are chosen again
    for (int i = warp; i * CL + rank < n_tok; i += kRouteWarps) {
        const int t = i * CL + rank;
        float x2 = 0.f;
#pragma unroll
        for (int w = 0; w < kRouteWarps; ++w) x2 += xn[w * TM + t];
        // of a pair both may be off; the bias addition rounds once more (relative to the logit)
        if (choose(logit + i * kMmaMaxExperts, 2.f * route_bound(H) * sqrtf(x2) * sqrtf(wmax), E, k, lane, todo[i], ids_out + (size_t)(t0 + t) * k,
                   w_out + (size_t)(t0 + t) * k))
            again |= 1u << i;
    }
    // One token in fifty is chosen again (64 experts of 2048), so every call of some size has one, and it is the call's tail: its
    // logits are spread over all warps, and its choice keeps its keys in registers: 333 tokens 12.0 -> 9.8 -> 8.3 us, 2048 17.2 -> 15.6 -> 14.1.
    if (!__syncthreads_or(again != 0)) return;
    __shared__ unsigned flagged;
    if (tid == 0) flagged = 0;
    __syncthreads();
    if (lane == 0 && again) atomicOr(&flagged, again);
    __syncthreads();
    int item = 0;
    for (unsigned toks = flagged; toks; toks &= toks - 1) {
        const int i = __ffs(toks) - 1;
        for (int b = 0; b < kMmaMaxExperts / 32; ++b)
            for (unsigned es = todo[i][b]; es; es &= es - 1, ++item) {
                if (item % kRouteWarps != warp) continue;
                const int e = 32 * b + __ffs(es) - 1;
                const float v = logit_again(hidden + (size_t)(t0 + i * CL + rank) * H, w_router + (size_t)e * H, H, lane);
                if (lane == 0) logit[i * kMmaMaxExperts + e] = v + (bias ? bias[e] : 0.f);
            }
    }
    __syncthreads();
    for (; again; again &= again - 1) {
        const int i = __ffs(again) - 1, t = i * CL + rank;
        softmax_topk_few(logit + i * kMmaMaxExperts, E, k, lane, ids_out + (size_t)(t0 + t) * k, w_out + (size_t)(t0 + t) * k);
    }
}

template <int NT, int CL, int U>
int launch_route_mma(const exmoe_shape& s, const __nv_bfloat16* hidden, const __nv_bfloat16* w, const float* bias, int T,
                     int32_t* ids, float* wts, cudaStream_t st) {
    constexpr int TM = 16, EC = 8 * NT;
    constexpr size_t smem = 4 * ((size_t)kRouteWarps * TM * (EC + 1) + (size_t)TM / CL * kMmaMaxExperts + kRouteWarps * (TM + EC) + 2 * CL);
    static SmemOnce once;
    if (!allow_smem(route_mma_kernel<NT, CL, U>, (int)smem, once)) return EXMOE_ERR_CUDA;
    return launch_dependent(route_mma_kernel<NT, CL, U>, (T + TM - 1) / TM * CL, CL, smem, s, hidden, w, bias, T, ids, wts, st);
}

// Which form a call takes.  All give the same bits but the tensor-core ones (see there).  One token per cluster of eight CTAs
// while the clusters find room on the chip at once, and for what nothing else fits; then four tokens per read of the
// matrix, by clusters of eight, or of four where these have a warp per expert or the calls are large; with few experts one
// CTA per token; then the tensor cores.  us, replayed from a graph, in the order one / four / four narrow / token / tensor
// cores (16 experts per CTA / 32):
//   64 experts, d_model 2048:  32 tokens 5.1 / 4.9 / - / - / 5.8         64: - / 5.1 / 6.5 / - / 6.8     192: - / 7.7 / - / - / 7.7     208: - / 9.1 / 10.9 / - / 7.8
//   16 experts, d_model 512:   64 tokens 5.2 / 3.5 / 3.3 / 3.9 / 6.8    223: - / 5.7 / 4.1 / 4.1 / 7.0   800: - / 13 / 7.4 / 4.7 / 7.8 / 7.7
//   16 experts, d_model 2048: 128 tokens 9.5 / 7.0 / 4.6 / 5.1 / 9.6    300: - / 9.8 / 7.3 / 5.4 / 9.7   900: - / 22 / 14 / 12 / 11 / 11
//   8 experts, d_model 256:    64 tokens 5.0 / 3.3 / 3.2 / 2.7 / 3.8   1024: - / 14 / 9.1 / 4.9 / 6.7 / 6.7   2048: - / 26 / 15 / 6.8 / 8.4 / 7.4
//   193 / 223 tokens, four and tensor cores, in calls with a near-tie (most at 1024 and more; without one the tensor cores take 2 us less):
//   64 experts, d_model 256: 5.7 / 6.0 and 6.6 / 6.7    48, 512: 6.1 / 6.3 and 6.8 / 6.8    64, 640: 6.7 / 7.2 and - / 6.9    64, 768: 6.9 / 7.3 and 6.9 / 6.9
//   64, 1024: 7.2 / 8.0 and 7.3 / 7.3    64, 4096: 13.3 / 14.5 and 10.6 / 10.7    128, 128: 8.7 / 9.1 and 7.6 / 7.7    128, 256: 8.7 / 9.2 and 8.3 / 8.3
//   256 experts, d_model 1024 (no tensor-core form): 256 tokens 31 / 21 / 22 / 26    1024: 104 / 58 / 55 / 70    4000: 387 / 205 / 178 / 195
//   20 experts, d_model 1000 (none either): 300 tokens 15 / 8.2 / 5.3 / 6.4          4000: 162 / 71 / 40 / 29
enum class RouteForm { One, Four, FourNarrow, Token, Mma, MmaWide };
constexpr RouteForm route_form(int E, int H, int k, int T) {
    const bool mma = H % 32 == 0 && H <= kMmaMaxModel && E <= kMmaMaxExperts && k <= 32;
    const bool four = 8 * (size_t)H + 4 * (size_t)E <= (size_t)kRouteSmemMax;
    const bool small = E * H <= 40000, few = E <= 32 && E * H <= 65536;    // 80 KB of matrix; 128 KB
    if (T < kRouteFewTokens) return RouteForm::One;
    if (few) {
        if (T >= (E <= 8 ? kRouteFewTokens : kRouteTokenTokens) && (!mma || T < (E <= 8 ? 1536 : small ? 896 : 600))) return RouteForm::Token;
        if (T < kRouteTokenTokens && four) return RouteForm::FourNarrow;
    }
    if (mma && T >= (E <= 64 && H < 640 ? kRouteMmaTokensShort : kRouteMmaTokens)) return T >= kRouteWideTokens ? RouteForm::MmaWide : RouteForm::Mma;
    if (small && !mma && T >= 2048) return RouteForm::Token;
    return four ? (T >= 512 ? RouteForm::FourNarrow : RouteForm::Four) : RouteForm::One;
}
static_assert(route_form(64, 2048, 8, 47) == RouteForm::One && route_form(64, 2048, 8, 48) == RouteForm::Four);
static_assert(route_form(64, 2048, 8, 192) == RouteForm::Four && route_form(64, 2048, 8, 193) == RouteForm::Mma);
static_assert(route_form(64, 640, 8, 193) == RouteForm::Mma && route_form(128, 128, 8, 193) == RouteForm::Mma);
static_assert(route_form(64, 512, 8, 223) == RouteForm::Four && route_form(48, 512, 8, 224) == RouteForm::Mma);
static_assert(route_form(64, 2048, 8, 1152) == RouteForm::MmaWide && route_form(16, 512, 4, 896) == RouteForm::Mma);
static_assert(route_form(16, 512, 4, 191) == RouteForm::FourNarrow && route_form(16, 512, 4, 192) == RouteForm::Token);
static_assert(route_form(16, 512, 4, 895) == RouteForm::Token && route_form(8, 256, 2, 48) == RouteForm::Token);
static_assert(route_form(32, 2048, 8, 599) == RouteForm::Token && route_form(32, 2048, 8, 600) == RouteForm::Mma);
static_assert(route_form(20, 1000, 3, 4000) == RouteForm::Token && route_form(256, 1024, 8, 4000) == RouteForm::FourNarrow);
static_assert(route_form(4096, 1024, 8, 256) == RouteForm::Four && route_form(64, 40000, 8, 4000) == RouteForm::One);

}  // namespace

extern "C" int exmoe_route(const exmoe_shape* shape, const void* hidden_bf16, const void* router_bf16, const float* bias,
                           int T, int32_t* topk_ids, float* topk_weights, void* stream) {
    if (!shape || T < 0) return EXMOE_ERR_ARG;
    if (shape->d_model <= 0 || shape->d_model % 8 || shape->num_experts <= 0 || shape->num_experts > 4096 ||
        shape->top_k <= 0 || shape->top_k > shape->num_experts)
        return EXMOE_ERR_SHAPE;
    if (T == 0) return EXMOE_OK;
    if (!hidden_bf16 || !router_bf16 || !topk_ids || !topk_weights) return EXMOE_ERR_ARG;
    if ((reinterpret_cast<uintptr_t>(hidden_bf16) | reinterpret_cast<uintptr_t>(router_bf16)) & 15) return EXMOE_ERR_ARG;
    const size_t row = (size_t)shape->d_model * 2, logits = (size_t)shape->num_experts * 4;
    if (row + logits > (size_t)kRouteSmemMax) return EXMOE_ERR_SHAPE;
    const exmoe_shape& s = *shape;
    const __nv_bfloat16* x = (const __nv_bfloat16*)hidden_bf16;
    const __nv_bfloat16* w = (const __nv_bfloat16*)router_bf16;
    cudaStream_t st = (cudaStream_t)stream;
    switch (route_form(s.num_experts, s.d_model, s.top_k, T)) {
        case RouteForm::One: return launch_route<8, 1>(s, x, w, bias, T, topk_ids, topk_weights, st);
        case RouteForm::Four: return launch_route<8, 4>(s, x, w, bias, T, topk_ids, topk_weights, st);
        case RouteForm::FourNarrow: return launch_route<4, 4>(s, x, w, bias, T, topk_ids, topk_weights, st);
        case RouteForm::Token: return launch_route_token(s, x, w, bias, T, topk_ids, topk_weights, st);
        case RouteForm::Mma: return launch_route_mma<2, 4, 4>(s, x, w, bias, T, topk_ids, topk_weights, st);
        case RouteForm::MmaWide: return launch_route_mma<4, 2, 2>(s, x, w, bias, T, topk_ids, topk_weights, st);
    }
    return EXMOE_ERR_STATE;
}

}  // namespace exmoe
