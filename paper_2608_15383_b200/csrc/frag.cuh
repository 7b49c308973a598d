// Device helpers shared by the kernels that feed the packed codes to mma.sync: the m16n8k16 MMAs with the
// conversions of the packed layout (Eq. 3 codes, offset-binary) and of the activations that go with them, block sums of
// activations, and the programmatic-dependent-launch controls.
#pragma once
#include <stdint.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace exmoe {

__device__ __forceinline__ void mma_m16n8k16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                             uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// sum of the 8 BF16 values of a 16-byte chunk, in binary32
__device__ __forceinline__ float sum8_bf16(const uint4& v) {
    const uint32_t r[4] = {v.x, v.y, v.z, v.w};
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) s += __uint_as_float(r[i] << 16) + __uint_as_float(r[i] & 0xffff0000u);
    return s;
}

// ---- codes as FP16 subnormals ---------------------------------------------------------------------------------------
// A nibble in bits 0-3 of a 16-bit half IS the FP16 subnormal u * 2^-24, and in bits 4-7 it is 16 u * 2^-24: four code pairs
// of a word take one shift and four ANDs (BF16 pairs 128 + u took three shifts and four lop3, at the same half rate), and the
// products need no bias as large as 136.  The activations go in as FP16 scaled by a power of two per row and 128-wide
// block: X = x * 2^(14-E), E the exponent of the block's largest value, and X / 16 for the k that meet bits 4-7.  FP16 has
// three bits more than BF16, so that is exact for values down to 2^-27 of the block's largest and off by less than
// 2^-35 of it below that.  The MMA takes FP16 subnormals exactly (checked) and sums in binary32, so a block contributes
//     s * ( 2^(E+10) D - 8 sum x )
// with the roundings of these binary32 operations.  Both factors are kept as 2^16 s and 2^-16 ( .. ): no overflow.
__device__ __forceinline__ void mma_m16n8k16_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                 uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// A word pair (rows q and q + 8) as MMA operands: a[0..3] meets x[0..1] of the lane's eight activations, a[4..7] x[2..3]
struct CodeFrag {
    uint32_t a[8];
    __device__ __forceinline__ CodeFrag(uint32_t wq, uint32_t wq8) {
        constexpr uint32_t L = 0x000f000fu, H = 0x00f000f0u;
        a[0] = wq & L;
        a[1] = wq8 & L;
        a[2] = wq & H;
        a[3] = wq8 & H;
        wq >>= 8;
        wq8 >>= 8;
        a[4] = wq & L;
        a[5] = wq8 & L;
        a[6] = wq & H;
        a[7] = wq8 & H;
    }
    __device__ __forceinline__ void first(float (&d)[4], const uint4& x) const { mma_m16n8k16_f16(d, a[0], a[1], a[2], a[3], x.x, x.y); }
    __device__ __forceinline__ void second(float (&d)[4], const uint4& x) const { mma_m16n8k16_f16(d, a[4], a[5], a[6], a[7], x.z, x.w); }
};
// One 128-wide block of a BF16 row by 16 lanes of eight consecutive values each: the FP16 operands of this lane's eight and
// cst = (2^(E-6), -2^-13 sum x), the same in all 16 lanes.  An infinity or NaN in the block makes the row's results NaN.
__device__ __forceinline__ uint4 f16_block(const uint4& raw, float2& cst) {
    const uint32_t in[4] = {raw.x, raw.y, raw.z, raw.w};
    uint32_t top = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) top = max(top, max((in[i] << 16) & 0x7fff0000u, in[i] & 0x7fff0000u));
    float sum = sum8_bf16(raw);
#pragma unroll
    for (int m = 8; m >= 1; m >>= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, m);
        top = max(top, __shfl_xor_sync(0xffffffffu, top, m));
    }
    const int eb = max((int)(top >> 23), 14);                              // biased E, so that 2^(14-E) is finite
    const float up = __uint_as_float((uint32_t)(268 - eb) << 23), up16 = up * 0.0625f;
    uint32_t out[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float f = i & 1 ? up16 : up;                                 // k 2,3,6,7 meet bits 4-7
        const __half2 h = __floats2half2_rn(__uint_as_float(in[i] << 16) * f, __uint_as_float(in[i] & 0xffff0000u) * f);
        out[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    cst.x = __uint_as_float(top >= 0x7f800000u ? 0x7fffffffu : (uint32_t)(eb - 6) << 23);
    cst.y = -0x1p-13f * sum;
    return make_uint4(out[0], out[1], out[2], out[3]);
}
// 2^16 times the FP16 group scales of rows q and q + 8
__device__ __forceinline__ float2 scales16(uint32_t sv) {
    const float2 s = __half22float2(*reinterpret_cast<const __half2*>(&sv));
    return make_float2(s.x * 65536.f, s.y * 65536.f);
}

__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// What a kernel reads behind grid_dependency_wait may be written while it runs: no const __restrict__ there (a load that the
// compiler takes for read-only may move in front of the wait), and where many such loads are issued together, these.  It may
// stand where the data are complete before the kernel starts: weights, a router's matrix and bias, tensor maps; and what the kernels
// in front of a down or a combine kernel have waited for before they let it start (ids, routing weights).
__device__ __forceinline__ int4 load_behind_wait_cg(const int4* p) {       // past L1
    int4 v;
    asm volatile("ld.global.cg.v4.s32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int load_behind_wait_cg(const int* p) {
    int v;
    asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace exmoe
