// What the two tree-attention kernels share: small device functions and the table of encoded tensor maps.
#pragma once
#include <cuda.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace mtv {

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// 2^x for two values on the FMA pipes: x = j + f with j the nearest integer (read off the low mantissa bits of
// x + 1.5 * 2^23) and f in [-0.5, 0.5]; 2^f by a cubic with the smallest largest relative error over that interval (7.5e-5, far
// below the bf16 rounding of P); 2^j by an add to the exponent field.  x <= 127; it is clamped at -126 (the result then underflows
// towards zero like ex2's).
__device__ __forceinline__ float2 exp2_poly2(float2 x) {
    const float magic = 12582912.f;
    x.x = fmaxf(x.x, -126.f);
    x.y = fmaxf(x.y, -126.f);
    const float2 t = __fadd2_rn(x, make_float2(magic, magic));
    const float2 jf = __fadd2_rn(t, make_float2(-magic, -magic));
    const float2 f = __fadd2_rn(x, make_float2(-jf.x, -jf.y));
    float2 q = __ffma2_rn(make_float2(0.055171650f, 0.055171650f), f, make_float2(0.24261113f, 0.24261113f));
    q = __ffma2_rn(q, f, make_float2(0.69326097f, 0.69326097f));
    q = __ffma2_rn(q, f, make_float2(0.99992806f, 0.99992806f));
    return make_float2(__int_as_float(__float_as_int(q.x) + (__float_as_int(t.x) << 23)),
                       __int_as_float(__float_as_int(q.y) + (__float_as_int(t.y) << 23)));
}
__device__ __forceinline__ uint32_t pack2_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// A word that another kernel may be writing: never an earlier load's value, nor moved over what orders it (a barrier, the wait
// for the previous kernel).
__device__ __forceinline__ int ld_relaxed(const int32_t *p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_acquire(const int32_t *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Tensor map over bf16 data (rank 2 to 5) with a 128-byte-swizzled box whose innermost extent is 64 elements, from a table
// of those already encoded.
bool tensor_map_bf16(CUtensorMap *map, const void *base, int rank, const cuuint64_t *dims, const cuuint64_t *strides_bytes,
                     const cuuint32_t *box);

}  // namespace mtv
