// Shared by the tensor-core kernels (pdit_mma.cu, pdit_concurrent.cu): bytes as
// f16 subnormals, mma.sync fragments, paired binary32 arithmetic.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace pdit {

constexpr float kMmUnit = 3.552713678800501e-15f;   // 2^-48: half a unit of energy (general form: one)
constexpr float kMmScale = 5.62949953421312e14f;    // 2^49: energy per 1.0 (general form: 2^48)
constexpr float kMmOne = 2.98023223876953125e-08f;  // 2^-25: the unit in its last place

// Two binary32 operations at once (each rounded as the single one).
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 d;
    asm("{ .reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; add.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z; }"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    float2 d;
    asm("{ .reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; sub.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z; }"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 d;
    asm("{ .reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; mul.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z; }"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{ .reg .b64 x, y, z, w; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; mov.b64 w, {%6, %7}; "
        "fma.rn.f32x2 z, x, y, w; mov.b64 {%0, %1}, z; }"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
// The smaller of two; not a number where one is not.
__device__ __forceinline__ float min_nan(float a, float b) {
    float d;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ float2 two(float v) { return make_float2(v, v); }

// Loads at 32-bit shared-window addresses (volatile: they stay on their side
// of the barriers).
__device__ __forceinline__ int lds_u8(uint32_t a) {
    int v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ float lds_f32(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ float2 lds_f64(uint32_t a) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ uint2 lds_u64(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], const uint2 b) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// The 16 x 16 fragment of rows row0.. of a table at depth step s. Depth order
// within a step: a thread's four consecutive bytes are the fragment's (2q,
// 2q + 1) and (2q + 8, 2q + 9), as in the vectors.
template <int DS>
__device__ __forceinline__ void mm_frag(const uint8_t *tab, int row0, int s, int lane, uint32_t (&a)[4]) {
    const uint8_t *p = tab + (row0 + (lane >> 2)) * DS + 16 * s + 4 * (lane & 3);
    const uint32_t x = *reinterpret_cast<const uint32_t *>(p);
    const uint32_t y = *reinterpret_cast<const uint32_t *>(p + 8 * DS);
    a[0] = __byte_perm(x, 0, 0x4140);
    a[1] = __byte_perm(y, 0, 0x4140);
    a[2] = __byte_perm(x, 0, 0x4342);
    a[3] = __byte_perm(y, 0, 0x4342);
}

}  // namespace pdit
