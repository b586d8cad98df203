// f32x2.cuh -- packed FP32 arithmetic (internal).
#pragma once

namespace lisa {

// packed FP32 pairs (Blackwell f32x2): one instruction, each lane rounded as its scalar
// counterpart
#define LISA_F32X2(op, ...)                                                                  \
    asm("{\n.reg .b64 ra, rb, rc, rd;\n"                                                      \
        "mov.b64 ra, {%2, %3};\nmov.b64 rb, {%4, %5};\nmov.b64 rc, {%6, %7};\n" op         \
        "\nmov.b64 {%0, %1}, rd;\n}"                                                          \
        : "=f"(d.x), "=f"(d.y)                                                              \
        : __VA_ARGS__)

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    LISA_F32X2("fma.rn.f32x2 rd, ra, rb, rc;", "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x),
               "f"(c.y));
    return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 d;
    LISA_F32X2("mul.rn.f32x2 rd, ra, rb;", "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(0.0f),
               "f"(0.0f));
    return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 d;
    LISA_F32X2("add.rn.f32x2 rd, ra, rb;", "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(0.0f),
               "f"(0.0f));
    return d;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    float2 d;
    LISA_F32X2("sub.rn.f32x2 rd, ra, rb;", "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(0.0f),
               "f"(0.0f));
    return d;
}
#undef LISA_F32X2

}  // namespace lisa
