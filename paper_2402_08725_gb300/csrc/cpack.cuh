// Packed FP32 pairs and the arithmetic of in-register DFTs over two value types (internal, device code).
//
// sm_103a issues add, multiply and fused multiply-add on two FP32 values per instruction
// (add/mul/fma.rn.f32x2).  The rate of the FP32 pipe is the same (78.7 against 77.2 TFLOP/s measured),
// but half the instructions are issued, which is what bounds the chunk kernel.  zdft of fft_pair.cuh runs on
//   float2  one complex value (x = real, y = imaginary): additions are packed;
//   C2      two complex values side by side (the same position of two epochs): every operation is.
#pragma once

#include <cuda_runtime.h>

namespace sr {

__device__ __forceinline__ float2 f2add(float2 a, float2 b) {
    float2 r;
    asm("{.reg .b64 p, q, s; mov.b64 p, {%2, %3}; mov.b64 q, {%4, %5}; add.rn.f32x2 s, p, q; mov.b64 {%0, %1}, s;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 f2sub(float2 a, float2 b) {
    float2 r;
    asm("{.reg .b64 p, q, s; mov.b64 p, {%2, %3}; mov.b64 q, {%4, %5}; sub.rn.f32x2 s, p, q; mov.b64 {%0, %1}, s;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 f2mul(float2 a, float2 b) {
    float2 r;
    asm("{.reg .b64 p, q, s; mov.b64 p, {%2, %3}; mov.b64 q, {%4, %5}; mul.rn.f32x2 s, p, q; mov.b64 {%0, %1}, s;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) {
    float2 r;
    asm("{.reg .b64 p, q, s, t; mov.b64 p, {%2, %3}; mov.b64 q, {%4, %5}; mov.b64 s, {%6, %7};"
        " fma.rn.f32x2 t, p, q, s; mov.b64 {%0, %1}, t;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
__device__ __forceinline__ float2 f2dup(float a) { return make_float2(a, a); }
// c - a b, elementwise (negation is free on the scalar instruction)
__device__ __forceinline__ float2 f2nfma(float2 a, float2 b, float2 c) {
    return make_float2(fmaf(-a.x, b.x, c.x), fmaf(-a.y, b.y, c.y));
}

struct C2 {
    float2 re, im;  // (real, real) and (imaginary, imaginary) of the two values
};

// a + b, a - b, c x, a + c x, a + i c x (c real), and a +- i b
__device__ __forceinline__ float2 zadd(float2 a, float2 b) { return f2add(a, b); }
__device__ __forceinline__ float2 zsub(float2 a, float2 b) { return f2sub(a, b); }
__device__ __forceinline__ float2 zscale(float c, float2 x) { return f2mul(x, f2dup(c)); }
__device__ __forceinline__ float2 zaxpy(float c, float2 x, float2 a) { return f2fma(x, f2dup(c), a); }
__device__ __forceinline__ float2 zaxpyi(float c, float2 x, float2 a) {
    return make_float2(fmaf(-c, x.y, a.x), fmaf(c, x.x, a.y));
}
__device__ __forceinline__ float2 zaddi(float2 a, float2 b) { return make_float2(a.x - b.y, a.y + b.x); }
__device__ __forceinline__ float2 zsubi(float2 a, float2 b) { return make_float2(a.x + b.y, a.y - b.x); }

__device__ __forceinline__ C2 zadd(C2 a, C2 b) { return {f2add(a.re, b.re), f2add(a.im, b.im)}; }
__device__ __forceinline__ C2 zsub(C2 a, C2 b) { return {f2sub(a.re, b.re), f2sub(a.im, b.im)}; }
__device__ __forceinline__ C2 zscale(float c, C2 x) { return {f2mul(x.re, f2dup(c)), f2mul(x.im, f2dup(c))}; }
__device__ __forceinline__ C2 zaxpy(float c, C2 x, C2 a) {
    return {f2fma(x.re, f2dup(c), a.re), f2fma(x.im, f2dup(c), a.im)};
}
__device__ __forceinline__ C2 zaxpyi(float c, C2 x, C2 a) {
    return {f2fma(x.im, f2dup(-c), a.re), f2fma(x.re, f2dup(c), a.im)};
}
__device__ __forceinline__ C2 zaddi(C2 a, C2 b) { return {f2sub(a.re, b.im), f2add(a.im, b.re)}; }
__device__ __forceinline__ C2 zsubi(C2 a, C2 b) { return {f2add(a.re, b.im), f2sub(a.im, b.re)}; }

// v w and v conj(w)
__device__ __forceinline__ float2 zmulw(float2 v, float2 w) {
    return make_float2(v.x * w.x - v.y * w.y, v.x * w.y + v.y * w.x);
}
__device__ __forceinline__ float2 zmulwc(float2 v, float2 w) {
    return make_float2(v.x * w.x + v.y * w.y, v.y * w.x - v.x * w.y);
}
__device__ __forceinline__ C2 zmulw(C2 v, float2 w) {
    const float2 wx = f2dup(w.x);
    return {f2fma(v.im, f2dup(-w.y), f2mul(v.re, wx)), f2fma(v.re, f2dup(w.y), f2mul(v.im, wx))};
}
__device__ __forceinline__ C2 zmulwc(C2 v, float2 w) {
    const float2 wx = f2dup(w.x);
    return {f2fma(v.im, f2dup(w.y), f2mul(v.re, wx)), f2fma(v.re, f2dup(-w.y), f2mul(v.im, wx))};
}
__device__ __forceinline__ void zneg(float2 &v) { v = make_float2(-v.x, -v.y); }
__device__ __forceinline__ void zneg(C2 &v) {
    zneg(v.re);
    zneg(v.im);
}
__device__ __forceinline__ float2 zmuli(float2 v) { return make_float2(-v.y, v.x); }
__device__ __forceinline__ float2 zmulni(float2 v) { return make_float2(v.y, -v.x); }
__device__ __forceinline__ C2 zmuli(C2 v) { return {make_float2(-v.im.x, -v.im.y), v.re}; }
__device__ __forceinline__ C2 zmulni(C2 v) { return {v.im, make_float2(-v.re.x, -v.re.y)}; }

}  // namespace sr
