// Complex numbers as float pairs (hi + lo per component, ~2^-44 relative) for FP64-quality
// arithmetic on the fp32 pipe, which is ~64x GB300's FP64 pipe: the error-free transforms
// TwoSum and TwoProduct (with fmaf) and a fused (h, l) += x y.  Device code only.
#pragma once

namespace afqmc {

struct __align__(16) ffc {   // 16-byte aligned: a peer CTA can receive it as one 16-byte store
    float rh, rl, ih, il;
};
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float v = s - a;
    e = (a - (s - v)) + (b - v);
}
// (h, l) + x y for float pairs: TwoProduct of the leading parts, first-order cross terms
__device__ __forceinline__ void ff_fma(float& h, float& l, float xh, float xl, float yh, float yl) {
    const float p = xh * yh;
    float pe = fmaf(xh, yh, -p);
    pe = fmaf(xh, yl, fmaf(xl, yh, pe));
    float s, e;
    two_sum(h, p, s, e);
    e += l + pe;
    h = s + e;
    l = e - (h - s);
}

// (double)x by integer operations for zero and normal numbers
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), e = (b >> 23) & 0xffu;
    if (e == 0xffu || (e == 0u && (b << 1) != 0u)) return (double)x;
    const unsigned hi = (b & 0x80000000u) | ((b & 0x7fffffffu) >> 3), up = e ? 896u << 20 : 0u;
    return __hiloint2double((int)(hi + up), (int)(b << 29));
}
// v as the float pair h = (float)v, l = (float)(v - h), by integer operations for zero and where
// neither half leaves the normal range
__device__ __forceinline__ void ff_split(double v, float& h, float& l) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ffu) - 1023;
    if (e < -70 || e > 126) {
        h = (float)v;
        l = (b << 1) == 0ull ? 0.f : (float)(v - (double)h);
        return;
    }
    const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
    const unsigned long long m = (b & 0xfffffffffffffull) | (1ull << 52);
    unsigned top = (unsigned)(m >> 29);                     // 24 bits
    int rest = (int)((unsigned)m & 0x1fffffffu);            // 29 bits
    const bool up = rest > (1 << 28) || (rest == (1 << 28) && (top & 1u));   // to nearest, ties to even
    top += up ? 1u : 0u;
    rest -= up ? 1 << 29 : 0;
    h = (float)top * __uint_as_float(sign | (unsigned)(e - 23 + 127) << 23);
    l = (float)rest * __uint_as_float(sign | (unsigned)(e - 52 + 127) << 23);
}

// Two floats in one 64-bit register and sm_100's packed fp32 arithmetic on them (each half rounded
// as the scalar operation is).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 f2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float f2_lo(f32x2 x) { return __uint_as_float((unsigned)x); }
__device__ __forceinline__ float f2_hi(f32x2 x) { return __uint_as_float((unsigned)(x >> 32)); }
__device__ __forceinline__ f32x2 f2_add(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 f2_sub(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 f2_mul(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 f2_fma(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// ff_fma on both halves, bit for bit; nxh = -xh (there is no packed negation)
__device__ __forceinline__ void ff_fma2(f32x2& h, f32x2& l, f32x2 xh, f32x2 nxh, f32x2 xl, f32x2 yh, f32x2 yl) {
    const f32x2 np = f2_mul(nxh, yh);
    const f32x2 pe = f2_fma(xh, yl, f2_fma(xl, yh, f2_fma(xh, yh, np)));
    const f32x2 s = f2_sub(h, np), v = f2_sub(s, h);
    f32x2 e = f2_sub(f2_sub(h, f2_sub(s, v)), f2_add(np, v));
    e = f2_add(e, f2_add(l, pe));
    h = f2_add(s, e);
    l = f2_sub(e, f2_sub(h, s));
}

}  // namespace afqmc
