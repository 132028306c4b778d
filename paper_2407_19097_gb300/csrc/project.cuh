// Four points at a time through the fixed FP32 projection of the render pass (raster.cu).
#pragma once
#include "internal.h"

namespace nrv {

// Pairs of FP32 values in one 64-bit register (mul/add/fma.f32x2, each half rounded on its
// own exactly as the scalar instruction rounds).
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_pack(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(f2 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_add_rz(f2 a, f2 b) {
    f2 r;
    asm("add.rz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// (of the gated network's epilogue)
__device__ __forceinline__ float ex2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// (.ftz: the depths it is used for, 2^-60 .. 2^125, and their reciprocals are normal; without
// it every call carries a scaling for subnormal arguments, a tenth of the pass's instructions.  The
// gate's denominators are at least 1.)
__device__ __forceinline__ float rcp_approx(float v) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// -1/w: one Newton-Raphson step on the hardware's approximation.
__device__ __forceinline__ f2 f2_neg_rcp(f2 w) {
    float w0, w1;
    f2_unpack(w, w0, w1);
    const f2 n0 = f2_pack(rcp_approx(-w0), rcp_approx(-w1));
    return f2_fma(n0, f2_fma(w, n0, f2_pack(1.0f, 1.0f)), n0);
}
// -(c / w) given n = -1/w: a quotient corrected twice by its exact remainder.
__device__ __forceinline__ f2 f2_neg_quot(f2 c, f2 w, f2 n) {
    const f2 q0 = f2_mul(c, n);
    const f2 q1 = f2_fma(f2_fma(w, q0, c), n, q0);
    return f2_fma(f2_fma(w, q1, c), n, q1);
}

// The depths for which project4's quotient is proven (below).
constexpr uint32_t FAST_W_LO = (127u - 60u) << 23;    // 2^-60
constexpr uint32_t FAST_W_HI = (127u + 125u) << 23;   // 2^125

// A view as project4 reads it: the matrix entries and screen factors doubled for the paired
// arithmetic, the depth range as float bits.
struct __align__(16) FView {
    f2 m[12];             // {m, m}
    f2 nhw, hh;           // {-W/2, -W/2}, {H/2, H/2}
    f2 one;               // {1, 1}, not known to the compiler (see project4)
    uint32_t wlo, wspan;  // depths [wlo, wlo + wspan] (float bits) take the fast path
    uint32_t width, height;
    unsigned long long* key;
    uint32_t wide;        // the depth range reaches past the fast path's
};
__device__ __forceinline__ void fview_init(FView& f, const RView& v) {
    for (int i = 0; i < 12; ++i) f.m[i] = f2_pack(v.m[i], v.m[i]);
    f.nhw = f2_pack(-v.hw, -v.hw);
    f.hh = f2_pack(v.hh, v.hh);
    const uint32_t lo = __float_as_uint(v.znear), hi = __float_as_uint(v.zfar);   // 0 < znear <= zfar
    f.wide = lo < FAST_W_LO || hi > FAST_W_HI;
    f.wlo = lo > FAST_W_LO ? lo : FAST_W_LO;
    const uint32_t h = hi < FAST_W_HI ? hi : FAST_W_HI;
    f.wspan = h >= f.wlo ? h - f.wlo : 0u;
    if (h < f.wlo) f.wlo = 0xFFFFFFFFu;   // no depth takes the fast path
    f.width = (uint32_t)v.width;
    f.height = (uint32_t)v.height;
    f.key = v.key;
    const float one = __fdiv_rn(v.hw, v.hw);
    f.one = f2_pack(one, one);
}

// Projection + clipping of four points (pairs 0,1 and 2,3) for one view, bit for bit the
// sequence of project_point, in about a third of its instructions:
//  * the transforms, quotients and screen maps run on pairs (f32x2).  The sums of the
//    transforms are written as product * one + sum: the compiler contracts a paired mul and
//    add into one fma even with explicit rounding, and cannot contract this;
//  * the quotients share one reciprocal.  n = -1/w correctly rounded: the hardware's
//    approximation after one Newton-Raphson step (checked against every mantissa by the
//    tests).  With n correctly rounded, Markstein's theorem (P. Markstein, "IA-64 and
//    Elementary Functions", 2000, ch. 8) makes a corrected quotient correctly rounded when
//    the quotient it starts from is within one unit: the first correction gives that, the
//    second the IEEE quotient.  No step overflows or loses bits to underflow for w in
//    [2^-60, 2^125] unless |q| < 2^-40, where (q + 1) and (1 - q) round to 1 whatever q's
//    last bits are; a quotient that overflows ends as NaN, off screen like the exact one.
//  * floor(s) for 0 <= s < 2^23 is the low mantissa of s + 2^23 rounded toward zero, and one
//    unsigned comparison of those bits rejects s < 0, s >= W and NaN alike (the conversion
//    instruction runs at an eighth of the rate).
// db: bits of w; pix: row-major pixel.
__device__ __forceinline__ void project4(const FView& v, const f2* X, const f2* Y, const f2* Z,
                                         uint32_t* pix, uint32_t* db, bool* ok) {
    const f2 one = f2_pack(1.0f, 1.0f), none = f2_pack(-1.0f, -1.0f);
    const f2 big = f2_pack(8388608.0f, 8388608.0f);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        auto row = [&](int r) {
            const f2 xy = f2_fma(f2_mul(v.m[4 * r + 1], Y[h]), v.one, f2_mul(v.m[4 * r], X[h]));
            return f2_add(f2_fma(f2_mul(v.m[4 * r + 2], Z[h]), v.one, xy), v.m[4 * r + 3]);
        };
        const f2 w = row(2);
        float w0, w1;
        f2_unpack(w, w0, w1);
        const f2 n = f2_neg_rcp(w);
        const f2 bx = f2_add_rz(f2_mul(f2_add(f2_neg_quot(row(0), w, n), none), v.nhw), big);
        const f2 by = f2_add_rz(f2_mul(f2_add(f2_neg_quot(row(1), w, n), one), v.hh), big);
        float bx0, bx1, by0, by1;
        f2_unpack(bx, bx0, bx1);
        f2_unpack(by, by0, by1);
        auto put = [&](int j, float wj, float fx, float fy) {
            const uint32_t px = __float_as_uint(fx) - 0x4B000000u, py = __float_as_uint(fy) - 0x4B000000u;
            db[j] = __float_as_uint(wj);
            ok[j] = (db[j] - v.wlo <= v.wspan) & (px < v.width) & (py < v.height);
            pix[j] = py * v.width + px;
        };
        put(2 * h, w0, bx0, by0);
        put(2 * h + 1, w1, bx1, by1);
    }
}

}  // namespace nrv
