// Two double-FP32 values at a time (df.cuh) in packed FP32 instructions
// (add / mul / fma.rn.f32x2): hi and lo hold the parts of both.  Every packed
// operation rounds as its scalar form does: on the host, without contraction,
// the results are the same bit for bit (a CPU test).  In device code nvcc may
// contract a product and a sum of the scalar functions into one FMA, never those
// of the packed asm, so there the two differ in the last bits (2^-43 relative
// in whole transforms; the error against FP64 is the same).  The FP32 pipe runs a packed instruction over two cycles, so its rate of
// operations is that of scalar instructions; what falls by half are the issue
// slots and the independent instructions a warp needs in flight.  Measured
// (N_side 512, l_max 1024, 4 maps, spin 2): transpose 11.1 -> 9.2 ms, synthesis
// 7.7 -> 6.6 ms (FP32 pipe 77 % busy).
// f32x2 instructions have no operand negation: differences are formed as fma(y,
// -1, x), which rounds like x - y.
#pragma once

#include "df.cuh"

namespace shtg {

// (on the host the two halves apart: a CPU test compares the results with the
// scalar functions bit for bit)
SHTG_DF_FN float2 ffma2(float2 a, float2 b, float2 c) {
    float2 d;
#ifdef __CUDA_ARCH__
    asm("{\n\t.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
        "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
#else
    d.x = fmaf(a.x, b.x, c.x);
    d.y = fmaf(a.y, b.y, c.y);
#endif
    return d;
}
SHTG_DF_FN float2 fmul2(float2 a, float2 b) {
    float2 d;
#ifdef __CUDA_ARCH__
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "mul.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
#else
    d.x = a.x * b.x;
    d.y = a.y * b.y;
#endif
    return d;
}
SHTG_DF_FN float2 fadd2(float2 a, float2 b) {
    float2 d;
#ifdef __CUDA_ARCH__
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "add.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
#else
    d.x = a.x + b.x;
    d.y = a.y + b.y;
#endif
    return d;
}
SHTG_DF_FN float2 fpair(float x, float y) {
    float2 d;
    d.x = x;
    d.y = y;
    return d;
}
SHTG_DF_FN float2 fsub2(float2 a, float2 b) { return ffma2(b, fpair(-1.f, -1.f), a); }
// sign change on the integer pipe
SHTG_DF_FN float fneg_bits(float x) {
#ifdef __CUDA_ARCH__
    return __int_as_float(__float_as_int(x) ^ 0x80000000);
#else
    return -x;
#endif
}
SHTG_DF_FN float2 fneg2(float2 a) { return fpair(fneg_bits(a.x), fneg_bits(a.y)); }

struct __align__(16) df2 {
    float2 hi, lo;
};

SHTG_DF_FN df2 df2_make(df a, df b) {
    df2 r;
    r.hi = fpair(a.hi, b.hi);
    r.lo = fpair(a.lo, b.lo);
    return r;
}
SHTG_DF_FN df2 df2_both(df a) { return df2_make(a, a); }
SHTG_DF_FN df df2_x(const df2 &a) { return df_make(a.hi.x, a.lo.x); }
SHTG_DF_FN df df2_y(const df2 &a) { return df_make(a.hi.y, a.lo.y); }

SHTG_DF_FN void df2_set_x(df2 &a, const df2 &b) {
    a.hi.x = b.hi.x;
    a.lo.x = b.lo.x;
}
SHTG_DF_FN void df2_set_y(df2 &a, const df2 &b) {
    a.hi.y = b.hi.y;
    a.lo.y = b.lo.y;
}

// a + b, a - b (df_add, df_sub)
SHTG_DF_FN df2 df2_add(const df2 &a, const df2 &b) {
    const float2 s = fadd2(a.hi, b.hi);
    const float2 bb = fsub2(s, a.hi);
    const float2 e = fadd2(fsub2(a.hi, fsub2(s, bb)), fsub2(b.hi, bb));
    const float2 f = fadd2(e, fadd2(a.lo, b.lo));
    df2 r;
    r.hi = fadd2(s, f);
    r.lo = fsub2(f, fsub2(r.hi, s));
    return r;
}
SHTG_DF_FN df2 df2_neg(const df2 &a) {
    df2 r;
    r.hi = fneg2(a.hi);
    r.lo = fneg2(a.lo);
    return r;
}
SHTG_DF_FN df2 df2_zero() { return df2_both(df_zero()); }
SHTG_DF_FN df2 df2_sub(const df2 &a, const df2 &b) {
    const float2 s = fsub2(a.hi, b.hi);            // a.hi + (-b.hi)
    const float2 bb = fsub2(s, a.hi);
    // (-b.hi) - bb = -(b.hi + bb)
    const float2 e = fsub2(fsub2(a.hi, fsub2(s, bb)), fadd2(b.hi, bb));
    const float2 f = fadd2(e, fsub2(a.lo, b.lo));
    df2 r;
    r.hi = fadd2(s, f);
    r.lo = fsub2(f, fsub2(r.hi, s));
    return r;
}
// a * b (df_mul)
SHTG_DF_FN df2 df2_mul(const df2 &a, const df2 &b) {
    const float2 np = fmul2(a.hi, fneg2(b.hi));   // -(a.hi b.hi), exactly negated
    float2 e = ffma2(a.hi, b.hi, np);
    e = ffma2(a.hi, b.lo, ffma2(a.lo, b.hi, e));
    // fast_two_sum(p, e), p = -np
    df2 r;
    r.hi = fsub2(e, np);
    r.lo = fsub2(e, fadd2(r.hi, np));
    return r;
}
// s += a * b (df_fma on two running sums); np = -(a.hi b.hi), which the caller
// forms from whichever operand it keeps a sign-changed copy of
SHTG_DF_FN void df2_fma(df2 &s, const df2 &a, const df2 &b, const float2 np) {
    float2 e = ffma2(a.hi, b.hi, np);
    e = ffma2(a.hi, b.lo, ffma2(a.lo, b.hi, e));
    // two_sum(s.hi, p), p = -np
    const float2 t = fsub2(s.hi, np);
    const float2 bb = fsub2(t, s.hi);
    const float2 e2 = fsub2(fsub2(s.hi, fsub2(t, bb)), fadd2(np, bb));   // (hi - (t - bb)) + (p - bb)
    s.hi = t;
    s.lo = fadd2(s.lo, fadd2(e2, e));
}
// df_acc_norm
SHTG_DF_FN void df2_norm(df2 &s) {
    const float2 t = fadd2(s.hi, s.lo);
    const float2 bb = fsub2(t, s.hi);
    const float2 l = fadd2(fsub2(s.hi, fsub2(t, bb)), fsub2(s.lo, bb));
    s.hi = t;
    s.lo = l;
}

}  // namespace shtg
