// Host driver for the packed double-FP32 functions of csrc/df2.cuh (built and
// run by tests/test_df2_host.py on the CPU; no GPU): counts the results whose
// halves differ in any bit from the scalar functions of csrc/df.cuh, and those
// of df_from that differ in value from the float conversions.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>

#include "df2.cuh"

using namespace shtg;

static uint64_t g_state = 0x2545F4914F6CDD1Dull;
static double draw(bool wide) {   // random sign, |x| in [1, 2) times 2^-30 .. 2^30 (wide) or 1
    g_state ^= g_state >> 12;
    g_state ^= g_state << 25;
    g_state ^= g_state >> 27;
    const uint64_t r = g_state * 0x2545F4914F6CDD1Dull;
    const double x = ldexp(1.0 + (double)(r >> 12) / 4503599627370496.0, wide ? (int)(r % 61) - 30 : 0);
    return (r & 2048) ? -x : x;
}
// bits, with -0 as 0: a difference formed as fma(y, -1, x) may give the other zero
static uint32_t bits(float x) {
    uint32_t u;
    x += 0.f;
    std::memcpy(&u, &x, 4);
    return u;
}
static int differs(df a, df b) { return bits(a.hi) != bits(b.hi) || bits(a.lo) != bits(b.lo); }
static int differs(const df2 &p, df x, df y) { return differs(df2_x(p), x) + differs(df2_y(p), y); }

int main() {
    int add = 0, sub = 0, mul = 0, acc = 0;
    df2 s2 = df2_zero();
    dfacc s[2];
    df_acc_zero(s[0]);
    df_acc_zero(s[1]);
    for (int i = 0; i < 20000; ++i) {
        df a[2], b[2];
        for (int h = 0; h < 2; ++h) {
            a[h] = df_from(draw(i & 1));
            b[h] = df_from(draw(i & 2));
            if (i % 64 == 5) b[h] = df_neg(a[h]);   // exact cancellation
            if (i % 64 == 6) b[h] = df_zero();
        }
        const df2 pa = df2_make(a[0], a[1]), pb = df2_make(b[0], b[1]);
        add += differs(df2_add(pa, pb), df_add(a[0], b[0]), df_add(a[1], b[1]));
        sub += differs(df2_sub(pa, pb), df_sub(a[0], b[0]), df_sub(a[1], b[1]));
        mul += differs(df2_mul(pa, pb), df_mul(a[0], b[0]), df_mul(a[1], b[1]));
        df2_fma(s2, pa, pb, fmul2(fneg2(pa.hi), pb.hi));
        for (int h = 0; h < 2; ++h) df_fma(s[h], a[h], b[h]);
        if (i % 32 == 31) {
            df2_norm(s2);
            for (int h = 0; h < 2; ++h) df_acc_norm(s[h]);
        }
        acc += differs(s2, df_make(s[0].hi, s[0].lo), df_make(s[1].hi, s[1].lo));
    }
    // df_from against the conversions it stands for, at both ends of its range
    // of exponents and beyond, ties, zeros and infinity
    int from = 0;
    auto check = [&](double x) {
        const df a = df_from(x);
        const float hi = (float)x, lo = (float)(x - (double)hi);
        const double sa = (double)a.hi + (double)a.lo, sb = (double)hi + (double)lo;
        from += !(sa == sb || (sa != sa && sb != sb)) || std::fabs(a.lo) > std::fabs(std::nextafter(hi, INFINITY) - hi) / 2;
    };
    for (int e = -200; e <= 130; ++e)
        for (int i = 0; i < 100; ++i) {
            const double x = ldexp(draw(false), e);
            check(x);
            check((double)(float)x * (1.0 + ldexp(1.0, -24)));   // halfway between floats
            check(ldexp(x < 0 ? -2.0 : 2.0, e) * (1.0 - ldexp(1.0, -30)));
        }
    check(0.0);
    check(-0.0);
    check(INFINITY);
    std::printf("from %d ", from);
    std::printf("add %d sub %d mul %d fma %d\n", add, sub, mul, acc);
    return 0;
}
