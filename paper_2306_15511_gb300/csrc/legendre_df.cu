// FP64-accurate Legendre sums in double-FP32 arithmetic (df.cuh).
//
// The same sums as the FP64 kernels: synthesis F_r(m) = sum_l a_lm
// lambda_lm(theta_r) with the even / odd split of App. A, and the transpose
// c_lm = sum_r lambda_lm(theta_r) G_r(m).  Inputs and outputs stay FP64 in
// HBM (the plan's FP64 recurrence coefficients, start states and tile
// states, FP64 alm and ring data); values are rounded to df when they are
// staged, and every multiply-add of the recurrence and the contraction runs
// in df on the FP32 pipe.  GB300 issues 64 FP32 operations per FP64
// operation, and a df multiply-add costs about twelve, so the FP64-accurate
// transforms (RHS and residual replacements of the mixed solver, the
// SHTG_DF64 transforms) leave the narrow FP64 pipe.  Rounding: ~2^-47
// relative per operation against 2^-53 for FP64; the recurrence carries O(l)
// of them, far below the 1e-10 the FP64 transforms are held to.
//
// The multiply-adds run on (re, im) pairs, the spin-2 recurrences on (y+, y-),
// in packed instructions (df2.cuh).  Synthesis: one thread per ring pair and
// NM maps, as the CUDA-core kernels, the recurrence in registers.  Transpose: the
// register-blocked contraction of legendre_blk.cuh.
#include "df2.cuh"
#include "legendre_blk.cuh"

namespace shtg {
namespace {

struct __align__(16) dfc2 {   // spin-0 coefficients (a, b)
    df a, b;
};
struct __align__(16) dfc4 {   // spin-2 coefficients: (alpha + beta, alpha - beta), alpha, gamma
    df2 yz;
    df x, w;
};

__device__ __forceinline__ dfc2 dfc2_from(double2 v) {
    dfc2 r;
    r.a = df_from(v.x);
    r.b = df_from(v.y);
    return r;
}
__device__ __forceinline__ dfc4 dfc4_from(double4_32a v) {
    dfc4 r;
    r.x = df_from(v.x);
    r.yz = df2_make(df_from(v.y), df_from(v.z));
    r.w = df_from(v.w);
    return r;
}

// recurrence state of one ring pair (u = 1 - cos theta; the start values s0,
// s1 enter at l = ls); spin 2 runs y+ and y- (from lsb) as the halves of one
// packed value
template <int SPIN> struct DfPair {
    int ls[1], lsb[1];
    df u, s0, s1, a1, a2;
};
template <> struct DfPair<2> {
    int ls[1], lsb[1];
    df u;
    df2 s0, s1, a1, a2;
};

// geometry and FP64 start states of ring pair pr for m, rounded to df
__device__ __forceinline__ void df_pair_load(const LegArgs<double> &a, int m, int pr, DfPair<0> &S) {
    S.a1 = S.a2 = S.s0 = S.s1 = df_zero();
    S.u = df_make(1.f, 0.f);
    S.ls[0] = S.lsb[0] = a.lmax + 1;
    if (pr >= a.npairs) return;
    S.u = df_from(a.u[pr]);
    const int64_t o = (int64_t)m * a.npairs + pr;
    S.ls[0] = a.ls[o];
    const double2 s = a.st[o];
    S.s0 = df_from(s.x);
    S.s1 = df_from(s.y);
}
__device__ __forceinline__ void df_pair_load(const LegArgs<double> &a, int m, int pr, DfPair<2> &S) {
    S.a1 = S.a2 = S.s0 = S.s1 = df2_zero();
    S.u = df_make(1.f, 0.f);
    S.ls[0] = S.lsb[0] = a.lmax + 1;
    if (pr >= a.npairs) return;
    S.u = df_from(a.u[pr]);
    const int64_t o = (int64_t)m * a.npairs + pr;
    const int2 q = a.ls2[o];
    S.ls[0] = q.x;
    S.lsb[0] = q.y;
    const double4_32a s = a.st2[o];
    S.s0 = df2_make(df_from(s.x), df_from(s.z));
    S.s1 = df2_make(df_from(s.y), df_from(s.w));
}

// spin 0: lambda_l = a (1 - u) lambda_{l-1} + b lambda_{l-2}, formed as
// t + b lambda_{l-2} - t u with t = a lambda_{l-1} (as the FP64 kernels do):
// near the poles u ~ 1e-6 keeps its full relative precision, which a
// rounded cos(theta) = 1 - u would not (2^-48 absolute on cos(theta) is
// 1e-8 relative on u at the first HEALPix ring of N_side 1024)
template <bool INJ>
__device__ __forceinline__ void df_step(DfPair<0> &S, const dfc2 *s_rec, const dfc4 *, int i, int l) {
    const dfc2 cf = s_rec[i];
    const df t = df_mul(cf.a, S.a1);
    const df n = df_sub(df_add(t, df_mul(cf.b, S.a2)), df_mul(t, S.u));
    S.a2 = S.a1;
    S.a1 = n;
    if (INJ && l == S.ls[0]) {
        S.a2 = S.s0;
        S.a1 = S.s1;
    }
}

// spin 2: y+-_l = ((alpha + -beta) - alpha u) y+-_{l-1} - gamma y+-_{l-2}
template <bool INJ>
__device__ __forceinline__ void df_step(DfPair<2> &S, const dfc2 *, const dfc4 *s_s2c, int i, int l) {
    const dfc4 cf = s_s2c[i];
    const df2 t = df2_sub(cf.yz, df2_both(df_mul(cf.x, S.u)));
    const df2 n = df2_sub(df2_mul(S.a1, t), df2_mul(S.a2, df2_both(cf.w)));
    S.a2 = S.a1;
    S.a1 = n;
    if (INJ) {
        if (l == S.ls[0]) {
            df2_set_x(S.a2, S.s0);
            df2_set_x(S.a1, S.s1);
        }
        if (l == S.lsb[0]) {
            df2_set_y(S.a2, S.s0);
            df2_set_y(S.a1, S.s1);
        }
    }
}

// (lw, lx) = (y+ + y-, y+ - y-)
__device__ __forceinline__ df2 df_wx(const DfPair<2> &S) {
    const df p = df2_x(S.a1), q = df2_y(S.a1);
    return df2_add(df2_both(p), df2_make(q, df_neg(q)));
}

// =========================================================== synthesis
template <int NM, int SPIN>
__global__ void __launch_bounds__(LEG_THREADS) k_leg_synth_df(const LegArgs<double> a) {
    constexpr int NA = (SPIN == 2) ? 4 * NM : NM;    // alm operands staged per l
    constexpr int NACC = (SPIN == 2) ? 4 : 1;         // complex sums per parity class per map
    __shared__ dfc2 s_rec[SPIN == 2 ? 1 : LEG_CHUNK];
    __shared__ dfc4 s_s2c[SPIN == 2 ? LEG_CHUNK : 1];
    // spin 0 (re, im); spin 2 per map E = (re, im), B, and for the lx terms
    // (B im, -B re), (-E im, E re)
    __shared__ df2 s_alm[NA][LEG_CHUNK];
    __shared__ int s_red[LEG_THREADS / 32];

    const int m = blockIdx.y;
    const int L = a.lmax;
    const int map0 = blockIdx.z * NM;
    const int nm = min(NM, a.nmaps - map0);
    const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2;

    DfPair<SPIN> S;
    const int pr = blockIdx.x * LEG_THREADS + threadIdx.x;
    df_pair_load(a, m, pr, S);
    int lo = min(S.ls[0], S.lsb[0]), hi = -1;
    if (S.ls[0] <= L) hi = max(hi, S.ls[0]);
    if (S.lsb[0] <= L) hi = max(hi, S.lsb[0]);
    const int warp_lo = __reduce_min_sync(0xffffffffu, lo);
    const int warp_hi = __reduce_max_sync(0xffffffffu, hi);
    const int clo = cta_min(warp_lo, s_red);

    df2 accE[NM][NACC], accO[NM][NACC];
#pragma unroll
    for (int k = 0; k < NM; ++k)
#pragma unroll
        for (int q = 0; q < NACC; ++q) accE[k][q] = accO[k][q] = df2_zero();

    // s += x * b with the sign-changed leading part nx of x
    auto fma = [](df2 &s, const df2 &x, const float2 nx, const df2 &b) { df2_fma(s, x, b, fmul2(nx, b.hi)); };
    auto accumulate = [&](const int i, df2(&acc)[NM][NACC]) {
        if constexpr (SPIN == 0) {
            const df2 lam = df2_both(S.a1);
            const float2 nl = fneg2(lam.hi);
#pragma unroll
            for (int k = 0; k < NM; ++k) fma(acc[k][0], lam, nl, s_alm[k][i]);
        } else {
            const df2 wx = df_wx(S);
            const df2 lx = df2_both(df2_y(wx)), nlw = df2_neg(df2_both(df2_x(wx)));
            const float2 nx = fneg2(lx.hi), nw = fpair(wx.hi.x, wx.hi.x);
#pragma unroll
            for (int k = 0; k < NM; ++k) {
                // W parts: Q = -E lw, U = -B lw ; X parts: Q = -i B lx, U = i E lx
                fma(acc[k][0], nlw, nw, s_alm[4 * k][i]);
                fma(acc[k][1], nlw, nw, s_alm[4 * k + 1][i]);
                fma(acc[k][2], lx, nx, s_alm[4 * k + 2][i]);
                fma(acc[k][3], lx, nx, s_alm[4 * k + 3][i]);
            }
        }
    };
    auto renorm = [&]() {
#pragma unroll
        for (int k = 0; k < NM; ++k)
#pragma unroll
            for (int q = 0; q < NACC; ++q) {
                df2_norm(accE[k][q]);
                df2_norm(accO[k][q]);
            }
    };

    for (int c0 = clo; c0 <= L; c0 += LEG_CHUNK) {
        const int c1 = min(c0 + LEG_CHUNK, L + 1);
        __syncthreads();
        for (int i = threadIdx.x; i < c1 - c0; i += LEG_THREADS) {
            const int l = c0 + i;
            const int64_t idx = base + l;
            if (SPIN == 2) s_s2c[i] = dfc4_from(a.s2c[idx]);
            else s_rec[i] = dfc2_from(a.rec[idx]);
            const double bm = a.beam ? a.beam[l] : 1.0;
#pragma unroll
            for (int k = 0; k < NM; ++k) {
                df2 v[2];
#pragma unroll
                for (int c = 0; c < (SPIN == 2 ? 2 : 1); ++c) {
                    double2 z = make_double2(0.0, 0.0);
                    if (k < nm) {
                        z = a.alm[((int64_t)(map0 + k) * a.rs + c) * a.nalm + idx];
                        if (m == 0) z.y = 0.0;
                        z.x *= bm;
                        z.y *= bm;
                    }
                    v[c] = df2_make(df_from(z.x), df_from(z.y));
                }
                if constexpr (SPIN == 0) {
                    s_alm[k][i] = v[0];
                } else {
                    s_alm[4 * k][i] = v[0];
                    s_alm[4 * k + 1][i] = v[1];
                    s_alm[4 * k + 2][i] = df2_make(df2_y(v[1]), df_neg(df2_x(v[1])));
                    s_alm[4 * k + 3][i] = df2_make(df_neg(df2_y(v[0])), df2_x(v[0]));
                }
            }
        }
        __syncthreads();
        int l = max(c0, warp_lo);
        const int la_end = min(c1 - 1, warp_hi);
        for (; l <= la_end; ++l) {   // start states still being injected
            df_step<true>(S, s_rec, s_s2c, l - c0, l);
            if ((l - m) & 1) accumulate(l - c0, accO);
            else accumulate(l - c0, accE);
        }
        if (l < c1 && ((l - m) & 1)) {
            df_step<false>(S, s_rec, s_s2c, l - c0, l);
            accumulate(l - c0, accO);
            ++l;
        }
        for (; l + 1 < c1; l += 2) {
            df_step<false>(S, s_rec, s_s2c, l - c0, l);
            accumulate(l - c0, accE);
            df_step<false>(S, s_rec, s_s2c, l + 1 - c0, l + 1);
            accumulate(l + 1 - c0, accO);
        }
        if (l < c1) {
            df_step<false>(S, s_rec, s_s2c, l - c0, l);
            accumulate(l - c0, accE);
        }
        renorm();   // at most 64 terms per class since the last one
    }

    if (pr >= a.npairs) return;
    const int rn = pr, rs = a.nring - 1 - pr;
#pragma unroll
    for (int k = 0; k < NM; ++k) {
        if (k >= nm) break;
        double E[2 * NACC], O[2 * NACC];
#pragma unroll
        for (int q = 0; q < NACC; ++q) {
            E[2 * q] = df_to(df2_x(accE[k][q]));
            E[2 * q + 1] = df_to(df2_y(accE[k][q]));
            O[2 * q] = df_to(df2_x(accO[k][q]));
            O[2 * q + 1] = df_to(df2_y(accO[k][q]));
        }
        if constexpr (SPIN == 0) {
            double2 *out = a.F + (int64_t)(map0 + k) * a.nring * (L + 1) + m;
            out[(int64_t)rn * (L + 1)] = make_double2(E[0] + O[0], E[1] + O[1]);
            if (rs != rn) out[(int64_t)rs * (L + 1)] = make_double2(E[0] - O[0], E[1] - O[1]);
        } else {
            // north: W + X over both classes; south: even W - X, odd X - W
            double2 *oq = a.F + (int64_t)(2 * (map0 + k)) * a.nring * (L + 1) + m;
            double2 *ou = a.F + (int64_t)(2 * (map0 + k) + 1) * a.nring * (L + 1) + m;
            oq[(int64_t)rn * (L + 1)] = make_double2(E[0] + O[0] + E[4] + O[4], E[1] + O[1] + E[5] + O[5]);
            ou[(int64_t)rn * (L + 1)] = make_double2(E[2] + O[2] + E[6] + O[6], E[3] + O[3] + E[7] + O[7]);
            if (rs != rn) {
                oq[(int64_t)rs * (L + 1)] = make_double2(E[0] - O[0] - E[4] + O[4], E[1] - O[1] - E[5] + O[5]);
                ou[(int64_t)rs * (L + 1)] = make_double2(E[2] - O[2] - E[6] + O[6], E[3] - O[3] - E[7] + O[7]);
            }
        }
    }
}

// =========================================================== transpose
// double-FP32 arithmetic of the register-blocked transpose (legendre_blk.cuh)
struct ArDf {
    typedef df V;
    typedef df2 Acc;
    struct Op {
        df2 v;
        float2 nh;   // -v.hi
    };
    typedef dfc2 C2;
    typedef dfc4 C4;
    template <int SPIN> using State = DfPair<SPIN>;
    static constexpr bool HALVES = true, GROUPS = false;
    static constexpr int OPB = sizeof(df2);
    static __device__ __forceinline__ V from(double x) { return df_from(x); }
    static __device__ __forceinline__ C2 c2(double2 v) { return dfc2_from(v); }
    static __device__ __forceinline__ C4 c4(double4_32a v) { return dfc4_from(v); }
    static __device__ __forceinline__ void put(unsigned char *p, double re, double im) {
        *reinterpret_cast<df2 *>(p) = df2_make(df_from(re), df_from(im));
    }
    static __device__ __forceinline__ Op get(const unsigned char *p) {
        Op o;
        o.v = *reinterpret_cast<const df2 *>(p);
        o.nh = fneg2(o.v.hi);
        return o;
    }
    static __device__ __forceinline__ void zero(Acc &s) { s = df2_zero(); }
    static __device__ __forceinline__ void fma(Acc &s, V x, const Op &y) {
        const df2 xx = df2_both(x);
        df2_fma(s, xx, y.v, fmul2(xx.hi, y.nh));
    }
    static __device__ __forceinline__ void norm(Acc &s) { df2_norm(s); }
    static __device__ __forceinline__ double2 to(const Acc &s) { return make_double2(df_to(df2_x(s)), df_to(df2_y(s))); }
    static __device__ __forceinline__ void restart(State<0> &S, double2 t) {
        S.a1 = df_from(t.x);
        S.a2 = df_from(t.y);
    }
    static __device__ __forceinline__ void restart(State<2> &S, double4_32a t) {
        S.a1 = df2_make(df_from(t.x), df_from(t.z));
        S.a2 = df2_make(df_from(t.y), df_from(t.w));
    }
    // lambda, or (lw, lx)
    template <int SPIN> static __device__ __forceinline__ void values(const State<SPIN> &S, V (&v)[2]) {
        if constexpr (SPIN == 2) {
            const df2 wx = df_wx(S);
            v[0] = df2_x(wx);
            v[1] = df2_y(wx);
        } else {
            v[0] = S.a1;
            v[1] = df_zero();
        }
    }
    template <int SPIN>
    static __device__ __forceinline__ void load(const LegArgs<double> &a, int m, int pr, State<SPIN> &S) {
        df_pair_load(a, m, pr, S);
    }
    template <int SPIN, bool INJ>
    static __device__ __forceinline__ void step(State<SPIN> &S, const C2 *s_rec, const C4 *s_s2c, int i, int l) {
        df_step<INJ>(S, s_rec, s_s2c, i, l);
    }
};

template <int NM, int SPIN>
int launch_synth_df(Plan *p, const double2 *alm, int rs, int nmaps, const double *beam, double2 *F,
                    cudaStream_t st) {
    LegArgs<double> a = leg_make_args<double>(p);
    a.alm = alm;
    a.rs = rs;
    a.F = F;
    a.beam = beam;
    a.nmaps = nmaps;
    dim3 grid((p->npairs + LEG_THREADS - 1) / LEG_THREADS, p->lmax + 1, (nmaps + NM - 1) / NM);
    prof_begin(p, K_LEG_SYN64, st);
    k_leg_synth_df<NM, SPIN><<<grid, LEG_THREADS, 0, st>>>(a);
    prof_end(p, st);
    SHTG_CHECK_LAUNCH("k_leg_synth_df");
    return SHTG_OK;
}

}  // namespace

// One ring pair per thread, maps per pass by the least work
// (leg_maps_per_pass: the recurrence and a map's multiply-adds stand in the
// same ratio as in native FP64).
int leg_synth_df(Plan *p, int spin, const double2 *alm, int rs, int nmaps, const double *beam, double2 *F,
                 cudaStream_t st) {
    static const int nm0[] = {8, 6, 4, 3, 2, 1}, nm2[] = {4, 3, 2, 1};
    if (spin == 2) {
        switch (leg_maps_per_pass(2, nmaps, nm2, 4)) {
            case 1: return launch_synth_df<1, 2>(p, alm, rs, nmaps, beam, F, st);
            case 2: return launch_synth_df<2, 2>(p, alm, rs, nmaps, beam, F, st);
            case 3: return launch_synth_df<3, 2>(p, alm, rs, nmaps, beam, F, st);
            default: return launch_synth_df<4, 2>(p, alm, rs, nmaps, beam, F, st);
        }
    }
    switch (leg_maps_per_pass(0, nmaps, nm0, 6)) {
        case 1: return launch_synth_df<1, 0>(p, alm, rs, nmaps, beam, F, st);
        case 2: return launch_synth_df<2, 0>(p, alm, rs, nmaps, beam, F, st);
        case 3: return launch_synth_df<3, 0>(p, alm, rs, nmaps, beam, F, st);
        case 4: return launch_synth_df<4, 0>(p, alm, rs, nmaps, beam, F, st);
        case 6: return launch_synth_df<6, 0>(p, alm, rs, nmaps, beam, F, st);
        default: return launch_synth_df<8, 0>(p, alm, rs, nmaps, beam, F, st);
    }
}

int leg_analysis_df(Plan *p, int spin, const double2 *G, int nmaps, const double *beam, double2 *alm, int rs,
                    cudaStream_t st, int vjp) {
    if (spin == 2) return analysis_blk<ArDf, 2>(p, G, nmaps, beam, alm, rs, st, vjp);
    return analysis_blk<ArDf, 0>(p, G, nmaps, beam, alm, rs, st, vjp);
}

}  // namespace shtg
