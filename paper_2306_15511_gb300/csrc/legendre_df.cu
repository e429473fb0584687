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
// Synthesis: one thread per ring pair (NR of them) and NM maps, as the
// CUDA-core kernels, the recurrence in registers.  Transpose: the
// register-blocked contraction of legendre_blk.cuh.
#include "df.cuh"
#include "legendre_blk.cuh"

namespace shtg {
namespace {

struct __align__(16) dfc2 {   // spin-0 coefficients (a, b)
    df a, b;
};
struct __align__(16) dfc4 {   // spin-2 coefficients (alpha, alpha + beta, alpha - beta, gamma)
    df x, y, z, w;
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
    r.y = df_from(v.y);
    r.z = df_from(v.z);
    r.w = df_from(v.w);
    return r;
}

template <int NR> struct DfPair {
    int pr[NR];
    df u[NR];   // u = 1 - cos theta
    int ls[NR], lsb[NR];
    df s0[NR], s1[NR], s2[NR], s3[NR];
    df a1[NR], a2[NR], b1[NR], b2[NR];
};

template <int NR>
__device__ __forceinline__ void df_pair_reset(DfPair<NR> &S, int j, int L) {
    S.a1[j] = S.a2[j] = S.b1[j] = S.b2[j] = df_zero();
    S.s0[j] = S.s1[j] = S.s2[j] = S.s3[j] = df_zero();
    S.u[j] = df_make(1.f, 0.f);
    S.ls[j] = S.lsb[j] = L + 1;
}

// geometry and FP64 start states of ring pair pr for m, rounded to df
template <int NR, int SPIN>
__device__ __forceinline__ void df_pair_load(const LegArgs<double> &a, int m, int pr, DfPair<NR> &S, int j) {
    S.pr[j] = pr;
    df_pair_reset(S, j, a.lmax);
    if (pr >= a.npairs) return;
    const double u = a.u[pr];
    S.u[j] = df_from(u);
    const int64_t o = (int64_t)m * a.npairs + pr;
    if (SPIN == 2) {
        const int2 q = a.ls2[o];
        S.ls[j] = q.x;
        S.lsb[j] = q.y;
        const double4_32a s = a.st2[o];
        S.s0[j] = df_from(s.x);
        S.s1[j] = df_from(s.y);
        S.s2[j] = df_from(s.z);
        S.s3[j] = df_from(s.w);
    } else {
        S.ls[j] = a.ls[o];
        const double2 s = a.st[o];
        S.s0[j] = df_from(s.x);
        S.s1[j] = df_from(s.y);
    }
}

// spin 0: lambda_l = a (1 - u) lambda_{l-1} + b lambda_{l-2}, formed as
// t + b lambda_{l-2} - t u with t = a lambda_{l-1} (as the FP64 kernels do):
// near the poles u ~ 1e-6 keeps its full relative precision, which a
// rounded cos(theta) = 1 - u would not (2^-48 absolute on cos(theta) is
// 1e-8 relative on u at the first HEALPix ring of N_side 1024)
template <int NR, bool INJ>
__device__ __forceinline__ void df_step0(DfPair<NR> &S, const dfc2 cf, int l) {
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        const df t = df_mul(cf.a, S.a1[j]);
        const df n = df_sub(df_add(t, df_mul(cf.b, S.a2[j])), df_mul(t, S.u[j]));
        S.a2[j] = S.a1[j];
        S.a1[j] = n;
        if (INJ && l == S.ls[j]) {
            S.a2[j] = S.s0[j];
            S.a1[j] = S.s1[j];
        }
    }
}

// spin 2: y+-_l = ((alpha + -beta) - alpha u) y+-_{l-1} - gamma y+-_{l-2}
template <int NR, bool INJ>
__device__ __forceinline__ void df_step2(DfPair<NR> &S, const dfc4 cf, int l) {
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        const df au = df_mul(cf.x, S.u[j]);
        const df tp = df_sub(cf.y, au), tm = df_sub(cf.z, au);
        const df pn = df_sub(df_mul(tp, S.a1[j]), df_mul(cf.w, S.a2[j]));
        const df mn = df_sub(df_mul(tm, S.b1[j]), df_mul(cf.w, S.b2[j]));
        S.a2[j] = S.a1[j];
        S.a1[j] = pn;
        S.b2[j] = S.b1[j];
        S.b1[j] = mn;
        if (INJ) {
            if (l == S.ls[j]) {
                S.a2[j] = S.s0[j];
                S.a1[j] = S.s1[j];
            }
            if (l == S.lsb[j]) {
                S.b2[j] = S.s2[j];
                S.b1[j] = S.s3[j];
            }
        }
    }
}

template <int NR, int SPIN, bool INJ>
__device__ __forceinline__ void df_stepx(DfPair<NR> &S, const dfc2 *s_rec, const dfc4 *s_s2c, int i, int l) {
    if (SPIN == 2) df_step2<NR, INJ>(S, s_s2c[i], l);
    else df_step0<NR, INJ>(S, s_rec[i], l);
}

// =========================================================== synthesis
template <int NR, int NM, int SPIN>
__global__ void __launch_bounds__(LEG_THREADS) k_leg_synth_df(const LegArgs<double> a) {
    constexpr int NA = (SPIN == 2) ? 2 * NM : NM;   // alm rows staged (E, B per map)
    constexpr int NACC = (SPIN == 2) ? 8 : 2;        // reals per parity class per map
    __shared__ dfc2 s_rec[SPIN == 2 ? 1 : LEG_CHUNK];
    __shared__ dfc4 s_s2c[SPIN == 2 ? LEG_CHUNK : 1];
    __shared__ dfc s_alm[NA][LEG_CHUNK];
    __shared__ int s_red[LEG_THREADS / 32];

    const int m = blockIdx.y;
    const int L = a.lmax;
    const int map0 = blockIdx.z * NM;
    const int nm = min(NM, a.nmaps - map0);
    const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2;

    DfPair<NR> S;
    int lo = L + 1, hi = -1;
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        df_pair_load<NR, SPIN>(a, m, blockIdx.x * (LEG_THREADS * NR) + j * LEG_THREADS + threadIdx.x, S, j);
        lo = min(lo, min(S.ls[j], S.lsb[j]));
        if (S.ls[j] <= L) hi = max(hi, S.ls[j]);
        if (S.lsb[j] <= L) hi = max(hi, S.lsb[j]);
    }
    const int warp_lo = __reduce_min_sync(0xffffffffu, lo);
    const int warp_hi = __reduce_max_sync(0xffffffffu, hi);
    const int clo = cta_min(warp_lo, s_red);

    dfacc accE[NR][NM][NACC], accO[NR][NM][NACC];
#pragma unroll
    for (int j = 0; j < NR; ++j)
#pragma unroll
        for (int k = 0; k < NM; ++k)
#pragma unroll
            for (int q = 0; q < NACC; ++q) {
                df_acc_zero(accE[j][k][q]);
                df_acc_zero(accO[j][k][q]);
            }

    auto accumulate = [&](const int i, dfacc(&acc)[NR][NM][NACC]) {
        if (SPIN == 0) {
#pragma unroll
            for (int k = 0; k < NM; ++k) {
                const dfc av = s_alm[k][i];
#pragma unroll
                for (int j = 0; j < NR; ++j) {
                    df_fma(acc[j][k][0], S.a1[j], av.re);
                    df_fma(acc[j][k][1], S.a1[j], av.im);
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < NR; ++j) {
                const df lw = df_add(S.a1[j], S.b1[j]), lx = df_sub(S.a1[j], S.b1[j]);
                const df nlw = df_neg(lw), nlx = df_neg(lx);
#pragma unroll
                for (int k = 0; k < NM; ++k) {
                    const dfc e = s_alm[2 * k][i];
                    const dfc b = s_alm[2 * k + 1][i];
                    // W parts: Q = -E lw, U = -B lw ; X parts: Q = -i B lx, U = i E lx
                    df_fma(acc[j][k][0], nlw, e.re);
                    df_fma(acc[j][k][1], nlw, e.im);
                    df_fma(acc[j][k][2], nlw, b.re);
                    df_fma(acc[j][k][3], nlw, b.im);
                    df_fma(acc[j][k][4], lx, b.im);
                    df_fma(acc[j][k][5], nlx, b.re);
                    df_fma(acc[j][k][6], nlx, e.im);
                    df_fma(acc[j][k][7], lx, e.re);
                }
            }
        }
    };
    auto renorm = [&]() {
#pragma unroll
        for (int j = 0; j < NR; ++j)
#pragma unroll
            for (int k = 0; k < NM; ++k)
#pragma unroll
                for (int q = 0; q < NACC; ++q) {
                    df_acc_norm(accE[j][k][q]);
                    df_acc_norm(accO[j][k][q]);
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
            for (int k = 0; k < NA; ++k) {
                double2 v = make_double2(0.0, 0.0);
                const int mk = (SPIN == 2) ? k / 2 : k;
                if (mk < nm) {
                    const int64_t row = (int64_t)(map0 + mk) * a.rs + ((SPIN == 2) ? (k & 1) : 0);
                    v = a.alm[row * a.nalm + idx];
                    if (m == 0) v.y = 0.0;
                    v.x *= bm;
                    v.y *= bm;
                }
                dfc d;
                d.re = df_from(v.x);
                d.im = df_from(v.y);
                s_alm[k][i] = d;
            }
        }
        __syncthreads();
        int l = max(c0, warp_lo);
        const int la_end = min(c1 - 1, warp_hi);
        for (; l <= la_end; ++l) {   // start states still being injected
            df_stepx<NR, SPIN, true>(S, s_rec, s_s2c, l - c0, l);
            if ((l - m) & 1) accumulate(l - c0, accO);
            else accumulate(l - c0, accE);
        }
        if (l < c1 && ((l - m) & 1)) {
            df_stepx<NR, SPIN, false>(S, s_rec, s_s2c, l - c0, l);
            accumulate(l - c0, accO);
            ++l;
        }
        for (; l + 1 < c1; l += 2) {
            df_stepx<NR, SPIN, false>(S, s_rec, s_s2c, l - c0, l);
            accumulate(l - c0, accE);
            df_stepx<NR, SPIN, false>(S, s_rec, s_s2c, l + 1 - c0, l + 1);
            accumulate(l + 1 - c0, accO);
        }
        if (l < c1) {
            df_stepx<NR, SPIN, false>(S, s_rec, s_s2c, l - c0, l);
            accumulate(l - c0, accE);
        }
        renorm();   // at most 64 terms per class since the last one
    }

#pragma unroll
    for (int j = 0; j < NR; ++j) {
        const int pr = S.pr[j];
        if (pr >= a.npairs) continue;
        const int rn = pr, rs = a.nring - 1 - pr;
#pragma unroll
        for (int k = 0; k < NM; ++k) {
            if (k >= nm) break;
            double E[NACC], O[NACC];
#pragma unroll
            for (int q = 0; q < NACC; ++q) {
                E[q] = df_acc_to(accE[j][k][q]);
                O[q] = df_acc_to(accO[j][k][q]);
            }
            if (SPIN == 0) {
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
}

// =========================================================== transpose
// double-FP32 arithmetic of the register-blocked transpose (legendre_blk.cuh)
struct ArDf {
    typedef df V;
    typedef dfacc Acc;
    typedef dfc2 C2;
    typedef dfc4 C4;
    typedef DfPair<1> State;
    static __device__ __forceinline__ V from(double x) { return df_from(x); }
    static __device__ __forceinline__ C2 c2(double2 v) { return dfc2_from(v); }
    static __device__ __forceinline__ C4 c4(double4_32a v) { return dfc4_from(v); }
    static __device__ __forceinline__ V add(V x, V y) { return df_add(x, y); }
    static __device__ __forceinline__ V sub(V x, V y) { return df_sub(x, y); }
    static __device__ __forceinline__ V neg(V x) { return df_neg(x); }
    static __device__ __forceinline__ void zero(Acc &s) { df_acc_zero(s); }
    static __device__ __forceinline__ void fma(Acc &s, V x, V y) { df_fma(s, x, y); }
    static __device__ __forceinline__ void norm(Acc &s) { df_acc_norm(s); }
    static __device__ __forceinline__ double to(const Acc &s) { return df_acc_to(s); }
    template <int SPIN>
    static __device__ __forceinline__ void load(const LegArgs<double> &a, int m, int pr, State &S) {
        df_pair_load<1, SPIN>(a, m, pr, S, 0);
    }
    template <int SPIN, bool INJ>
    static __device__ __forceinline__ void step(State &S, const C2 *s_rec, const C4 *s_s2c, int i, int l) {
        df_stepx<1, SPIN, INJ>(S, s_rec, s_s2c, i, l);
    }
};

template <int NR, int NM, int SPIN>
int launch_synth_df(Plan *p, const double2 *alm, int rs, int nmaps, const double *beam, double2 *F,
                    cudaStream_t st) {
    LegArgs<double> a = leg_make_args<double>(p);
    a.alm = alm;
    a.rs = rs;
    a.F = F;
    a.beam = beam;
    a.nmaps = nmaps;
    dim3 grid((p->npairs + LEG_THREADS * NR - 1) / (LEG_THREADS * NR), p->lmax + 1, (nmaps + NM - 1) / NM);
    prof_begin(p, K_LEG_SYN64, st);
    k_leg_synth_df<NR, NM, SPIN><<<grid, LEG_THREADS, 0, st>>>(a);
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
            case 1: return launch_synth_df<1, 1, 2>(p, alm, rs, nmaps, beam, F, st);
            case 2: return launch_synth_df<1, 2, 2>(p, alm, rs, nmaps, beam, F, st);
            case 3: return launch_synth_df<1, 3, 2>(p, alm, rs, nmaps, beam, F, st);
            default: return launch_synth_df<1, 4, 2>(p, alm, rs, nmaps, beam, F, st);
        }
    }
    switch (leg_maps_per_pass(0, nmaps, nm0, 6)) {
        case 1: return launch_synth_df<1, 1, 0>(p, alm, rs, nmaps, beam, F, st);
        case 2: return launch_synth_df<1, 2, 0>(p, alm, rs, nmaps, beam, F, st);
        case 3: return launch_synth_df<1, 3, 0>(p, alm, rs, nmaps, beam, F, st);
        case 4: return launch_synth_df<1, 4, 0>(p, alm, rs, nmaps, beam, F, st);
        case 6: return launch_synth_df<1, 6, 0>(p, alm, rs, nmaps, beam, F, st);
        default: return launch_synth_df<1, 8, 0>(p, alm, rs, nmaps, beam, F, st);
    }
}

int leg_analysis_df(Plan *p, int spin, const double2 *G, int nmaps, const double *beam, double2 *alm, int rs,
                    cudaStream_t st, int vjp) {
    if (spin == 2) return analysis_blk<ArDf, 2>(p, G, nmaps, beam, alm, rs, st, vjp);
    return analysis_blk<ArDf, 0>(p, G, nmaps, beam, alm, rs, st, vjp);
}

}  // namespace shtg
