// FP64-accurate Legendre transpose (Y^T) as a register-blocked contraction,
// for native FP64 (legendre_g64.cu) and double-FP32 (legendre_df.cu)
// arithmetic.
//
// c_lm = sum_r lambda_lm(theta_r) G_r(m): CTA = one m, 128 l and NMT maps.
// Per stage of 32 ring pairs each of the four warps generates one 32-l
// segment of the recurrences (a lane per pair) from the FP64 states
// tabulated every SHTG_TS64 l into shared memory ([row = l - lbase][pair]),
// and every thread accumulates a block of outputs over all ring pairs in
// registers: NMT rows of one parity class of l - m (App. A: lambda_lm(pi -
// theta) = (-1)^(l+m) lambda_lm(theta), so class-E rows take G_N + G_S and
// class-O rows G_N - G_S) times the 2 (spin 0) or 4 (spin 2: E re, E im, B
// re, B im) outputs of one map.  Each recurrence runs once per (l, ring
// pair) for the CTA's maps, and the sum over ring pairs needs no
// cross-thread reduction.
//
// What bounds it: the arithmetic.  An FP64 warp instruction occupies its
// scheduler's FP64 unit for 64 cycles (two lanes per clock and SM), a
// double-FP32 multiply-add costs about twelve FP32 instructions, so the
// loop is as fast as its count of useful operations per scheduler:
// - all four warps generate (one half-warp generating 16 pairs over 128 l,
//   the FP64 kernel's first form, kept three of four FP64 units idle for
//   longer than the contraction of eight maps takes);
// - NMT follows the number of maps that the call has (1, 2, 4 or 8), so that
//   few threads multiply maps that are not there;
// - row blocks beyond l_max, or before the first significant l of the stage's
//   pairs, are left out.
// Measured (FP64; before: the best of the 8-map form and the warp-reduction
// kernels, which stay candidates of the spin-0 FP64 transpose, legendre64.cu):
// N_side 300, l_max 500, 3 maps, spin 0 / 2:
// 2.87 / 7.3 -> 1.65 / 5.5 ms; N_side 512, l_max 1024, 8 maps: 28.4 / 115 ->
// 15.1 / 56 ms.  The ring data as 16-byte (re, im) operands, signs and the
// lw / lx exchange folded in when they are staged: N_side 128, l_max 256, 2
// T+E+B maps, both transposes and both syntheses in FP64 1.93 -> 1.81 ms.
// Double-FP32, N_side 512, l_max 1024, 4 maps, spin 2: 15.8 -> 11.1 ms, 9.2 ms
// with packed arithmetic (df2.cuh), 7.1 ms with the value tile in two halves
// and integer conversions (df.cuh).
#pragma once

#include <string>

#include "legendre_kernels.cuh"

namespace shtg {

constexpr int B_LR = 128;        // l per CTA (rows): four 32-l segments, one per warp
constexpr int B_KP = 32;         // ring pairs per stage (a warp's lanes)
constexpr int B_NT = 128;        // threads
constexpr int B_LS = B_KP + 1;   // row stride of the value tile (odd: rows in distinct banks)
static_assert(SHTG_TS64 == 32, "a warp restarts its 32-l segment from a tabulated state");

// maps per pass of an FP64-accurate Legendre sum out of the n sizes nms
// (legendre64.cu)
int leg_maps_per_pass(int spin, int nmaps, const int *nms, int n);

// Ar: the arithmetic.  V value, Acc two running sums (re, im), Op one ring-data
// operand (re, im) in registers and OPB its bytes in shared memory, C2 / C4
// staged coefficients, State<SPIN> recurrence state of one pair.
//
// Ring-data operands of a (ring pair, map, class c): spin 0 one, the class's
// set G_c; spin 2 four, those of the lw terms -Q_c, -U_c (the class's set) and
// of the lx terms (U_im, -U_re), (-Q_im, Q_re) of the other class's set:
//   E^ = -lw G_Q - i lx G_U,  B^ = i lx G_Q - lw G_U.
template <class Ar, int SPIN, int NMT> struct BlkLayout {
    typedef typename Ar::V V;
    // Parts of a segment generated at a time.  Two (double-FP32): the value tile
    // takes 34 instead of 68 KB at spin 2, and four CTAs share an SM instead of
    // two, so one's generation and staging run beside another's contraction (the
    // FP32 pipe was 56 % busy).  One map: a half would leave threads without rows.
    // FP64: its pipe is the bound with two CTAs as well.
    static constexpr int HV = Ar::HALVES && NMT > 1 ? 2 : 1;   // parts of a segment generated at a time
    static constexpr int TR = B_LR / HV;                       // rows of the value tile
    static constexpr int NV = SPIN == 2 ? 2 : 1;   // value tiles: lambda, or (lw, lx)
    static constexpr int NO = SPIN == 2 ? 4 : 2;   // outputs per map
    static constexpr int NOP = SPIN == 2 ? 4 : 1;  // ring-data operands per (pair, map, class)
    static constexpr int COEF = SPIN == 2 ? sizeof(typename Ar::C4) : sizeof(typename Ar::C2);
    static constexpr int LAM = 0;
    static constexpr int GSET = (LAM + NV * TR * B_LS * (int)sizeof(V) + 15) & ~15;
    static constexpr int CO = (GSET + B_KP * NOP * NMT * 2 * Ar::OPB + 31) & ~31;
    static constexpr int RED = CO + B_LR * COEF;
    static constexpr int BYTES = RED + 16;
};

// Ring-data operands of stage s (32 ring pairs) for NMT maps
template <class Ar, int SPIN, int NMT>
__device__ __forceinline__ void stage_ops(const LegArgs<double> &a, int m, int s, int map0, int nm, int tid,
                                          unsigned char *gset) {
    constexpr int NOP = BlkLayout<Ar, SPIN, NMT>::NOP;
    constexpr int OS = NMT * 2 * Ar::OPB;   // stride of the operands
    const int64_t rowsz = (int64_t)a.nring * (a.lmax + 1);
    for (int it = tid; it < B_KP * NMT; it += B_NT) {
        const int pp = it / NMT, kk = it % NMT;
        const int pr = s * B_KP + pp;
        // z: spin 0 G_E, G_O; spin 2 Q_E, Q_O, U_E, U_O
        double2 z[4] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0), make_double2(0.0, 0.0),
                        make_double2(0.0, 0.0)};
        if (pr < a.npairs && kk < nm) {
            const int rn = pr, rs = a.nring - 1 - pr;
#pragma unroll
            for (int cc = 0; cc < (SPIN == 2 ? 2 : 1); ++cc) {
                const int64_t row = SPIN == 2 ? 2 * (map0 + kk) + cc : map0 + kk;
                const double2 *gr = a.F + row * rowsz + m;
                const double2 gn = gr[(int64_t)rn * (a.lmax + 1)];
                const double2 gs = rs != rn ? gr[(int64_t)rs * (a.lmax + 1)] : make_double2(0.0, 0.0);
                z[2 * cc] = make_double2(gn.x + gs.x, gn.y + gs.y);       // even set
                z[2 * cc + 1] = make_double2(gn.x - gs.x, gn.y - gs.y);   // odd set
            }
        }
#pragma unroll
        for (int cl = 0; cl < 2; ++cl) {
            unsigned char *g = gset + ((pp * NOP * NMT + kk) * 2 + cl) * Ar::OPB;
            if (SPIN == 0) {
                Ar::put(g, z[cl].x, z[cl].y);
            } else {
                const double2 xq = z[1 - cl], xu = z[3 - cl];
                Ar::put(g, -z[cl].x, -z[cl].y);
                Ar::put(g + OS, -z[2 + cl].x, -z[2 + cl].y);
                Ar::put(g + 2 * OS, xu.y, -xu.x);
                Ar::put(g + 3 * OS, -xq.y, xq.x);
            }
        }
    }
}

// NG groups of 128 threads, each with its own tiles, take the stages in turn;
// group 0 adds the sums of group 1 and writes.  Two groups (FP64, grids that
// leave SMs idle): a CTA with few significant l keeps one or two of its warps
// busy, so the second group's warps sit two schedulers further on.
template <class Ar, int SPIN, int NMT, int NG>
__global__ void __launch_bounds__(B_NT * NG) k_leg_analysis_blk(const LegArgs<double> a) {
    typedef BlkLayout<Ar, SPIN, NMT> Ly;
    typedef typename Ar::V V;
    constexpr int NO = Ly::NO, NOP = Ly::NOP, NJ = NMT, RG = 64 / NJ;
    constexpr int HV = Ly::HV, TR = Ly::TR, SR = 32 / HV, NJH = NJ / HV;
    extern __shared__ __align__(32) unsigned char smem[];
    const int grp = NG == 1 ? 0 : threadIdx.x / B_NT;
    const int tid = NG == 1 ? threadIdx.x : (threadIdx.x % B_NT) ^ (64 * grp);
    unsigned char *tiles = smem + grp * Ly::CO;
    V *lam = reinterpret_cast<V *>(tiles + Ly::LAM);     // [NV][TR][B_LS]
    unsigned char *gset = tiles + Ly::GSET;              // [B_KP][NOP][NMT][class] operands
    typename Ar::C2 *s_rec = reinterpret_cast<typename Ar::C2 *>(smem + NG * Ly::CO);
    typename Ar::C4 *s_s2c = reinterpret_cast<typename Ar::C4 *>(smem + NG * Ly::CO);
    int *s_first = reinterpret_cast<int *>(smem + (NG - 1) * Ly::CO + Ly::RED);

    const int m = blockIdx.y;
    const int L = a.lmax;
    const int lbase = m + blockIdx.x * B_LR;
    if (lbase > L) return;
    const int lend = min(L, lbase + B_LR - 1);
    const int map0 = blockIdx.z * NMT;
    const int nm = min(NMT, a.nmaps - map0);
    const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2;

    for (int i = threadIdx.x; i < B_LR; i += B_NT * NG) {
        const int l = lbase + i;
        const bool in = l <= L;
        if (SPIN == 2) s_s2c[i] = Ar::c4(in ? a.s2c[base + l] : make_double4_32a(0.0, 0.0, 0.0, 0.0));
        else s_rec[i] = Ar::c2(in ? a.rec[base + l] : make_double2(0.0, 0.0));
    }
    // first ring pair whose recurrence starts at or before lend (the start l
    // falls towards the equator; a later pair without significant values only
    // adds exact zeros)
    if (threadIdx.x == 0) *s_first = a.npairs;
    __syncthreads();
    for (int pr = threadIdx.x; pr < a.npairs; pr += B_NT * NG) {
        const int64_t o = (int64_t)m * a.npairs + pr;
        int lsp;
        if (SPIN == 2) {
            const int2 q = a.ls2[o];
            lsp = min(q.x, q.y);
        } else {
            lsp = a.ls[o];
        }
        if (lsp <= lend) {
            atomicMin(s_first, pr);
            break;
        }
    }
    __syncthreads();
    const int s0 = *s_first / B_KP;
    const int nps = (a.npairs + B_KP - 1) / B_KP;

    // this thread's outputs: map k, class c, in part h of the segments the tile
    // rows c + 2 (rg + RG j), j < NJH; tile row r is row lrow(h, r)
    auto lrow = [](int h, int r) { return HV == 1 ? r : 32 * (r / SR) + SR * h + r % SR; };
    const int k = tid & (NMT - 1), c = (tid / NMT) & 1, rg = tid / (2 * NMT);
    typename Ar::Acc acc[NJ][NO / 2];
#pragma unroll
    for (int j = 0; j < NJ; ++j)
#pragma unroll
        for (int q = 0; q < NO / 2; ++q) Ar::zero(acc[j][q]);

    // this warp's tile rows of block j: WR consecutive ones from row0 + 2 RG j
    constexpr int WR = 32 / NMT;
    const int row0 = 2 * ((tid & ~31) / (2 * NMT));
    auto sync = [&]() {   // of the group
        if (NG == 1) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(B_NT) : "memory");
    };
    for (int s = s0 + grp; s < nps; s += NG) {
        // ---- recurrences of the stage's 32 ring pairs: warp w runs rows
        // 32 w .. 32 w + 31 of pair s * 32 + lane from the FP64 state
        // tabulated at l0 = lbase + 32 w
        const int pp = tid & 31, seg = tid >> 5;
        const int pr = s * B_KP + pp;
        const int l0 = lbase + 32 * seg;
        typename Ar::template State<SPIN> S;
        Ar::template load<SPIN>(a, m, pr, S);
        const bool live = pr < a.npairs && l0 <= L;
        // no pair of the stage has a significant value below this l
        const int first_l = __reduce_min_sync(0xffffffffu, SPIN == 2 ? min(S.ls[0], S.lsb[0]) : S.ls[0]);
        if (live) {
            const int64_t e = (a.toff64[m] + (l0 - m) / SHTG_TS64) * a.npairs + pr;
            if constexpr (SPIN == 2) Ar::restart(S, a.tst64_2[e]);
            else Ar::restart(S, a.tst64_0[e]);
        }
        // injection steps only if some pair of the warp starts in this segment
        const bool inj = __any_sync(0xffffffffu, live && ((S.ls[0] >= l0 && S.ls[0] < l0 + 32) ||
                                                          (SPIN == 2 && S.lsb[0] >= l0 && S.lsb[0] < l0 + 32)));
        const bool gen = __any_sync(0xffffffffu, live) && l0 + 31 >= first_l;
#pragma unroll
        for (int h = 0; h < HV; ++h) {
            sync();   // the previous part's (stage's) tiles are consumed
            if (gen) {
                for (int r = SR * seg; r < SR * seg + SR; ++r) {
                    const int i = lrow(h, r);
                    if (inj) Ar::template step<SPIN, true>(S, s_rec, s_s2c, i, lbase + i);
                    else Ar::template step<SPIN, false>(S, s_rec, s_s2c, i, lbase + i);
                    V v[2];
                    Ar::template values<SPIN>(S, v);
                    lam[r * B_LS + pp] = live ? v[0] : Ar::from(0.0);
                    if (SPIN == 2) lam[(TR + r) * B_LS + pp] = live ? v[1] : Ar::from(0.0);
                }
            } else {   // beyond l_max or before every start
                for (int r = SR * seg; r < SR * seg + SR; ++r) {
                    lam[r * B_LS + pp] = Ar::from(0.0);
                    if (SPIN == 2) lam[(TR + r) * B_LS + pp] = Ar::from(0.0);
                }
            }
            // ---- ring data of the stage: per (pair, map, class) the operands
            if (h == 0) stage_ops<Ar, SPIN, NMT>(a, m, s, map0, nm, tid, gset);
            sync();
            // ---- contraction over the stage's ring pairs; row blocks beyond
            // l_max or before every start of the stage (exact zeros) are left out
            bool on[NJH];
#pragma unroll
            for (int j = 0; j < NJH; ++j) {
                const int l = lbase + lrow(h, row0 + 2 * RG * j);
                on[j] = l <= L && l + WR > first_l;
            }
#pragma unroll 2
            for (int p = 0; p < B_KP; ++p) {
                typename Ar::Op g[NOP];
#pragma unroll
                for (int o = 0; o < NOP; ++o) g[o] = Ar::get(gset + (((p * NOP + o) * NMT + k) * 2 + c) * Ar::OPB);
#pragma unroll
                for (int j = 0; j < NJH; ++j) {
                    if (!on[j]) continue;   // warp-uniform
                    const int r = c + 2 * (rg + RG * j);
                    typename Ar::Acc *ac = acc[h * NJH + j];
                    const V lw = lam[r * B_LS + p];
                    if (SPIN == 0) {
                        Ar::fma(ac[0], lw, g[0]);
                    } else {
                        const V lx = lam[(TR + r) * B_LS + p];
                        Ar::fma(ac[0], lx, g[NOP / 2]);
                        Ar::fma(ac[0], lw, g[0]);
                        Ar::fma(ac[NO / 2 - 1], lx, g[NOP - 1]);
                        Ar::fma(ac[NO / 2 - 1], lw, g[NOP / 2 - 1]);
                    }
                }
            }
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int q = 0; q < NO / 2; ++q) Ar::norm(acc[j][q]);   // 64 terms at most since the last
    }
    if constexpr (NG == 2) {
        __syncthreads();   // both groups' tiles are consumed
        typename Ar::Acc *sum = reinterpret_cast<typename Ar::Acc *>(smem);
        if (grp == 1) {
#pragma unroll
            for (int j = 0; j < NJ; ++j)
#pragma unroll
                for (int q = 0; q < NO / 2; ++q) sum[(j * (NO / 2) + q) * B_NT + tid] = acc[j][q];
        }
        __syncthreads();
        if (grp == 1) return;
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int q = 0; q < NO / 2; ++q) Ar::add(acc[j][q], sum[(j * (NO / 2) + q) * B_NT + tid]);
    }
    // ---- epilogue: every alm of this CTA's l range written once
    if (k >= nm) return;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int l = lbase + lrow(j / NJH, c + 2 * (rg + RG * (j % NJH)));
        if (l > L) continue;
        const double bm = (a.beam ? a.beam[l] : 1.0) * ((a.vjp && m > 0) ? 2.0 : 1.0);
#pragma unroll
        for (int cc = 0; cc < NO / 2; ++cc) {
            const int64_t row = (int64_t)(map0 + k) * a.rs + cc;
            double2 *dst = const_cast<double2 *>(a.alm) + row * a.nalm + base + l;
            const double2 v = Ar::to(acc[j][cc]);
            *dst = make_double2(v.x * bm, m == 0 ? 0.0 : v.y * bm);
        }
    }
}

template <class Ar, int SPIN, int NMT, int NG>
int launch_analysis_blk_g(Plan *p, const double2 *G, int nmaps, const double *beam, double2 *alm, int rs,
                        cudaStream_t st, int vjp) {
    LegArgs<double> a = leg_make_args<double>(p);
    a.alm = alm;
    a.rs = rs;
    a.vjp = vjp;
    a.F = const_cast<double2 *>(G);
    a.beam = beam;
    a.nmaps = nmaps;
    if (!a.toff64 || !a.tst64_0 || (SPIN == 2 && !a.tst64_2)) {
        set_error("FP64-accurate transpose: the plan has no FP64 recurrence tile states");
        return SHTG_ERR_ARG;
    }
    typedef BlkLayout<Ar, SPIN, NMT> Ly;
    static_assert(NG == 1 || B_NT * NMT * Ly::NO / 2 * sizeof(typename Ar::Acc) <= Ly::CO, "sums of a group");
    const int smem = Ly::BYTES + (NG - 1) * Ly::CO;
    auto kern = k_leg_analysis_blk<Ar, SPIN, NMT, NG>;
    if (smem > 48 * 1024) SHTG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    dim3 grid((p->lmax + B_LR) / B_LR, p->lmax + 1, (nmaps + NMT - 1) / NMT);
    prof_begin(p, K_LEG_ANA64, st);
    kern<<<grid, B_NT * NG, smem, st>>>(a);
    prof_end(p, st);
    SHTG_CHECK_LAUNCH("k_leg_analysis_blk");
    return SHTG_OK;
}

// NG: two groups where CTAs of one group would not give every SM one and there
// are stages for both (N_side 32, l_max 64, one map: 25.3 -> 17.2 us).
template <class Ar, int SPIN, int NMT>
int launch_analysis_blk(Plan *p, const double2 *G, int nmaps, const double *beam, double2 *alm, int rs,
                        cudaStream_t st, int vjp) {
    if constexpr (Ar::GROUPS) {
        const int64_t ctas = (int64_t)((p->lmax + B_LR) / B_LR) * (p->lmax + 1) * ((nmaps + NMT - 1) / NMT);
        if (ctas <= p->nsm && p->npairs > B_KP)
            return launch_analysis_blk_g<Ar, SPIN, NMT, 2>(p, G, nmaps, beam, alm, rs, st, vjp);
    }
    return launch_analysis_blk_g<Ar, SPIN, NMT, 1>(p, G, nmaps, beam, alm, rs, st, vjp);
}

// NMT: the least work over the call's maps (leg_maps_per_pass)
template <class Ar, int SPIN>
int analysis_blk(Plan *p, const double2 *G, int nmaps, const double *beam, double2 *alm, int rs, cudaStream_t st,
                 int vjp) {
    static const int nmt[] = {8, 4, 2, 1};
    switch (leg_maps_per_pass(SPIN, nmaps, nmt, 4)) {
        case 1: return launch_analysis_blk<Ar, SPIN, 1>(p, G, nmaps, beam, alm, rs, st, vjp);
        case 2: return launch_analysis_blk<Ar, SPIN, 2>(p, G, nmaps, beam, alm, rs, st, vjp);
        case 4: return launch_analysis_blk<Ar, SPIN, 4>(p, G, nmaps, beam, alm, rs, st, vjp);
        default: return launch_analysis_blk<Ar, SPIN, 8>(p, G, nmaps, beam, alm, rs, st, vjp);
    }
}

}  // namespace shtg
