// Native FP64 arithmetic of the register-blocked Legendre transpose
// (legendre_blk.cuh), and the FP64 recurrence states tabulated every
// SHTG_TS64 l that it (and its double-FP32 form) restarts from: built once
// at plan creation by the same steps, so the values equal those of one
// continuous run.
#include <algorithm>
#include <string>
#include <vector>

#include "legendre_blk.cuh"

namespace shtg {
namespace {

struct ArF64 {
    typedef double V;
    typedef double2 Acc;
    typedef double2 Op;
    typedef double2 C2;
    typedef double4_32a C4;
    template <int SPIN> using State = PairState<double, 1>;
    static constexpr bool HALVES = false, GROUPS = true;
    static __device__ __forceinline__ void add(Acc &s, const Acc &t) {
        s.x += t.x;
        s.y += t.y;
    }
    static constexpr int OPB = sizeof(double2);
    static __device__ __forceinline__ V from(double x) { return x; }
    static __device__ __forceinline__ C2 c2(double2 v) { return v; }
    static __device__ __forceinline__ C4 c4(double4_32a v) { return v; }
    static __device__ __forceinline__ void put(unsigned char *p, double re, double im) {
        *reinterpret_cast<double2 *>(p) = make_double2(re, im);
    }
    static __device__ __forceinline__ Op get(const unsigned char *p) { return *reinterpret_cast<const double2 *>(p); }
    static __device__ __forceinline__ void zero(Acc &s) { s = make_double2(0.0, 0.0); }
    static __device__ __forceinline__ void fma(Acc &s, V x, const Op &y) {
        s.x = ::fma(x, y.x, s.x);
        s.y = ::fma(x, y.y, s.y);
    }
    static __device__ __forceinline__ void norm(Acc &) {}
    static __device__ __forceinline__ double2 to(const Acc &s) { return s; }
    static __device__ __forceinline__ void restart(State<2> &S, double2 t) {
        S.a1[0] = t.x;
        S.a2[0] = t.y;
    }
    static __device__ __forceinline__ void restart(State<2> &S, double4_32a t) {
        S.a1[0] = t.x;
        S.a2[0] = t.y;
        S.b1[0] = t.z;
        S.b2[0] = t.w;
    }
    // lambda, or (lw, lx)
    template <int SPIN> static __device__ __forceinline__ void values(const State<SPIN> &S, V (&v)[2]) {
        v[0] = SPIN == 2 ? S.a1[0] + S.b1[0] : S.a1[0];
        v[1] = SPIN == 2 ? S.a1[0] - S.b1[0] : 0.0;
    }
    template <int SPIN>
    static __device__ __forceinline__ void load(const LegArgs<double> &a, int m, int pr, State<SPIN> &S) {
        S.a1[0] = S.a2[0] = S.b1[0] = S.b2[0] = 0.0;
        S.u[0] = 1.0;
        S.ls[0] = S.lsb[0] = a.lmax + 1;
        S.s0[0] = S.s1[0] = S.s2[0] = S.s3[0] = 0.0;
        if (pr >= a.npairs) return;
        const int64_t o = (int64_t)m * a.npairs + pr;
        S.u[0] = a.u[pr];
        if (SPIN == 2) {
            const int2 q = a.ls2[o];
            S.ls[0] = q.x;
            S.lsb[0] = q.y;
            const double4_32a s4 = a.st2[o];
            S.s0[0] = s4.x;
            S.s1[0] = s4.y;
            S.s2[0] = s4.z;
            S.s3[0] = s4.w;
        } else {
            S.ls[0] = a.ls[o];
            const double2 s2 = a.st[o];
            S.s0[0] = s2.x;
            S.s1[0] = s2.y;
        }
    }
    template <int SPIN, bool INJ>
    static __device__ __forceinline__ void step(State<SPIN> &S, const C2 *s_rec, const C4 *s_s2c, int i, int l) {
        stepx<double, 1, SPIN, INJ>(S, s_rec, s_s2c, i, l);
    }
};

// Synthesis on small grids: CTA = one m, 32 ring pairs (a lane each) and NM
// maps; warp w runs the 32-l segments w, w + 4, ... from the tabulated states
// and the warps' sums are added in their order.  The serial chain of a CTA is
// then a quarter of the l range, and all four FP64 units of an SM work where the
// one-thread-per-pair kernel keeps one per 32 pairs busy over the whole range.
template <int NM, int SPIN>
__global__ void __launch_bounds__(LEG_THREADS) k_leg_synth_seg(const LegArgs<double> a) {
    constexpr int NW = LEG_THREADS / 32, NA = SPIN == 2 ? 2 * NM : NM, NACC = SPIN == 2 ? 8 : 2;
    constexpr int NS = 2 * NM * NACC;   // sums of a pair
    extern __shared__ __align__(32) unsigned char smem[];
    const int m = blockIdx.y, L = a.lmax, n = L + 1 - m;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int map0 = blockIdx.z * NM, nm = min(NM, a.nmaps - map0);
    const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2;
    // coefficients and alm of every l, then (same memory) the warps' sums
    double4_32a *s_s2c = reinterpret_cast<double4_32a *>(smem);
    double2 *s_rec = reinterpret_cast<double2 *>(smem);
    double2 *s_alm = reinterpret_cast<double2 *>(smem + n * (SPIN == 2 ? sizeof(double4_32a) : sizeof(double2)));
    for (int i = threadIdx.x; i < n; i += LEG_THREADS) {
        const int l = m + i;
        if (SPIN == 2) s_s2c[i] = a.s2c[base + l];
        else s_rec[i] = a.rec[base + l];
        const double bm = a.beam ? a.beam[l] : 1.0;
#pragma unroll
        for (int k = 0; k < NA; ++k) {
            double2 v = make_double2(0.0, 0.0);
            const int mk = SPIN == 2 ? k / 2 : k;
            if (mk < nm) {
                v = a.alm[((int64_t)(map0 + mk) * a.rs + (SPIN == 2 ? (k & 1) : 0)) * a.nalm + base + l];
                if (m == 0) v.y = 0.0;
                v.x *= bm;
                v.y *= bm;
            }
            s_alm[k * n + i] = v;
        }
    }
    const int pr = blockIdx.x * 32 + lane;
    ArF64::State<SPIN> S;
    ArF64::load<SPIN>(a, m, pr, S);
    const int first_l = __reduce_min_sync(0xffffffffu, SPIN == 2 ? min(S.ls[0], S.lsb[0]) : S.ls[0]);
    __syncthreads();
    double acc[2][NM][NACC];   // class l - m even, odd
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int k = 0; k < NM; ++k)
#pragma unroll
            for (int q = 0; q < NACC; ++q) acc[c][k][q] = 0.0;
    auto add = [&](int i, double(&ac)[NM][NACC]) {
        stepx<double, 1, SPIN, true>(S, s_rec, s_s2c, i, m + i);
        double v[2];
        ArF64::values<SPIN>(S, v);
        const double lw = v[0], lx = v[1];
#pragma unroll
        for (int k = 0; k < NM; ++k) {
            if (SPIN == 0) {
                const double2 e = s_alm[k * n + i];
                ac[k][0] = fma(lw, e.x, ac[k][0]);
                ac[k][1] = fma(lw, e.y, ac[k][1]);
            } else {
                // W parts: Q = -E lw, U = -B lw ; X parts: Q = -i B lx, U = i E lx
                const double2 e = s_alm[2 * k * n + i], b = s_alm[(2 * k + 1) * n + i];
                ac[k][0] = fma(-lw, e.x, ac[k][0]);
                ac[k][1] = fma(-lw, e.y, ac[k][1]);
                ac[k][2 % NACC] = fma(-lw, b.x, ac[k][2 % NACC]);
                ac[k][3 % NACC] = fma(-lw, b.y, ac[k][3 % NACC]);
                ac[k][4 % NACC] = fma(lx, b.y, ac[k][4 % NACC]);
                ac[k][5 % NACC] = fma(-lx, b.x, ac[k][5 % NACC]);
                ac[k][6 % NACC] = fma(-lx, e.y, ac[k][6 % NACC]);
                ac[k][7 % NACC] = fma(lx, e.x, ac[k][7 % NACC]);
            }
        }
    };
    for (int t = w; t * SHTG_TS64 < n; t += NW) {
        const int i0 = t * SHTG_TS64, i1 = min(n, i0 + SHTG_TS64);
        if (m + i1 <= first_l) continue;   // before every start of the warp's pairs
        if (pr < a.npairs) {
            const int64_t e = (a.toff64[m] + t) * a.npairs + pr;
            if constexpr (SPIN == 2) ArF64::restart(S, a.tst64_2[e]);
            else ArF64::restart(S, a.tst64_0[e]);
        }
        int i = i0;
        for (; i + 1 < i1; i += 2) {
            add(i, acc[0]);
            add(i + 1, acc[1]);
        }
        if (i < i1) add(i, acc[0]);
    }
    __syncthreads();   // coefficients and alm are consumed
    double *s_sum = reinterpret_cast<double *>(smem);   // [NW][NS][32]
#pragma unroll
    for (int q = 0; q < NS; ++q) s_sum[(w * NS + q) * 32 + lane] = acc[q / (NM * NACC)][q / NACC % NM][q % NACC];
    __syncthreads();
    // warp w finishes the maps w, w + 4, ...
    if (pr >= a.npairs) return;
    const int rn = pr, rs = a.nring - 1 - pr;
    for (int k = w; k < nm; k += NW) {
        double E[NACC], O[NACC];
#pragma unroll
        for (int q = 0; q < NACC; ++q) {
            E[q] = O[q] = 0.0;
#pragma unroll
            for (int v = 0; v < NW; ++v) {
                E[q] += s_sum[(v * NS + k * NACC + q) * 32 + lane];
                O[q] += s_sum[(v * NS + (NM + k) * NACC + q) * 32 + lane];
            }
        }
        double2 *oq = a.F + (int64_t)((SPIN == 2 ? 2 : 1) * (map0 + k)) * a.nring * (L + 1) + m;
        if constexpr (SPIN == 0) {
            oq[(int64_t)rn * (L + 1)] = make_double2(E[0] + O[0], E[1] + O[1]);
            if (rs != rn) oq[(int64_t)rs * (L + 1)] = make_double2(E[0] - O[0], E[1] - O[1]);
        } else {
            // north: W + X over both classes; south: even W - X, odd X - W
            double2 *ou = oq + (int64_t)a.nring * (L + 1);
            oq[(int64_t)rn * (L + 1)] = make_double2(E[0] + O[0] + E[4] + O[4], E[1] + O[1] + E[5] + O[5]);
            ou[(int64_t)rn * (L + 1)] = make_double2(E[2] + O[2] + E[6] + O[6], E[3] + O[3] + E[7] + O[7]);
            if (rs != rn) {
                oq[(int64_t)rs * (L + 1)] = make_double2(E[0] - O[0] - E[4] + O[4], E[1] - O[1] - E[5] + O[5]);
                ou[(int64_t)rs * (L + 1)] = make_double2(E[2] - O[2] - E[6] + O[6], E[3] - O[3] - E[7] + O[7]);
            }
        }
    }
}

template <int NM, int SPIN>
int launch_synth_seg(Plan *p, const double2 *alm, int rs, int nmaps, const double *beam, double2 *F, cudaStream_t st) {
    LegArgs<double> a = leg_make_args<double>(p);
    a.alm = alm;
    a.rs = rs;
    a.F = F;
    a.beam = beam;
    a.nmaps = nmaps;
    const size_t in = (size_t)(p->lmax + 1) * ((SPIN == 2 ? 32 : 16) + 16 * (SPIN == 2 ? 2 * NM : NM));
    const size_t sums = sizeof(double) * LEG_THREADS * 2 * NM * (SPIN == 2 ? 8 : 2);
    const size_t smem = std::max(in, sums);
    auto kern = k_leg_synth_seg<NM, SPIN>;
    if (smem > 48 * 1024) SHTG_CUDA(allow_max_smem(kern));
    dim3 grid((p->npairs + 31) / 32, p->lmax + 1, (nmaps + NM - 1) / NM);
    prof_begin(p, K_LEG_SYN64, st);
    kern<<<grid, LEG_THREADS, smem, st>>>(a);
    prof_end(p, st);
    SHTG_CHECK_LAUNCH("k_leg_synth_seg");
    return SHTG_OK;
}

// FP64 recurrence state before every l = m + SHTG_TS64 t of every (m, ring
// pair), [m][t][pair]: the steps of the Legendre kernels, one thread per
// (m, pair).
template <int SPIN>
__global__ void __launch_bounds__(LEG_THREADS) k_tile_states64(const LegArgs<double> a, const int64_t *toff,
                                                               double2 *out0, double4_32a *out2) {
    const int m = blockIdx.y;
    const int L = a.lmax;
    PairState<double, 1> S;
    int wlo, whi;
    load_pairs<double, 1, SPIN>(a, blockIdx.x, m, S, wlo, whi);
    const int pr = S.pr[0];
    if (pr >= a.npairs) return;
    const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2;
    const int64_t o = toff[m] * a.npairs + pr;
    for (int l = m; l <= L; ++l) {
        if (((l - m) & (SHTG_TS64 - 1)) == 0) {
            const int64_t e = o + (int64_t)((l - m) / SHTG_TS64) * a.npairs;
            if (SPIN == 2) out2[e] = make_double4_32a(S.a1[0], S.a2[0], S.b1[0], S.b2[0]);
            else out0[e] = make_double2(S.a1[0], S.a2[0]);
        }
        stepx<double, 1, SPIN, true>(S, a.rec + base, a.s2c + base, l, l);
    }
}

}  // namespace

int build_tile_states64(Plan *p) {
    const int L = p->lmax;
    std::vector<int64_t> toff(L + 2);
    toff[0] = 0;
    for (int m = 0; m <= L; ++m) toff[m + 1] = toff[m] + (L + 1 - m + SHTG_TS64 - 1) / SHTG_TS64;
    const size_t nent = (size_t)toff[L + 1] * p->npairs;
    auto alloc = [&](void **ptr, size_t bytes) -> int {
        cudaError_t e = cudaMalloc(ptr, bytes);
        if (e != cudaSuccess) {
            *ptr = nullptr;
            cudaGetLastError();
            set_error(std::string("cudaMalloc of ") + std::to_string(bytes) +
                      " bytes (FP64 recurrence tile states) failed: " + cudaGetErrorString(e));
            return SHTG_ERR_NOMEM;
        }
        p->device_bytes += (int64_t)bytes;
        return SHTG_OK;
    };
    SHTG_TRY(alloc((void **)&p->d_toff64, sizeof(int64_t) * toff.size()));
    SHTG_CUDA(cudaMemcpy(p->d_toff64, toff.data(), sizeof(int64_t) * toff.size(), cudaMemcpyHostToDevice));
    SHTG_TRY(alloc((void **)&p->d_tst64_0, sizeof(double2) * nent));
    LegArgs<double> a = leg_make_args<double>(p);
    dim3 grid((p->npairs + LEG_THREADS - 1) / LEG_THREADS, L + 1);
    k_tile_states64<0><<<grid, LEG_THREADS>>>(a, p->d_toff64, p->d_tst64_0, nullptr);
    SHTG_CHECK_LAUNCH("k_tile_states64");
    if (p->flags & SHTG_SPIN2) {
        SHTG_TRY(alloc((void **)&p->d_tst64_2, sizeof(double4_32a) * nent));
        k_tile_states64<2><<<grid, LEG_THREADS>>>(a, p->d_toff64, nullptr, p->d_tst64_2);
        SHTG_CHECK_LAUNCH("k_tile_states64");
    }
    SHTG_CUDA(cudaDeviceSynchronize());
    return SHTG_OK;
}

// Whether the FP64 synthesis takes the segment kernel: the plan has the
// tabulated states, and one thread per pair gives fewer CTAs than there are SMs
// (l_max < 152).  With more, every SM has several warps of FP64 work anyway.
// N_side 32, l_max 64, one map: 15.5 -> 11.4 us.
bool leg_synth_seg_fits(const Plan *p, int groups) {
    return p->d_tst64_0 && (int64_t)((p->npairs + LEG_THREADS - 1) / LEG_THREADS) * (p->lmax + 1) * groups <= p->nsm;
}
int leg_synth_seg(Plan *p, int spin, int nm, const double2 *alm, int rs, int nmaps, const double *beam, double2 *F,
                  cudaStream_t st) {
    if (spin == 2) {
        switch (nm) {
            case 1: return launch_synth_seg<1, 2>(p, alm, rs, nmaps, beam, F, st);
            case 2: return launch_synth_seg<2, 2>(p, alm, rs, nmaps, beam, F, st);
            case 3: return launch_synth_seg<3, 2>(p, alm, rs, nmaps, beam, F, st);
            default: return launch_synth_seg<4, 2>(p, alm, rs, nmaps, beam, F, st);
        }
    }
    switch (nm) {
        case 1: return launch_synth_seg<1, 0>(p, alm, rs, nmaps, beam, F, st);
        case 2: return launch_synth_seg<2, 0>(p, alm, rs, nmaps, beam, F, st);
        case 3: return launch_synth_seg<3, 0>(p, alm, rs, nmaps, beam, F, st);
        case 4: return launch_synth_seg<4, 0>(p, alm, rs, nmaps, beam, F, st);
        case 6: return launch_synth_seg<6, 0>(p, alm, rs, nmaps, beam, F, st);
        default: return launch_synth_seg<8, 0>(p, alm, rs, nmaps, beam, F, st);
    }
}

int leg_analysis_g64(Plan *p, int spin, const double2 *G, int nmaps, const double *beam, double2 *alm, int rs,
                     cudaStream_t st, int vjp) {
    if (spin == 2) return analysis_blk<ArF64, 2>(p, G, nmaps, beam, alm, rs, st, vjp);
    return analysis_blk<ArF64, 0>(p, G, nmaps, beam, alm, rs, st, vjp);
}

}  // namespace shtg
