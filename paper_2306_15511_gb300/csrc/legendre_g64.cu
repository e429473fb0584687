// Native FP64 arithmetic of the register-blocked Legendre transpose
// (legendre_blk.cuh), and the FP64 recurrence states tabulated every
// SHTG_TS64 l that it (and its double-FP32 form) restarts from: built once
// at plan creation by the same steps, so the values equal those of one
// continuous run.
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
    static constexpr bool HALVES = false;
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

int leg_analysis_g64(Plan *p, int spin, const double2 *G, int nmaps, const double *beam, double2 *alm, int rs,
                     cudaStream_t st, int vjp) {
    if (spin == 2) return analysis_blk<ArF64, 2>(p, G, nmaps, beam, alm, rs, st, vjp);
    return analysis_blk<ArF64, 0>(p, G, nmaps, beam, alm, rs, st, vjp);
}

}  // namespace shtg
