// Ring stage of the spherical-harmonic transforms: on each iso-latitude ring
// the field is f(phi_j) = sum_{m=-L..L} F(m) e^{i m (phi0 + 2 pi j / n)} with
// F(-m) = conj(F(m)) (a real field), phi0 = shift * pi / n.
//
// One CTA per ring pair.  The north and south rings of a pair have the same
// n and phi0, so one complex FFT of z = f_N + i f_S serves both.  Frequencies
// are folded modulo n (rings with n < 2L + 1 alias).  The length-n DFT is a
// Stockham autosort FFT in shared memory (natural order in and out): every
// pass loads R elements per butterfly into registers, applies the twiddles,
// does the radix-R DFT in registers and writes the R outputs to their sorted
// places (Govindaraju et al. 2008, "High performance discrete Fourier
// transforms on graphics processors"; radix 8 in FP32, 4 in FP64, with one
// radix-2 or -4 pass first where the length needs it).  The buffer is padded
// by one element per 16 so that the scattered writes of the early passes hit
// distinct banks.  Rings whose n is
// not a power of two (HEALPix polar caps) use Bluestein's chirp convolution
// with precomputed kernel spectra.  The fused variant applies N^-1 between
// the inverse and the forward transform, so the pixel map never goes to
// global memory inside an operator application.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "common.cuh"

namespace shtg {

// Radix of the passes and threads per CTA.  FP64: radix 4, M / 4 threads (1024
// with two butterflies at M = 8192).  An FP64 warp instruction takes 64 cycles
// of its scheduler's FP64 unit, so a ring's transform takes as long as its
// busiest scheduler's FP64 instructions: radix-16 butterflies (272 FP64
// instructions each, M / 16 of them, two of three twiddles computed) left a
// short ring's work on one or two warps of an SM; radix-4 ones take 28 on four
// times as many threads, spread over all four schedulers.  Fused stage of one
// map at N_side 32: 104 -> 30 us; of 12 T, Q, U maps at N_side 128, l_max 256:
// 1009 -> 584 us; synthesis of 8 maps at N_side 512, M = 4096: 1.85 -> 1.71
// ms (near the FP64 pipe).  FP64 lengths up to 256: radix 2, M / 2 threads: 8
// FP64 instructions a pass on all four schedulers (radix 4: 28 on the first one
// or two, and half as many passes): synthesis of one map at N_side 32, l_max 64,
// with its Legendre sums 30 -> 27 us.  FP32 lengths up to 1024: radix 8, 128
// threads (latency bound: one radix-16 butterfly a pass on 64 threads took
// longer); the same 12 maps at N_side 128: 80 -> 50 us.  Launches of lengths up
// to 1024 run one kernel for all their lengths with the threads of the longest.
template <typename T> __host__ __device__ constexpr int ring_lr(int logm) {   // log2 of the radix
    return sizeof(T) == 4 ? 3 : logm <= 8 ? 1 : 2;
}
template <typename T> __host__ __device__ constexpr int ring_nt(int logm) {
    return logm <= 10 ? 1 << (10 - ring_lr<T>(10))
                      : (1 << (logm - ring_lr<T>(logm))) > 1024 ? 1024 : 1 << (logm - ring_lr<T>(logm));
}
// Which passes a launch runs: radix 4 / 8 as above (FP64; FP32 lengths up to
// 1024 in the analysis and the fused stage), or FP32 radix 16 with M / 16
// threads, of one length (FIX > 0) or (64 threads) of any length up to 1024.
enum { RING_R48 = 0, RING_R16 = 1, RING_R16_ANY = 2 };
template <typename T, int MODE, int FIX> struct RingCore {
    static constexpr int kind = sizeof(T) == 8 ? RING_R48 : FIX > 0 ? RING_R16 : MODE == 0 ? RING_R16_ANY : RING_R48;
    static constexpr int nt = kind == RING_R48 ? ring_nt<T>(FIX > 0 ? FIX : 10) : kind == RING_R16 ? (1 << FIX) / 16 : 64;
    static constexpr int sm_threads = kind == RING_R16_ANY ? 512 : 1024;   // at 64 (R16_ANY: 128) registers
};

__device__ __forceinline__ int rpad(int i) { return i + (i >> 4); }

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }

// ---------------------------------------------------------------------------
// Radix-R DFTs in registers, forward (e^{-2 pi i r s / R}), natural order in
// and out.
template <typename C>
__device__ __forceinline__ void dft2(C &a, C &b) {
    const C t = a;
    a = cadd(t, b);
    b = csub(t, b);
}
template <typename C>
__device__ __forceinline__ void dft4(C &x0, C &x1, C &x2, C &x3) {
    const C t0 = cadd(x0, x2), t1 = csub(x0, x2), t2 = cadd(x1, x3);
    const C d = csub(x1, x3);
    const C t3 = C{d.y, -d.x};
    x0 = cadd(t0, t2);
    x2 = csub(t0, t2);
    x1 = cadd(t1, t3);
    x3 = csub(t1, t3);
}
template <int R, typename C> struct Dft;
template <typename C> struct Dft<2, C> {
    static __device__ __forceinline__ void run(C *v) { dft2(v[0], v[1]); }
};
template <typename C> struct Dft<4, C> {
    static __device__ __forceinline__ void run(C *v) { dft4(v[0], v[1], v[2], v[3]); }
};
// r = 4 r1 + r2, s = s1 + 2 s2: four DFTs of length 2, twiddles w_8^(r2 s1),
// two DFTs of length 4
template <typename C> struct Dft<8, C> {
    static __device__ __forceinline__ void run(C *v) {
        typedef decltype(v[0].x) T;
        const T h = T(0.70710678118654752440);
        C y[4][2];
#pragma unroll
        for (int r2 = 0; r2 < 4; ++r2) {
            y[r2][0] = v[r2];
            y[r2][1] = v[4 + r2];
            dft2(y[r2][0], y[r2][1]);
        }
        C t = y[1][1];
        y[1][1] = C{h * (t.x + t.y), h * (t.y - t.x)};      // w_8
        t = y[2][1];
        y[2][1] = C{t.y, -t.x};                             // w_8^2
        t = y[3][1];
        y[3][1] = C{h * (t.y - t.x), -(h * (t.x + t.y))};   // w_8^3
#pragma unroll
        for (int s1 = 0; s1 < 2; ++s1) {
            dft4(y[0][s1], y[1][s1], y[2][s1], y[3][s1]);
#pragma unroll
            for (int s2 = 0; s2 < 4; ++s2) v[s1 + 2 * s2] = y[s2][s1];
        }
    }
};

// Stockham FFT of length M = 2^LOGM, forward, unnormalized, natural order in
// and out, in place in shared memory (all reads of a pass finish before its
// writes).  Passes: NS = 1 with radix 2^(LOGM mod LR) where that is above one,
// then radix 2^LR with NS growing by the radix.  Butterfly j of a pass (k = j
// mod NS) takes x[j + r M / R], multiplies element r by w^r (w = e^{-2 pi i
// k / (R NS)}), does a radix-R DFT and writes output s to (j - k) R + k + s NS.
//
// Twiddles of the passes with NS > 1 come from a table rounded once from
// FP64 (ring_twiddles): FP64 holds w, w^2, w^3 (radix 2: w) at k, NS + k, 2 NS + k; FP32
// holds w and w^4 and forms the others as products (at most three extra
// roundings).  A warp's consecutive k read consecutive entries.
//
// Padded addresses: rpad(i) = i + i / 16.  Loads: rpad(j + r NB) is rpad(j) +
// r (NB + NB / 16) where 16 divides NB = M / R.  Stores to o = d + r NS, d =
// (j - k) R + k: NS >= 16: rpad(d) + r (NS + NS / 16); NS < 16 (NS divides 16,
// k < NS): d + (d - k) / 16 + r NS + (r NS) / 16.
template <int R, int LOGM, int NS, int NT, typename C>
__device__ __forceinline__ void fft_pass(C *buf, const C *__restrict__ tw) {
    constexpr int M = 1 << LOGM, NB = M / R, BPT = (NB + NT - 1) / NT;
    C v[BPT][R];
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        const int j = threadIdx.x + b * NT;
        if (NB % NT == 0 || j < NB) {
#pragma unroll
            for (int r = 0; r < R; ++r)
                v[b][r] = NB % 16 == 0 ? buf[rpad(j) + r * (NB + NB / 16)] : buf[rpad(j + r * NB)];
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        const int j = threadIdx.x + b * NT;
        if (NB % NT == 0 || j < NB) {
            const int k = j & (NS - 1);
            if constexpr (NS > 1 && R == 2) v[b][1] = cmul(v[b][1], tw[k]);
            if constexpr (NS > 1 && R == 4) {
                v[b][1] = cmul(v[b][1], tw[k]);
                v[b][2] = cmul(v[b][2], tw[NS + k]);
                v[b][3] = cmul(v[b][3], tw[2 * NS + k]);
            }
            if constexpr (NS > 1 && R == 8) {
                const C w1 = tw[k], w4 = tw[NS + k];
                const C w2 = cmul(w1, w1), w3 = cmul(w2, w1);
                v[b][1] = cmul(v[b][1], w1);
                v[b][2] = cmul(v[b][2], w2);
                v[b][3] = cmul(v[b][3], w3);
                v[b][4] = cmul(v[b][4], w4);
                v[b][5] = cmul(v[b][5], cmul(w4, w1));
                v[b][6] = cmul(v[b][6], cmul(w4, w2));
                v[b][7] = cmul(v[b][7], cmul(w4, w3));
            }
            Dft<R, C>::run(v[b]);
            const int d = (j - k) * R + k;
            const int bo = NS >= 16 ? d + (d >> 4) : d + ((d - k) >> 4);
#pragma unroll
            for (int r = 0; r < R; ++r) buf[bo + (NS >= 16 ? r * (NS + NS / 16) : r * NS + (r * NS) / 16)] = v[b][r];
        }
    }
    __syncthreads();
}
// table entries of the passes of one length before the pass with this NS
template <typename T> __host__ __device__ constexpr int ring_tw_off(int logm, int ns) {
    const int LR = ring_lr<T>(logm), PER = sizeof(T) == 8 ? (1 << LR) - 1 : 2;
    int o = 0;
    for (int q = 1 << (logm % LR); q < ns; q <<= LR)
        if (q > 1) o += PER * q;
    return o;
}
template <typename T> __host__ __device__ constexpr int ring_tw_len(int logm) {
    return ring_tw_off<T>(logm, 1 << logm);
}
template <int LOGM, int NS, int NT, typename C>
__device__ __forceinline__ void fft_passes(C *buf, const C *__restrict__ tw) {
    typedef decltype(buf[0].x + buf[0].x) T;
    constexpr int LR = ring_lr<T>(LOGM);
    if constexpr (NS < (1 << LOGM)) {
        fft_pass<(1 << LR), LOGM, NS, NT>(buf, tw + ring_tw_off<T>(LOGM, NS));
        fft_passes<LOGM, (NS << LR), NT>(buf, tw);
    }
}
template <int LOGM, int NT, typename C>
__device__ __forceinline__ void fft_fixed(C *buf, const C *__restrict__ tw) {
    typedef decltype(buf[0].x + buf[0].x) T;
    constexpr int R0 = 1 << (LOGM % ring_lr<T>(LOGM));
    if constexpr (R0 > 1) fft_pass<R0, LOGM, 1, NT>(buf, tw);
    fft_passes<LOGM, R0, NT>(buf, tw);
}
// One of the lengths of a launch that holds several (FIX 0), as a function
// of its own: inlined side by side, the ten lengths' addresses are all kept
// in registers across the calls and spill (1.7 KB a thread).  The buffer is
// passed as its offset in the dynamic shared memory (a pointer would lose
// its address space).
template <int LOGM, int NT, typename C>
__device__ __noinline__ void fft_small(const int buf_off, const C *__restrict__ tw) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    fft_fixed<LOGM, NT>(reinterpret_cast<C *>(s_raw) + buf_off, tw);
}
// any length up to 1024 (FIX 0), or 2^FIX
template <int FIX, int NT, typename C>
__device__ __forceinline__ void fft_run(C *buf, const int buf_off, const int logM, const C *__restrict__ tw) {
    if constexpr (FIX > 0) {
        fft_fixed<FIX, NT>(buf, tw);
    } else {
        switch (logM) {
            case 1: fft_small<1, NT>(buf_off, tw); break;
            case 2: fft_small<2, NT>(buf_off, tw); break;
            case 3: fft_small<3, NT>(buf_off, tw); break;
            case 4: fft_small<4, NT>(buf_off, tw); break;
            case 5: fft_small<5, NT>(buf_off, tw); break;
            case 6: fft_small<6, NT>(buf_off, tw); break;
            case 7: fft_small<7, NT>(buf_off, tw); break;
            case 8: fft_small<8, NT>(buf_off, tw); break;
            case 9: fft_small<9, NT>(buf_off, tw); break;
            case 10: fft_small<10, NT>(buf_off, tw); break;
            default: break;   // length 1
        }
    }
}

// ---------------------------------------------------------------------------
// FP32 radix-16 passes (M / 16 threads): the long rings, where they move the
// least shared memory per point (radix 8 with M / 8 threads was 3 % slower on
// the whole transform of 8 Q/U maps at N_side 1024), and the synthesis of the
// short ones, so that FP32 maps (and what is summed over them, such as the
// log-posterior's value) keep their rounding.
// butterflies per thread of the first radix-R pass of a 64-thread launch (M <= 1024;
// a radix-8 pass goes first at M = 8, 128 only)
__host__ __device__ constexpr int ring_first_bpt(int R) { return R == 8 ? 1 : 4; }
// v * e^{-2 pi i k / 16}; k is a compile-time constant after unrolling, so the
// switch folds away
template <typename C>
__device__ __forceinline__ C rot16(const C v, const int k) {
    typedef decltype(v.x) T;
    const T c1 = T(0.92387953251128675613), s1 = T(0.38268343236508977173), h = T(0.70710678118654752440);
    T c, s;   // cos, sin of k pi / 8
    switch (k & 15) {
        case 0: return v;
        case 4: return C{v.y, -v.x};
        case 8: return C{-v.x, -v.y};
        case 12: return C{-v.y, v.x};
        case 1: c = c1; s = s1; break;
        case 2: c = h; s = h; break;
        case 3: c = s1; s = c1; break;
        case 5: c = -s1; s = c1; break;
        case 6: c = -h; s = h; break;
        case 7: c = -c1; s = s1; break;
        case 9: c = -c1; s = -s1; break;
        case 10: c = -h; s = -h; break;
        case 11: c = -s1; s = -c1; break;
        case 13: c = s1; s = -c1; break;
        case 14: c = h; s = -h; break;
        default: c = c1; s = -s1; break;   // 15
    }
    return C{v.x * c + v.y * s, v.y * c - v.x * s};
}

template <typename C> struct Dft8s {   // N1 = 2, N2 = 4
    static __device__ __forceinline__ void run(C *v) {
        C y[4][2];
#pragma unroll
        for (int r2 = 0; r2 < 4; ++r2) {
            y[r2][0] = v[r2];
            y[r2][1] = v[4 + r2];
            dft2(y[r2][0], y[r2][1]);
            y[r2][1] = rot16(y[r2][1], 2 * r2);   // w_8^{r2} = w_16^{2 r2}
        }
#pragma unroll
        for (int s1 = 0; s1 < 2; ++s1) {
            dft4(y[0][s1], y[1][s1], y[2][s1], y[3][s1]);
#pragma unroll
            for (int s2 = 0; s2 < 4; ++s2) v[s1 + 2 * s2] = y[s2][s1];
        }
    }
};
template <typename C> struct Dft16s {   // N1 = N2 = 4
    static __device__ __forceinline__ void run(C *v) {
        C y[4][4];
#pragma unroll
        for (int r2 = 0; r2 < 4; ++r2) {
            y[r2][0] = v[r2];
            y[r2][1] = v[4 + r2];
            y[r2][2] = v[8 + r2];
            y[r2][3] = v[12 + r2];
            dft4(y[r2][0], y[r2][1], y[r2][2], y[r2][3]);
#pragma unroll
            for (int s1 = 1; s1 < 4; ++s1) y[r2][s1] = rot16(y[r2][s1], r2 * s1);
        }
#pragma unroll
        for (int s1 = 0; s1 < 4; ++s1) {
            dft4(y[0][s1], y[1][s1], y[2][s1], y[3][s1]);
#pragma unroll
            for (int s2 = 0; s2 < 4; ++s2) v[s1 + 4 * s2] = y[s2][s1];
        }
    }
};

template <int R, typename C> struct DftS;
template <typename C> struct DftS<2, C> : Dft<2, C> {};
template <typename C> struct DftS<4, C> : Dft<4, C> {};
template <typename C> struct DftS<8, C> : Dft8s<C> {};
template <typename C> struct DftS<16, C> : Dft16s<C> {};

// Twiddles from the two-level table in shared memory: e^{-2 pi i t / Mmax}
template <typename C> struct TwTab {
    const C *lo, *hi;
    int blo, logmax;
    __device__ __forceinline__ C at(int t) const {
        return cmul(hi[t >> blo], lo[t & ((1 << blo) - 1)]);
    }
};

// One Stockham pass of radix R over a length-M transform whose sub-transforms
// of length Ns are done: butterfly j (k = j mod Ns) takes x[j + r M/R],
// multiplies element r by w^{r k} (w = e^{-+2 pi i / (Ns R)}), does a radix-R
// DFT and writes output s to (j - k) R + k + s Ns.  Each thread handles BPT
// butterflies; all reads finish (barrier) before any write, so the pass runs
// in place.  With post != null the outputs are multiplied by post[index];
// with cj they are conjugated (after the multiplication).
template <int R, int BPT, int NT, bool TW, typename C>
__device__ __forceinline__ void spass(C *buf, const int M, const int Ns, const TwTab<C> &tw,
                                      const C *__restrict__ post, const bool cj) {
    const int nb = M / R;
    C v[BPT][R];
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        const int j = threadIdx.x + b * NT;
        if (j < nb) {
#pragma unroll
            for (int r = 0; r < R; ++r) v[b][r] = buf[rpad(j + r * nb)];
        }
    }
    __syncthreads();
    int lsr = 0;   // log2(Ns R)
    while ((1 << lsr) < Ns * R) ++lsr;
    const int lshift = tw.logmax - lsr;
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        const int j = threadIdx.x + b * NT;
        if (j < nb) {
            const int k = j & (Ns - 1);
            if (TW && Ns > 1) {
                // w^r = w^{4a} w^b (r = 4a + b): table values at r = 1, 2, 4, 8,
                // products elsewhere (at most three roundings per twiddle)
                const int t = k << lshift;
                C wb[4], wa[4];
                wb[1] = tw.at(t);
                if (R >= 4) {
                    wb[2] = tw.at(2 * t);
                    wb[3] = cmul(wb[2], wb[1]);
                }
                if (R >= 8) wa[1] = tw.at(4 * t);
                if (R >= 16) {
                    wa[2] = tw.at(8 * t);
                    wa[3] = cmul(wa[2], wa[1]);
                }
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    const int ra = r >> 2, rb = r & 3;
                    const C w = ra == 0 ? wb[rb] : (rb == 0 ? wa[ra] : cmul(wa[ra], wb[rb]));
                    v[b][r] = cmul(v[b][r], w);
                }
            }
            DftS<R, C>::run(v[b]);
            const int d = (j - k) * R + k;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int o = d + r * Ns;
                C y = post ? cmul(v[b][r], post[o]) : v[b][r];
                if (cj) y.y = -y.y;
                buf[rpad(o)] = y;
            }
        }
    }
    __syncthreads();
}

// Length-2^logM forward DFT (e^{-2 pi i jk/M}, unnormalized) of buf in
// place, natural order in and out; the last pass multiplies by post (if not
// null) and conjugates when cj is set.  The inverse transform is
// conj(DFT(conj x)): callers conjugate on the way in and out.  Passes: one
// radix-8, -4 or -2 pass when log2 M is not a multiple of four, then radix
// 16.  One call site, inlined once.
template <int NT, typename C>
__device__ __forceinline__ void fft_stockham(C *buf, const int logM, const TwTab<C> tw,
                                          const C *__restrict__ post, const bool cj) {
    static_assert(NT == 64, "ring_first_bpt");
    // M <= 16 NT (the plan checks it).  A radix-2, -4 or -8 pass (when log2 M is
    // not a multiple of four) goes first, where it needs no twiddles (Ns = 1),
    // with ring_first_bpt butterflies per thread (M / R <= 256 for R = 2 and 4, 16
    // for R = 8); the radix-16 passes follow with at most one butterfly per
    // thread, the last of them applying post / cj.
    const int M = 1 << logM;
    int Ns = 1, rem = logM;
    const int r0 = logM & 3;
    if (r0 != 0) {
        const bool last = rem == r0;
        if (r0 == 3) spass<8, ring_first_bpt(8), NT, false>(buf, M, 1, tw, last ? post : nullptr, last && cj);
        else if (r0 == 2) spass<4, ring_first_bpt(4), NT, false>(buf, M, 1, tw, last ? post : nullptr, last && cj);
        else spass<2, ring_first_bpt(2), NT, false>(buf, M, 1, tw, last ? post : nullptr, last && cj);
        Ns = 1 << r0;
        rem -= r0;
    }
    while (rem > 0) {
        const bool last = rem == 4;
        spass<16, 1, NT, true>(buf, M, Ns, tw, last ? post : nullptr, last && cj);
        Ns <<= 4;
        rem -= 4;
    }
}

// ---------------------------------------------------------------------------
// FP32 fixed-length Stockham FFT (M = 2^LOGM known at compile time), used by
// the launches of the long rings.  Same passes as fft_stockham (one radix-2, -4 or
// -8 pass when log2 M is not a multiple of four, then radix-16 passes), but
// every shared-memory address of a pass is a per-thread base plus a
// compile-time offset, and the twiddles of each radix-16 pass come from a
// precomputed table (twf_*): entries k and NS + k of pass p hold w^1 and w^4
// for w = e^{-2 pi i k / (16 NS)}, k < NS = 2^(LOGM mod 4) 16^p (passes with
// NS = 1 need none), rounded once from FP64; the other powers are products
// of those.  A warp's 32 consecutive k read 32 consecutive entries.
//
// Padded addresses: rpad(i) = i + i / 16.  For a pass with NB = M / R
// butterflies (NB a multiple of 16), butterfly j reads j + r NB, whose padded
// address is rpad(j) + r (NB + NB / 16).  Radix-16 outputs go to
// o = d + r NS with d = 16 (j - k) + k: for NS >= 16, rpad(o) = d + (j - k) +
// k / 16 + r (NS + NS / 16); for NS = 1, 2, 4, 8 (NS divides 16, k < NS),
// rpad(o) = d + (j - k) + r NS + (r NS) / 16.  The first pass (NS = 1)
// writes o = R j + r at rpad(R j) + r.
__host__ __device__ constexpr int twf_pass_ns(int logm, int p) { return (1 << (logm & 3)) << (4 * p); }
__host__ __device__ constexpr int twf_pass_off(int logm, int p) {
    int o = 0;
    for (int q = 0; q < p; ++q)
        if (twf_pass_ns(logm, q) > 1) o += 2 * twf_pass_ns(logm, q);
    return o;
}

// Radix-16 DFT in place with its outputs left transposed: X[s] ends at
// v[4 (s mod 4) + s / 4] (the same 4 x 4 decomposition as Dft16s: DFT-4 down
// the columns r2, twiddles w16^(r2 s1), DFT-4 along the rows s1), so no second
// array of 16 values is live; callers read the outputs through the
// compile-time permutation dft16_at.
__host__ __device__ constexpr int dft16_at(int s) { return 4 * (s & 3) + (s >> 2); }
template <typename C>
__device__ __forceinline__ void dft16_tp(C *v) {
#pragma unroll
    for (int r2 = 0; r2 < 4; ++r2) {
        dft4(v[r2], v[r2 + 4], v[r2 + 8], v[r2 + 12]);
        v[r2 + 4] = rot16(v[r2 + 4], r2);
        v[r2 + 8] = rot16(v[r2 + 8], 2 * r2);
        v[r2 + 12] = rot16(v[r2 + 12], 3 * r2);
    }
#pragma unroll
    for (int s1 = 0; s1 < 4; ++s1) dft4(v[4 * s1], v[4 * s1 + 1], v[4 * s1 + 2], v[4 * s1 + 3]);
}

__host__ __device__ constexpr int twf_len(int logm) { return twf_pass_off(logm, logm >> 2); }

template <int R, int LOGM, int NT, typename C>
__device__ __forceinline__ void fpass_first(C *buf) {
    constexpr int M = 1 << LOGM, NB = M / R, BPT = (NB + NT - 1) / NT;
    constexpr int SIN = NB + NB / 16;
    static_assert(NB % 16 == 0, "first pass needs M / R to be a multiple of 16");
    C v[BPT][R];
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        const int j = threadIdx.x + b * NT;
        if (NB % NT == 0 || j < NB) {
            const int bi = j + (j >> 4);
#pragma unroll
            for (int r = 0; r < R; ++r) v[b][r] = buf[bi + r * SIN];
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        const int j = threadIdx.x + b * NT;
        if (NB % NT == 0 || j < NB) {
            DftS<R, C>::run(v[b]);
            const int o0 = j * R;
            const int bo = o0 + (o0 >> 4);
#pragma unroll
            for (int r = 0; r < R; ++r) buf[bo + r] = v[b][r];
        }
    }
    __syncthreads();
}

template <int LOGM, int NS, int NT, typename C>
__device__ __forceinline__ void fpass16(C *buf, const C *__restrict__ twp) {
    constexpr int M = 1 << LOGM, NB = M / 16, BPT = (NB + NT - 1) / NT;
    constexpr int SIN = NB + NB / 16;
    static_assert(NB % 16 == 0, "radix-16 pass needs M / 16 to be a multiple of 16");
    C v[BPT][16];
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        const int j = threadIdx.x + b * NT;
        if (NB % NT == 0 || j < NB) {
            const int bi = j + (j >> 4);
#pragma unroll
            for (int r = 0; r < 16; ++r) v[b][r] = buf[bi + r * SIN];
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        const int j = threadIdx.x + b * NT;
        if (NB % NT == 0 || j < NB) {
            const int k = j & (NS - 1);
            if (NS > 1) {
                // w^r for r = 4a + c from the two table values w and w^4:
                // w^2, w^3 = w^2 w; w^8 = (w^4)^2, w^12 = w^8 w^4; w^(4a + c) =
                // w^(4a) w^c: at most five roundings, ten live registers
                const C w1 = twp[k], w4 = twp[NS + k];
                const C w2 = cmul(w1, w1), w3 = cmul(w2, w1);
                v[b][1] = cmul(v[b][1], w1);
                v[b][2] = cmul(v[b][2], w2);
                v[b][3] = cmul(v[b][3], w3);
                C wa = w4;
#pragma unroll
                for (int a = 1; a < 4; ++a) {
                    if (a > 1) wa = cmul(wa, w4);
                    v[b][4 * a] = cmul(v[b][4 * a], wa);
                    v[b][4 * a + 1] = cmul(v[b][4 * a + 1], cmul(wa, w1));
                    v[b][4 * a + 2] = cmul(v[b][4 * a + 2], cmul(wa, w2));
                    v[b][4 * a + 3] = cmul(v[b][4 * a + 3], cmul(wa, w3));
                }
            }
            dft16_tp(v[b]);
            const int d = 16 * (j - k) + k;
            const int bo = NS >= 16 ? d + (j - k) + (k >> 4) : d + (j - k);
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int off = NS >= 16 ? r * (NS + NS / 16) : r * NS + (r * NS) / 16;
                buf[bo + off] = v[b][dft16_at(r)];
            }
        }
    }
    __syncthreads();
}

template <int LOGM, int NT, int P, typename C>
__device__ __forceinline__ void fft16_passes(C *buf, const C *__restrict__ tw) {
    if constexpr (P < (LOGM >> 2)) {
        fpass16<LOGM, twf_pass_ns(LOGM, P), NT>(buf, tw + twf_pass_off(LOGM, P));
        fft16_passes<LOGM, NT, P + 1>(buf, tw);
    }
}

// Length-2^LOGM forward DFT of buf in place (natural order in and out).
template <int LOGM, int NT, typename C>
__device__ __forceinline__ void fft16_fixed(C *buf, const C *__restrict__ tw) {
    static_assert(LOGM >= 8, "fixed-length passes need M >= 256");
    constexpr int R0L = LOGM & 3;
    if constexpr (R0L != 0) fpass_first<(1 << R0L), LOGM, NT>(buf);
    fft16_passes<LOGM, NT, 0>(buf, tw);
}

// One transform direction in place: a DFT for power-of-two rings (bh null), a
// Bluestein convolution with kernel spectrum bh otherwise (buf then holds its
// conjugate); one FFT call site.
template <int KIND, int FIX, int NT, typename C>
__device__ __forceinline__ void transform_dir(C *buf, const int buf_off, const int logM, const C *__restrict__ tw,
                                              const TwTab<C> &tw2, const C *__restrict__ bh) {
    const int nf = bh ? 2 : 1;
    if constexpr (KIND == RING_R16_ANY) {
        for (int k = 0; k < nf; ++k)
            fft_stockham<NT>(buf, logM, tw2, k == 0 ? bh : nullptr, bh != nullptr && k == 0);
        return;
    }
    const int M = 1 << logM;
#pragma unroll 1
    for (int k = 0; k < nf; ++k) {
        if (k == 1) {
#pragma unroll 4
            for (int i = threadIdx.x; i < M; i += NT) {
                C y = cmul(buf[rpad(i)], __ldg(bh + i));
                y.y = -y.y;
                buf[rpad(i)] = y;
            }
            __syncthreads();
        }
        if constexpr (KIND == RING_R16) fft16_fixed<(FIX > 0 ? FIX : 8), NT>(buf, tw);
        else fft_run<FIX, NT>(buf, buf_off, logM, tw);
    }
}

template <typename T> struct RingArgs {
    typedef typename VT<T>::C C;
    int lmax, nring, npairs, nmaps;
    int64_t npix;
    const RingFFT *rf;
    const int64_t *ofs;
    const double *wring;
    const C *chirp, *bfwd, *binv;
    const C *rph;     // ring phase tables e^{i pi k / n}
    // twiddles: RING_R48 pass tables of every length, those of M = 2^logM at
    // tw_off[logM]; RING_R16 the pass table of M = 2^FIX; RING_R16_ANY the
    // two-level table [lo | hi]
    const C *tw;
    int tw_off[SHTG_FFT_LOGMAX + 1];
    int tw_blo, tw_nlo, logmax;   // RING_R16_ANY
    int tw_len;       // entries staged in shared memory
    int mpg;          // maps per CTA: CTA (pair, y) handles maps [y mpg, min(nmaps, (y + 1) mpg))
    C *FG;            // [map][ring][m]
    T *map;           // [map][npix]
    const T *ninv;    // fused: [comp][npix]
    int nT;           // fused: rows [0, nT) use N^-1 component 0 (T), later rows component 1 (Q, U)
    int weighted;     // analysis: multiply by the quadrature weight
    int buf_len;      // shared transform buffer length (padded) of this launch
    int chirp_len;    // shared chirp buffer length (longest Bluestein ring of the launch)
    const int *pairs; // ring pairs handled by this launch (one CTA each)
};

// The transforms of one map: [fold or load] -> one (MODE 0, 1) or two
// (MODE 2, with the N^-1 weighting between) transform directions -> [write
// map or unfold].  A direction is one FFT (power-of-two rings) or, for
// Bluestein rings, a convolution = DFT, times the kernel spectrum and
// conjugated in the last pass, DFT again: buf then holds the conjugate of the
// convolution.  The directions run in a loop, so the FFT is inlined once.
// The work of one CTA: ring pair a.pairs[pidx], maps [y mpg, (y + 1) mpg).
// Called by the plan's kernel (the block indices) and by the grouped kernel
// (one work item of a list that spans several geometries).
template <typename T, int MODE, int FIX>
__device__ __forceinline__ void ring_cta(const RingArgs<T> &a, const int pidx, const int y) {
    typedef typename VT<T>::C C;
    extern __shared__ __align__(16) unsigned char s_raw[];
    // FIX > 0: every ring of the launch has M = 2^FIX
    constexpr bool fixed = FIX > 0;
    constexpr int KIND = RingCore<T, MODE, FIX>::kind, NT = RingCore<T, MODE, FIX>::nt;
    // FP32 launches stage their twiddles in shared memory, FP64 ones read them
    // through L1 (the FP64 8192-point buffer and chirp leave no room)
    constexpr bool tw_smem = sizeof(T) == 4;
    C *s_tw = reinterpret_cast<C *>(s_raw);
    C *buf = s_tw + a.tw_len;
    C *s_chirp = buf + a.buf_len;          // this ring's chirp (Bluestein rings)
    C *scr_p = s_chirp + a.chirp_len;      // aliased fold: partial sums [north | south][NT] (generic launches)

    const int pr = a.pairs[pidx];
    const int rn = pr, rs = a.nring - 1 - pr;
    const bool single = (rn == rs);
    const RingFFT f = a.rf[rn];
    const int n = f.n, logM = f.logM, M = 1 << logM;
    const int L = a.lmax;
    const C *tw = KIND == RING_R48 ? a.tw + a.tw_off[logM] : a.tw;
    if (tw_smem) {
        const int ntw = KIND == RING_R48 ? ring_tw_len<T>(logM) : a.tw_len;
        for (int i = threadIdx.x; i < ntw; i += NT) s_tw[i] = tw[i];
        tw = s_tw;
    }
    TwTab<C> tw2;   // RING_R16_ANY
    tw2.lo = s_tw;
    tw2.hi = s_tw + a.tw_nlo;
    tw2.blo = a.tw_blo;
    tw2.logmax = a.logmax;
    // the chirp is read up to five times per element and map: stage it once
    const C *chirp = a.chirp + f.chirp_off;
    if (f.blue) {
        for (int i = threadIdx.x; i < n; i += NT) s_chirp[i] = chirp[i];
        chirp = s_chirp;
    }
    __syncthreads();
    const C *ph = a.rph + f.ph_off;   // e^{i pi k / n} (shifted rings)
    const C zero = {T(0), T(0)};
    constexpr int NDIR = MODE == 2 ? 2 : 1;

    const int q0 = y * a.mpg, q1 = min(a.nmaps, q0 + a.mpg);
    for (int q = q0; q < q1; ++q) {
        if (MODE != 1 && n >= 2 * L) {
            // ---- fold without aliasing (n >= 2 l_max): F(m) alone fills bin m
            // and conj F(m) bin n - m (phase e^{+-i pi s m / n}); with n = 2 l_max
            // both land in bin n / 2 = l_max; bins strictly between l_max and
            // n - l_max are zero.  One thread per m: independent loads.
            const C *Fn = a.FG + ((int64_t)q * a.nring + rn) * (L + 1);
            const C *Fs = a.FG + ((int64_t)q * a.nring + rs) * (L + 1);
#pragma unroll 4
            for (int mm = threadIdx.x; mm <= L; mm += NT) {
                C hn = Fn[mm], hs = single ? zero : Fs[mm];
                if (f.shift) {
                    const C phk = ph[mm];
                    hn = cmul(hn, phk);
                    hs = cmul(hs, phk);
                }
                C z1 = {hn.x - hs.y, hn.y + hs.x};      // bin mm
                C z2 = {hn.x + hs.y, -hn.y + hs.x};     // bin n - mm: conj(hn) + i conj(hs)
                if (mm == 0) z2 = zero;
                const int k2 = n - mm;
                if (2 * mm == n) {                      // bin n / 2 collects both
                    z1.x += z2.x;
                    z1.y += z2.y;
                }
                buf[rpad(mm)] = f.blue ? cmul(z1, cconj(chirp[mm])) : cconj(z1);
                if (mm > 0 && 2 * mm != n)
                    buf[rpad(k2)] = f.blue ? cmul(z2, cconj(chirp[k2])) : cconj(z2);
            }
            for (int k = L + 1 + threadIdx.x; k < n - L; k += NT) buf[rpad(k)] = zero;
        } else if (MODE != 1) {
            // ---- aliased fold (n < 2 l_max) into the length-n spectrum of
            // z = f_N + i f_S.  Per residue r: Q(r) = sum_t (-1)^{s t} F(r + t n)
            // (phi0 = s pi / n); then H(k) = e^{i pi s k / n} [Q(k) + (-1)^s
            // conj Q(n - k)] for k > 0 and H(0) = Q(0) + conj(Q(0) - F(0)).
            // Rings with n < NT / 2 split each residue's sum over S = NT / n
            // thread segments (coalesced reads, fixed summation order), so a
            // small polar ring costs no more time than a long one.
            const C *Fn = a.FG + ((int64_t)q * a.nring + rn) * (L + 1);
            const C *Fs = a.FG + ((int64_t)q * a.nring + rs) * (L + 1);
            // Q of the south ring in buf[n, 2n) (the launch's buffer holds 2n
            // for every aliased ring; Bluestein rings: M >= 2n)
            auto qsr = [&](int k) -> C & { return buf[rpad(n + k)]; };
            const int S = (!fixed && n <= NT / 2) ? NT / n : 1;   // fixed launches: n > NT / 2
            if (S > 1) {
                const int k = threadIdx.x % n, s = threadIdx.x / n;
                if (s < S) {
                    C pn = zero, ps = zero;
                    T sg = (f.shift && (s & 1)) ? T(-1) : T(1);   // (-1)^{s t}, t = s + j S
                    const bool flip = f.shift && (S & 1);
                    for (int mm = k + s * n; mm <= L; mm += S * n) {
                        const C vn = Fn[mm];
                        pn.x += sg * vn.x;
                        pn.y += sg * vn.y;
                        if (!single) {
                            const C vs = Fs[mm];
                            ps.x += sg * vs.x;
                            ps.y += sg * vs.y;
                        }
                        if (flip) sg = -sg;
                    }
                    scr_p[s * n + k] = pn;
                    scr_p[NT + s * n + k] = ps;
                }
                __syncthreads();
                for (int kk = threadIdx.x; kk < n; kk += NT) {
                    C qn = zero, qq = zero;
                    for (int s2 = 0; s2 < S; ++s2) {
                        qn = cadd(qn, scr_p[s2 * n + kk]);
                        qq = cadd(qq, scr_p[NT + s2 * n + kk]);
                    }
                    buf[rpad(kk)] = qn;
                    qsr(kk) = qq;
                }
            } else {
                for (int k = threadIdx.x; k < n; k += NT) {
                    C qn = zero, qq = zero;
                    T sg = T(1);
                    for (int mm = k; mm <= L; mm += n) {
                        const C vn = Fn[mm];
                        qn.x += sg * vn.x;
                        qn.y += sg * vn.y;
                        if (!single) {
                            const C vs = Fs[mm];
                            qq.x += sg * vs.x;
                            qq.y += sg * vs.y;
                        }
                        if (f.shift) sg = -sg;
                    }
                    buf[rpad(k)] = qn;
                    qsr(k) = qq;
                }
            }
            __syncthreads();
            // bins k and n - k from one thread, in place over Q_N
            const T sig = f.shift ? T(-1) : T(1);
            for (int j = threadIdx.x; 2 * j <= n; j += NT) {
                const int k1 = j, k2 = j ? n - j : 0;
                const C qn1 = buf[rpad(k1)], qn2 = buf[rpad(k2)];
                const C qs1 = qsr(k1), qs2 = qsr(k2);
                C hn1, hs1, hn2, hs2;
                if (j == 0) {
                    const C f0n = Fn[0], f0s = single ? zero : Fs[0];
                    hn1 = {qn1.x + (qn1.x - f0n.x), qn1.y - (qn1.y - f0n.y)};
                    hs1 = {qs1.x + (qs1.x - f0s.x), qs1.y - (qs1.y - f0s.y)};
                } else {
                    hn1 = {qn1.x + sig * qn2.x, qn1.y - sig * qn2.y};
                    hs1 = {qs1.x + sig * qs2.x, qs1.y - sig * qs2.y};
                }
                hn2 = {qn2.x + sig * qn1.x, qn2.y - sig * qn1.y};
                hs2 = {qs2.x + sig * qs1.x, qs2.y - sig * qs1.y};
                if (f.shift) {
                    // e^{i pi (n - k) / n} = -conj e^{i pi k / n}
                    const C ph1 = ph[k1];
                    const C ph2 = {-ph1.x, ph1.y};
                    hn1 = cmul(hn1, ph1);
                    hs1 = cmul(hs1, ph1);
                    hn2 = cmul(hn2, ph2);
                    hs2 = cmul(hs2, ph2);
                }
                const C z1 = {hn1.x - hs1.y, hn1.y + hs1.x};
                buf[rpad(k1)] = f.blue ? cmul(z1, cconj(chirp[k1])) : cconj(z1);
                if (k2 != k1) {
                    const C z2 = {hn2.x - hs2.y, hn2.y + hs2.x};
                    buf[rpad(k2)] = f.blue ? cmul(z2, cconj(chirp[k2])) : cconj(z2);
                }
            }
            // (Bluestein rings keep Q_S in buf[n, 2n): zero the tail only after)
            if (f.blue) __syncthreads();
        } else {
            // ---- load z = w (m_N + i m_S)
            const T *mn = a.map + (int64_t)q * a.npix + a.ofs[rn];
            const T *ms = a.map + (int64_t)q * a.npix + a.ofs[rs];
            const T w = a.weighted ? T(a.wring[rn]) : T(1);
#pragma unroll 4
            for (int j = threadIdx.x; j < n; j += NT) {
                const C z = {mn[j] * w, single ? T(0) : ms[j] * w};
                buf[rpad(j)] = f.blue ? cmul(z, chirp[j]) : z;
            }
        }
        if (f.blue)
            for (int k = n + threadIdx.x; k < M; k += NT) buf[rpad(k)] = zero;
        __syncthreads();
#pragma unroll 1
        for (int dir = 0; dir < NDIR; ++dir) {
            // inverse (e^{+2 pi i jk/n}) for MODE 0 and the first direction of
            // MODE 2, forward (e^{-2 pi i jk/n}) otherwise
            const bool fwd = MODE == 1 || dir == 1;
            const C *bh = f.blue ? (fwd ? a.bfwd : a.binv) + f.bhat_off : nullptr;
            transform_dir<KIND, FIX, NT>(buf, a.tw_len, logM, tw, tw2, bh);
            if (MODE == 2 && dir == 0) {
                // ---- N^-1 weighting (each thread rewrites the elements it reads)
                const int comp = q < a.nT ? 0 : 1;
                const T *wn = a.ninv + (int64_t)comp * a.npix + a.ofs[rn];
                const T *ws = a.ninv + (int64_t)comp * a.npix + a.ofs[rs];
#pragma unroll 4
                for (int j = threadIdx.x; j < n; j += NT) {
                    C z = buf[rpad(j)];
                    if (f.blue) z = cmul(z, chirp[j]);
                    z.y = -z.y;
                    C y = {z.x * wn[j], single ? T(0) : z.y * ws[j]};
                    if (f.blue) y = cmul(y, chirp[j]);
                    buf[rpad(j)] = y;
                }
                if (f.blue)
                    for (int k = n + threadIdx.x; k < M; k += NT) buf[rpad(k)] = zero;
                __syncthreads();
            }
        }
        if (MODE == 0) {
            // ---- ring pixels: z = conj(buf) (direct) or conj(buf c) (Bluestein)
            T *mn = a.map + (int64_t)q * a.npix + a.ofs[rn];
            T *ms = a.map + (int64_t)q * a.npix + a.ofs[rs];
            for (int j = threadIdx.x; j < n; j += NT) {
                C z = buf[rpad(j)];
                if (f.blue) z = cmul(z, chirp[j]);
                z.y = -z.y;
                mn[j] = z.x;
                if (!single) ms[j] = z.y;
            }
        } else {
            // ---- unfold: G(m) = e^{-i m phi0} Y(m mod n), split north / south
            C *Gn = a.FG + ((int64_t)q * a.nring + rn) * (L + 1);
            C *Gs = a.FG + ((int64_t)q * a.nring + rs) * (L + 1);
            // G(k + t n) = (-1)^{s t} e^{-i pi s k / n} Y(k), one phase per bin
            if (n > L) {
                for (int k = threadIdx.x; k <= L; k += NT) {
                    const int k2 = k ? n - k : 0;
                    C w1 = buf[rpad(k)], w2 = buf[rpad(k2)];
                    if (f.blue) {
                        w1 = cmul(cconj(w1), chirp[k]);
                        w2 = cmul(cconj(w2), chirp[k2]);
                    }
                    C yn = {T(0.5) * (w1.x + w2.x), T(0.5) * (w1.y - w2.y)};
                    C ys = {T(0.5) * (w1.y + w2.y), T(-0.5) * (w1.x - w2.x)};
                    if (f.shift) {
                        const C phk = cconj(ph[k]);
                        yn = cmul(yn, phk);
                        ys = cmul(ys, phk);
                    }
                    Gn[k] = yn;
                    if (!single) Gs[k] = ys;
                }
            } else {
                // aliased rings: Y_N(k), Y_S(k) for bins k and n - k from one
                // thread (Y_N in place over buf, Y_S beside it), then every m
                // written once, coalesced
                auto ysr = [&](int k) -> C & { return buf[rpad(n + k)]; };
                for (int j = threadIdx.x; 2 * j <= n; j += NT) {
                    const int k1 = j, k2 = j ? n - j : 0;
                    C w1 = buf[rpad(k1)], w2 = buf[rpad(k2)];
                    if (f.blue) {
                        w1 = cmul(cconj(w1), chirp[k1]);
                        w2 = cmul(cconj(w2), chirp[k2]);
                    }
                    C yn1 = {T(0.5) * (w1.x + w2.x), T(0.5) * (w1.y - w2.y)};
                    C ys1 = {T(0.5) * (w1.y + w2.y), T(-0.5) * (w1.x - w2.x)};
                    C yn2 = {yn1.x, -yn1.y};
                    C ys2 = {ys1.x, -ys1.y};
                    if (f.shift) {
                        // e^{-i pi (n - k) / n} = -conj e^{-i pi k / n}
                        const C ph1 = cconj(ph[k1]);
                        const C ph2 = {-ph1.x, ph1.y};
                        yn1 = cmul(yn1, ph1);
                        ys1 = cmul(ys1, ph1);
                        yn2 = cmul(yn2, ph2);
                        ys2 = cmul(ys2, ph2);
                    }
                    buf[rpad(k1)] = yn1;
                    ysr(k1) = ys1;
                    if (k2 != k1) {
                        buf[rpad(k2)] = yn2;
                        ysr(k2) = ys2;
                    }
                }
                __syncthreads();
                int k = threadIdx.x % n, t = threadIdx.x / n;
                const int dk = NT % n, dt = NT / n;
                for (int mm = threadIdx.x; mm <= L; mm += NT) {
                    C yn = buf[rpad(k)], ys = ysr(k);
                    if (f.shift && (t & 1)) {
                        yn = {-yn.x, -yn.y};
                        ys = {-ys.x, -ys.y};
                    }
                    Gn[mm] = yn;
                    if (!single) Gs[mm] = ys;
                    k += dk;
                    t += dt;
                    if (k >= n) {
                        k -= n;
                        t += 1;
                    }
                }
            }
        }
        __syncthreads();
    }
}

template <typename T, int MODE, int FIX>
__global__ void __launch_bounds__((RingCore<T, MODE, FIX>::nt), (RingCore<T, MODE, FIX>::sm_threads / RingCore<T, MODE, FIX>::nt))
    k_ring(const RingArgs<T> a) {
    ring_cta<T, MODE, FIX>(a, blockIdx.x, blockIdx.y);
}

// Grouped launch (chains of several geometries): one launch per
// transform-length class (the template's FIX) over the launch buckets
// of that class of every plan; entry e is one (plan, bucket) with its own
// arguments, flat CTA i belongs to the entry with first[e] <= i <
// first[e + 1] and runs ring pair i' % count[e], map group i' / count[e]
// (i' = i - first[e]).  Entries whose plan group's device flag is 0 are
// skipped.
#define SHTG_RING_ENTRIES (2 * SHTG_MAX_GROUPS)
template <typename T> struct RingGroups {
    int ne;
    int first[SHTG_RING_ENTRIES + 1];
    int count[SHTG_RING_ENTRIES];
    const int *active[SHTG_RING_ENTRIES];   // the entry's plan group flag (null: always active)
    RingArgs<T> a[SHTG_RING_ENTRIES];
};

template <typename T, int MODE, int FIX>
__global__ void __launch_bounds__((RingCore<T, MODE, FIX>::nt), (RingCore<T, MODE, FIX>::sm_threads / RingCore<T, MODE, FIX>::nt))
    k_ring_grp(const __grid_constant__ RingGroups<T> G) {
    const int i = blockIdx.x;
    int e = 0;
    while (e + 1 < G.ne && i >= G.first[e + 1]) ++e;
    if (G.active[e] && *G.active[e] == 0) return;
    const int li = i - G.first[e];
    ring_cta<T, MODE, FIX>(G.a[e], li % G.count[e], li / G.count[e]);
}

template <typename T> static RingArgs<T> ring_args(Plan *p);
template <> RingArgs<float> ring_args<float>(Plan *p) {
    RingArgs<float> a{};
    a.chirp = p->d_chirp32;
    a.rph = p->d_rph32;
    a.bfwd = p->d_bfwd32;
    a.binv = p->d_binv32;
    return a;
}
template <> RingArgs<double> ring_args<double>(Plan *p) {
    RingArgs<double> a{};
    a.chirp = p->d_chirp64;
    a.rph = p->d_rph64;
    a.bfwd = p->d_bfwd64;
    a.binv = p->d_binv64;
    return a;
}

template <typename T, typename C>
static void ring_twiddles_t(int logmax, std::vector<C> &t, int *off) {
    const double PI = 3.14159265358979323846;
    for (int lg = 0; lg <= logmax; ++lg) {
        const int LR = ring_lr<T>(lg);
        off[lg] = (int)t.size();
        for (int ns = 1 << (lg % LR); ns < (1 << lg); ns <<= LR) {
            if (ns == 1) continue;
            for (int r = 1; r < (1 << LR); ++r) {
                if (sizeof(T) == 4 && r != 1 && r != 4) continue;
                for (int k = 0; k < ns; ++k) {
                    const double ang = -2.0 * PI * (double)((int64_t)r * k) / ((double)(1 << LR) * ns);
                    t.push_back(C{T(cos(ang)), T(sin(ang))});
                }
            }
        }
    }
}
void ring_twiddles(std::vector<double2> &t64, int *off64, std::vector<float2> &t32, int *off32) {
    ring_twiddles_t<double>(SHTG_FFT_LOGMAX, t64, off64);
    ring_twiddles_t<float>(10, t32, off32);
}

template <typename T> static const typename VT<T>::C *ring_tab(Plan *p);
template <> const float2 *ring_tab<float>(Plan *p) { return p->d_twr32; }
template <> const double2 *ring_tab<double>(Plan *p) { return p->d_twr64; }

// launch arguments and shared memory of one bucket of plan p.  Buckets above
// 1024 hold rings of one transform length M = 2^FIX (FIX = g.fix: 2^logm, or
// 2^(logm - 1) for aliased direct rings, whose buffer still holds 2^logm:
// checked at plan creation).
template <typename T, int MODE, int FIX>
static void ring_bucket_args(Plan *p, const Plan::RingLaunch &g, RingArgs<T> &a, size_t &smem) {
    typedef typename VT<T>::C C;
    typedef RingCore<T, MODE, FIX> Core;
    a.lmax = p->lmax;
    a.nring = p->nring;
    a.npairs = p->npairs;
    a.npix = p->npix;
    a.rf = p->d_rfft;
    a.ofs = p->d_ofs;
    a.wring = p->d_wring;
    a.logmax = p->fft_logmax;
    a.tw_blo = p->tw_blo;
    a.tw_nlo = p->tw_nlo;
    const int M = 1 << g.logm;
    a.buf_len = M + M / 16;
    a.chirp_len = g.chirp;
    a.tw_len = 0;
    if constexpr (Core::kind == RING_R48) {
        a.tw = ring_tab<T>(p);
        for (int lg = 0; lg <= SHTG_FFT_LOGMAX; ++lg)
            a.tw_off[lg] = sizeof(T) == 8 ? p->twr_off64[lg] : p->twr_off32[lg];
        if (sizeof(T) == 4)   // room for the longest table of the launch
            for (int lg = 0; lg <= 10; ++lg) a.tw_len = std::max(a.tw_len, ring_tw_len<T>(lg));
    } else if constexpr (Core::kind == RING_R16) {
        a.tw = p->d_twf32 + p->twf_off[FIX];
        a.tw_len = twf_len(FIX);
    } else {
        a.tw = p->d_tw32;
        a.tw_len = p->tw_nlo + p->tw_nhi;
    }
    // shared memory: twiddles, buffer, chirp, and the aliased fold's partial
    // sums (FIX = 0 only: the other launches' rings have n > NT / 2, so they
    // never split a residue's sum)
    smem = sizeof(C) * ((size_t)a.tw_len + a.buf_len + a.chirp_len + ((g.alias && FIX == 0) ? 2 * Core::nt : 0));
    a.pairs = p->d_ring_groups + g.off;
}

template <typename T, int MODE, int FIX>
static int launch_ring_fix(Plan *p, const Plan::RingLaunch &g, RingArgs<T> a, cudaStream_t st) {
    typedef RingCore<T, MODE, FIX> Core;
    size_t smem = 0;
    ring_bucket_args<T, MODE, FIX>(p, g, a, smem);
    const int ctas = g.count;
    auto kern = k_ring<T, MODE, FIX>;
    if (smem > 48 * 1024) SHTG_CUDA(allow_max_smem(kern));
    // The maps of a ring pair are split over grid.y when the pairs alone give
    // fewer than four waves of resident CTAs (a CTA still handles at least
    // two maps, so its chirp and twiddle staging stay amortized)
    const int per = std::max(1, std::min(Core::sm_threads / Core::nt, smem ? (int)((227 * 1024) / (smem + 1024)) : 32));
    const int want = 4 * p->nsm * per;
    int groups = (want + ctas - 1) / ctas;
    groups = std::max(1, std::min(groups, (a.nmaps + 1) / 2));
    a.mpg = (a.nmaps + groups - 1) / groups;
    groups = (a.nmaps + a.mpg - 1) / a.mpg;
    kern<<<dim3(ctas, groups), Core::nt, smem, st>>>(a);
    return SHTG_OK;
}

template <typename T, int MODE>
static int launch_ring(Plan *p, RingArgs<T> a, cudaStream_t st) {
    // one launch per length bucket, each with the thread count and shared
    // memory of its longest transform.  The buckets touch disjoint ring
    // pairs, so all but the first run on the plan's side streams, forked from
    // and joined back into st with events (parallel branches when st is
    // being captured into a graph): the short single-wave launches of the
    // small polar rings then overlap with the long ones.
    prof_begin(p, sizeof(T) == 8 ? K_RING64 : K_RING32, st);
    int nl = 0, nside = 0;
    const int nb = (int)p->ring_launch.size();
    if (nb > 1) SHTG_CUDA(cudaEventRecord(p->ring_fork, st));
    for (int gi = 0; gi < nb; ++gi) {
        const Plan::RingLaunch &g = p->ring_launch[gi];
        if (g.count == 0) continue;
        cudaStream_t ls = st;
        if (gi > 0 && nside < Plan::RING_SIDE) {
            ls = p->ring_side[nside];
            SHTG_CUDA(cudaStreamWaitEvent(ls, p->ring_fork, 0));
        }
        int rc = SHTG_OK;
        switch (g.fix) {
            case 10: rc = launch_ring_fix<T, MODE, 10>(p, g, a, ls); break;
            case 11: rc = launch_ring_fix<T, MODE, 11>(p, g, a, ls); break;
            case 12: rc = launch_ring_fix<T, MODE, 12>(p, g, a, ls); break;
            case 13: rc = launch_ring_fix<T, MODE, 13>(p, g, a, ls); break;
            default: rc = launch_ring_fix<T, MODE, 0>(p, g, a, ls); break;
        }
        if (rc != SHTG_OK) return rc;
        if (ls != st) {
            SHTG_CUDA(cudaEventRecord(p->ring_join[nside], ls));
            SHTG_CUDA(cudaStreamWaitEvent(st, p->ring_join[nside], 0));
            ++nside;
        }
        ++nl;
    }
    prof_end(p, st, nl);
    SHTG_CHECK_LAUNCH("k_ring");
    return SHTG_OK;
}

// the buckets of one transform-length class (FIX; 0: lengths up to 1024) of
// every plan as one launch; nl counts the launches made
template <typename T, int FIX>
static int ring_grp_class(int ng, Plan *const *ps, typename VT<T>::C *const *FG, const int *nmaps, const int *nT,
                          const T *const *ninv, const int *const *active, cudaStream_t st, int &nl) {
    typedef RingCore<T, 2, FIX> Core;
    RingGroups<T> G{};
    size_t smem = 0;
    int npair = 0;
    for (int g = 0; g < ng; ++g)
        for (const Plan::RingLaunch &b : ps[g]->ring_launch)
            if (b.fix == FIX && b.count > 0) {
                if (G.ne == SHTG_RING_ENTRIES) {
                    set_error("grouped ring launch: more than " + std::to_string(SHTG_RING_ENTRIES) +
                              " launch buckets of one length");
                    return SHTG_ERR_ARG;
                }
                RingArgs<T> a = ring_args<T>(ps[g]);
                size_t sm = 0;
                ring_bucket_args<T, 2, FIX>(ps[g], b, a, sm);
                a.FG = FG[g];
                a.nmaps = nmaps[g];
                a.nT = nT[g];
                a.ninv = ninv[g];
                smem = std::max(smem, sm);
                G.a[G.ne] = a;
                G.count[G.ne] = b.count;
                G.active[G.ne] = active ? active[g] : nullptr;
                G.ne += 1;
                npair += b.count;
            }
    if (G.ne == 0) return SHTG_OK;
    // maps per CTA as in the plan's launches: enough CTAs for about four
    // waves, at least two maps per CTA
    const int want = 4 * ps[0]->nsm * std::max(1, Core::sm_threads / Core::nt);
    int64_t total = 0;
    for (int e = 0; e < G.ne; ++e) {
        RingArgs<T> &a = G.a[e];
        int groups = (want + npair - 1) / npair;
        groups = std::max(1, std::min(groups, (a.nmaps + 1) / 2));
        a.mpg = (a.nmaps + groups - 1) / groups;
        groups = (a.nmaps + a.mpg - 1) / a.mpg;
        G.first[e] = (int)total;
        total += (int64_t)G.count[e] * groups;
        if (total > 0x7fffffff) {
            set_error("grouped ring launch: too many CTAs");
            return SHTG_ERR_ARG;
        }
    }
    G.first[G.ne] = (int)total;
    auto kern = k_ring_grp<T, 2, FIX>;
    if (smem > 48 * 1024) SHTG_CUDA(allow_max_smem(kern));
    kern<<<(unsigned)total, Core::nt, smem, st>>>(G);
    ++nl;
    return SHTG_OK;
}

template <typename T>
int ring_fused_grp(int ng, Plan *const *ps, typename VT<T>::C *const *FG, const int *nmaps, const int *nT,
                   const T *const *ninv, const int *const *active, cudaStream_t st) {
    if (ng < 1 || ng > SHTG_MAX_GROUPS) {
        set_error("grouped ring launch: 1 to " + std::to_string(SHTG_MAX_GROUPS) + " groups");
        return SHTG_ERR_ARG;
    }
    Plan *acct = ps[0];
    prof_begin(acct, sizeof(T) == 8 ? K_RING64 : K_RING32, st);
    int nl = 0;
    SHTG_TRY((ring_grp_class<T, 13>(ng, ps, FG, nmaps, nT, ninv, active, st, nl)));
    SHTG_TRY((ring_grp_class<T, 12>(ng, ps, FG, nmaps, nT, ninv, active, st, nl)));
    SHTG_TRY((ring_grp_class<T, 11>(ng, ps, FG, nmaps, nT, ninv, active, st, nl)));
    SHTG_TRY((ring_grp_class<T, 10>(ng, ps, FG, nmaps, nT, ninv, active, st, nl)));
    SHTG_TRY((ring_grp_class<T, 0>(ng, ps, FG, nmaps, nT, ninv, active, st, nl)));
    prof_end(acct, st, nl);
    SHTG_CHECK_LAUNCH("k_ring_grp");
    return SHTG_OK;
}
template int ring_fused_grp<float>(int, Plan *const *, float2 *const *, const int *, const int *,
                                   const float *const *, const int *const *, cudaStream_t);

template <typename T>
int ring_synth(Plan *p, const typename VT<T>::C *F, int nmaps, T *map, cudaStream_t st) {
    RingArgs<T> a = ring_args<T>(p);
    a.FG = const_cast<typename VT<T>::C *>(F);
    a.map = map;
    a.nmaps = nmaps;
    return launch_ring<T, 0>(p, a, st);
}
template <typename T>
int ring_analysis(Plan *p, const T *map, int nmaps, int weighted, typename VT<T>::C *G,
                  cudaStream_t st) {
    RingArgs<T> a = ring_args<T>(p);
    a.FG = G;
    a.map = const_cast<T *>(map);
    a.nmaps = nmaps;
    a.weighted = weighted;
    return launch_ring<T, 1>(p, a, st);
}
template <typename T>
int ring_fused(Plan *p, typename VT<T>::C *FG, int nmaps, int nT, const T *ninv,
               cudaStream_t st) {
    RingArgs<T> a = ring_args<T>(p);
    a.FG = FG;
    a.nmaps = nmaps;
    a.nT = nT;
    a.ninv = ninv;
    return launch_ring<T, 2>(p, a, st);
}

template int ring_synth<float>(Plan *, const float2 *, int, float *, cudaStream_t);
template int ring_synth<double>(Plan *, const double2 *, int, double *, cudaStream_t);
template int ring_analysis<float>(Plan *, const float *, int, int, float2 *, cudaStream_t);
template int ring_analysis<double>(Plan *, const double *, int, int, double2 *, cudaStream_t);
template int ring_fused<float>(Plan *, float2 *, int, int, const float *, cudaStream_t);
template int ring_fused<double>(Plan *, double2 *, int, int, const double *, cudaStream_t);

}  // namespace shtg
