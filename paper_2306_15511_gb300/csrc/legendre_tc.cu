// Legendre synthesis on the 5th-generation tensor cores (tcgen05).
//
// F_r(m) = sum_l lambda_lm(theta_r) a_lm is, for one m and a block of 128
// ring pairs, the product of a [pair x l] matrix (the recurrence values,
// generated on the fly) with an [l x column] matrix (the alm of all maps),
// split by the parity of l - m into the even / odd sums E, O (App. A:
// lambda_lm(pi - theta) = (-1)^(l+m) lambda_lm(theta)), F_N = E + O,
// F_S = E - O.  Spin 2 uses the two Wigner recurrences y+, y- with
// lw = y+ + y-, lx = y+ - y- as two A matrices and the (E, B) -> (Q, U)
// sign pattern folded into the B matrices.
//
// Precision: every thread runs the FP32 recurrence of its ring pair exactly
// as the FP32 CUDA-core kernels do (same FP64 start states), and each value
// x is split into bf16 x_hi + x_lo (x_lo = bf16(x - x_hi)); the alm are split
// the same way.  Three products hi*hi + lo*hi + hi*lo are accumulated in
// FP32 in tensor memory, which keeps ~16 of the 24 mantissa bits of every
// product (relative error ~2^-17 per term) at bf16 tensor-core rates.
//
// Two kernels.  k_tc_records builds, once per m and chunk of 32 l (16 per
// parity class, one MMA K of 16 each), a record in global memory: the B tiles
// (the alm of up to 8 or 16 maps, times the beam, as bf16 hi / lo in the
// layout the MMA reads) and the recurrence coefficients.  k_leg_synth_tc, one
// CTA per m and 128 ring pairs, then loops over the chunks: the record arrives
// by a bulk copy issued one chunk ahead, the 128 threads generate the A tiles
// (bf16 hi / lo) in tensor memory, lane = ring pair, and one thread issues the
// tcgen05.mma of the chunk and commits them to an mbarrier.  While
// the tensor core works on one CTA's chunk, the other three on the SM
// generate.  Every TC_FLUSH chunks the accumulators move from tensor memory to
// FP32 sums in shared memory; the F_N / F_S epilogue reads those.
//
// What bounds it: the generation, 13.7 instructions per (l, ring pair) at spin
// 2 (coefficients 1.5, recurrence 3 packed fma.f32x2 on the (y+, y-) pair, lw
// and lx 2, bf16 split 5, the rest stores, waits and the epilogue), issued at
// 44 % of the issue rate: the waits for the chunk's MMAs and the barrier take
// the rest with four warps per scheduler.  Measured (N_side 512, l_max 1024, 8
// Q/U maps): every CTA of an m building the same B tiles between barriers, 28
// instructions, A tiles in shared memory: 657 us; records and packed
// operations, 504 us + 43 us for the records, the shared-memory pipe 67 % busy
// (A tiles written once and read by two MMAs); A tiles in tensor memory, 451 us
// + 43.  N_side 1024, l_max 2048, 8 Q/U maps, with the ring stage: 5.42 -> 4.2
// ms.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdlib>

#include "legendre_kernels.cuh"

namespace shtg {
namespace {

constexpr int TC_M = 128;        // ring pairs per CTA = MMA M = threads
constexpr int TC_ATILE = 4096;   // one A tile: 128 rows x 16 bf16 (K-major core matrices)
constexpr uint32_t TC_WAIT_LIMIT = 1u << 22;   // bounded mbarrier polling

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor, no swizzle: start address, LBO = byte
// stride between core matrices adjacent in K, SBO = byte stride between
// core matrices adjacent in M (or N); version 1 at bit 46.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor of kind::f16 with bf16 A and B (both K-major) and an
// FP32 accumulator: D format bit 4, A / B format 1 (bf16) at bits 7 / 10,
// N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t da, uint64_t db, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// Every statement below that orders memory (waits, fences, commits, the MMAs and
// the tensor-memory accesses) clobbers "memory": the compiler then keeps plain
// loads and stores of shared memory on their side of it.  A tcgen05.ld and its
// wait are one statement, since the registers hold nothing before the wait.

// Wait (bounded) for the completion of the mbarrier phase with the given
// parity; false if the limit ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
    uint32_t done = 0;
    for (uint32_t it = 0; it < TC_WAIT_LIMIT && !done; ++it) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
    }
    return done != 0;
}

// 32 consecutive TMEM columns of this warp's 32 lanes: thread = lane
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
          "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
          "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// D += A B with A in tensor memory (lane = row, two bf16 of K per column) and
// B in shared memory
__device__ __forceinline__ void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t db, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(db), "r"(idesc), "r"(accumulate)
        : "memory");
}

// 4 consecutive TMEM columns of this warp's 32 lanes <- 4 registers per thread
__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(a), "r"(b), "r"(c),
                 "r"(d)
                 : "memory");
}

// Packed pairs of FP32 operations (one issue slot for two; the same rounding
// as the scalar ones)
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n\t.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
        "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float2 fmul2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "mul.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}

// (a, b) -> bf16x2 hi and lo words, element a in the low half
__device__ __forceinline__ void split2(float a, float b, uint32_t &hi, uint32_t &lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    // the lo parts a - hi, b - hi (exact) in one packed operation
    const float2 hf = make_float2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
    const float2 d = ffma2(hf, make_float2(-1.f, -1.f), make_float2(a, b));
    const __nv_bfloat162 l = __floats2bfloat162_rn(d.x, d.y);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}

// 8 values -> one 16-byte core-matrix row of hi and one of lo
__device__ __forceinline__ void store_row8(unsigned char *hi_row, unsigned char *lo_row, const float (&x)[8]) {
    uint4 h, l;
    split2(x[0], x[1], h.x, l.x);
    split2(x[2], x[3], h.y, l.y);
    split2(x[4], x[5], h.z, l.z);
    split2(x[6], x[7], h.w, l.w);
    *reinterpret_cast<uint4 *>(hi_row) = h;
    *reinterpret_cast<uint4 *>(lo_row) = l;
}

// Tile configuration of NMT maps.  NCOL: B rows of one product block (spin 0:
// re, im per map; spin 2: Q re, Q im, U re, U im per map); a B tile holds
// NCOL hi rows then NCOL lo rows, 16 K (l of one parity class) each.  A record
// is the B tiles of one chunk of 32 l followed by its coefficients.
constexpr int TC_NREC = 2;    // record stages of the synthesis (chunk c uses stage c % 2)
constexpr int TC_FLUSH = 4;   // chunks summed in tensor memory before they move to the FP32 sums
template <int SPIN, int NMT> struct TcCfg {
    static constexpr int NCOL = SPIN == 2 ? 4 * NMT : 2 * NMT;
    static constexpr int NA = SPIN == 2 ? 2 * NMT : NMT;      // alm rows of the maps
    static constexpr int NTA = SPIN == 2 ? 8 : 4, NTB = SPIN == 2 ? 4 : 2;
    // tensor memory: two accumulators of NCOL columns, then the A tiles of one
    // chunk (8 columns each)
    static constexpr int ACOL = 2 * NCOL;
    static constexpr int TMEM = ACOL + 8 * NTA <= 64 ? 64 : 128;
    static_assert(ACOL + 8 * NTA <= TMEM, "accumulators and A tiles fit the allocation");
    static constexpr int BTILE = 2 * NCOL * 32;
    static constexpr int COEF = NTB * BTILE;                  // offset of the coefficients in a record
    static constexpr int REC = COEF + 32 * (SPIN == 2 ? 24 : 8);
    // shared memory of the synthesis CTA: the record stages, the FP32 sums of
    // the flushed chunks [column][thread], mbarriers (one per stage, one for
    // the MMAs), the TMEM address, scratch
    static constexpr int SUMS = TC_NREC * REC;
    static constexpr int BARS = SUMS + 2 * NCOL * TC_M * 4;
    static constexpr int TMEMA = BARS + 8 * (TC_NREC + 1);
    static constexpr int RED = TMEMA + 16;
    static constexpr int BYTES = RED + 16;
    static_assert(REC % 16 == 0, "a bulk copy moves multiples of 16 bytes");
};

// Recurrence coefficients of one l as the recurrence uses them: spin 2 (alpha
// + beta, alpha - beta, -alpha, -gamma), spin 0 (a, b).
__device__ __forceinline__ float4 tc_coef(const float4 s) { return make_float4(s.y, s.z, -s.x, -s.w); }

// The recurrence state of one ring pair: spin 0 p1.x, p2.x = lambda_{l-1},
// lambda_{l-2}; spin 2 the (y+, y-) pairs.  step: the same operations and
// roundings as step0 / step2 of the CUDA-core kernels.
template <int SPIN> struct TcState {
    float2 p1, p2;
    float u;
    // spin 2: yz = (alpha + beta, alpha - beta), xx = (-alpha, -alpha), ww =
    // (-gamma, -gamma); spin 0: yz = (a, b)
    __device__ __forceinline__ void step(const float2 yz, const float2 xx, const float2 ww) {
        if (SPIN == 2) {
            const float2 t = ffma2(xx, make_float2(u, u), yz);
            const float2 n = ffma2(t, p1, fmul2(ww, p2));
            p2 = p1;
            p1 = n;
        } else {
            rstep(p1.x, p2.x, yz.x, yz.y, u);
        }
    }
    // the start values of the recurrences that start at l
    __device__ __forceinline__ void inject(const int l, const int ls, const int lsb, const float s0, const float s1,
                                           const float s2, const float s3) {
        if (l == ls) {
            p2.x = s0;
            p1.x = s1;
        }
        if (SPIN == 2 && l == lsb) {
            p2.y = s2;
            p1.y = s3;
        }
    }
    __device__ __forceinline__ float w() const { return SPIN == 2 ? p1.x + p1.y : p1.x; }   // lw (spin 0: lambda)
    __device__ __forceinline__ float x() const { return SPIN == 2 ? p1.x - p1.y : 0.f; }    // lx
};

// B tiles of one chunk from the staged alm (already times the beam).  Tile
// b: spin 0 -> class b (0 even, 1 odd); spin 2 -> b = 2 w + class with
// W columns (-E re, -E im, -B re, -B im) and X columns (B im, -B re, -E im,
// E re) per map, feeding (Q re, Q im, U re, U im).  Column c, K index k:
// hi at row c, lo at row NCOL + c (K-major core matrices, LBO = 32 NCOL).
template <int SPIN, int NMT, int ALMS>
__device__ __forceinline__ void gen_btiles(const float2 *s_alm, unsigned char *bt) {
    typedef TcCfg<SPIN, NMT> Cfg;
    constexpr int NCOL = Cfg::NCOL, NTB = Cfg::NTB;
    // item = (tile b, K group kg, column c): one 16-byte core-matrix row of
    // hi and one of lo (the 8 K values, l = off + 16 kg + 2 j, of column c),
    // consecutive threads on consecutive rows.  Column c of tile b reads one
    // component of one staged alm row: spin 0 (re, im) of map c / 2; spin 2 W
    // tiles (b < 2) -(E re, E im, B re, B im), X tiles (B im, -B re, -E im, E
    // re) of map c / 4, component c % 4.
    for (int it = threadIdx.x; it < NTB * 2 * NCOL; it += TC_M) {
        const int c = it % NCOL, kg = (it / NCOL) & 1, b = it / (2 * NCOL);
        const int off = b & 1;
        int row, ri;
        float sg;
        if (SPIN == 0) {
            row = c >> 1;
            ri = c & 1;
            sg = 1.f;
        } else {
            const int mk = c >> 2, comp = c & 3;
            if (b < 2) {
                row = 2 * mk + (comp >= 2 ? 1 : 0);
                ri = comp & 1;
                sg = -1.f;
            } else {
                row = 2 * mk + (comp < 2 ? 1 : 0);
                ri = (comp & 1) ^ 1;
                sg = (comp == 1 || comp == 2) ? -1.f : 1.f;
            }
        }
        const float *src = reinterpret_cast<const float *>(s_alm + row * ALMS + off + 16 * kg) + ri;
        float x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = sg * src[4 * j];
        unsigned char *r = bt + b * Cfg::BTILE + kg * (32 * NCOL) + c * 16;
        store_row8(r, r + NCOL * 16, x);
    }
}

// The record of the chunk of 32 l from l0 for the maps from map0 on, by the CTA's
// threads: its inputs in registers (loaded a chunk ahead where a CTA builds one
// after the other), then the coefficients and the B tiles from them
constexpr int TC_ALMS = 33;   // float2 per staged alm row (odd: rows fall in distinct banks)
template <int SPIN, int NMT> struct RecIn {
    static constexpr int N = TcCfg<SPIN, NMT>::NA * 32 / TC_M;
    float2 v[N];
    float4 c;   // threads below 32: coefficients of l0 + threadIdx.x
};
template <int SPIN, int NMT>
__device__ __forceinline__ void load_record(const LegArgs<float> &a, int m, int l0, int map0, RecIn<SPIN, NMT> &R) {
    const int L = a.lmax;
    const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2;
    const int i = threadIdx.x & 31, l = l0 + i;
    const float bm = a.beam && l <= L ? a.beam[l] : 1.f;
#pragma unroll
    for (int e = 0; e < RecIn<SPIN, NMT>::N; ++e) {
        const int k = (threadIdx.x + e * TC_M) >> 5, mk = SPIN == 2 ? k / 2 : k;
        float2 v = make_float2(0.f, 0.f);
        if (l <= L && map0 + mk < a.nmaps) {
            const int64_t row = (int64_t)(map0 + mk) * a.rs + (SPIN == 2 ? (k & 1) : 0);
            v = a.alm[row * a.nalm + base + l];
            if (m == 0) v.y = 0.f;
            v.x *= bm;
            v.y *= bm;
        }
        R.v[e] = v;
    }
    R.c = make_float4(0.f, 0.f, 0.f, 0.f);
    if (threadIdx.x < 32 && l <= L) {
        if (SPIN == 2) {
            R.c = tc_coef(a.s2c[base + l]);
        } else {
            const float2 c = a.rec[base + l];
            R.c = make_float4(c.x, c.y, 0.f, 0.f);
        }
    }
}
template <int SPIN, int NMT>
__device__ __forceinline__ void store_coefs(const RecIn<SPIN, NMT> &R, unsigned char *rec) {
    const int i = threadIdx.x;
    if (i >= 32) return;
    if (SPIN == 2) {
        // per two l, three 16-byte loads for the generation: (yz, xx) of
        // the first, (ww, ww) of both, (yz, xx) of the second
        float4 *dst = reinterpret_cast<float4 *>(rec + TcCfg<SPIN, NMT>::COEF) + 3 * (i >> 1);
        dst[2 * (i & 1)] = make_float4(R.c.x, R.c.y, R.c.z, R.c.z);
        reinterpret_cast<float2 *>(dst + 1)[i & 1] = make_float2(R.c.w, R.c.w);
    } else {
        reinterpret_cast<float2 *>(rec + TcCfg<SPIN, NMT>::COEF)[i] = make_float2(R.c.x, R.c.y);
    }
}
// B tiles straight from the registers (the words of gen_btiles): a warp holds one
// alm row, lane i the l of class i & 1 and K index i / 2, so lanes i and i ^ 2
// exchange one component and each stores the 4-byte words (two K) of the other:
// lanes with bit 1 clear re, the others im.
template <int SPIN, int NMT>
__device__ __forceinline__ void store_btiles(const RecIn<SPIN, NMT> &R, unsigned char *bt) {
    typedef TcCfg<SPIN, NMT> Cfg;
    constexpr int NCOL = Cfg::NCOL, LO = NCOL * 16;   // offset of the lo rows
    const int i = threadIdx.x & 31, im = (i >> 1) & 1;
    unsigned char *t = bt + (i & 1) * Cfg::BTILE + (i >> 4) * (32 * NCOL) + ((i >> 2) & 3) * 4;
#pragma unroll
    for (int e = 0; e < RecIn<SPIN, NMT>::N; ++e) {
        const int k = (threadIdx.x + e * TC_M) >> 5;
        const float2 v = R.v[e];
        const float o = __shfl_xor_sync(0xffffffffu, im ? v.x : v.y, 2);
        uint32_t hi, lo;
        split2(im ? o : v.x, im ? v.y : o, hi, lo);
        auto put = [&](int tile, int c, uint32_t sign) {   // class pair of tiles, column, sign of both words
            unsigned char *q = t + tile * Cfg::BTILE + c * 16;
            *reinterpret_cast<uint32_t *>(q) = hi ^ sign;
            *reinterpret_cast<uint32_t *>(q + LO) = lo ^ sign;
        };
        if (SPIN == 0) {
            put(0, 2 * k + im, 0u);
        } else {
            // row k = (map, E or B); W -(E re, E im, B re, B im), X (B im, -B re, -E im, E re)
            const int c0 = 4 * (k >> 1), B = k & 1;
            put(0, c0 + 2 * B + im, 0x80008000u);
            put(2, c0 + (B ? 1 - im : 3 - im), B == im ? 0u : 0x80008000u);
        }
    }
}

// Records of every (m, chunk): grid (chunk, m, map group); entry (group,
// toff[m] + chunk).
template <int SPIN, int NMT>
__global__ void __launch_bounds__(TC_M) k_tc_records(const LegArgs<float> a) {
    typedef TcCfg<SPIN, NMT> Cfg;
    __shared__ float2 s_alm[Cfg::NA * TC_ALMS];
    const int m = blockIdx.y, l0 = m + 32 * blockIdx.x;
    if (l0 > a.lmax) return;
    RecIn<SPIN, NMT> R;
    load_record<SPIN, NMT>(a, m, l0, blockIdx.z * NMT, R);
    unsigned char *rec = a.rec_tc + ((int64_t)blockIdx.z * a.nrec + a.toff[m] + blockIdx.x) * Cfg::REC;
#pragma unroll
    for (int e = 0; e < RecIn<SPIN, NMT>::N; ++e)
        s_alm[((threadIdx.x + e * TC_M) >> 5) * TC_ALMS + (threadIdx.x & 31)] = R.v[e];
    store_coefs<SPIN, NMT>(R, rec);
    __syncthreads();
    gen_btiles<SPIN, NMT, TC_ALMS>(s_alm, rec);   // (whole 16-byte rows: coalesced in global memory)
}

// Recurrence over one chunk of 32 l (l = q0 .. q0 + 31, coefficients cf of the
// record); values of the even class (l - m even, K index (l - q0) / 2) and the
// odd class go to their A tiles in tensor memory as bf16 hi / lo (ta: this
// warp's lanes of the first tile's first column).  Lane = this thread's ring
// pair; half h = 0, 1 holds K 0..7, 8..15 (columns 4 h .. 4 h + 3 of a tile).
// wait() returns once the A tiles are free: it is called after the first
// half's recurrence, which so overlaps with the MMAs of the chunk before.
template <int SPIN, bool INJ, typename Wait>
__device__ __forceinline__ void gen_atiles(TcState<SPIN> &T, const PairState<float, 1> &S, const float4 *cf,
                                           const int q0, const uint32_t ta, Wait wait) {
    auto store = [&](int tile, int h, const float (&x)[8]) {   // tile: hi, tile + 1: lo
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) split2(x[2 * i], x[2 * i + 1], hi[i], lo[i]);
        tmem_st4(ta + 8 * tile + 4 * h, hi[0], hi[1], hi[2], hi[3]);
        tmem_st4(ta + 8 * tile + 8 + 4 * h, lo[0], lo[1], lo[2], lo[3]);
    };
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float wE[8], wO[8], xE[8], xO[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int d = 16 * h + 2 * i;
            if (SPIN == 2) {
                const float4 k0 = cf[3 * (d / 2)], g = cf[3 * (d / 2) + 1], k1 = cf[3 * (d / 2) + 2];
                T.step(make_float2(k0.x, k0.y), make_float2(k0.z, k0.w), make_float2(g.x, g.y));
                if (INJ) T.inject(q0 + d, S.ls[0], S.lsb[0], S.s0[0], S.s1[0], S.s2[0], S.s3[0]);
                wE[i] = T.w();
                xE[i] = T.x();
                T.step(make_float2(k1.x, k1.y), make_float2(k1.z, k1.w), make_float2(g.z, g.w));
            } else {
                const float4 k = cf[d / 2], z = make_float4(0.f, 0.f, 0.f, 0.f);
                T.step(make_float2(k.x, k.y), make_float2(z.x, z.y), make_float2(z.z, z.w));
                if (INJ) T.inject(q0 + d, S.ls[0], S.lsb[0], S.s0[0], S.s1[0], S.s2[0], S.s3[0]);
                wE[i] = T.w();
                T.step(make_float2(k.z, k.w), make_float2(z.x, z.y), make_float2(z.z, z.w));
            }
            if (INJ) T.inject(q0 + d + 1, S.ls[0], S.lsb[0], S.s0[0], S.s1[0], S.s2[0], S.s3[0]);
            wO[i] = T.w();
            xO[i] = T.x();
        }
        if (h == 0) wait();
        // tiles: (lw) E hi, lo | O hi, lo; spin 2 also lx E hi, lo | O hi, lo
        store(0, h, wE);
        store(2, h, wO);
        if (SPIN == 2) {
            store(4, h, xE);
            store(6, h, xO);
        }
    }
}

// bulk copy of one record into shared memory, completing on bar
__device__ __forceinline__ void bulk_load(unsigned char *dst, const unsigned char *src, uint32_t bytes,
                                          uint64_t *bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// REC: the records are in global memory; otherwise the CTA builds each chunk's (at
// spin 2 three CTAs per SM: with 128 registers it spills, N_side 128, l_max 256, 4
// Q/U maps 31.3 us, with 168 28.4).  Alone on an SM or nearly so, a CTA takes as
// long as its serial chain per chunk.  So one barrier per chunk: the coefficients
// of the next chunk are stored before it, the B tiles go from registers to their
// places without a staging pass, and the sums move out of tensor memory after the
// generation, when the MMAs they wait for are done.  With the staging pass, its
// second barrier and a wait of its own for the move: N_side 48, l_max 100, 8 Q/U
// maps 19.7 -> 18.0 us, N_side 64, l_max 150, 3 maps 20.4 -> 18.6 us (the form
// before the records: 17.5 and 18.3 us).
template <int SPIN, int NMT, bool REC>
__global__ void __launch_bounds__(TC_M, (REC || SPIN == 0 ? 4 : 3)) k_leg_synth_tc(const LegArgs<float> a) {
    typedef TcCfg<SPIN, NMT> Cfg;
    constexpr int NCOL = Cfg::NCOL;
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + Cfg::BARS);
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + Cfg::TMEMA);
    int *s_red = reinterpret_cast<int *>(smem + Cfg::RED);

    const int tid = threadIdx.x, warp = tid >> 5;
    const int m = blockIdx.y;
    const int L = a.lmax;
    const int map0 = blockIdx.z * NMT;
    const int nm = min(NMT, a.nmaps - map0);

    PairState<float, 1> S;
    int warp_lo, warp_hi;
    load_pairs<float, 1, SPIN>(a, blockIdx.x, m, S, warp_lo, warp_hi);
    const int lo = cta_min(warp_lo, s_red);
    const int pr = S.pr[0];
    const int rn = pr, rs = a.nring - 1 - pr;
    const int nrow = SPIN == 2 ? 2 * nm : nm;   // output rows of this CTA
    const int64_t rowsz = (int64_t)a.nring * (L + 1);
    float2 *out = a.F + (int64_t)(SPIN == 2 ? 2 * map0 : map0) * rowsz + m;

    if (lo > L) {   // no significant l for any pair of this CTA: zero output
        if (pr < a.npairs) {
            for (int k = 0; k < nrow; ++k) {
                out[k * rowsz + (int64_t)rn * (L + 1)] = make_float2(0.f, 0.f);
                if (rs != rn) out[k * rowsz + (int64_t)rs * (L + 1)] = make_float2(0.f, 0.f);
            }
        }
        return;
    }

    const int ch0 = (lo - m) >> 5;                 // chunks start at l - m = 0 mod 32
    const int n = ((L - m) >> 5) - ch0 + 1;        // chunks of this CTA
    RecIn<SPIN, NMT> R;
    if (!REC) load_record<SPIN, NMT>(a, m, m + 32 * ch0, map0, R);
    if (tid == 0) {
        for (int i = 0; i <= TC_NREC; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bars[i])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)),
                     "r"(Cfg::TMEM) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (!REC) store_coefs<SPIN, NMT>(R, smem);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *s_tmem;

    const unsigned char *rec = a.rec_tc + ((int64_t)blockIdx.z * a.nrec + a.toff[m] + ch0) * Cfg::REC;
    if (REC && tid == 0) {
        bulk_load(smem, rec, Cfg::REC, &bars[0]);
        if (n > 1) bulk_load(smem + Cfg::REC, rec + Cfg::REC, Cfg::REC, &bars[1]);
    }
    const uint64_t descB = sdesc(smem_u32(smem), 32 * NCOL, 128);
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);   // this warp's lanes
    TcState<SPIN> T;
    T.p1 = T.p2 = make_float2(0.f, 0.f);
    T.u = S.u[0];
    bool ok = true;
    uint64_t *mma_bar = &bars[TC_NREC];
    // The tensor core truncates at every accumulation, so a sum left in tensor
    // memory over all chunks drifts (relative 1e-6 of the result at l_max
    // 2048): every TC_FLUSH chunks it moves to sums that round to nearest.
    float *sums = reinterpret_cast<float *>(smem + Cfg::SUMS) + tid;
    auto flush = [&](bool first) {
#pragma unroll
        for (int h = 0; h < 2 * NCOL / 16; ++h) {
            float v[16];
            tmem_ld16(trow + 16 * h, v);
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                float *q = sums + (16 * h + c) * TC_M;
                *q = first ? v[c] : *q + v[c];
            }
        }
    };
    const int fl = n <= 8 ? 2 : TC_FLUSH;   // short sums: the start of the sum weighs more
    int st = 0, ph = 0;   // record stage of chunk c and its barrier's phase
    for (int c = 0; c < n; ++c) {
        unsigned char *bt = smem + st * Cfg::REC;
        if (REC) {
            ok = mbar_wait(&bars[st], ph) && ok;        // the record
        } else {   // (chunk c - 2 used this stage; its MMAs were waited for in chunk c - 1)
            store_btiles<SPIN, NMT>(R, bt);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (c + 1 < n) load_record<SPIN, NMT>(a, m, m + 32 * (ch0 + c + 1), map0, R);
        }
        // the MMAs of chunk c - 1: the A tiles are free, and so is its record
        // stage (its coefficients were read before the last barrier)
        auto free_tiles = [&]() {
            if (c == 0) return;
            ok = mbar_wait(mma_bar, (c - 1) & 1) && ok;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (REC && tid == 0 && c + TC_NREC - 1 < n) {
                const int sp = st == 0 ? TC_NREC - 1 : st - 1;
                bulk_load(smem + sp * Cfg::REC, rec + (int64_t)(c + TC_NREC - 1) * Cfg::REC, Cfg::REC, &bars[sp]);
            }
        };
        const int q0 = m + 32 * (ch0 + c);
        const float4 *cf = reinterpret_cast<const float4 *>(bt + Cfg::COEF);
        // injection steps only where some pair of the warp starts in this chunk
        const bool starts = (S.ls[0] >= q0 && S.ls[0] < q0 + 32) ||
                            (SPIN == 2 && S.lsb[0] >= q0 && S.lsb[0] < q0 + 32);
        if (__any_sync(0xffffffffu, starts)) gen_atiles<SPIN, true>(T, S, cf, q0, trow + Cfg::ACOL, free_tiles);
        else gen_atiles<SPIN, false>(T, S, cf, q0, trow + Cfg::ACOL, free_tiles);
        // (that stage's coefficients were read before the last barrier)
        if (!REC && c + 1 < n) store_coefs<SPIN, NMT>(R, smem + (st ^ 1) * Cfg::REC);
        // the sums up to chunk c - 1, whose MMAs free_tiles waited for
        if (c > 0 && (c & (fl - 1)) == 0) flush(c == fl);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t id = idesc_bf16(TC_M, NCOL);
            const uint32_t acc = (c & (fl - 1)) != 0;
            // (the address field counts 16-byte units)
            const uint64_t db = descB + (uint32_t)(st * (Cfg::REC >> 4));
            // A tiles t, t + 1 (hi, lo) and B tile b: D += A_lo B_hi + A_hi B_lo
            // (small; first, so that a new sum truncates little), D += A_hi B_hi
            auto ah = [&](int t) { return tmem + Cfg::ACOL + 8 * t; };
            auto bh = [&](int b) { return db + (uint32_t)(b * (Cfg::BTILE >> 4)); };
            auto low = [&](uint32_t d, int t, int b, uint32_t accumulate) {
                mma_bf16_ts(d, ah(t) + 8, bh(b), id, accumulate);
                mma_bf16_ts(d, ah(t), bh(b) + NCOL, id, 1);
            };
            auto high = [&](uint32_t d, int t, int b) { mma_bf16_ts(d, ah(t), bh(b), id, 1); };
            const uint32_t dE = tmem, dO = tmem + NCOL;
            // spin 2: symmetric part: lw even with W even, lx odd with X odd;
            // antisymmetric part: lw odd with W odd, lx even with X even
            low(dE, 0, 0, acc);
            low(dO, 2, 1, acc);
            if (SPIN == 2) {
                low(dE, 6, 3, 1);
                low(dO, 4, 2, 1);
            }
            high(dE, 0, 0);
            high(dO, 2, 1);
            if (SPIN == 2) {
                high(dE, 6, 3);
                high(dO, 4, 2);
            }
            mma_commit(mma_bar);
        }
        if (++st == TC_NREC) {
            st = 0;
            ph ^= 1;
        }
    }
    // ---- the last commit covers every MMA issued before it
    ok = mbar_wait(mma_bar, (n - 1) & 1) && ok;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!ok && tid == 0 && a.err) atomicExch(a.err, 1);

    // ---- epilogue: this thread's TMEM lane is its ring pair; columns [0,
    // NCOL) the even (spin 2: symmetric) part, [NCOL, 2 NCOL) the odd one
    if (n > fl) flush(false);
    float e[NCOL], o[NCOL];
    if (n > fl) {
#pragma unroll
        for (int c = 0; c < NCOL; ++c) {
            e[c] = sums[c * TC_M];
            o[c] = sums[(NCOL + c) * TC_M];
        }
    } else if (NCOL == 16) {
        tmem_ld16(trow, *reinterpret_cast<float(*)[16]>(e));
        tmem_ld16(trow + NCOL, *reinterpret_cast<float(*)[16]>(o));
    } else {
        tmem_ld32(trow, *reinterpret_cast<float(*)[32]>(e));
        tmem_ld32(trow + NCOL, *reinterpret_cast<float(*)[32]>(o));
    }
    if (ok && pr < a.npairs) {
        // output row k: columns 2 k, 2 k + 1
#pragma unroll
        for (int k = 0; k < NCOL / 2; ++k) {
            if (k >= nrow) break;
            out[k * rowsz + (int64_t)rn * (L + 1)] = make_float2(e[2 * k] + o[2 * k], e[2 * k + 1] + o[2 * k + 1]);
            if (rs != rn)
                out[k * rowsz + (int64_t)rs * (L + 1)] = make_float2(e[2 * k] - o[2 * k], e[2 * k + 1] - o[2 * k + 1]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Cfg::TMEM) : "memory");
}

template <int SPIN, int NMT, bool REC>
int launch_synth_tc(Plan *p, const float2 *alm, int rs, int nmaps, const float *beam, float2 *F,
                    cudaStream_t st) {
    typedef TcCfg<SPIN, NMT> Cfg;
    LegArgs<float> a = leg_make_args<float>(p);
    a.rs = rs;
    a.beam = beam;
    a.err = p->d_flag;
    a.rec_tc = p->d_tcrec[SPIN / 2];
    a.nrec = p->tc_nrec;
    const int smem = Cfg::BYTES;
    auto kern = k_leg_synth_tc<SPIN, NMT, REC>;
    SHTG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    // as many map groups per pass as the plan's record buffer holds
    const int groups = (nmaps + NMT - 1) / NMT;
    const int fit = !REC ? groups : (int)std::max<int64_t>(1, std::min<int64_t>(groups, p->tcrec_bytes[SPIN / 2] / (p->tc_nrec * Cfg::REC)));
    prof_begin(p, K_LEG_SYN32, st);
    int nl = 0;
    for (int g0 = 0; g0 < groups; g0 += fit) {
        const int ng = std::min(fit, groups - g0);
        a.nmaps = std::min(nmaps - g0 * NMT, ng * NMT);
        a.alm = alm + (int64_t)g0 * NMT * rs * p->nalm;
        a.F = F + (int64_t)g0 * NMT * (SPIN == 2 ? 2 : 1) * p->nring * (p->lmax + 1);
        if (REC) k_tc_records<SPIN, NMT><<<dim3(p->lmax / 32 + 1, p->lmax + 1, ng), TC_M, 0, st>>>(a);
        kern<<<dim3((p->npairs + TC_M - 1) / TC_M, p->lmax + 1, ng), TC_M, smem, st>>>(a);
        nl += REC ? 2 : 1;
    }
    prof_end(p, st, nl);
    SHTG_CHECK_LAUNCH("k_leg_synth_tc");
    return SHTG_OK;
}

// FP32 recurrence state before every l = m + 32 t of every (m, ring pair):
// the same steps (rstep / step2 with the same injections) as the Legendre
// kernels, so a kernel that restarts from an entry reproduces the values of
// one continuous run bit for bit.  One thread per (m, pair); entries
// [m][t][pair] so that a warp's stores are contiguous.
template <int SPIN>
__global__ void __launch_bounds__(LEG_THREADS) k_tile_states(const LegArgs<float> a, const int64_t *toff,
                                                             float2 *out0, float4 *out2) {
    const int m = blockIdx.y;
    const int L = a.lmax;
    PairState<float, 1> S;
    int wlo, whi;
    load_pairs<float, 1, SPIN>(a, blockIdx.x, m, S, wlo, whi);
    const int pr = S.pr[0];
    if (pr >= a.npairs) return;
    const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2;
    const int64_t o = toff[m] * a.npairs + pr;
    for (int l = m; l <= L; ++l) {
        if (((l - m) & 31) == 0) {
            const int64_t e = o + (int64_t)((l - m) >> 5) * a.npairs;
            if (SPIN == 2) out2[e] = make_float4(S.a1[0], S.a2[0], S.b1[0], S.b2[0]);
            else out0[e] = make_float2(S.a1[0], S.a2[0]);
        }
        stepx<float, 1, SPIN, true>(S, a.rec + base, a.s2c + base, l, l);
    }
}

}  // namespace

int build_tile_states(Plan *p) {
    const int L = p->lmax;
    std::vector<int64_t> toff(L + 2);
    toff[0] = 0;
    for (int m = 0; m <= L; ++m) toff[m + 1] = toff[m] + (L + 1 - m + 31) / 32;
    const size_t nent = (size_t)toff[L + 1] * p->npairs;
    auto alloc = [&](void **ptr, size_t bytes) -> int {
        cudaError_t e = cudaMalloc(ptr, bytes);
        if (e != cudaSuccess) {
            *ptr = nullptr;
            cudaGetLastError();
            set_error(std::string("cudaMalloc of ") + std::to_string(bytes) +
                      " bytes (recurrence tile states) failed: " + cudaGetErrorString(e));
            return SHTG_ERR_NOMEM;
        }
        p->device_bytes += (int64_t)bytes;
        return SHTG_OK;
    };
    SHTG_TRY(alloc((void **)&p->d_toff, sizeof(int64_t) * toff.size()));
    SHTG_CUDA(cudaMemcpy(p->d_toff, toff.data(), sizeof(int64_t) * toff.size(), cudaMemcpyHostToDevice));
    SHTG_TRY(alloc((void **)&p->d_tst0, sizeof(float2) * nent));
    LegArgs<float> a = leg_make_args<float>(p);
    dim3 grid((p->npairs + LEG_THREADS - 1) / LEG_THREADS, L + 1);
    k_tile_states<0><<<grid, LEG_THREADS>>>(a, p->d_toff, p->d_tst0, nullptr);
    SHTG_CHECK_LAUNCH("k_tile_states");
    if (p->flags & SHTG_SPIN2) {
        SHTG_TRY(alloc((void **)&p->d_tst2, sizeof(float4) * nent));
        k_tile_states<2><<<grid, LEG_THREADS>>>(a, p->d_toff, nullptr, p->d_tst2);
        SHTG_CHECK_LAUNCH("k_tile_states");
    }
    p->tc_nrec = toff[L + 1];
    SHTG_CUDA(cudaDeviceSynchronize());
    return SHTG_OK;
}

namespace {

// ===================================================== transpose (Y^T)
// c_lm = sum_r lambda_lm(theta_r) G_r(m) for one m and a range of 256 l:
// rows = l (two 128-row tiles: l - m even, l - m odd), K = ring pairs in
// stages of 16, columns = (map, output) with the north / south combination
// G_N + G_S (rows with the parity of lambda) or G_N - G_S folded into the B
// tiles.  k_ta_records writes the B tiles of every (m, stage) as records in
// global memory, eight m at a time; k_leg_analysis_tc fetches them by bulk
// copies, one stage ahead.  A tiles hold the recurrence values l-major
// (MN-major core matrices: 8 pairs x 8 consecutive rows of one class), which
// is how a thread produces them: thread (pair p, segment s) runs the FP32
// recurrence of pair p over 32 l from the tabulated state at l = m + 32 t.
// The CTA accumulates over all ring pairs in tensor memory, so every alm is
// written once, by one CTA, without atomics.
//
// What bounds it: the shared-memory / L1 data path, which the MMAs' operand
// reads share.  Before the records every CTA copied its ring data with 8-byte
// cp.async (neighbouring m lie side by side in memory, so each took a line of
// its own) and built the same B tiles: about 1100 wavefronts per stage and 256
// l at spin 2, and the MMAs read 12 A tiles of 4 KB (384 wavefronts).  Now the
// products with hi and lo of B are one MMA of twice the columns into separate
// sums, so each of the 8 A tiles is read once.  Measured (N_side 1024, l_max
// 2048, 8 Q/U maps, with the ring stage): 7.18 -> 5.20 ms.  Spin 0 (8 maps) has
// half the shared and tensor memory, and 71 registers let six CTAs share an SM:
// N_side 512, l_max 1024, 4 maps, 0.38 -> 0.28 ms.
constexpr int TA_K = 16;        // ring pairs per stage (MMA K)
template <int SPIN, int NMT> struct TaCfg {   // NMT maps per CTA
    static constexpr int NO = SPIN == 2 ? 4 * NMT : 2 * NMT, NAT = SPIN == 2 ? 8 : 4, NBT = SPIN == 2 ? 4 : 2;
};
// Staged ring data of one (m, stage): [pair][north rows | south rows] float2
// with pair stride GS = 2 NROW + 2: the builder's warp reads 8 consecutive
// floats per K pair and its four K pairs sit 4 GS = 8 (mod 32) floats apart,
// so every load hits 32 distinct banks.
template <int SPIN, int NMT> struct TaRing {
    static constexpr int NROW = SPIN == 2 ? 2 * NMT : NMT;
    static constexpr int GS = 2 * NROW + 2;
    static constexpr int SG = TA_K * GS + 4;   // stride of the m
};
// Shared memory of the transpose CTA: NAS A buffers (the tiles of one stage),
// NAS + 1 B buffers, without records (REC false) the ring data of one stage,
// the coefficients of 256 l, the mbarriers (NAS of the
// MMAs, NAS + 1 of the records) and the TMEM address.  With one A buffer (53 KB
// at spin 2) four CTAs share an SM, and each waits for its own MMAs while the
// others generate.
template <int SPIN, int NMT, int NAS, bool REC> struct TaLayout {
    typedef TaCfg<SPIN, NMT> Cfg;
    static constexpr int BT = 64 * Cfg::NO;                         // B tile: 2 NO rows x 16 K bf16
    static constexpr int ASTAGE = Cfg::NAT * TC_ATILE;
    static constexpr int BSTAGE = Cfg::NBT * BT;                    // one record
    static constexpr int NBS = NAS + 1;
    static constexpr int BOFF = NAS * ASTAGE;
    static constexpr int GOFF = BOFF + NBS * BSTAGE;
    static constexpr int COEF = GOFF + (REC ? 0 : ((TA_K * TaRing<SPIN, NMT>::GS * 8) + 15) & ~15);
    // coefficients of 256 l, one padding entry after every 32 (ta_cpad)
    static constexpr int BARS = COEF + 264 * (SPIN == 2 ? 16 : 8);
    static constexpr int TMEM = 4 * Cfg::NO;   // two classes, products with B hi and with B lo
    static constexpr int TMEMA = BARS + 48;
    static constexpr int BYTES = TMEMA + 16;
};
constexpr int TA_MB = 8;   // m per CTA of the records: 64-byte runs of the ring data

// Shared index of the recurrence coefficients of l = lbase + i in the
// transpose: one padding entry after every 32, so the two 32-l segments that
// a warp's threads step through at once (256 or 512 bytes apart unpadded,
// the same banks) read distinct banks.
__device__ __forceinline__ int ta_cpad(int i) { return i + (i >> 5); }

// MN-major A (bit 15), K-major B, bf16 in, FP32 accumulator
__host__ __device__ constexpr uint32_t idesc_bf16_amn(int m, int n) {
    return idesc_bf16(m, n) | (1u << 15);
}

// Start data of one ring pair for m (from the FP64 start states) and the
// tabulated FP32 recurrence state before l0 = m + 32 t.
struct PairStart {
    int ls, lsb;
    float s0, s1, s2, s3, u;
};
template <int SPIN>
__device__ __forceinline__ PairStart load_pair_start(const LegArgs<float> &a, int m, int pr) {
    PairStart q;
    q.ls = q.lsb = a.lmax + 1;
    q.s0 = q.s1 = q.s2 = q.s3 = 0.f;
    q.u = 1.f;
    if (pr < a.npairs) {
        const int64_t o = (int64_t)m * a.npairs + pr;
        q.u = a.u[pr];
        if (SPIN == 2) {
            const int2 l2 = a.ls2[o];
            const float4 s4 = a.st2[o];
            q.ls = l2.x;
            q.lsb = l2.y;
            q.s0 = s4.x;
            q.s1 = s4.y;
            q.s2 = s4.z;
            q.s3 = s4.w;
        } else {
            const float2 s2 = a.st[o];
            q.ls = a.ls[o];
            q.s0 = s2.x;
            q.s1 = s2.y;
        }
    }
    return q;
}
template <int SPIN>
__device__ __forceinline__ float4 load_tile_state(const LegArgs<float> &a, int m, int pr, int l0) {
    if (pr >= a.npairs || l0 > a.lmax) return make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t e = (a.toff[m] + ((l0 - m) >> 5)) * a.npairs + pr;
    if (SPIN == 2) return a.tst2[e];
    const float2 t = a.tst0[e];
    return make_float4(t.x, t.y, 0.f, 0.f);
}

// A tiles of one (stage, 256-l tile): this thread's pair (column pin of the
// K = 16 slice) over l = l0 .. l0 + 31, l0 = tstart + 32 seg, from state ts;
// values of class E (l - m even) go to rows 16 seg + j of the E tiles, class
// O to the same rows of the O tiles.  Pairs beyond npairs (state 0) and l
// beyond lmax (coefficients and state 0) give 0.  INJ: some pair of the warp
// starts its recurrence inside the segment (the tabulated state already holds
// every earlier start).  wait() as in the synthesis.
template <int SPIN, bool INJ, typename Wait>
__device__ __forceinline__ void gen_atiles_ana(const PairStart &q, const float4 ts, const int pin, const int seg,
                                               const int l0, const int lbase, const void *s_cf, unsigned char *at,
                                               Wait wait) {
    TcState<SPIN> T;
    T.u = q.u;
    if (SPIN == 2) {   // ts = (y+_{l-1}, y+_{l-2}, y-_{l-1}, y-_{l-2})
        T.p1 = make_float2(ts.x, ts.z);
        T.p2 = make_float2(ts.y, ts.w);
    } else {
        T.p1 = make_float2(ts.x, 0.f);
        T.p2 = make_float2(ts.y, 0.f);
    }
    const int kg = pin >> 3, krow = pin & 7;
    // padded shared index of l0 + d: l0 - lbase is a multiple of 32 and d <= 31,
    // so ta_cpad(l0 - lbase + d) = ta_cpad(l0 - lbase) + d
    const int cb = ta_cpad(l0 - lbase);
    const float4 *c4 = reinterpret_cast<const float4 *>(s_cf) + cb;
    const float2 *c2 = reinterpret_cast<const float2 *>(s_cf) + cb;
    auto step = [&](int d) {
        if (SPIN == 2) {
            const float4 k = c4[d];
            T.step(make_float2(k.x, k.y), make_float2(k.z, k.z), make_float2(k.w, k.w));
        } else {
            T.step(c2[d], make_float2(0.f, 0.f), make_float2(0.f, 0.f));
        }
        if (INJ) T.inject(l0 + d, q.ls, q.lsb, q.s0, q.s1, q.s2, q.s3);
    };
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        // rows 16 seg + 8 h .. + 7: core matrix (M group 2 seg + h, K group kg)
        unsigned char *t = at + (kg * 16 + 2 * seg + h) * 128 + krow * 16;
        float wE[8], wO[8], xE[8], xO[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int d = 16 * h + 2 * i;
            step(d);
            wE[i] = T.w();
            xE[i] = T.x();
            step(d + 1);
            wO[i] = T.w();
            xO[i] = T.x();
        }
        if (h == 0) wait();
        store_row8(t, t + TC_ATILE, wE);
        store_row8(t + 2 * TC_ATILE, t + 3 * TC_ATILE, wO);
        if (SPIN == 2) {
            store_row8(t + 4 * TC_ATILE, t + 5 * TC_ATILE, xE);
            store_row8(t + 6 * TC_ATILE, t + 7 * TC_ATILE, xO);
        }
    }
}

// Asynchronous copy (cp.async) of the ring data of stage ps into sg:
// element (pair p, row q, ring z) at sg[p GS + z NROW + q]; rows are the maps of
// this CTA (spin 2: Q, U of each); zeros for pairs beyond npairs, missing
// maps and the south ring of the equator pair.
template <int SPIN, int NMT>
__device__ __forceinline__ void stage_ring_data(const LegArgs<float> &a, const int m, const int ps, const int map0,
                                                const int nm, float2 *sg) {
    typedef TaRing<SPIN, NMT> Lay;
    const int L = a.lmax;
    const int64_t rowsz = (int64_t)a.nring * (L + 1);
    const int nrow = SPIN == 2 ? 2 * nm : nm;
    for (int it = threadIdx.x; it < TA_K * Lay::NROW * 2; it += TC_M) {
        const int z = it & 1;
        const int q = (it >> 1) % Lay::NROW;
        const int pp = it / (2 * Lay::NROW);
        const int pr = ps * TA_K + pp;
        float2 *dst = sg + pp * Lay::GS + z * Lay::NROW + q;
        const int rn = pr, rs = a.nring - 1 - pr;
        if (pr < a.npairs && q < nrow && !(z && rs == rn)) {
            const int64_t grow = (SPIN == 2 ? 2 * map0 : map0) + q;
            const float2 *src = a.F + grow * rowsz + (int64_t)(z ? rs : rn) * (L + 1) + m;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
        } else {
            *dst = make_float2(0.f, 0.f);
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// B tiles of one stage from the staged ring data.  Tile b: spin 0 -> rows
// for class b (0: G_N + G_S, 1: G_N - G_S) with columns (re, im) per map;
// spin 2 -> b = 2 x + class' with lw columns (x = 0, class' = b) and lx
// columns (x = 1, class' = the other one):
//   E^ = -lw G_Q - i lx G_U,  B^ = i lx G_Q - lw G_U
// (columns E re, E im, B re, B im per map).  hi at row c, lo at row NO + c.
// One thread per (K group kg, K pair kq, column c) writes that column's word
// (two consecutive ring pairs) in every tile: a warp covers 8 consecutive
// columns x 4 K pairs, i.e. 32 distinct banks per store, and reads only the
// two scalars per ring pair that its column needs.
template <int SPIN, int NMT>
__device__ __forceinline__ void gen_btiles_ana(const float2 *sg, unsigned char *bt) {
    typedef TaRing<SPIN, NMT> Lay;
    constexpr int NO = TaCfg<SPIN, NMT>::NO, BT = 64 * NO;
    const float *sgf = reinterpret_cast<const float *>(sg);
    for (int it = threadIdx.x; it < 8 * NO; it += TC_M) {
        const int kq = it & 3;
        const int c = (it >> 2) % NO;
        const int kg = it / (4 * NO);
        const int k0 = 8 * kg + 2 * kq;
        unsigned char *tile = bt + kg * (32 * NO) + kq * 4;
        if (SPIN == 0) {
            // column c: component c & 1 of map c >> 1, i.e. float c of the
            // north rows and float 2 NROW + c (the south rows)
            float vp[2], vm[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float *g = sgf + 2 * (k0 + q) * Lay::GS;
                const float gn = g[c], gs = g[2 * Lay::NROW + c];
                vp[q] = gn + gs;
                vm[q] = gn + (-1.f) * gs;
            }
            uint32_t hi, lo;
            split2(vp[0], vp[1], hi, lo);
            *reinterpret_cast<uint32_t *>(tile + c * 16) = hi;
            *reinterpret_cast<uint32_t *>(tile + (NO + c) * 16) = lo;
            split2(vm[0], vm[1], hi, lo);
            *reinterpret_cast<uint32_t *>(tile + BT + c * 16) = hi;
            *reinterpret_cast<uint32_t *>(tile + BT + (NO + c) * 16) = lo;
        } else {
            // column c = 4 k + comp of map k; the lw tiles take w = (-Q re,
            // -Q im, -U re, -U im)[comp], the lx tiles x = (U im, -U re,
            // -Q im, Q re)[comp], each as N + S or N - S
            const int k = c >> 2, comp = c & 3;
            const int wf = comp < 2 ? 0 : 1, wc = comp & 1;            // field (Q 0, U 1), re / im
            const int xf = comp < 2 ? 1 : 0, xc = (comp & 1) ^ 1;
            const float xs = (comp == 1 || comp == 2) ? -1.f : 1.f;
            // (row 2 k + field of the north rows at float 2 (2 k + field) + re/im,
            // the south rows 2 NROW floats later)
            float wp[2], wm[2], xp[2], xm[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float *g = sgf + 2 * (k0 + q) * Lay::GS + 4 * k;
                const float wn = g[2 * wf + wc], wsv = g[2 * Lay::NROW + 2 * wf + wc];
                const float xn = g[2 * xf + xc], xsv = g[2 * Lay::NROW + 2 * xf + xc];
                wp[q] = -(wn + wsv);
                wm[q] = -(wn + (-1.f) * wsv);
                xp[q] = xs * (xn + xsv);
                xm[q] = xs * (xn + (-1.f) * xsv);
            }
            uint32_t hi, lo;
            split2(wp[0], wp[1], hi, lo);   // b = 0: lw, class 0
            *reinterpret_cast<uint32_t *>(tile + c * 16) = hi;
            *reinterpret_cast<uint32_t *>(tile + (NO + c) * 16) = lo;
            split2(wm[0], wm[1], hi, lo);   // b = 1: lw, class 1
            *reinterpret_cast<uint32_t *>(tile + BT + c * 16) = hi;
            *reinterpret_cast<uint32_t *>(tile + BT + (NO + c) * 16) = lo;
            split2(xm[0], xm[1], hi, lo);   // b = 2: lx, class 1
            *reinterpret_cast<uint32_t *>(tile + 2 * BT + c * 16) = hi;
            *reinterpret_cast<uint32_t *>(tile + 2 * BT + (NO + c) * 16) = lo;
            split2(xp[0], xp[1], hi, lo);   // b = 3: lx, class 0
            *reinterpret_cast<uint32_t *>(tile + 3 * BT + c * 16) = hi;
            *reinterpret_cast<uint32_t *>(tile + 3 * BT + (NO + c) * 16) = lo;
        }
    }
}

// Records of stage blockIdx.x for m = a.m0 + 8 blockIdx.y .. + 7 (below a.m0 +
// a.mcnt) and map group blockIdx.z: entry ((group mcnt + m - m0) stages + stage).
template <int SPIN, int NMT>
__global__ void __launch_bounds__(TC_M) k_ta_records(const LegArgs<float> a) {
    typedef TaRing<SPIN, NMT> Ring;
    constexpr int BSTAGE = TaLayout<SPIN, NMT, 1, true>::BSTAGE;
    __shared__ float2 sg[TA_MB * Ring::SG];
    const int L = a.lmax, ps = blockIdx.x;
    const int i0 = TA_MB * blockIdx.y, ni = min(TA_MB, a.mcnt - i0);
    const int map0 = blockIdx.z * NMT;
    const int nrow = (SPIN == 2 ? 2 : 1) * min(NMT, a.nmaps - map0);
    const float2 *src = a.F + (int64_t)(SPIN == 2 ? 2 * map0 : map0) * a.nring * (L + 1) + a.m0 + i0;
    // rows are the maps of the group (spin 2: Q, U of each); zeros for pairs
    // beyond npairs, missing maps and the south ring of the equator pair
#pragma unroll 8
    for (int it = threadIdx.x; it < TA_K * 2 * Ring::NROW * TA_MB; it += TC_M) {
        const int mi = it & (TA_MB - 1), q = (it / TA_MB) % Ring::NROW;
        const int z = (it / (TA_MB * Ring::NROW)) & 1, pp = it / (2 * TA_MB * Ring::NROW);
        const int rn = ps * TA_K + pp, rs = a.nring - 1 - rn;
        float2 v = make_float2(0.f, 0.f);
        if (mi < ni && rn < a.npairs && q < nrow && !(z && rs == rn))
            v = src[((int64_t)q * a.nring + (z ? rs : rn)) * (L + 1) + mi];
        sg[mi * Ring::SG + pp * Ring::GS + z * Ring::NROW + q] = v;
    }
    __syncthreads();
    unsigned char *rec = a.rec_tc + (((int64_t)blockIdx.z * a.mcnt + i0) * gridDim.x + ps) * BSTAGE;
    for (int mi = 0; mi < ni; ++mi)
        gen_btiles_ana<SPIN, NMT>(sg + mi * Ring::SG, rec + (int64_t)mi * gridDim.x * BSTAGE);
}

template <int SPIN, int NMT, int NAS, bool REC>
__global__ void __launch_bounds__(TC_M, (SPIN == 0 && NMT == 8 ? 6 : 4)) k_leg_analysis_tc(const LegArgs<float> a) {
    typedef TaLayout<SPIN, NMT, NAS, REC> Lay;
    constexpr int NO = Lay::Cfg::NO, NBS = Lay::NBS, BSTAGE = Lay::BSTAGE;
    extern __shared__ __align__(1024) unsigned char smem[];
    float4 *s_c4 = reinterpret_cast<float4 *>(smem + Lay::COEF);   // spin 2 (tc_coef)
    float2 *s_c2 = reinterpret_cast<float2 *>(smem + Lay::COEF);   // spin 0 (a, b)
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + Lay::BARS), *full = bars + NAS;
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + Lay::TMEMA);

    const int tid = threadIdx.x, warp = tid >> 5;
    const int m = a.m0 + blockIdx.y;
    const int L = a.lmax;
    const int lbase = m + blockIdx.x * 256;
    if (lbase > L) return;
    const int lend = min(L, lbase + 255);
    const int map0 = blockIdx.z * NMT;
    const int nm = min(NMT, a.nmaps - map0);
    const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2;

    for (int i = tid; i < 256; i += TC_M) {
        const int l = lbase + i;
        const bool in = l <= L;
        if (SPIN == 2) s_c4[ta_cpad(i)] = tc_coef(in ? a.s2c[base + l] : make_float4(0.f, 0.f, 0.f, 0.f));
        else s_c2[ta_cpad(i)] = in ? a.rec[base + l] : make_float2(0.f, 0.f);
    }
    if (tid == 0) {
        for (int i = 0; i < NAS + NBS; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bars[i])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)),
                     "r"(Lay::TMEM) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *s_tmem;

    const int pin = tid & (TA_K - 1), seg = tid >> 4;
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
    float2 *sgb = reinterpret_cast<float2 *>(smem + Lay::GOFF);
    int *s_first = reinterpret_cast<int *>(smem + Lay::TMEMA + 4);

    // first stage with a pair whose recurrence starts at or before lend; the
    // start l falls towards the equator, so every later stage is worked too
    // (a stage without significant values contributes exact zeros)
    if (tid == 0) *s_first = a.npairs;
    __syncthreads();
    {
        int first = a.npairs;
        for (int pr = tid; pr < a.npairs; pr += TC_M) {
            const int64_t o = (int64_t)m * a.npairs + pr;
            int lsp;
            if (SPIN == 2) {
                const int2 q = a.ls2[o];
                lsp = min(q.x, q.y);
            } else {
                lsp = a.ls[o];
            }
            if (lsp <= lend) {
                first = pr;
                break;
            }
        }
        if (first < a.npairs) atomicMin(s_first, first);
    }
    __syncthreads();
    const int s0 = *s_first / TA_K;
    const int nps = (a.npairs + TA_K - 1) / TA_K;
    const int nst = s0 < nps ? nps - s0 : 0;

    const uint64_t descA = sdesc(smem_u32(smem), 2048, 128), descB = sdesc(smem_u32(smem + Lay::BOFF), 32 * NO, 128);
    const unsigned char *rec = a.rec_tc + (((int64_t)blockIdx.z * a.mcnt + blockIdx.y) * nps + s0) * BSTAGE;
    bool ok = true;
    PairStart pst{}, pnext{};
    float4 tcur = make_float4(0.f, 0.f, 0.f, 0.f);
    const int l0 = lbase + 32 * seg;
    if (nst > 0) {
        if (!REC) stage_ring_data<SPIN, NMT>(a, m, s0, map0, nm, sgb);
        else if (tid == 0) bulk_load(smem + Lay::BOFF, rec, BSTAGE, &full[0]);
        pst = load_pair_start<SPIN>(a, m, s0 * TA_K + pin);
        tcur = load_tile_state<SPIN>(a, m, s0 * TA_K + pin, l0);
    }
    // Stage si commits its MMAs to barrier si % NAS, completing that barrier's
    // phase si / NAS, and its record sits in B buffer si % NBS.
    int bsel = 0, bph = 0;
    for (int si = 0; si < nst; ++si) {
        const int pr = (s0 + si) * TA_K + pin;
        const bool more = si + 1 < nst;
        float4 tnext = make_float4(0.f, 0.f, 0.f, 0.f);
        if (more) {   // in flight during this stage
            pnext = load_pair_start<SPIN>(a, m, pr + TA_K);
            tnext = load_tile_state<SPIN>(a, m, pr + TA_K, l0);
        }
        if (!REC) {   // (this B buffer was read by stage si - NBS, waited for in stage si - 1)
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            gen_btiles_ana<SPIN, NMT>(sgb, smem + Lay::BOFF + bsel * BSTAGE);
        }
        const int asel = si % NAS;
        unsigned char *at = smem + asel * Lay::ASTAGE;
        // the MMAs of stage si - NAS are done: its A buffer is free, and so is
        // the B buffer that the next stage's record goes to
        auto free_tiles = [&]() {
            if (si >= NAS) ok = mbar_wait(&bars[asel], ((si - NAS) / NAS) & 1) && ok;
            if (REC && tid == 0 && more) {
                const int bn = bsel + 1 == NBS ? 0 : bsel + 1;
                bulk_load(smem + Lay::BOFF + bn * BSTAGE, rec + (int64_t)(si + 1) * BSTAGE, BSTAGE, &full[bn]);
            }
        };
        const bool starts = (pst.ls >= l0 && pst.ls < l0 + 32) || (SPIN == 2 && pst.lsb >= l0 && pst.lsb < l0 + 32);
        if (__any_sync(0xffffffffu, starts && l0 <= L))
            gen_atiles_ana<SPIN, true>(pst, tcur, pin, seg, l0, lbase, s_c4, at, free_tiles);
        else
            gen_atiles_ana<SPIN, false>(pst, tcur, pin, seg, l0, lbase, s_c4, at, free_tiles);
        tcur = tnext;
        pst = pnext;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        // (the ring data are consumed: the next stage's copy runs beside this
        // stage's MMAs and the next generation)
        if (!REC && more) stage_ring_data<SPIN, NMT>(a, m, s0 + si + 1, map0, nm, sgb);
        if (tid == 0) {
            if (REC) ok = mbar_wait(&full[bsel], bph) && ok;   // the stage's record
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // id2: hi and lo rows of B side by side (2 NO columns); id: hi only
            const uint32_t id2 = idesc_bf16_amn(TC_M, 2 * NO), id = idesc_bf16_amn(TC_M, NO);
            const uint32_t acc = si > 0;
            // (the address field counts 16-byte units)
            const uint64_t da = descA + (uint32_t)(asel * (Lay::ASTAGE >> 4));
            const uint64_t db = descB + (uint32_t)(bsel * (BSTAGE >> 4));
            auto A = [&](int t) { return da + (uint32_t)(t * (TC_ATILE >> 4)); };
            auto B = [&](int t) { return db + (uint32_t)(t * (Lay::BT >> 4)); };
            const uint32_t dE = tmem, dO = tmem + 2 * NO;
            // A hi with B hi and B lo, A lo with B hi; spin 2: even rows lw with
            // W from G_N + G_S, lx with X from G_N - G_S, odd rows the others
            mma_bf16(dE, A(0), B(0), id2, acc);
            mma_bf16(dE, A(1), B(0), id, 1);
            mma_bf16(dO, A(2), B(1), id2, acc);
            mma_bf16(dO, A(3), B(1), id, 1);
            if (SPIN == 2) {
                mma_bf16(dE, A(4), B(2), id2, 1);
                mma_bf16(dE, A(5), B(2), id, 1);
                mma_bf16(dO, A(6), B(3), id2, 1);
                mma_bf16(dO, A(7), B(3), id, 1);
            }
            mma_commit(&bars[asel]);
        }
        if (++bsel == NBS) {
            bsel = 0;
            bph ^= 1;
        }
    }
    if (nst > 0) ok = mbar_wait(&bars[(nst - 1) % NAS], ((nst - 1) / NAS) & 1) && ok;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    ok = __syncthreads_and(ok);   // (the records' waits are one thread's)
    if (!ok && tid == 0 && a.err) atomicExch(a.err, 1);

    // ---- epilogue: lane = row i, l = lbase + 2 i (E tile) and + 1 (O tile)
#pragma unroll
    for (int cls = 0; cls < 2; ++cls) {
        const int l = lbase + 2 * tid + cls;
        float d[NO], e[NO];
        if constexpr (NO == 16) {
            tmem_ld16(trow + cls * 2 * NO, d);
            tmem_ld16(trow + cls * 2 * NO + NO, e);
        } else {
            tmem_ld32(trow + cls * 2 * NO, d);
            tmem_ld32(trow + cls * 2 * NO + NO, e);
        }
        if (!ok || l > L) continue;
        const float bm = (a.beam ? a.beam[l] : 1.f) * ((a.vjp && m > 0) ? 2.f : 1.f);
#pragma unroll
        for (int k = 0; k < NMT; ++k) {
            if (k >= nm) break;
#pragma unroll
            for (int c = 0; c < (SPIN == 2 ? 2 : 1); ++c) {
                const int j = SPIN == 2 ? 4 * k + 2 * c : 2 * k;
                float re = 0.f, im = 0.f;
                if (nst > 0) {
                    re = (d[j] + e[j]) * bm;
                    im = m == 0 ? 0.f : (d[j + 1] + e[j + 1]) * bm;
                }
                const int64_t row = (int64_t)(map0 + k) * a.rs + c;
                float2 *dst = const_cast<float2 *>(a.alm) + row * a.nalm + base + l;
                *dst = make_float2(re, im);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Lay::TMEM) : "memory");
}

template <int SPIN, int NMT, int NAS, bool REC>
int launch_analysis_tc(Plan *p, const float2 *G, int nmaps, const float *beam, float2 *alm, int rs,
                       cudaStream_t st, int vjp) {
    LegArgs<float> a = leg_make_args<float>(p);
    typedef TaLayout<SPIN, NMT, NAS, REC> Lay;
    a.rs = rs;
    a.vjp = vjp;
    a.beam = beam;
    a.err = p->d_flag;
    a.rec_tc = p->d_tcrec[SPIN / 2];
    if (!a.toff || !a.tst0 || (SPIN == 2 && !a.tst2)) {
        set_error("tensor-core transpose: the plan has no recurrence tile states");
        return SHTG_ERR_ARG;
    }
    const int smem = Lay::BYTES;
    auto kern = k_leg_analysis_tc<SPIN, NMT, NAS, REC>;
    SHTG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    // with records as many map groups, then as many m per pass as the plan's
    // buffer holds (all of them up to its cap)
    const int nps = (p->npairs + TA_K - 1) / TA_K, groups = (nmaps + NMT - 1) / NMT;
    const int64_t per_m = (int64_t)nps * Lay::BSTAGE, bytes = p->tcrec_bytes[SPIN / 2];
    const int gfit = REC ? (int)std::max<int64_t>(1, std::min<int64_t>(groups, bytes / per_m)) : groups;
    const int mfit = REC ? (int)std::max<int64_t>(1, std::min<int64_t>(p->lmax + 1, bytes / (per_m * gfit))) : p->lmax + 1;
    prof_begin(p, K_LEG_ANA32, st);
    int nl = 0;
    for (int g0 = 0; g0 < groups; g0 += gfit) {
        const int ng = std::min(gfit, groups - g0);
        a.nmaps = std::min(nmaps - g0 * NMT, ng * NMT);
        a.alm = alm + (int64_t)g0 * NMT * rs * p->nalm;
        a.F = const_cast<float2 *>(G) + (int64_t)g0 * NMT * (SPIN == 2 ? 2 : 1) * p->nring * (p->lmax + 1);
        for (a.m0 = 0; a.m0 <= p->lmax; a.m0 += mfit) {
            a.mcnt = std::min(mfit, p->lmax + 1 - a.m0);
            if (REC) k_ta_records<SPIN, NMT><<<dim3(nps, (a.mcnt + TA_MB - 1) / TA_MB, ng), TC_M, 0, st>>>(a);
            kern<<<dim3((p->lmax - a.m0 + 256) / 256, a.mcnt, ng), TC_M, smem, st>>>(a);
            nl += REC ? 2 : 1;
        }
    }
    prof_end(p, st, nl);
    SHTG_CHECK_LAUNCH("k_leg_analysis_tc");
    return SHTG_OK;
}

// bytes of all records of the transpose for mb maps
template <int SPIN, int NMT> int64_t ta_record_bytes(const Plan *p, int mb) {
    const int64_t per_m = (int64_t)((p->npairs + TA_K - 1) / TA_K) * TaLayout<SPIN, NMT, 1, true>::BSTAGE;
    return per_m * (p->lmax + 1) * ((mb + NMT - 1) / NMT);
}
}  // namespace

// The plan's record buffers, one per spin, which synthesis and transpose use in
// turn: every record of a full batch, at most 1 GB for the synthesis and 4 GB
// for the transpose (whose passes each end on a nearly empty wave), and no more
// than an eighth of the device's free memory; what does not fit takes several
// passes.  The buffer is optional: it is reserved by the plan's first
// tensor-core call at this spin, after everything that the plan cannot do
// without, and where it does not hold one map group (synthesis) and one m
// (transpose), the CTAs build their own operands.  Returns whether the plan has
// it.  The calls that come here are host-synchronous (the wait flag) or captured
// in the solver's relaxed mode; the allocation runs in that mode too, so that a
// capture of another thread stands.
static bool reserve_records(Plan *p, int spin) {
    const int k = spin / 2;
    if (p->tcrec_tried[k]) return p->d_tcrec[k] != nullptr;
    p->tcrec_tried[k] = true;
    const int mb = p->max_batch;
    const int64_t cap = (int64_t)1 << 30;
    const int64_t rec = k == 1 ? TcCfg<2, 8>::REC : mb > 8 ? TcCfg<0, 16>::REC : TcCfg<0, 8>::REC;
    const int64_t groups = k == 0 && mb > 8 ? (mb + 15) / 16 : (mb + 7) / 8;
    const int64_t ana = k == 1 ? ta_record_bytes<2, 8>(p, mb)
                               : mb > 8 ? ta_record_bytes<0, 16>(p, mb)
                                        : ta_record_bytes<0, 8>(p, mb);
    const int64_t least = std::max(p->tc_nrec * rec, ana / ((p->lmax + 1) * groups));
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    size_t avail = 0, total = 0;
    const bool known = cudaMemGetInfo(&avail, &total) == cudaSuccess;
    if (!known) cudaGetLastError();
    int64_t room = known ? (int64_t)(avail / 8) : 0;
    // SHTG_TC_RECORD_BYTES: this many bytes in place of the eighth (for tests of
    // several passes and of a plan without the buffer)
    if (const char *e = getenv("SHTG_TC_RECORD_BYTES")) room = atoll(e);
    int64_t bytes = std::max(least, std::max(std::min(p->tc_nrec * rec * groups, cap), std::min(ana, 4 * cap)));
    bytes = std::min(bytes, room);
    for (; bytes >= least; bytes /= 2) {
        if (cudaMalloc((void **)&p->d_tcrec[k], (size_t)bytes) == cudaSuccess) {
            p->tcrec_bytes[k] = bytes;
            p->device_bytes += bytes;
            break;
        }
        p->d_tcrec[k] = nullptr;
        cudaGetLastError();
    }
    cudaThreadExchangeStreamCaptureMode(&mode);
    return p->d_tcrec[k] != nullptr;
}

// Synthesis: 8 maps per CTA, or 16 at spin 0 when the call has more than 8 (the
// recurrence is then generated once for all of them) and the CTAs of one map
// group are more than the SMs (N_side 64, l_max 128, 10 maps, 129 CTAs: two
// groups of 8 side by side 15.9 us, one of 16 17.0).  From records, or with the
// CTAs building each chunk's themselves; both give the same bits.  Up to two
// waves of CTAs the autotuner tries both (N_side 24, l_max 60, 5 Q/U maps: 15.8 us
// from records, 13.1 without, in calls with the ring stage; N_side 128, l_max
// 380, 1 Q/U map: 37.2 and 38.4).  Beyond, the records: each is read by more
// than one CTA, and the alm come from further away between other calls than in
// the tuner's runs (N_side 256, l_max 500, 8 Q/U maps: 125 and 117 us in the
// tuner's runs, 130 and 140 in calls).
template <int SPIN, int NMT>
static int synth_tc_shape(int v, Plan *p, const float2 *alm, int rs, int nmaps, const float *beam, float2 *F,
                          cudaStream_t st) {
    if (v == 1) return launch_synth_tc<SPIN, NMT, false>(p, alm, rs, nmaps, beam, F, st);
    return launch_synth_tc<SPIN, NMT, true>(p, alm, rs, nmaps, beam, F, st);
}
int leg_synth_tc(Plan *p, int spin, const float2 *alm, int rs, int nmaps, const float *beam, float2 *F,
                 cudaStream_t st) {
    const int64_t ctas = (int64_t)((p->npairs + TC_M - 1) / TC_M) * (p->lmax + 1);   // of a map group
    const int v0 = reserve_records(p, spin) ? 0 : 1;   // the first shape that the plan can run
    const int nv = v0 == 0 && ctas * ((nmaps + 7) / 8) > 8 * p->nsm ? 1 : 2 - v0;
    return tune(p, 2, spin == 2 ? 1 : 0, nmaps, nv, st, [&](int w) {
        const int v = v0 + w;
        if (spin == 2) return synth_tc_shape<2, 8>(v, p, alm, rs, nmaps, beam, F, st);
        if (nmaps > 8 && ctas > p->nsm)
            return synth_tc_shape<0, 16>(v, p, alm, rs, nmaps, beam, F, st);
        return synth_tc_shape<0, 8>(v, p, alm, rs, nmaps, beam, F, st);
    });
}

// Transpose: maps per CTA likewise; one or two A buffers, with records or with
// the CTAs building their own B tiles (small grids, where the records' launch
// costs more than it saves: N_side 64, l_max 128, 10 maps, spin 0, 23 against 16
// us; N_side 512, l_max 1024, 4 maps, spin 2, 0.63 against 0.69 ms), tried by the autotuner (key kind 2).  All
// sum the same products in the same order, so the choice does not change a bit of
// the result.
template <int SPIN, int NMT>
static int analysis_tc_shape(int v, Plan *p, const float2 *G, int nmaps, const float *beam, float2 *alm, int rs,
                             cudaStream_t st, int vjp) {
    switch (v) {
        case 1: return launch_analysis_tc<SPIN, NMT, 2, true>(p, G, nmaps, beam, alm, rs, st, vjp);
        case 2: return launch_analysis_tc<SPIN, NMT, 1, false>(p, G, nmaps, beam, alm, rs, st, vjp);
        case 3: return launch_analysis_tc<SPIN, NMT, 2, false>(p, G, nmaps, beam, alm, rs, st, vjp);
        default: return launch_analysis_tc<SPIN, NMT, 1, true>(p, G, nmaps, beam, alm, rs, st, vjp);
    }
}

int leg_analysis_tc(Plan *p, int spin, const float2 *G, int nmaps, const float *beam, float2 *alm, int rs,
                    cudaStream_t st, int vjp) {
    const int v0 = reserve_records(p, spin) ? 0 : 2;
    return tune(p, 2, spin == 2 ? 3 : 2, nmaps, 4 - v0, st, [&](int w) {
        const int v = v0 + w;
        if (spin == 2) return analysis_tc_shape<2, 8>(v, p, G, nmaps, beam, alm, rs, st, vjp);
        if (nmaps > 8) return analysis_tc_shape<0, 16>(v, p, G, nmaps, beam, alm, rs, st, vjp);
        return analysis_tc_shape<0, 8>(v, p, G, nmaps, beam, alm, rs, st, vjp);
    });
}

}  // namespace shtg
