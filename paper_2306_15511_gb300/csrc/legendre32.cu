// FP32 Legendre kernel shapes (ring pairs per thread, maps per pass) for the
// autotuner.  The candidates follow the number of maps, so that no pass
// multiplies maps that are not there (at one map a pass over two maps issues
// 11 instructions per (l, ring pair), one over a single map 5.5); the first is
// the one kept without tuning.  Every shape of the synthesis gives the same
// bits.  N_side 512, l_max 1024, one map: synthesis 189 -> 132 us, transpose
// 259 -> 222 us (with the pairs of a warp consecutive, load_pairs).
#include "legendre_kernels.cuh"

namespace shtg {
namespace {

typedef int (*SynthFn)(Plan *, const float2 *, int, int, const float *, float2 *, cudaStream_t);
typedef int (*AnaFn)(Plan *, const float2 *, int, const float *, float2 *, int, cudaStream_t, int);
template <typename Fn> struct Shapes {
    int n;
    Fn fn[4];
};
#define SV(SP, NR, NM) &launch_synth_v<float, SP, NR, NM>
#define AV(SP, NR, NM) &launch_analysis_v<float, SP, NR, NM>

// by the number of maps: 1, 2, 3 and more
const Shapes<SynthFn> &synth_shapes(int spin, int nmaps) {
    static const Shapes<SynthFn> s0[3] = {{4, {SV(0, 4, 1), SV(0, 8, 1), SV(0, 2, 1), SV(0, 1, 1)}},
                                          {3, {SV(0, 4, 2), SV(0, 2, 2), SV(0, 1, 2)}},
                                          {4, {SV(0, 4, 2), SV(0, 4, 4), SV(0, 2, 4), SV(0, 8, 2)}}};
    static const Shapes<SynthFn> s2[3] = {{3, {SV(2, 2, 1), SV(2, 4, 1), SV(2, 1, 1)}},
                                          {3, {SV(2, 2, 2), SV(2, 1, 2), SV(2, 2, 1)}},
                                          {4, {SV(2, 2, 2), SV(2, 2, 1), SV(2, 4, 1), SV(2, 1, 4)}}};
    return (spin == 2 ? s2 : s0)[nmaps >= 3 ? 2 : nmaps - 1];
}
const Shapes<AnaFn> &ana_shapes(int spin, int nmaps) {
    static const Shapes<AnaFn> a0[3] = {{4, {AV(0, 8, 1), AV(0, 4, 1), AV(0, 2, 1), AV(0, 1, 1)}},
                                        {4, {AV(0, 4, 2), AV(0, 8, 2), AV(0, 8, 1), AV(0, 2, 2)}},
                                        {4, {AV(0, 4, 2), AV(0, 8, 1), AV(0, 8, 2), AV(0, 6, 2)}}};
    static const Shapes<AnaFn> a2[3] = {{3, {AV(2, 4, 1), AV(2, 2, 1), AV(2, 1, 1)}},
                                        {4, {AV(2, 2, 2), AV(2, 4, 1), AV(2, 4, 2), AV(2, 1, 2)}},
                                        {4, {AV(2, 2, 2), AV(2, 4, 1), AV(2, 3, 2), AV(2, 4, 2)}}};
    return (spin == 2 ? a2 : a0)[nmaps >= 3 ? 2 : nmaps - 1];
}

}  // namespace

int leg_synth32_count(int spin, int nmaps) { return synth_shapes(spin, nmaps).n; }
int leg_synth32_shape(Plan *p, int spin, int v, const float2 *alm, int rs, int nmaps, const float *beam, float2 *F,
                      cudaStream_t st) {
    return synth_shapes(spin, nmaps).fn[v](p, alm, rs, nmaps, beam, F, st);
}
int leg_analysis32_count(int spin, int nmaps) { return ana_shapes(spin, nmaps).n; }
int leg_analysis32_shape(Plan *p, int spin, int v, const float2 *G, int nmaps, const float *beam, float2 *alm, int rs,
                         cudaStream_t st, int vjp) {
    return ana_shapes(spin, nmaps).fn[v](p, G, nmaps, beam, alm, rs, st, vjp);
}

}  // namespace shtg
