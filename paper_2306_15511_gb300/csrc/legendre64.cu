// FP64 Legendre synthesis: maps per pass by the number of maps.
#include "legendre_blk.cuh"

namespace shtg {

// small grids (legendre_g64.cu)
bool leg_synth_seg_fits(const Plan *p, int groups);
int leg_synth_seg(Plan *p, int spin, int nm, const double2 *alm, int rs, int nmaps, const double *beam, double2 *F,
                  cudaStream_t st);

// Maps per pass: the FP64 pipe bounds this kernel (a warp instruction takes
// 64 cycles of its scheduler's FP64 unit), and a pass over NM maps costs
// R + W NM multiply-adds per (l, m, ring pair), whether or not all NM are
// there: the recurrence (R = 3, spin 2: 8) and the sums (W = 2, spin 2: 8).
// The pass count times that cost is smallest for the NM taken here.
int leg_maps_per_pass(int spin, int nmaps, const int *nms, int n) {
    const int R = spin == 2 ? 8 : 3, W = spin == 2 ? 8 : 2;
    int best = nms[0];
    long long cost = -1;
    for (int i = 0; i < n; ++i) {
        const long long c = (long long)((nmaps + nms[i] - 1) / nms[i]) * (R + W * nms[i]);
        if (cost < 0 || c < cost) {
            cost = c;
            best = nms[i];
        }
    }
    return best;
}

// One ring pair per thread: with two the kernel is 1.05 to 1.5 times slower
// (N_side 512, l_max 1024, 8 maps: 12.8 against 13.7 ms at spin 0, 54.3
// against 59.0 ms at spin 2; N_side 300, one map: 0.61 against 0.93 ms).
// Before, at most four maps shared a recurrence and none of the shapes was
// made for one or three maps (N_side 32, l_max 64, one map: 51 us, with this
// kernel 15.5; such small grids now take the segment kernel, 11.4).
// At spin 2 and two or more maps the autotuner may take another shape: where the
// grid is a wave and a bit, a shape with more or smaller CTAs can win (304
// Gauss-Legendre rings, l_max 300, 4 maps: four maps per pass 1.31 ms with the
// ring stage, the tuned shape 1.09).  No shape changes a bit of the result.
static int leg_synth64_count(const Plan *p, int spin, int nmaps, int nm) {
    return spin == 2 && nmaps > 1 && !leg_synth_seg_fits(p, (nmaps + nm - 1) / nm) ? 4 : 1;
}
static int leg_synth64_shape(Plan *p, int spin, int v, int nm, const double2 *alm, int rs, int nmaps,
                             const double *beam, double2 *F, cudaStream_t st) {
    if (v == 1) return launch_synth_v<double, 2, 2, 2>(p, alm, rs, nmaps, beam, F, st);
    if (v == 2) return launch_synth_v<double, 2, 1, 2>(p, alm, rs, nmaps, beam, F, st);
    if (v == 3) return launch_synth_v<double, 2, 2, 1>(p, alm, rs, nmaps, beam, F, st);
    if ((spin == 0 || p->d_tst64_2) && leg_synth_seg_fits(p, (nmaps + nm - 1) / nm))
        return leg_synth_seg(p, spin, nm, alm, rs, nmaps, beam, F, st);
    if (spin == 2) {
        switch (nm) {
            case 1: return launch_synth_v<double, 2, 1, 1>(p, alm, rs, nmaps, beam, F, st);
            case 2: return launch_synth_v<double, 2, 1, 2>(p, alm, rs, nmaps, beam, F, st);
            case 3: return launch_synth_v<double, 2, 1, 3>(p, alm, rs, nmaps, beam, F, st);
            default: return launch_synth_v<double, 2, 1, 4>(p, alm, rs, nmaps, beam, F, st);
        }
    }
    switch (nm) {
        case 1: return launch_synth_v<double, 0, 1, 1>(p, alm, rs, nmaps, beam, F, st);
        case 2: return launch_synth_v<double, 0, 1, 2>(p, alm, rs, nmaps, beam, F, st);
        case 3: return launch_synth_v<double, 0, 1, 3>(p, alm, rs, nmaps, beam, F, st);
        case 4: return launch_synth_v<double, 0, 1, 4>(p, alm, rs, nmaps, beam, F, st);
        case 6: return launch_synth_v<double, 0, 1, 6>(p, alm, rs, nmaps, beam, F, st);
        default: return launch_synth_v<double, 0, 1, 8>(p, alm, rs, nmaps, beam, F, st);
    }
}

static int synth64_nm(int spin, int nmaps) {
    static const int nm0[] = {8, 6, 4, 3, 2, 1}, nm2[] = {4, 3, 2, 1};
    return spin == 2 ? leg_maps_per_pass(2, nmaps, nm2, 4) : leg_maps_per_pass(0, nmaps, nm0, 6);
}
int leg_synth_g64(Plan *p, int spin, const double2 *alm, int rs, int nmaps, const double *beam, double2 *F,
                  cudaStream_t st) {
    return leg_synth64_shape(p, spin, 0, synth64_nm(spin, nmaps), alm, rs, nmaps, beam, F, st);
}
template <>
int leg_synth<double>(Plan *p, int spin, const double2 *alm, int rs, int nmaps, const double *beam, double2 *F,
                      cudaStream_t st) {
    const int nm = synth64_nm(spin, nmaps);
    return tune(p, 0, spin == 2 ? 1 : 0, nmaps, leg_synth64_count(p, spin, nmaps, nm), st,
                [&](int v) { return leg_synth64_shape(p, spin, v, nm, alm, rs, nmaps, beam, F, st); });
}

// Transpose: the register-blocked contraction, or (spin 0, one CTA per m and no
// atomic additions) the warp-reduction kernels, which fill the chip better where
// the contraction's 128-l tiles leave a ragged last wave (N_side 128, l_max 256, 5
// maps, with the ring stage: 0.92 ms, the tuned kernel 0.63); the autotuner decides.
template <>
int leg_analysis<double>(Plan *p, int spin, const double2 *G, int nmaps, const double *beam, double2 *alm, int rs,
                         cudaStream_t st, int vjp) {
    const bool small = (int64_t)((p->lmax + B_LR) / B_LR) * (p->lmax + 1) <= p->nsm;
    const int n = spin == 2 || small || p->npairs > 4 * LEG_THREADS ? 1 : p->npairs > 2 * LEG_THREADS ? 2 : 4;
    return tune(p, 0, spin == 2 ? 3 : 2, nmaps, n, st, [&](int v) {
        if (v == 1) return launch_analysis_v<double, 0, 4, 1>(p, G, nmaps, beam, alm, rs, st, vjp);
        if (v == 2) return launch_analysis_v<double, 0, 2, 1>(p, G, nmaps, beam, alm, rs, st, vjp);
        if (v == 3) return launch_analysis_v<double, 0, 2, 2>(p, G, nmaps, beam, alm, rs, st, vjp);
        return leg_analysis_g64(p, spin, G, nmaps, beam, alm, rs, st, vjp);
    });
}

}  // namespace shtg
