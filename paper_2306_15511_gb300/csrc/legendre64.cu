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
// made for one or three maps (N_side 32, l_max 64, one map: 51 us, now 21).
template <>
int leg_synth<double>(Plan *p, int spin, const double2 *alm, int rs, int nmaps, const double *beam, double2 *F,
                      cudaStream_t st) {
    static const int nm0[] = {8, 6, 4, 3, 2, 1}, nm2[] = {4, 3, 2, 1};
    const int nm = spin == 2 ? leg_maps_per_pass(2, nmaps, nm2, 4) : leg_maps_per_pass(0, nmaps, nm0, 6);
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

}  // namespace shtg
