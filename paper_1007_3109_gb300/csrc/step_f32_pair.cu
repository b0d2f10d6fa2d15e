// Temporal blocking to depth K with two columns per lane: the single-grid
// launch variants (the kernel is in step_f32_pair_kernel.cuh).
#include "step_f32_pair_kernel.cuh"

namespace lbrd {

namespace {

template <int K, int NW, int NS, int MINB, bool PP, bool ANY = false, bool EA = false, int SML = 0>
cudaError_t dispatch_pair(int Q, int S, const StepArgs &a, cudaStream_t st) {
    if (Q == 9 && S == 1) return launch_pair<9, 1, K, NW, NS, MINB, PP, ANY, EA, SML>(a, st);
    if (Q == 9 && S == 2) return launch_pair<9, 2, K, NW, NS, MINB, PP, ANY, EA, SML>(a, st);
    if (Q == 5 && S == 1) return launch_pair<5, 1, K, NW, NS, MINB, PP, ANY, EA, SML>(a, st);
    if (Q == 5 && S == 2) return launch_pair<5, 2, K, NW, NS, MINB, PP, ANY, EA, SML>(a, st);
    return cudaErrorInvalidValue;
}

// Levels SML in shared memory and rows staged early (EA) for two D2Q9 species only,
// which spill without; the other kernels pull from earlier rows first (PP).
template <int K, int NW, int NS, int MINB, bool PP, bool ANY, bool EA, int SML>
cudaError_t dispatch_pair2(int Q, int S, const StepArgs &a, cudaStream_t st) {
    if (Q == 9 && S == 2) return launch_pair<9, 2, K, NW, NS, MINB, false, ANY, EA, SML>(a, st);
    if (Q == 9 && S == 1) return launch_pair<9, 1, K, NW, NS, MINB, PP, ANY>(a, st);
    if (Q == 5 && S == 1) return launch_pair<5, 1, K, NW, NS, MINB, PP, ANY>(a, st);
    if (Q == 5 && S == 2) return launch_pair<5, 2, K, NW, NS, MINB, PP, ANY>(a, st);
    return cudaErrorInvalidValue;
}

}  // namespace

// K time steps per launch, two columns per lane.  v: depth and launch shape.
cudaError_t launch_step_f32_pair(int v, int Q, int S, const StepArgs &a, cudaStream_t st) {
    switch (v) {
        case 0: return dispatch_pair<4, 4, 2, 2, false>(Q, S, a, st);
        case 1: return dispatch_pair<4, 4, 2, 2, true>(Q, S, a, st);
        case 2: return dispatch_pair<4, 4, 3, 2, false>(Q, S, a, st);
        case 3: return dispatch_pair<4, 4, 3, 2, true>(Q, S, a, st);
        case 4: return dispatch_pair2<5, 4, 2, 2, false, false, true, 4>(Q, S, a, st);
        case 5: return dispatch_pair<5, 4, 2, 2, true>(Q, S, a, st);
        case 6: return dispatch_pair<6, 4, 2, 1, true>(Q, S, a, st);
        case 7: return dispatch_pair<4, 2, 3, 4, true>(Q, S, a, st);
        case 8: return dispatch_pair<3, 4, 3, 2, true>(Q, S, a, st);
        case 9: return dispatch_pair<5, 4, 3, 2, true>(Q, S, a, st);
        case 10: return dispatch_pair<5, 4, 3, 2, false>(Q, S, a, st);
        // any nx
        case 11: return dispatch_pair<5, 4, 2, 2, true, true>(Q, S, a, st);
        case 12: return dispatch_pair<4, 4, 2, 2, false, true>(Q, S, a, st);
        case 13: return dispatch_pair<6, 4, 2, 1, true, true>(Q, S, a, st);
        case 14: return dispatch_pair<3, 4, 3, 2, true, true>(Q, S, a, st);
        // more rows staged ahead (two to four): the smaller D2Q5 rows leave L1 its share
        case 15: return dispatch_pair<6, 4, 3, 1, true>(Q, S, a, st);
        case 16: return dispatch_pair<6, 4, 5, 1, true>(Q, S, a, st);
        case 17: return dispatch_pair<5, 4, 4, 2, false>(Q, S, a, st);
        // eight warps per block, one block per SM: the SM's warps walk eight adjacent strips
        case 18: return dispatch_pair2<5, 8, 2, 1, false, false, true, 4>(Q, S, a, st);
        case 19: return dispatch_pair<6, 8, 3, 1, true>(Q, S, a, st);
        case 20: return dispatch_pair2<5, 8, 2, 1, true, true, false, 4>(Q, S, a, st);
        // a row staged as soon as level 1 has read the oldest one (one more row in flight;
        // D2Q5: the D2Q9 forms are slower so)
        case 21: return dispatch_pair<6, 4, 3, 1, true, false, true>(Q, S, a, st);
        // three rows in flight: grids that stay in L2 (320 x 256 2.15 us per step against 2.26 for the
        // best K = 5 form, 512^2 3.26 / 3.23, 768^2 4.89 / 5.27)
        case 22: return dispatch_pair<4, 4, 3, 1, true, false, true>(Q, S, a, st);
        // level 4's rows in shared memory (the any-nx form stages late: early, its spills took 1531 x 1021
        // from 12.4 to 18.7 us; 11.3 now)
        case 23: return dispatch_pair<6, 8, 2, 1, false, false, true, 8>(Q, S, a, st);
        case 24: return dispatch_pair<6, 4, 2, 2, false, false, false, 8>(Q, S, a, st);
        case 25: return dispatch_pair<6, 8, 2, 1, false, true, false, 8>(Q, S, a, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbrd
