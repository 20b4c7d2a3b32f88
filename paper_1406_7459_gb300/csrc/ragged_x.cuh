// ragged_x.cuh -- x kernels of ragged films per carrier length (ragged.cuh).
#pragma once
#include "ragged.cuh"

namespace mmk {

// Rows per tile: two up to N = 256 (per L2-resident step against four rows:
// 250x250x4 18.9 against 19.4 us, 200x60x3 9.6 against 11.7, 180x180x6 22.3
// against 23.0: more blocks in flight), four above (600x400x1 28.5 against
// 36.8 us with two, 500x500x2 51.0 against 63.0: two rows leave 32-thread
// transform groups too few per block and read 16-byte runs of the spectrum)
// where their shared memory fits.
template <int N> __host__ __device__ constexpr int rag_rows() {
    return N <= 256 || XstepLayout<N, 4>::BYTES > 200 * 1024 ? 2 : 4;
}

template <int N> void rag_fill_x(FastStepFns* f) {
    constexpr int R = rag_rows<N>();
    f->kb[kModeDemag] = k_xstep_pdl<N, R, kModeDemag, true>;
    f->kb[kModeHeff] = k_xstep_pdl<N, R, kModeHeff, true>;
    f->kb[kModeStep] = k_xstep_pdl<N, R, kModeStep, true>;
    f->kst[0] = k_xstep_stage<N, R, kModeStage, true>;
    f->kst[1] = k_xstep_stage<N, R, kModeErr, true>;
    f->rb = R;
    f->tb = XstepLayout<N, R>::THREADS;
    f->sb = XstepLayout<N, R>::BYTES;
    constexpr int R1 = 4;                     // small tiles: a run's first transform is one wave
    f->p1 = k_pass1_rag<N, R1>;
    f->p1c = k_pass1_comb<N, R1, true>;
    f->r1 = R1;
    f->t1 = R1 * Fft2<N>::G;
    f->s1 = pass1_fast_smem<N, R1, true>();
}

}  // namespace mmk
