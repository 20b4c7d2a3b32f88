// ragged.cuh -- carrier lengths of ragged films.
//
// A film whose sides are no powers of two runs on the compile-time kernels
// of the two-kernel step (fast_step.cuh, RAG) with each side carried in the
// smallest length N >= n that has a compile-time transform: any padded
// length >= 2n - 1 gives the exact linear convolution (Sec. 2), so the rows
// and lines are zero past the sample and the outputs past it are dropped.
// Lengths between the powers of two (3 and 5 times a power of two) keep the
// waste of a carried side below a half, and below a third above 256.
//
// The general mixed-radix kernels transform the whole padded line in three
// or four shared-memory stages with a block barrier, an index computation
// and a twiddle load per stage; here a line is two unpadded register
// transforms with one exchange.  Bound by the latency of two single-wave
// kernels on small films and by shared memory and the FP32 pipes on large
// ones, like the power-of-two step.  Per L2-resident Euler step, general
// kernels against these: 200x60x3 25 against 9.6 us, 600x400x1 field
// evaluation and stage 55 against 34 us.
#pragma once
#include "fast_step.cuh"

namespace mmk {

constexpr int kRagLens[] = {16, 32, 48, 64, 96, 128, 192, 256, 320, 384, 512, 640, 768, 1024};

// The smallest carrier length >= n, or 0.
inline int ragged_len(int n) {
    for (int N : kRagLens)
        if (n <= N) return N;
    return 0;
}

// Plane kernels exist where a plane's threads and shared memory fit.
template <int NY, int NZ> constexpr bool rag_plane_fits() {
    return PlaneLayout<NY, NZ>::THREADS <= 768 && PlaneLayout<NY, NZ>::BYTES <= 227 * 1024;
}

template <int NY, int NZ> bool rag_fill_plane(FastStepFns* f) {
    if constexpr (rag_plane_fits<NY, NZ>()) {
        f->ka = k_plane_pdl<NY, NZ, true>;
        f->ta = PlaneLayout<NY, NZ>::THREADS;
        f->sa = PlaneLayout<NY, NZ>::BYTES;
        return true;
    } else {
        return false;
    }
}

// NZ layers, carrier NY, for the lengths of [0, 7) or [7, 14) of kRagLens
template <int NZ> bool rag_lookup_plane_lo(int NY, FastStepFns* f) {
    switch (NY) {
        case 16: return rag_fill_plane<16, NZ>(f);
        case 32: return rag_fill_plane<32, NZ>(f);
        case 48: return rag_fill_plane<48, NZ>(f);
        case 64: return rag_fill_plane<64, NZ>(f);
        case 96: return rag_fill_plane<96, NZ>(f);
        case 128: return rag_fill_plane<128, NZ>(f);
        case 192: return rag_fill_plane<192, NZ>(f);
        default: return false;
    }
}
template <int NZ> bool rag_lookup_plane_hi(int NY, FastStepFns* f) {
    switch (NY) {
        case 256: return rag_fill_plane<256, NZ>(f);
        case 320: return rag_fill_plane<320, NZ>(f);
        case 384: return rag_fill_plane<384, NZ>(f);
        case 512: return rag_fill_plane<512, NZ>(f);
        case 640: return rag_fill_plane<640, NZ>(f);
        case 768: return rag_fill_plane<768, NZ>(f);
        case 1024: return rag_fill_plane<1024, NZ>(f);
        default: return false;
    }
}

}  // namespace mmk
