// ragged.cuh -- carrier lengths of ragged films.
//
// A film whose sides are no powers of two runs on the compile-time kernels
// of the two-kernel step (fast_step.cuh, RAG) with each side carried in the
// smallest length N >= n that has a compile-time transform: any padded
// length >= 2n - 1 gives the exact linear convolution (Sec. 2), so the rows
// and lines are zero past the sample and the outputs past it are dropped.
// Lengths between the powers of two (3 and 5 times a power of two) keep the
// waste of a carried side of more than 8 cells below a half, and below a third
// above 256.  Shorter sides, single rows and columns among them, are carried in 16
// all the same: what they waste is less than the general kernels' barriers
// cost (per L2-resident Euler step, general kernels against these: 600x1x1
// 18.5 against 13.1 us, 1x200x2 15.9 against 6.0, 5x5x5 14.9 against 4.9,
// 1x1x100 16.6 against 14.6, 2x2x1 7.6 against 4.0).  The nearest are single
// columns of one layer, whose general kernels transform nothing along x: 1x32x1 4.1
// against 4.4, 1x64x1 4.4 against 4.5, 1x128x1 4.9 against 4.7, and an RK4
// step of them 25 against 17.
//
// The general mixed-radix kernels transform the whole padded line in three
// or four shared-memory stages with a block barrier, an index computation
// and a twiddle load per stage; here a line is two unpadded register
// transforms with one exchange.  Bound by the latency of two single-wave
// kernels on small films and by shared memory and the FP32 pipes on large
// ones, like the power-of-two step.  Per L2-resident Euler step, general
// kernels against these: 200x60x3 22.0 against 9.5 us, 300x300x3 52.8 against
// 42.9, 1000x1000x1 174.6 against 105.1, an RK4 step of it 756 against 405.
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

// k_plane_pdl exists where a plane's threads and shared memory fit, the
// large-plane kernel for transform groups of a warp where its lines fit.
template <int NY, int NZ> constexpr bool rag_plane_fits() {
    return PlaneLayout<NY, NZ>::THREADS <= 768 && PlaneLayout<NY, NZ>::BYTES <= 227 * 1024;
}
template <int NY, int NZ> constexpr bool big_plane_fits() {
    if constexpr (Fft2<NY>::G == 32) return BigPlane<NY, NZ>::BYTES <= 226 * 1024;
    else return false;
}

// many: the planes fill the SMs (kBigPlanes).  Then the large-plane kernel
// takes the planes of more than 512 threads, whose registers spill in
// k_plane_pdl, and those that do not fit it.  With fewer planes these stay on
// k_plane_pdl or on the split pass, which is the better side for the widest
// planes (per L2-resident Euler step, as it is against the large-plane kernel:
// 64x512x8 24.5 against 32.3 us, 20x400x6 15.5 against 26.1) but not for four
// and five layers (128x512x4 25.8 against 21.6, 64x640x4 33.6 against 22.4,
// 100x400x5 38.6 against 30.0).
template <int NY, int NZ> bool rag_fill_plane(bool many, FastStepFns* f) {
    if constexpr (big_plane_fits<NY, NZ>() &&
                  (PlaneLayout<NY, NZ>::THREADS > 512 || !rag_plane_fits<NY, NZ>())) {
        if (many) {
            f->ka = k_plane_big<NY, NZ, true>;
            f->ta = BigPlane<NY, NZ>::THREADS;
            f->sa = BigPlane<NY, NZ>::BYTES;
            f->big = true;
            return true;
        }
    }
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
template <int NZ> bool rag_lookup_plane_lo(int NY, bool many, FastStepFns* f) {
    switch (NY) {
        case 16: return rag_fill_plane<16, NZ>(many, f);
        case 32: return rag_fill_plane<32, NZ>(many, f);
        case 48: return rag_fill_plane<48, NZ>(many, f);
        case 64: return rag_fill_plane<64, NZ>(many, f);
        case 96: return rag_fill_plane<96, NZ>(many, f);
        case 128: return rag_fill_plane<128, NZ>(many, f);
        case 192: return rag_fill_plane<192, NZ>(many, f);
        default: return false;
    }
}
template <int NZ> bool rag_lookup_plane_hi(int NY, bool many, FastStepFns* f) {
    switch (NY) {
        case 256: return rag_fill_plane<256, NZ>(many, f);
        case 320: return rag_fill_plane<320, NZ>(many, f);
        case 384: return rag_fill_plane<384, NZ>(many, f);
        case 512: return rag_fill_plane<512, NZ>(many, f);
        case 640: return rag_fill_plane<640, NZ>(many, f);
        case 768: return rag_fill_plane<768, NZ>(many, f);
        case 1024: return rag_fill_plane<1024, NZ>(many, f);
        default: return false;
    }
}

}  // namespace mmk
