// fast_step_plane_big.cu -- the large-plane kernel of power-of-two films.
#include "fast_step.cuh"

namespace mmk {

template <int NY, int NZ>
static bool fill_big(FastStepFns* f) {
    static_assert(BigPlane<NY, NZ>::BYTES <= 226 * 1024, "shared memory of a plane");
    f->ka = k_plane_big<NY, NZ>;
    f->ta = BigPlane<NY, NZ>::THREADS;
    f->sa = BigPlane<NY, NZ>::BYTES;
    f->big = true;
    return true;
}

bool fast_step_lookup_plane_big(int ny, int nz, FastStepFns* f) {
    if (ny == 512 && nz == 4) return fill_big<512, 4>(f);
    if (ny == 512 && nz == 8) return fill_big<512, 8>(f);
    if (ny == 1024 && nz == 4) return fill_big<1024, 4>(f);
    return false;
}

}  // namespace mmk
