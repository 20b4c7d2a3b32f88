// ragged_plane_nz2.cu -- the plane kernel of ragged films of 2 layers.
#include "ragged.cuh"

namespace mmk {

bool ragged_lookup_plane_nz2(int NY, bool many, FastStepFns* f) {
    return rag_lookup_plane_lo<2>(NY, many, f) || rag_lookup_plane_hi<2>(NY, many, f);
}

}  // namespace mmk
