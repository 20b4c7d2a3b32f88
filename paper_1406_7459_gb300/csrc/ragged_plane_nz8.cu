// ragged_plane_nz8.cu -- the plane kernel of ragged films of 8 layers.
#include "ragged.cuh"

namespace mmk {

bool ragged_lookup_plane_nz8(int NY, bool many, FastStepFns* f) {
    return rag_lookup_plane_lo<8>(NY, many, f) || rag_lookup_plane_hi<8>(NY, many, f);
}

}  // namespace mmk
