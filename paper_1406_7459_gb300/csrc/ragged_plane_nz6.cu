// ragged_plane_nz6.cu -- the plane kernel of ragged films of 6 layers.
#include "ragged.cuh"

namespace mmk {

bool ragged_lookup_plane_nz6(int NY, bool many, FastStepFns* f) {
    return rag_lookup_plane_lo<6>(NY, many, f) || rag_lookup_plane_hi<6>(NY, many, f);
}

}  // namespace mmk
