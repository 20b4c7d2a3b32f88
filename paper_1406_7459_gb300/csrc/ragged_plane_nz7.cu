// ragged_plane_nz7.cu -- the plane kernel of ragged films of 7 layers.
#include "ragged.cuh"

namespace mmk {

bool ragged_lookup_plane_nz7(int NY, bool many, FastStepFns* f) {
    return rag_lookup_plane_lo<7>(NY, many, f) || rag_lookup_plane_hi<7>(NY, many, f);
}

}  // namespace mmk
