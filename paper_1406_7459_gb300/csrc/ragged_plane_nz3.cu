// ragged_plane_nz3.cu -- the plane kernel of ragged films of 3 layers.
#include "ragged.cuh"

namespace mmk {

bool ragged_lookup_plane_nz3(int NY, bool many, FastStepFns* f) {
    return rag_lookup_plane_lo<3>(NY, many, f) || rag_lookup_plane_hi<3>(NY, many, f);
}

}  // namespace mmk
