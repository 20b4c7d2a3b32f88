// ragged_plane_nz1.cu -- the plane kernel of ragged films of 1 layer.
#include "ragged.cuh"

namespace mmk {

bool ragged_lookup_plane_nz1(int NY, bool many, FastStepFns* f) {
    return rag_lookup_plane_lo<1>(NY, many, f) || rag_lookup_plane_hi<1>(NY, many, f);
}

}  // namespace mmk
