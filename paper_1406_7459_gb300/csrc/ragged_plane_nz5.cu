// ragged_plane_nz5.cu -- the plane kernel of ragged films of 5 layers.
#include "ragged.cuh"

namespace mmk {

bool ragged_lookup_plane_nz5(int NY, bool many, FastStepFns* f) {
    return rag_lookup_plane_lo<5>(NY, many, f) || rag_lookup_plane_hi<5>(NY, many, f);
}

}  // namespace mmk
