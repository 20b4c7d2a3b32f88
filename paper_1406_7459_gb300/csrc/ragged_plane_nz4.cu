// ragged_plane_nz4.cu -- the plane kernel of ragged films of 4 layers.
#include "ragged.cuh"

namespace mmk {

bool ragged_lookup_plane_nz4(int NY, bool many, FastStepFns* f) {
    return rag_lookup_plane_lo<4>(NY, many, f) || rag_lookup_plane_hi<4>(NY, many, f);
}

}  // namespace mmk
