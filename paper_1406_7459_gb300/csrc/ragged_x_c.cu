// ragged_x_c.cu -- the x kernels of ragged films: the row transform that
// starts a run, and the inverse-x + field + LLG + forward-x kernel with its
// field-only variants, carrier lengths 320 to 512.
#include "ragged_x.cuh"

namespace mmk {

bool ragged_lookup_x_c(int N, FastStepFns* f) {
    switch (N) {
        case 320: rag_fill_x<320>(f); return true;
        case 384: rag_fill_x<384>(f); return true;
        case 512: rag_fill_x<512>(f); return true;
        default: return false;
    }
}

}  // namespace mmk
