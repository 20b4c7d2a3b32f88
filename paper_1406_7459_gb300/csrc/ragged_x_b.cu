// ragged_x_b.cu -- the x kernels of ragged films: the row transform that
// starts a run, and the inverse-x + field + LLG + forward-x kernel with its
// field-only variants, carrier lengths 128 to 256.
#include "ragged_x.cuh"

namespace mmk {

bool ragged_lookup_x_b(int N, FastStepFns* f) {
    switch (N) {
        case 128: rag_fill_x<128>(f); return true;
        case 192: rag_fill_x<192>(f); return true;
        case 256: rag_fill_x<256>(f); return true;
        default: return false;
    }
}

}  // namespace mmk
