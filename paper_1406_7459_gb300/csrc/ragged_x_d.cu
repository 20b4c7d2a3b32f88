// ragged_x_d.cu -- the x kernels of ragged films: the row transform that
// starts a run, and the inverse-x + field + LLG + forward-x kernel with its
// field-only variants, carrier lengths 640 to 1024.
#include "ragged_x.cuh"

namespace mmk {

bool ragged_lookup_x_d(int N, FastStepFns* f) {
    switch (N) {
        case 640: rag_fill_x<640>(f); return true;
        case 768: rag_fill_x<768>(f); return true;
        case 1024: rag_fill_x<1024>(f); return true;
        default: return false;
    }
}

}  // namespace mmk
