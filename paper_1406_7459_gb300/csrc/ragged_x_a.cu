// ragged_x_a.cu -- the x kernels of ragged films: the row transform that
// starts a run, and the inverse-x + field + LLG + forward-x kernel with its
// field-only variants, carrier lengths 16 to 96.
#include "ragged_x.cuh"

namespace mmk {

bool ragged_lookup_x_a(int N, FastStepFns* f) {
    switch (N) {
        case 16: rag_fill_x<16>(f); return true;
        case 32: rag_fill_x<32>(f); return true;
        case 48: rag_fill_x<48>(f); return true;
        case 64: rag_fill_x<64>(f); return true;
        case 96: rag_fill_x<96>(f); return true;
        default: return false;
    }
}

}  // namespace mmk
