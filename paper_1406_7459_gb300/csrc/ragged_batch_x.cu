// ragged_batch_x.cu -- x kernels of the batched ragged step, per class.
#include "ragged_batch.cuh"

namespace mmk {

template <int N> static RagXFns x_fns() {
    RagXFns f;
    f.p1 = k_rag_batch_pass1<N>;
    f.t1 = kRagRows1 * Fft2<N>::G;
    f.s1 = pass1_fast_smem<N, kRagRows1, true>();
    f.xs = k_rag_batch_xstep<N>;
    f.rows = rag_rows<N>();
    f.tx = XstepLayout<N, rag_rows<N>()>::THREADS;
    f.sx = XstepLayout<N, rag_rows<N>()>::BYTES;
    return f;
}

RagXFns rag_x_fns(int cls) {
    switch (cls) {
        case 0: return x_fns<16>();
        case 1: return x_fns<32>();
        case 2: return x_fns<48>();
        case 3: return x_fns<64>();
        case 4: return x_fns<96>();
        case 5: return x_fns<128>();
        case 6: return x_fns<192>();
        case 7: return x_fns<256>();
        default: return RagXFns{};
    }
}

}  // namespace mmk
