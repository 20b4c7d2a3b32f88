// ragged_batch_planes.cu -- plane kernels of the batched ragged step, per class.
#include "ragged_batch.cuh"

namespace mmk {

template <int NY, int NZ> static RagPlaneFns plane_fns() {
    RagPlaneFns f;
    f.k = k_rag_batch_plane<NY, NZ>;
    f.t = PlaneLayout<NY, NZ>::THREADS;
    f.smem = PlaneLayout<NY, NZ>::BYTES;
    return f;
}

RagPlaneFns rag_plane_fns(int cls) {
    switch (cls) {
        case 0: return plane_fns<16, 1>();
        case 1: return plane_fns<16, 2>();
        case 2: return plane_fns<16, 3>();
        case 3: return plane_fns<16, 4>();
        case 4: return plane_fns<32, 1>();
        case 5: return plane_fns<32, 2>();
        case 6: return plane_fns<32, 3>();
        case 7: return plane_fns<32, 4>();
        case 8: return plane_fns<48, 1>();
        case 9: return plane_fns<48, 2>();
        case 10: return plane_fns<48, 3>();
        case 11: return plane_fns<48, 4>();
        case 12: return plane_fns<64, 1>();
        case 13: return plane_fns<64, 2>();
        case 14: return plane_fns<64, 3>();
        case 15: return plane_fns<64, 4>();
        case 16: return plane_fns<96, 1>();
        case 17: return plane_fns<96, 2>();
        case 18: return plane_fns<128, 1>();
        case 19: return plane_fns<128, 2>();
        case 20: return plane_fns<192, 1>();
        case 21: return plane_fns<192, 2>();
        case 22: return plane_fns<256, 1>();
        case 23: return plane_fns<256, 2>();
        default: return RagPlaneFns{};
    }
}

}  // namespace mmk
