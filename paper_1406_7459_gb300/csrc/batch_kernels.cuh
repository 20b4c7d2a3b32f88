// batch_kernels.cuh -- what the batched kernels share (batch.cu,
// batch_persist.cu): the descriptor of a sample on the general kernels, its
// lookup, and the plane tile.
#pragma once
#include "pass_bodies.cuh"
#include "plane_kernel.cuh"
#include "ragged_batch.cuh"

namespace mmk {

struct BatchDesc {
    Geom g;
    LlgCoef cf;
    float* M0;
    float* M1;
    float2* S;
    int r1, r3;
    int r2;                                   // kx planes per plane-pass CTA
};

__device__ __forceinline__ int find_sample(const int* __restrict__ pre, int ns, int b) {
    int lo = 0, hi = ns - 1;                  // largest s with pre[s] <= b
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(pre + mid) <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// plane-pass tile `tile` of a sample: r2 consecutive kx planes (fewer at
// the end), all their lines transformed together
__device__ __forceinline__ void batch_plane_tile(const BatchDesc& b, int tile) {
    const int kx0 = tile * b.r2;
    const int np = min(b.r2, b.g.Hx - kx0);
    const int nl = 3 * b.g.nz * np;
    switch (b.g.Lz) {
        case 1: plane_body_multi<1>(b.g, nl, b.S, kx0, np); break;
        case 4: plane_body_multi<4>(b.g, nl, b.S, kx0, np); break;
        case 5: plane_body_multi<5>(b.g, nl, b.S, kx0, np); break;
        default: plane_body_multi<8>(b.g, nl, b.S, kx0, np); break;
    }
}

// Work of one pass of a batch: the items of the ragged classes, then the
// tiles of the samples on the general kernels (prefix table `pre`).
struct BatchPass {
    const RagItem* items;
    const int* pre;
    int n_items, n_tiles;
};

// The persistent launch (batch_persist.cu).
struct GridBar;
typedef void (*BatchPersistFn)(const BatchDesc*, const RagDesc*, BatchPass, BatchPass, BatchPass, int, int, int, float,
                               int, int*, GridBar*, long long);
BatchPersistFn batch_persist_fn();

}  // namespace mmk
