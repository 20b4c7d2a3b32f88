// ragged_batch.cuh -- the batched step on the ragged-film kernels.
//
// Samples whose sides have carrier lengths (ragged.cuh) and whose plane and
// x blocks stay within 256 threads step on the bodies of the two-kernel step
// (fast_step.cuh, RAG), in place on their spectra: a plane block reads its
// whole kx plane before it writes it, an x tile its rows of every plane.
// Samples are grouped by class, the (NY, NZ) of the plane kernel and the N of
// the x kernels; each class is one launch over a list of (sample, tile)
// items, the classes of a pass side by side.  The same tile functions serve
// the persistent launch (any block size that holds the tile's groups).
//
// The item lists replace the search for a block's sample in a prefix table.
// 512 samples of 16..256 x 16..64 x 1..2 cells, per step: general kernels
// 2.18 ms as created and 0.84 ms with autotuned tiles, these 0.37 ms (0.19
// in planes, 0.18 in x tiles, each many waves of small blocks bound by the
// latency of their copy, transform and barrier chains).  The class border is
// the 256-thread block of the persistent launch.
#pragma once
#include "ragged_x.cuh"

namespace mmk {

// One sample as the tile functions need it.
struct RagDesc {
    int nx, ny, nz, N, Jst;
    int xcls, pcls;            // classes of the x and plane kernels; -1: on the general kernels
    const float2 *twx, *twy;
    const float* Kd;
    float* M[2];
    float2* S;
    LlgCoef cf;
};
struct RagItem {
    int s, tile;
};

constexpr int kRagBatchThreads = 256;      // block of the persistent launch

__device__ __forceinline__ Geom rag_geom(const RagDesc& d) {
    Geom g;
    g.nx = d.nx;
    g.ny = d.ny;
    g.nz = d.nz;
    g.N = d.N;
    g.Jst = d.Jst;
    g.Jr = d.Jst;
    g.twx = d.twx;
    g.twy = d.twy;
    return g;
}

// Plane kx of a sample.  The barriers are initialised here and invalidated
// at the end, so the function can run again in the same block; false,
// uniformly over the block, when a copy wait gave up (nothing is written
// then, and the barriers stay: the block must not run a plane again).
template <int NY, int NZ, int T>
__device__ __forceinline__ bool rag_plane_tile(const RagDesc& d, int kx, int* __restrict__ flag) {
    using Lay = PlaneLayout<NY, NZ>;
    using F = Fft2<NY>;
    constexpr int Q = F::Q, LY = Lay::LY, ZS = Lay::ZS, NL = Lay::NL;
    extern __shared__ __align__(16) float2 sm[];
    __shared__ __align__(8) uint64_t bars[3];             // twiddles, S lines, spectrum slice
    float2* tw = sm + Lay::TW_OFF;
    float2* ta = sm + Lay::TA_OFF;
    float* Ks = reinterpret_cast<float*>(sm + Lay::KT_OFF);
    float2* zb = sm + Lay::WORK_OFF;
    const Geom g = rag_geom(d);
    const uint32_t b_tw = smem_addr(&bars[0]), b_s = smem_addr(&bars[1]), b_k = smem_addr(&bars[2]);
    if (threadIdx.x == 0) {
        mbar_init(b_tw, 1);
        mbar_init(b_s, 1);
        mbar_init(b_k, 1);
        mbar_init_fence();
        proxy_fence_shared();                             // the block's earlier tiles used this memory
        proxy_fence_global();                             // S came from ordinary stores
        const float2* plane = d.S + (size_t)kx * NL * g.Jst;
        const uint32_t ln = (uint32_t)(g.Jst * sizeof(float2));
        mbar_expect_tx(b_s, NL * ln);
#pragma unroll 1
        for (int l = 0; l < NL; ++l) bulk_g2s(smem_addr(zb + l * ZS), plane + (size_t)l * g.Jst, ln, b_s);
        mbar_expect_tx(b_tw, LY * sizeof(float2));
        bulk_g2s(smem_addr(tw), g.twy, LY * sizeof(float2), b_tw);
        mbar_expect_tx(b_k, Lay::KT_FLOATS * sizeof(float));
        bulk_g2s(smem_addr(Ks), d.Kd + (size_t)kx * Lay::KT_FLOATS, Lay::KT_FLOATS * sizeof(float), b_k);
    }
    __syncthreads();
    const bool ok = mbar_wait(b_tw, 0);
    if (ok) fill_ta<NY, Q, T>(ta, tw);
    if (!plane_body<NY, NZ, T, true>(g, kx, ok, tw, ta, Ks, zb, b_s, 0, b_k, d.S)) {
        if (threadIdx.x == 0) {
            atomicOr(flag, kFlagTimeout);
            mbar_wait(b_tw, 0);                           // the copies in flight land first (bounded)
            mbar_wait(b_s, 0);
            mbar_wait(b_k, 0);
        }
        __syncthreads();
        return false;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        mbar_inval(b_tw);
        mbar_inval(b_s);
        mbar_inval(b_k);
    }
    __syncthreads();
    return true;
}

// x tile `tile` of a sample: the Euler step of its rows from M[par] to
// M[par ^ 1], and their next spectrum.
// OWN (load_m): the persistent launch, whose steps swap M[0] and M[1].
template <int N, int T, bool OWN>
__device__ __forceinline__ void rag_xstep_tile(const RagDesc& d, int tile, int par, float dt, int* __restrict__ flag) {
    constexpr int R = rag_rows<N>();
    using Lay = XstepLayout<N, R>;
    using F = Fft2<N>;
    constexpr int L = Lay::L;
    extern __shared__ __align__(16) float2 sm[];
    float2* tw = sm + Lay::TW_OFF;
    float2* ta = sm + Lay::TA_OFF;
    float* Mt = reinterpret_cast<float*>(sm + Lay::MT_OFF);
    float2* sb = sm + Lay::SB_OFF;
    float2* wk = sm + Lay::W_OFF;
    const Geom g = rag_geom(d);
    LlgCoef cf = d.cf;
    cf.dt = dt;
#pragma unroll
    for (int i = threadIdx.x; i < L / 2; i += T) copy16(tw + 2 * i, g.twx + 2 * i);
    F::template load_ta<T>(ta, g.twx);
    __pipeline_commit();
    const float* M = d.M[par];
    RagCells<(R * N + T - 1) / T> rc;
    load_rag_cells<N, R, T, OWN>(g, cf, tile, M, Mt, rc);
    xstep_body<N, R, kModeStep, T, true>(g, cf, tile, tw, ta, Mt, sb, wk, d.S, d.S, d.M[par ^ 1], flag, nullptr,
                                         XTma{}, &rc);
    __syncthreads();
}

// Row transform of 4 rows (tile) of M[par] into S, one row group per tile
// as in k_pass1_rag<N, 4>.
constexpr int kRagRows1 = 4;
template <int N, int T, bool OWN>
__device__ __forceinline__ void rag_pass1_tile(const RagDesc& d, int tile, int par) {
    const Geom g = rag_geom(d);
    pass1_rows<N, kRagRows1, T, true, false, OWN>(g, tile, d.M[par], d.S, nullptr);
    __syncthreads();
}

template <int NY, int NZ>
__global__ void __launch_bounds__(PlaneLayout<NY, NZ>::THREADS)
    k_rag_batch_plane(const RagDesc* __restrict__ d, const RagItem* __restrict__ items, int* __restrict__ flag) {
    const RagItem it = items[blockIdx.x];
    rag_plane_tile<NY, NZ, PlaneLayout<NY, NZ>::THREADS>(d[it.s], it.tile, flag);
}

template <int N>
__global__ void __launch_bounds__(XstepLayout<N, rag_rows<N>()>::THREADS)
    k_rag_batch_xstep(const RagDesc* __restrict__ d, const RagItem* __restrict__ items, int par, float dt,
                      int* __restrict__ flag) {
    const RagItem it = items[blockIdx.x];
    rag_xstep_tile<N, XstepLayout<N, rag_rows<N>()>::THREADS, false>(d[it.s], it.tile, par, dt, flag);
}

template <int N>
__global__ void __launch_bounds__(kRagRows1 * Fft2<N>::G)
    k_rag_batch_pass1(const RagDesc* __restrict__ d, const RagItem* __restrict__ items, int par) {
    const RagItem it = items[blockIdx.x];
    rag_pass1_tile<N, kRagRows1 * Fft2<N>::G, false>(d[it.s], it.tile, par);
}

// Kernels of one plane class / x class (batch.cu).
struct RagPlaneFns {
    void (*k)(const RagDesc*, const RagItem*, int*) = nullptr;
    int t = 0;
    size_t smem = 0;
};
struct RagXFns {
    void (*p1)(const RagDesc*, const RagItem*, int) = nullptr;
    void (*xs)(const RagDesc*, const RagItem*, int, float, int*) = nullptr;
    int t1 = 0, tx = 0, rows = 0;
    size_t s1 = 0, sx = 0;
};

// The classes: x lengths, and (NY, NZ) of the planes (NZ <= 4 up to NY = 64,
// <= 2 up to 256), so that every block fits 256 threads.
constexpr int kRagXClasses = 8, kRagPlaneClasses = 24;
inline int rag_x_class(int NX) {
    constexpr int len[kRagXClasses] = {16, 32, 48, 64, 96, 128, 192, 256};
    for (int i = 0; i < kRagXClasses; ++i)
        if (len[i] == NX) return i;
    return -1;
}
inline int rag_plane_class(int NY, int nz) {
    const int i = rag_x_class(NY);             // the same eight lengths
    if (i < 0 || nz < 1 || nz > (i < 4 ? 4 : 2)) return -1;
    return i < 4 ? i * 4 + nz - 1 : 16 + (i - 4) * 2 + nz - 1;
}

RagPlaneFns rag_plane_fns(int cls);
RagXFns rag_x_fns(int cls);

}  // namespace mmk
