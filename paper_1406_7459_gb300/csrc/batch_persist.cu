// batch_persist.cu -- the persistent batch step: one cooperative launch for
// many steps of every sample.
#include "batch_kernels.cuh"
#include "grid_sync.cuh"

namespace mmk {

// One function per class, not inlined: the kernel calls the class of the
// item it took.
template <int NY, int NZ> __device__ __noinline__ bool plane_item(const RagDesc& d, int tile, int* flag) {
    return rag_plane_tile<NY, NZ, kRagBatchThreads>(d, tile, flag);
}
template <int N> __device__ __noinline__ void xstep_item(const RagDesc& d, int tile, int par, float dt, int* flag) {
    rag_xstep_tile<N, kRagBatchThreads, true>(d, tile, par, dt, flag);
}
template <int N> __device__ __noinline__ void pass1_item(const RagDesc& d, int tile, int par) {
    rag_pass1_tile<N, kRagBatchThreads, true>(d, tile, par);
}

__device__ __forceinline__ bool any_plane(const RagDesc& d, int tile, int* flag) {
    switch (d.pcls) {
        case 0: return plane_item<16, 1>(d, tile, flag);
        case 1: return plane_item<16, 2>(d, tile, flag);
        case 2: return plane_item<16, 3>(d, tile, flag);
        case 3: return plane_item<16, 4>(d, tile, flag);
        case 4: return plane_item<32, 1>(d, tile, flag);
        case 5: return plane_item<32, 2>(d, tile, flag);
        case 6: return plane_item<32, 3>(d, tile, flag);
        case 7: return plane_item<32, 4>(d, tile, flag);
        case 8: return plane_item<48, 1>(d, tile, flag);
        case 9: return plane_item<48, 2>(d, tile, flag);
        case 10: return plane_item<48, 3>(d, tile, flag);
        case 11: return plane_item<48, 4>(d, tile, flag);
        case 12: return plane_item<64, 1>(d, tile, flag);
        case 13: return plane_item<64, 2>(d, tile, flag);
        case 14: return plane_item<64, 3>(d, tile, flag);
        case 15: return plane_item<64, 4>(d, tile, flag);
        case 16: return plane_item<96, 1>(d, tile, flag);
        case 17: return plane_item<96, 2>(d, tile, flag);
        case 18: return plane_item<128, 1>(d, tile, flag);
        case 19: return plane_item<128, 2>(d, tile, flag);
        case 20: return plane_item<192, 1>(d, tile, flag);
        case 21: return plane_item<192, 2>(d, tile, flag);
        case 22: return plane_item<256, 1>(d, tile, flag);
        case 23: return plane_item<256, 2>(d, tile, flag);
        default: return true;
    }
}
__device__ __forceinline__ void any_xstep(const RagDesc& d, int tile, int par, float dt, int* flag) {
    switch (d.xcls) {
        case 0: xstep_item<16>(d, tile, par, dt, flag); break;
        case 1: xstep_item<32>(d, tile, par, dt, flag); break;
        case 2: xstep_item<48>(d, tile, par, dt, flag); break;
        case 3: xstep_item<64>(d, tile, par, dt, flag); break;
        case 4: xstep_item<96>(d, tile, par, dt, flag); break;
        case 5: xstep_item<128>(d, tile, par, dt, flag); break;
        case 6: xstep_item<192>(d, tile, par, dt, flag); break;
        case 7: xstep_item<256>(d, tile, par, dt, flag); break;
        default: break;
    }
}
__device__ __forceinline__ void any_pass1(const RagDesc& d, int tile, int par) {
    switch (d.xcls) {
        case 0: pass1_item<16>(d, tile, par); break;
        case 1: pass1_item<32>(d, tile, par); break;
        case 2: pass1_item<48>(d, tile, par); break;
        case 3: pass1_item<64>(d, tile, par); break;
        case 4: pass1_item<96>(d, tile, par); break;
        case 5: pass1_item<128>(d, tile, par); break;
        case 6: pass1_item<192>(d, tile, par); break;
        case 7: pass1_item<256>(d, tile, par); break;
        default: break;
    }
}

// n steps of every sample in one cooperative launch.  Work queue 0 holds
// the row transforms of the starting state (only when the spectra are not
// already those of that state), queue 1 the plane tiles, queue 2 the update
// tiles, which also form the next step's x spectra in place: a tile reads
// exactly the spectrum entries it writes.  The state goes M[par0] ->
// M[par0 ^ 1] -> ..., so every load of M is an ordinary one (load_m).  A
// grid-barrier wait that runs out of polls, or a copy wait that gives up,
// sets kFlagTimeout.  Bound by the latency of a tile (queue, copies,
// barriers), so four blocks share an SM although their 64
// registers spill: 512 samples of up to 256 x 64 x 2 cells take 1.37 ms per
// step with two blocks, 1.05 with three and 0.95 with four.
__global__ void __launch_bounds__(kRagBatchThreads, 4)
    k_batch_persist(const BatchDesc* __restrict__ d, const RagDesc* __restrict__ rd, BatchPass q1, BatchPass q2,
                    BatchPass q3, int ns, int par0, int nsteps, float dt, int first_x, int* __restrict__ flag,
                    GridBar* __restrict__ gb, long long limit) {
    __shared__ int slot;
    unsigned bar = 0;
    bool ok = true;
    if (first_x) {
        for (int i; (i = queue_next(gb, 0, q1.n_items + q1.n_tiles, 0, &slot)) >= 0;) {
            if (i < q1.n_items) {
                const RagItem it = q1.items[i];
                any_pass1(rd[it.s], it.tile, par0);
                continue;
            }
            i -= q1.n_items;
            const int s = find_sample(q1.pre, ns, i);
            const BatchDesc& b = d[s];
            pass1_body<true>(b.g, b.r1, b.r1 / 2, par0 ? b.M1 : b.M0, b.S, i - __ldg(q1.pre + s));
        }
        ok = grid_sync(gb, bar++, limit);
    }
    for (int st = 0; ok && st < nsteps; ++st) {
        const int par = (par0 + st) & 1;
        for (int i; ok && (i = queue_next(gb, 1, q2.n_items + q2.n_tiles, st, &slot)) >= 0;) {
            if (i < q2.n_items) {
                const RagItem it = q2.items[i];
                ok = any_plane(rd[it.s], it.tile, flag);
                continue;
            }
            i -= q2.n_items;
            const int s = find_sample(q2.pre, ns, i);
            batch_plane_tile(d[s], i - __ldg(q2.pre + s));
        }
        ok = ok && grid_sync(gb, bar++, limit);
        if (!ok) break;
        for (int i; (i = queue_next(gb, 2, q3.n_items + q3.n_tiles, st, &slot)) >= 0;) {
            if (i < q3.n_items) {
                const RagItem it = q3.items[i];
                any_xstep(rd[it.s], it.tile, par, dt, flag);
                continue;
            }
            i -= q3.n_items;
            const int s = find_sample(q3.pre, ns, i);
            const BatchDesc& b = d[s];
            LlgCoef cf = b.cf;
            cf.dt = dt;
            pass3_body<kModeStepX, true>(b.g, b.r3, 3 * b.r3 / 2, cf, b.S, par ? b.M1 : b.M0, par ? b.M0 : b.M1, flag,
                                   i - __ldg(q3.pre + s), b.S);
        }
        if (st + 1 < nsteps) ok = grid_sync(gb, bar++, limit);
    }
    if (!ok && threadIdx.x == 0) atomicOr(flag, kFlagTimeout);
    grid_exit(gb);
}

BatchPersistFn batch_persist_fn() { return k_batch_persist; }

}  // namespace mmk
