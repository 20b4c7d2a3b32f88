// ragged_select.cu -- picks the kernels and carrier lengths of a ragged film
// (ragged.cuh) and launches its row transform.
#include "ragged_batch.cuh"

namespace mmk {

bool ragged_lookup_x_a(int N, FastStepFns* f);
bool ragged_lookup_x_b(int N, FastStepFns* f);
bool ragged_lookup_x_c(int N, FastStepFns* f);
bool ragged_lookup_x_d(int N, FastStepFns* f);
bool ragged_lookup_plane_nz1(int NY, bool many, FastStepFns* f);
bool ragged_lookup_plane_nz2(int NY, bool many, FastStepFns* f);
bool ragged_lookup_plane_nz3(int NY, bool many, FastStepFns* f);
bool ragged_lookup_plane_nz4(int NY, bool many, FastStepFns* f);
bool ragged_lookup_plane_nz5(int NY, bool many, FastStepFns* f);
bool ragged_lookup_plane_nz6(int NY, bool many, FastStepFns* f);
bool ragged_lookup_plane_nz7(int NY, bool many, FastStepFns* f);
bool ragged_lookup_plane_nz8(int NY, bool many, FastStepFns* f);

bool ragged_lookup_x(int nx, FastStepFns* f, int* NX) {
    *NX = ragged_len(nx);
    return ragged_lookup_x_a(*NX, f) || ragged_lookup_x_b(*NX, f) || ragged_lookup_x_c(*NX, f) ||
           ragged_lookup_x_d(*NX, f);
}

bool ragged_lookup(int nx, int ny, int nz, FastStepFns* f, int* NX, int* NY) {
    *NY = ragged_len(ny);
    const bool many = ragged_len(nx) + 1 >= kBigPlanes;
    bool ok = false;
    switch (nz) {
        case 1: ok = ragged_lookup_plane_nz1(*NY, many, f); break;
        case 2: ok = ragged_lookup_plane_nz2(*NY, many, f); break;
        case 3: ok = ragged_lookup_plane_nz3(*NY, many, f); break;
        case 4: ok = ragged_lookup_plane_nz4(*NY, many, f); break;
        case 5: ok = ragged_lookup_plane_nz5(*NY, many, f); break;
        case 6: ok = ragged_lookup_plane_nz6(*NY, many, f); break;
        case 7: ok = ragged_lookup_plane_nz7(*NY, many, f); break;
        case 8: ok = ragged_lookup_plane_nz8(*NY, many, f); break;
        default: break;
    }
    return ok && ragged_lookup_x(nx, f, NX);
}

int plan_ragged_len(int n) { return ragged_len(n); }

bool ragged_batchable(int nx, int ny, int nz) {
    return rag_x_class(ragged_len(nx)) >= 0 && rag_plane_class(ragged_len(ny), nz) >= 0;
}

// The plane kernel's trigger (fast_step.cuh), per L2-resident step, early
// against late.  Early wins where the x tiles cover the SMs (250x250x4 18.9
// against 20.2 us, 300x300x3 42.5 against 44.2), where the planes do so
// evenly, several to each (600x400x1 28.5 against 30.7, 700x64x1 17.9 against
// 19.5, 400x300x2 33.2 against 33.7), and where planes and tiles together
// leave each SM one block (30x30x1 4.4 against 4.9).  In between the early
// tiles crowd onto the SMs with fewer planes (200x60x3 12.3 against 9.6,
// 100x100x1 7.1 against 6.7).
int ragged_early_trigger(const Geom& g, const FastStepFns& f, int sms) {
    const int tiles = g.nz * (g.Jr / f.rb);
    return tiles >= sms || g.Hx >= 3 * sms || tiles + g.Hx <= sms;
}

cudaError_t launch_ragged_pass1(const Geom& g, const FastStepFns& f, const float* M, float2* S, cudaStream_t s,
                                float* Mcopy, const XComb& comb) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = launch_config(dim3(3 * g.nz * ((g.Jr + f.r1 - 1) / f.r1)), f.t1, f.s1, s, attr);
    if (comb.K) return cudaLaunchKernelEx(&cfg, f.p1c, g, M, S, Mcopy, comb);
    return cudaLaunchKernelEx(&cfg, f.p1, g, M, S, Mcopy);
}

}  // namespace mmk
