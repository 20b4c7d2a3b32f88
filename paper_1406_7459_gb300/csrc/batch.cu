// batch.cu -- many independent samples of uneven size stepped together.
//
// Samples with sides in the carrier lengths of the ragged-film kernels
// (ragged_batch.cuh) step on those, one launch per class of lengths and pass,
// the classes side by side; the others on the general mixed-radix kernels
// described next.  512 samples of 16..256 x 16..64 x 1..2 cells: see
// ragged_batch.cuh for both sides' times.
//
// Each sample is a complete problem of its own (grid, cell, material, field)
// with its own tensor spectrum; the step of every sample is the paper's
// three phases (Sec. 3: forward FFTs, member-wise product, inverse FFTs,
// then the field and Euler update).  All samples advance in lock step: one
// batched kernel per pass covers the tiles of every sample, each CTA
// finding its (sample, tile) in a prefix table over a per-sample
// descriptor array, and the three launches of a step replay from one CUDA
// graph.  Or (MM_STEP_PERSISTENT) one cooperative launch runs many steps,
// captured once in a CUDA graph and replayed on later calls:
// its blocks take (sample, tile) items from a work queue per pass, passes
// separated by bounded grid barriers, the x R2C of the next step fused into
// the update pass.  The tile shapes (rows per CTA in the x passes, threads
// per CTA) come from an autotuner that times candidate shapes on the batch
// itself.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/mm.h"
#include "batch_kernels.cuh"
#include "bulk_copy.cuh"
#include "grid_sync.cuh"

using namespace mmk;

namespace mmk {

__global__ void __launch_bounds__(256) k_batch_pass1(const BatchDesc* __restrict__ d, const int* __restrict__ pre,
                                                      int ns, int par) {
    const int s = find_sample(pre, ns, blockIdx.x);
    const BatchDesc& b = d[s];
    pass1_body(b.g, b.r1, b.r1 / 2, par ? b.M1 : b.M0, b.S, blockIdx.x - __ldg(pre + s));
}

__global__ void __launch_bounds__(256) k_batch_plane(const BatchDesc* __restrict__ d, const int* __restrict__ pre,
                                                      int ns) {
    const int s = find_sample(pre, ns, blockIdx.x);
    batch_plane_tile(d[s], blockIdx.x - __ldg(pre + s));
}

// The update pass; it also forms the x spectra of the new states in place
// (kModeStepX: a tile reads exactly the spectrum entries it writes), the
// first pass of the next step.
__global__ void __launch_bounds__(256) k_batch_pass3(const BatchDesc* __restrict__ d, const int* __restrict__ pre,
                                                      int ns, int par, float dt, int* __restrict__ flag) {
    const int s = find_sample(pre, ns, blockIdx.x);
    const BatchDesc& b = d[s];
    LlgCoef cf = b.cf;
    cf.dt = dt;
    pass3_body<kModeStepX>(b.g, b.r3, 3 * b.r3 / 2, cf, b.S, par ? b.M1 : b.M0, par ? b.M0 : b.M1, flag,
                           blockIdx.x - __ldg(pre + s), b.S);
}

}  // namespace mmk

// Steps per launch of the persistent batch step.
static constexpr int kBatchChunk = 1024;
// Steps of one dt that launch directly before their graphs are captured.
static constexpr int kBatchWarm = 8;

struct mm_batch {
    int ns = 0;
    cudaStream_t stream = nullptr;
    cudaStream_t cap = nullptr;
    std::vector<int> grid;                     // 3 per sample
    std::vector<double> cell, Ms, A, Ku, alpha, gamma, Hext;
    std::vector<BatchDesc> desc;               // host copy
    std::vector<size_t> moff;                  // float offset of each sample's M
    size_t mtotal = 0;                         // floats per M buffer (sum 3 N_s)
    long long cells = 0;
    float* M0 = nullptr;
    float* M1 = nullptr;
    float2* S = nullptr;
    float* Kt = nullptr;
    float2* tw = nullptr;
    BatchDesc* d_desc = nullptr;
    int* d_pre = nullptr;                      // 3 prefix arrays of ns + 1
    int* flag = nullptr;
    int tiles[3] = {0, 0, 0};                  // of the samples on the general kernels
    size_t smem[3] = {0, 0, 0};
    // samples on the ragged-film kernels, grouped by class (ragged_batch.cuh)
    struct Group {
        int first = 0, count = 0;              // of its items
    };
    std::vector<RagDesc> rag;
    RagDesc* d_rag = nullptr;
    RagItem* d_items = nullptr;
    Group g1[kRagXClasses], g2[kRagPlaneClasses], g3[kRagXClasses];   // row transform, plane, update
    int n_items[3] = {0, 0, 0}, off_items[3] = {0, 0, 0};
    size_t rag_smem = 0;                       // largest tile, for the persistent launch
    static constexpr int kSide = 3;            // streams beside the batch's own
    cudaStream_t side[kSide] = {};
    cudaEvent_t fork = nullptr, join[kSide] = {};
    int threads = 256, r1 = 4, r3 = 2, r2 = 1;
    int par = 0;
    int warm = 0;                              // steps launched directly with warm_dt, warm_ver
    double warm_dt = 0;
    unsigned long long warm_ver = 0;
    cudaGraphExec_t exec[2] = {nullptr, nullptr};
    double exec_dt[2] = {0, 0};
    unsigned long long exec_ver[2] = {0, 0};
    unsigned long long ver = 1;
    // persistent step: counters, co-resident grid, shared memory, choice
    GridBar* gb = nullptr;
    int pgrid = 0;
    size_t psmem = 0;
    int path = MM_STEP_AUTO;
    long long wait_limit = kGridWaitLimit;
    bool spec_valid = false;                   // S holds the x spectra of the current state
    // the persistent launch captured in a graph, for the arguments it was
    // captured with; pgraph_ok false once a capture failed (direct launches)
    cudaGraphExec_t pexec = nullptr;
    int pexec_m = 0, pexec_par = 0, pexec_first = 0;
    double pexec_dt = 0;
    long long pexec_limit = 0;
    unsigned long long pexec_ver = 0;
    bool pgraph_ok = true;
    int form = -1;                             // mm_batch_launch_form of the last step
};

#define BCU(expr)                                                                                    \
    do {                                                                                             \
        cudaError_t _e = (expr);                                                                     \
        if (_e != cudaSuccess) {                                                                     \
            char _m[256];                                                                            \
            snprintf(_m, sizeof(_m), "%s: %s", #expr, cudaGetErrorString(_e));                       \
            return set_error(_e == cudaErrorMemoryAllocation ? MM_ENOMEM : MM_ECUDA, _m);            \
        }                                                                                            \
    } while (0)

static LlgCoef batch_coef(const mm_batch* b, int s) {
    LlgCoef f;
    const double Ms = b->Ms[s], Ms2 = Ms * Ms, al = b->alpha[s], den = 1.0 + al * al;
    const double mu0 = 4.0e-7 * 3.14159265358979323846;
    f.Ms = (float)Ms;
    f.pexch = (float)(2.0 * b->A[s] / (mu0 * Ms2));
    f.panis = (float)(-2.0 * b->Ku[s] / (mu0 * Ms2));
    f.c1 = (float)(-b->gamma[s] / den);
    f.c2 = (float)(-al * b->gamma[s] / (den * Ms));
    f.idx2 = (float)(1.0 / (b->cell[3 * s] * b->cell[3 * s]));
    f.idy2 = (float)(1.0 / (b->cell[3 * s + 1] * b->cell[3 * s + 1]));
    f.idz2 = (float)(1.0 / (b->cell[3 * s + 2] * b->cell[3 * s + 2]));
    f.hx = (float)b->Hext[3 * s];
    f.hy = (float)b->Hext[3 * s + 1];
    f.hz = (float)b->Hext[3 * s + 2];
    f.dt = 0.f;
    return f;
}

// Tile counts, prefix tables, shared-memory sizes and descriptors for the
// current shape choice (r1, r3, threads); uploads them.
static int batch_layout(mm_batch* b) {
    std::vector<int> pre(3 * (b->ns + 1));
    size_t sm[3] = {0, 0, 0};
    int acc[3] = {0, 0, 0};
    for (int s = 0; s < b->ns; ++s) {
        BatchDesc& d = b->desc[s];
        const Geom& g = d.g;
        d.r1 = b->r1;
        d.r3 = b->r3;
        d.r2 = b->r2;
        d.cf = batch_coef(b, s);
        b->rag[s].cf = d.cf;
        for (int q = 0; q < 3; ++q) pre[q * (b->ns + 1) + s] = acc[q];
        if (b->rag[s].xcls >= 0) continue;
        const int t1 = 3 * g.nz * ((g.ny + b->r1 - 1) / b->r1);
        const int t2 = (g.Hx + b->r2 - 1) / b->r2;
        const int t3 = g.nz * ((g.ny + b->r3 - 1) / b->r3);
        acc[0] += t1;
        acc[1] += t2;
        acc[2] += t3;
        const size_t lx = (size_t)padded_len(g.Lx) * sizeof(float2), ly = (size_t)padded_len(g.Ly) * sizeof(float2);
        const size_t a1 = 2 * (size_t)(b->r1 / 2) * lx, a2 = 2 * (size_t)3 * g.nz * b->r2 * ly,
                     a3 = 2 * (size_t)(3 * b->r3 / 2) * lx;
        sm[0] = a1 > sm[0] ? a1 : sm[0];
        sm[1] = a2 > sm[1] ? a2 : sm[1];
        sm[2] = a3 > sm[2] ? a3 : sm[2];
    }
    for (int q = 0; q < 3; ++q) {
        pre[q * (b->ns + 1) + b->ns] = acc[q];
        b->tiles[q] = acc[q];
        b->smem[q] = sm[q];
        if (sm[q] > 227 * 1024) return set_error(MM_EUNSUPPORTED, "batch sample exceeds shared memory");
    }
    BCU(allow_smem(k_batch_pass1));
    BCU(allow_smem(k_batch_plane));
    BCU(allow_smem(k_batch_pass3));
    {
        size_t ps = sm[0] > sm[1] ? sm[0] : sm[1];
        ps = ps > sm[2] ? ps : sm[2];
        ps = ps > b->rag_smem ? ps : b->rag_smem;
        b->psmem = ps;
        BCU(allow_smem(batch_persist_fn()));
        int dev = 0, sms = 0, per_sm = 0;
        BCU(cudaGetDevice(&dev));
        BCU(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        BCU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_persist_fn(), kRagBatchThreads, ps));
        b->pgrid = per_sm * sms;
    }
    // on the batch's stream, behind the steps in flight that read the old
    // tables (the legacy stream waits for no non-blocking one)
    BCU(cudaMemcpyAsync(b->d_rag, b->rag.data(), sizeof(RagDesc) * b->ns, cudaMemcpyHostToDevice, b->stream));
    BCU(cudaMemcpyAsync(b->d_desc, b->desc.data(), sizeof(BatchDesc) * b->ns, cudaMemcpyHostToDevice, b->stream));
    BCU(cudaMemcpyAsync(b->d_pre, pre.data(), sizeof(int) * pre.size(), cudaMemcpyHostToDevice, b->stream));
    BCU(cudaStreamSynchronize(b->stream));      // before the host tables change or go
    b->ver++;
    return MM_OK;
}

// The class launches of a pass run side by side: fork the side streams off
// s, deal the launches out over s and them, join back into s.
struct Lanes {
    mm_batch* b;
    cudaStream_t s;
    int next = 0;
    cudaError_t begin() {
        cudaError_t e = cudaEventRecord(b->fork, s);
        for (int q = 0; q < mm_batch::kSide && e == cudaSuccess; ++q) e = cudaStreamWaitEvent(b->side[q], b->fork, 0);
        return e;
    }
    cudaStream_t lane() {
        const int q = next++ % (mm_batch::kSide + 1);
        return q == 0 ? s : b->side[q - 1];
    }
    cudaError_t end() {
        cudaError_t e = cudaGetLastError();
        for (int q = 0; q < mm_batch::kSide; ++q) {
            cudaError_t r = cudaEventRecord(b->join[q], b->side[q]);
            if (r == cudaSuccess) r = cudaStreamWaitEvent(s, b->join[q], 0);
            if (e == cudaSuccess) e = r;
        }
        return e;
    }
};

// x R2C of every sample's state M[par] into its spectrum
static int batch_pass1(mm_batch* b, int par, cudaStream_t s) {
    Lanes l{b, s};
    BCU(l.begin());
    if (b->tiles[0])
        k_batch_pass1<<<b->tiles[0], b->threads, b->smem[0], l.lane()>>>(b->d_desc, b->d_pre, b->ns, par);
    for (int c = 0; c < kRagXClasses; ++c)
        if (b->g1[c].count) {
            const RagXFns f = rag_x_fns(c);
            f.p1<<<b->g1[c].count, f.t1, f.s1, l.lane()>>>(b->d_rag, b->d_items + b->g1[c].first, par);
        }
    BCU(l.end());
    return MM_OK;
}

// One step from spectra that hold the x transforms of M[par]: the plane
// pass, then the update, which leaves the x transforms of M[par ^ 1].
static int batch_enqueue(mm_batch* b, int par, double dt, cudaStream_t s) {
    const int P = b->ns + 1;
    Lanes l{b, s};
    BCU(l.begin());
    if (b->tiles[1])
        k_batch_plane<<<b->tiles[1], b->threads, b->smem[1], l.lane()>>>(b->d_desc, b->d_pre + P, b->ns);
    for (int c = 0; c < kRagPlaneClasses; ++c)
        if (b->g2[c].count) {
            const RagPlaneFns f = rag_plane_fns(c);
            f.k<<<b->g2[c].count, f.t, f.smem, l.lane()>>>(b->d_rag, b->d_items + b->g2[c].first, b->flag);
        }
    BCU(l.end());
    Lanes u{b, s};
    BCU(u.begin());
    if (b->tiles[2])
        k_batch_pass3<<<b->tiles[2], b->threads, b->smem[2], u.lane()>>>(b->d_desc, b->d_pre + 2 * P, b->ns, par,
                                                                         (float)dt, b->flag);
    for (int c = kRagXClasses - 1; c >= 0; --c)               // the long rows first
        if (b->g3[c].count) {
            const RagXFns f = rag_x_fns(c);
            f.xs<<<b->g3[c].count, f.tx, f.sx, u.lane()>>>(b->d_rag, b->d_items + b->g3[c].first, par, (float)dt,
                                                           b->flag);
        }
    BCU(u.end());
    return MM_OK;
}

static void batch_release(mm_batch* b) {
    for (int p = 0; p < 2; ++p)
        if (b->exec[p]) cudaGraphExecDestroy(b->exec[p]);
    if (b->pexec) cudaGraphExecDestroy(b->pexec);
    cudaFree(b->M0);
    cudaFree(b->M1);
    cudaFree(b->S);
    cudaFree(b->Kt);
    cudaFree(b->tw);
    cudaFree(b->d_desc);
    cudaFree(b->d_pre);
    cudaFree(b->flag);
    cudaFree(b->gb);
    cudaFree(b->d_rag);
    cudaFree(b->d_items);
    for (int q = 0; q < mm_batch::kSide; ++q) {
        if (b->side[q]) cudaStreamDestroy(b->side[q]);
        if (b->join[q]) cudaEventDestroy(b->join[q]);
    }
    if (b->fork) cudaEventDestroy(b->fork);
    if (b->cap) cudaStreamDestroy(b->cap);
}

// The carrier lengths and classes of a sample the ragged-film kernels take.
static bool batch_classes(const Geom& g, int* NX, int* NY, int* xc, int* pc) {
    *NX = plan_ragged_len(g.nx);
    *NY = plan_ragged_len(g.ny);
    *xc = rag_x_class(*NX);
    *pc = rag_plane_class(*NY, g.nz);
    return *xc >= 0 && *pc >= 0;
}

// Item lists per class (they depend on the grids only) and the kernels'
// shared memory.
static int batch_items(mm_batch* b) {
    std::vector<RagItem> items;
    auto fill = [&](mm_batch::Group* g, int ncls, int pass) {
        b->off_items[pass] = (int)items.size();
        for (int c = 0; c < ncls; ++c) {
            g[c].first = (int)items.size();
            for (int s = 0; s < b->ns; ++s) {
                const RagDesc& d = b->rag[s];
                if (d.xcls < 0 || (pass == 1 ? d.pcls : d.xcls) != c) continue;
                const int n = pass == 0   ? 3 * d.nz * ((d.Jst + kRagRows1 - 1) / kRagRows1)
                              : pass == 1 ? b->desc[s].g.Hx
                                          : d.nz * (d.Jst / rag_x_fns(c).rows);
                for (int t = 0; t < n; ++t) items.push_back(RagItem{s, t});
            }
            g[c].count = (int)items.size() - g[c].first;
        }
        b->n_items[pass] = (int)items.size() - b->off_items[pass];
    };
    fill(b->g1, kRagXClasses, 0);
    fill(b->g2, kRagPlaneClasses, 1);
    fill(b->g3, kRagXClasses, 2);
    for (int c = 0; c < kRagXClasses; ++c)
        if (b->g1[c].count) {
            const RagXFns f = rag_x_fns(c);
            BCU(allow_smem(f.p1));
            BCU(allow_smem(f.xs));
            b->rag_smem = std::max(b->rag_smem, std::max(f.s1, f.sx));
        }
    for (int c = 0; c < kRagPlaneClasses; ++c)
        if (b->g2[c].count) {
            const RagPlaneFns f = rag_plane_fns(c);
            BCU(allow_smem(f.k));
            b->rag_smem = std::max(b->rag_smem, f.smem);
        }
    BCU(cudaMalloc(&b->d_items, sizeof(RagItem) * (items.empty() ? 1 : items.size())));
    BCU(cudaMemcpyAsync(b->d_items, items.data(), sizeof(RagItem) * items.size(), cudaMemcpyHostToDevice, b->stream));
    BCU(cudaStreamSynchronize(b->stream));
    return MM_OK;
}

extern "C" int mm_batch_create(mm_batch** out, int n, const int* grids, const double* cells, const double* Ms,
                               const double* A, const double* Ku, const double* alpha, const double* gamma,
                               void* cuda_stream) {
    if (!out) return set_error(MM_EINVAL, "out is NULL");
    *out = nullptr;
    if (n < 1 || !grids || !cells || !Ms || !A || !Ku || !alpha || !gamma)
        return set_error(MM_EINVAL, "n < 1 or null array");
    mm_batch* b = new (std::nothrow) mm_batch();
    if (!b) return set_error(MM_ENOMEM, "host allocation failed");
    b->ns = n;
    b->stream = (cudaStream_t)cuda_stream;
    b->grid.assign(grids, grids + 3 * n);
    b->cell.assign(cells, cells + 3 * n);
    b->Ms.assign(Ms, Ms + n);
    b->A.assign(A, A + n);
    b->Ku.assign(Ku, Ku + n);
    b->alpha.assign(alpha, alpha + n);
    b->gamma.assign(gamma, gamma + n);
    b->Hext.assign(3 * n, 0.0);
    b->desc.resize(n);
    b->moff.resize(n);
    b->rag.resize(n);
    int rc = [&]() -> int {
        size_t mt = 0, st = 0, kt = 0, tt = 0, wmax = 0, nmax = 0;
        std::vector<size_t> soff(n), koff(n), toff(n);
        for (int s = 0; s < n; ++s) {
            const int nx = grids[3 * s], ny = grids[3 * s + 1], nz = grids[3 * s + 2];
            if (nx < 1 || ny < 1 || nz < 1) return set_error(MM_EINVAL, "grid entries must be >= 1");
            for (int a = 0; a < 3; ++a)
                if (!(cells[3 * s + a] > 0.0)) return set_error(MM_EINVAL, "cell sizes must be > 0");
            if (!(Ms[s] > 0.0) || !(A[s] >= 0.0) || !(alpha[s] >= 0.0) || !(gamma[s] > 0.0) || !std::isfinite(Ku[s]))
                return set_error(MM_EINVAL, "bad material value");
            Geom& g = b->desc[s].g;
            memset(&g, 0, sizeof(g));
            g.nx = nx;
            g.ny = ny;
            g.nz = nz;
            g.N = nx * ny * nz;
            g.Lx = plan_padded_length(nx);
            g.Ly = plan_padded_length(ny);
            g.Lz = plan_padded_length(nz);
            if (g.Lx > kMaxLen || g.Ly > kMaxLen || g.Lz > 8)
                return set_error(MM_EUNSUPPORTED, "batch samples need padded lengths <= 4096 and nz <= 4");
            g.Hx = g.Lx / 2 + 1;
            g.Hy = g.Ly / 2 + 1;
            g.Hz = g.Lz / 2 + 1;
            g.Jst = ny;
            if (!plan_axis(g.Lx, &g.px) || !plan_axis(g.Ly, &g.py) || !plan_axis(g.Lz, &g.pz))
                return set_error(MM_EUNSUPPORTED, "no radix plan");
            RagDesc& rd = b->rag[s];
            memset(&rd, 0, sizeof(rd));
            int NX = 0, NY = 0;
            if (batch_classes(g, &NX, &NY, &rd.xcls, &rd.pcls)) {
                g.Lx = 2 * NX;
                g.Ly = 2 * NY;
                g.Lz = 1;                                     // the z sum is direct
                g.Hx = NX + 1;
                g.Hy = NY + 1;
                g.Hz = 1;
                g.Jst = (ny + 3) & ~3;
            } else {
                rd.xcls = rd.pcls = -1;
            }
            b->moff[s] = mt;
            mt += 3 * (size_t)g.N;
            // every sample's spectra start on 16 bytes (bulk copies)
            soff[s] = st;
            st += ((size_t)g.Hx * 3 * nz * g.Jst + 1) & ~(size_t)1;
            koff[s] = kt;
            kt += rd.xcls >= 0 ? (size_t)6 * g.Hx * kd_row(g.Hy) * nz
                               : ((size_t)6 * g.Hx * g.Hy * g.Hz + 3) & ~(size_t)3;
            tt += tt & 1;
            toff[s] = tt;
            tt += (size_t)(g.Lx + g.Ly + g.Lz);
            const int L[3] = {g.Lx, g.Ly, g.Lz};
            const size_t w = tensor_work_elems(&grids[3 * s], L);
            wmax = w > wmax ? w : wmax;
            nmax = (size_t)g.N > nmax ? (size_t)g.N : nmax;
            b->cells += g.N;
        }
        b->mtotal = mt;
        BCU(cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking));
        BCU(cudaMalloc(&b->M0, sizeof(float) * mt));
        BCU(cudaMalloc(&b->M1, sizeof(float) * mt));
        BCU(cudaMalloc(&b->S, sizeof(float2) * st));
        BCU(cudaMalloc(&b->Kt, sizeof(float) * kt));
        BCU(cudaMalloc(&b->tw, sizeof(float2) * tt));
        BCU(cudaMalloc(&b->d_desc, sizeof(BatchDesc) * n));
        BCU(cudaMalloc(&b->d_pre, sizeof(int) * 3 * (n + 1)));
        BCU(cudaMalloc(&b->d_rag, sizeof(RagDesc) * n));
        BCU(cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming));
        for (int q = 0; q < mm_batch::kSide; ++q) {
            BCU(cudaStreamCreateWithFlags(&b->side[q], cudaStreamNonBlocking));
            BCU(cudaEventCreateWithFlags(&b->join[q], cudaEventDisableTiming));
        }
        BCU(cudaMalloc(&b->flag, sizeof(int)));
        BCU(cudaMemset(b->flag, 0, sizeof(int)));
        BCU(cudaMalloc(&b->gb, sizeof(GridBar)));
        BCU(cudaMemset(b->gb, 0, sizeof(GridBar)));
        std::vector<float2> htw(tt);
        std::vector<float> hm(mt);
        for (int s = 0; s < n; ++s) {
            Geom& g = b->desc[s].g;
            float2* t = htw.data() + toff[s];
            plan_twiddles(g.Lx, t);
            plan_twiddles(g.Ly, t + g.Lx);
            plan_twiddles(g.Lz, t + g.Lx + g.Ly);
            g.twx = b->tw + toff[s];
            g.twy = g.twx + g.Lx;
            g.twz = g.twy + g.Ly;
            g.Kt = b->Kt + koff[s];
            g.Kd = nullptr;
            g.Kd0 = nullptr;
            b->desc[s].M0 = b->M0 + b->moff[s];
            b->desc[s].M1 = b->M1 + b->moff[s];
            b->desc[s].S = b->S + soff[s];
            RagDesc& rd = b->rag[s];
            rd.nx = g.nx;
            rd.ny = g.ny;
            rd.nz = g.nz;
            rd.N = g.N;
            rd.Jst = g.Jst;
            rd.twx = g.twx;
            rd.twy = g.twy;
            rd.Kd = g.Kt;
            rd.M[0] = b->desc[s].M0;
            rd.M[1] = b->desc[s].M1;
            rd.S = b->desc[s].S;
            for (int i = 0; i < g.N; ++i) {
                hm[b->moff[s] + i] = (float)Ms[s];
                hm[b->moff[s] + g.N + i] = 0.f;
                hm[b->moff[s] + 2 * (size_t)g.N + i] = 0.f;
            }
        }
        BCU(cudaMemcpy(b->tw, htw.data(), sizeof(float2) * tt, cudaMemcpyHostToDevice));
        BCU(cudaMemcpy(b->M0, hm.data(), sizeof(float) * mt, cudaMemcpyHostToDevice));
        // per-sample FP64 tensor set-up into each sample's spectrum slice
        double *Nd = nullptr, *w1 = nullptr, *w2 = nullptr;
        cudaError_t e = cudaMalloc(&Nd, sizeof(double) * 6 * nmax);
        if (e == cudaSuccess) e = cudaMalloc(&w1, sizeof(double) * wmax);
        if (e == cudaSuccess) e = cudaMalloc(&w2, sizeof(double) * wmax);
        for (int s = 0; s < n && e == cudaSuccess; ++s) {
            const Geom& g = b->desc[s].g;
            const int L[3] = {g.Lx, g.Ly, g.Lz};
            e = tensor_octant_fp64(&grids[3 * s], &cells[3 * s], Nd, b->stream);
            float* Ks = b->Kt + koff[s];
            if (e == cudaSuccess)
                e = b->rag[s].xcls >= 0 ? tensor_spectrum(&grids[3 * s], L, Nd, nullptr, w1, w2, b->stream, Ks,
                                                          ExchangeFold{}, nullptr, true)
                                        : tensor_spectrum(&grids[3 * s], L, Nd, Ks, w1, w2, b->stream);
        }
        if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
        cudaFree(Nd);
        cudaFree(w1);
        cudaFree(w2);
        BCU(e);
        const int rc2 = batch_items(b);
        return rc2 != MM_OK ? rc2 : batch_layout(b);
    }();
    if (rc != MM_OK) {
        batch_release(b);
        delete b;
        return rc;
    }
    *out = b;
    return MM_OK;
}

extern "C" int mm_batch_destroy(mm_batch* b) {
    if (!b) return MM_OK;
    cudaStreamSynchronize(b->stream);
    batch_release(b);
    delete b;
    return MM_OK;
}

extern "C" int mm_batch_set_field(mm_batch* b, const double* H) {
    if (!b || !H) return set_error(MM_EINVAL, "null argument");
    for (int i = 0; i < 3 * b->ns; ++i) {
        if (!std::isfinite(H[i])) return set_error(MM_EINVAL, "H_ext must be finite");
        b->Hext[i] = H[i];
    }
    return batch_layout(b);
}

extern "C" int mm_batch_set_m(mm_batch* b, const float* M) {
    if (!b || !M) return set_error(MM_EINVAL, "null argument");
    BCU(cudaMemcpyAsync(b->par ? b->M1 : b->M0, M, sizeof(float) * b->mtotal, cudaMemcpyDefault, b->stream));
    BCU(cudaMemsetAsync(b->flag, 0, sizeof(int), b->stream));
    BCU(cudaStreamSynchronize(b->stream));
    b->spec_valid = false;
    return MM_OK;
}

extern "C" int mm_batch_get_m(mm_batch* b, float* M) {
    if (!b || !M) return set_error(MM_EINVAL, "null argument");
    BCU(cudaMemcpyAsync(M, b->par ? b->M1 : b->M0, sizeof(float) * b->mtotal, cudaMemcpyDefault, b->stream));
    BCU(cudaStreamSynchronize(b->stream));
    return MM_OK;
}

// The persistent batch step is taken when asked for (MM_STEP_PERSISTENT)
// and when every block of its grid fits on the device at once.
static bool batch_uses_persist(const mm_batch* b) { return b->path == MM_STEP_PERSISTENT && b->pgrid > 0; }

extern "C" int mm_batch_set_path(mm_batch* b, int path) {
    if (!b) return set_error(MM_EINVAL, "null batch");
    if (path != MM_STEP_AUTO && path != MM_STEP_GRAPH && path != MM_STEP_PERSISTENT)
        return set_error(MM_EINVAL, "unknown step path");
    if (path == MM_STEP_PERSISTENT && b->pgrid < 1)
        return set_error(MM_EUNSUPPORTED, "the persistent batch step does not fit on this device");
    b->path = path;
    return MM_OK;
}

extern "C" int mm_batch_set_wait_limit(mm_batch* b, long long polls) {
    if (!b) return set_error(MM_EINVAL, "null batch");
    if (polls < 0) return set_error(MM_EINVAL, "polls must be >= 0");
    b->wait_limit = polls;
    return MM_OK;
}

// One cooperative launch of m steps on stream s.
static cudaError_t batch_launch_persist(const mm_batch* b, int m, double dt, int first, cudaStream_t s) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(b->pgrid);
    cfg.blockDim = dim3(kRagBatchThreads);
    cfg.dynamicSmemBytes = b->psmem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    BatchPass q[3];
    for (int i = 0; i < 3; ++i)
        q[i] = BatchPass{b->d_items + b->off_items[i], b->d_pre + i * (b->ns + 1), b->n_items[i], b->tiles[i]};
    return cudaLaunchKernelEx(&cfg, batch_persist_fn(), (const BatchDesc*)b->d_desc, (const RagDesc*)b->d_rag, q[0],
                              q[1], q[2], b->ns, b->par, m, (float)dt, first, b->flag, b->gb, b->wait_limit);
}

// The launch of m steps as a graph replay: captured (on the capture stream)
// the first time and again whenever its arguments change.  A capture or
// instantiation the runtime refuses switches the batch to direct launches.
static cudaError_t batch_replay_persist(mm_batch* b, int m, double dt, int first) {
    const bool same = b->pexec && b->pexec_m == m && b->pexec_dt == dt && b->pexec_par == b->par &&
                      b->pexec_first == first && b->pexec_limit == b->wait_limit && b->pexec_ver == b->ver;
    if (!same) {
        if (b->pexec) {
            cudaGraphExecDestroy(b->pexec);
            b->pexec = nullptr;
        }
        cudaError_t e = cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return e;
        const cudaError_t el = batch_launch_persist(b, m, dt, first, b->cap);
        cudaGraph_t graph = nullptr;
        e = cudaStreamEndCapture(b->cap, &graph);
        if (el != cudaSuccess || e != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            return el != cudaSuccess ? el : e;
        }
        e = cudaGraphInstantiate(&b->pexec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            b->pexec = nullptr;
            return e;
        }
        b->pexec_m = m;
        b->pexec_dt = dt;
        b->pexec_par = b->par;
        b->pexec_first = first;
        b->pexec_limit = b->wait_limit;
        b->pexec_ver = b->ver;
    }
    return cudaGraphLaunch(b->pexec, b->stream);
}

static int batch_step_persist(mm_batch* b, int n, double dt) {
    for (int s = 0; s < n;) {
        const int m = n - s < kBatchChunk ? n - s : kBatchChunk;
        const int first = b->spec_valid ? 0 : 1;
        cudaError_t e = cudaErrorNotSupported;
        if (b->pgraph_ok) {
            e = batch_replay_persist(b, m, dt, first);
            if (e != cudaSuccess) {
                cudaGetLastError();                       // a refused capture leaves no sticky error
                b->pgraph_ok = false;
            }
        }
        if (e != cudaSuccess) BCU(batch_launch_persist(b, m, dt, first, b->stream));
        b->form = e == cudaSuccess ? 1 : 2;
        b->par = (b->par + m) & 1;
        b->spec_valid = true;
        s += m;
    }
    return MM_OK;
}

extern "C" int mm_batch_step(mm_batch* b, int n, double dt) {
    if (!b) return set_error(MM_EINVAL, "null batch");
    if (n < 0 || !(dt > 0.0) || !std::isfinite(dt)) return set_error(MM_EINVAL, "n >= 0 and dt > 0 required");
    if (n == 0) return MM_OK;
    if (batch_uses_persist(b)) return batch_step_persist(b, n, dt);
    if (!b->spec_valid) {
        int rc = batch_pass1(b, b->par, b->stream);
        if (rc != MM_OK) return rc;
        b->spec_valid = true;
    }
    for (int s = 0; s < n; ++s) {
        const int p = b->par;
        // the first steps of a dt launch directly: capturing and instantiating
        // the step's graph (once per parity) takes longer than a few steps'
        // launches
        if (b->warm_dt != dt || b->warm_ver != b->ver) {
            b->warm_dt = dt;
            b->warm_ver = b->ver;
            b->warm = 0;
        }
        if (b->warm < kBatchWarm) {
            int rc = batch_enqueue(b, p, dt, b->stream);
            if (rc != MM_OK) return rc;
            ++b->warm;
            b->form = 3;
            b->par = 1 - p;
            continue;
        }
        if (!b->exec[p] || b->exec_dt[p] != dt || b->exec_ver[p] != b->ver) {
            if (b->exec[p]) {
                cudaGraphExecDestroy(b->exec[p]);
                b->exec[p] = nullptr;
            }
            BCU(cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal));
            int rc = batch_enqueue(b, p, dt, b->cap);
            cudaGraph_t graph = nullptr;
            cudaError_t e = cudaStreamEndCapture(b->cap, &graph);
            if (rc != MM_OK) {
                if (graph) cudaGraphDestroy(graph);
                return rc;
            }
            BCU(e);
            e = cudaGraphInstantiate(&b->exec[p], graph, 0);
            cudaGraphDestroy(graph);
            BCU(e);
            b->exec_dt[p] = dt;
            b->exec_ver[p] = b->ver;
        }
        BCU(cudaGraphLaunch(b->exec[p], b->stream));
        b->form = 0;
        b->par = 1 - p;
    }
    return MM_OK;
}

extern "C" int mm_batch_sync(mm_batch* b) {
    if (!b) return set_error(MM_EINVAL, "null batch");
    BCU(cudaStreamSynchronize(b->stream));
    int f = 0;
    BCU(cudaMemcpy(&f, b->flag, sizeof(int), cudaMemcpyDeviceToHost));
    if (f & kFlagTimeout) return set_error(MM_ETIMEOUT, "a grid-barrier wait of the batch step gave up");
    if (f) return set_error(MM_ENONFINITE, "a batch step produced a non-finite magnetisation");
    return MM_OK;
}

extern "C" long long mm_batch_cells(const mm_batch* b) { return b ? b->cells : -1; }

extern "C" int mm_batch_launch_form(const mm_batch* b) { return b ? b->form : -1; }

extern "C" int mm_batch_autotune(mm_batch* b, double dt, int choice[4], float* ms_out) {
    if (!b || !(dt > 0.0)) return set_error(MM_EINVAL, "null batch or dt <= 0");
    // keep the state: tuning steps run on a saved copy
    float* save = nullptr;
    BCU(cudaMalloc(&save, sizeof(float) * b->mtotal));
    float* cur = b->par ? b->M1 : b->M0;
    BCU(cudaMemcpyAsync(save, cur, sizeof(float) * b->mtotal, cudaMemcpyDeviceToDevice, b->stream));
    static const int cand[][3] = {{2, 2, 128}, {4, 2, 128}, {8, 2, 128}, {2, 4, 128}, {4, 4, 128}, {8, 4, 128},
                                  {2, 2, 256}, {4, 2, 256}, {8, 2, 256}, {2, 4, 256}, {4, 4, 256}, {8, 4, 256}};
    const int nc = (int)(sizeof(cand) / sizeof(cand[0]));
    cudaEvent_t e0, e1;
    BCU(cudaEventCreate(&e0));
    BCU(cudaEventCreate(&e1));
    float best = 1e30f;
    int bi = 0;
    int rc = MM_OK;
    b->r2 = 1;
    for (int c = 0; c < nc && rc == MM_OK; ++c) {
        b->r1 = cand[c][0];
        b->r3 = cand[c][1];
        b->threads = cand[c][2];
        rc = batch_layout(b);
        if (rc != MM_OK) break;
        rc = batch_pass1(b, b->par, b->stream);
        if (rc == MM_OK) rc = batch_enqueue(b, b->par, dt, b->stream);   // warm-up
        if (rc != MM_OK) break;
        b->par = 1 - b->par;
        cudaEventRecord(e0, b->stream);
        for (int k = 0; k < 3 && rc == MM_OK; ++k) {
            rc = batch_enqueue(b, b->par, dt, b->stream);
            b->par = 1 - b->par;
        }
        cudaEventRecord(e1, b->stream);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        ms /= 3.f;
        if (ms_out) ms_out[c] = ms;
        if (ms < best) {
            best = ms;
            bi = c;
        }
    }
    // second stage: kx planes per plane-pass CTA with the best x-pass shapes
    static const int cand2[] = {1, 2, 4, 8};
    int b2 = 0;
    float best2 = 1e30f;
    for (int c = 0; c < 4 && rc == MM_OK; ++c) {
        b->r1 = cand[bi][0];
        b->r3 = cand[bi][1];
        b->threads = cand[bi][2];
        b->r2 = cand2[c];
        rc = batch_layout(b);
        if (rc != MM_OK) break;
        rc = batch_pass1(b, b->par, b->stream);
        if (rc == MM_OK) rc = batch_enqueue(b, b->par, dt, b->stream);   // warm-up
        if (rc != MM_OK) break;
        b->par = 1 - b->par;
        cudaEventRecord(e0, b->stream);
        for (int k = 0; k < 3 && rc == MM_OK; ++k) {
            rc = batch_enqueue(b, b->par, dt, b->stream);
            b->par = 1 - b->par;
        }
        cudaEventRecord(e1, b->stream);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        ms /= 3.f;
        if (ms_out) ms_out[nc + c] = ms;
        if (ms < best2) {
            best2 = ms;
            b2 = c;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc == MM_OK) {
        b->r1 = cand[bi][0];
        b->r3 = cand[bi][1];
        b->threads = cand[bi][2];
        b->r2 = cand2[b2];
        rc = batch_layout(b);
    }
    cudaMemcpyAsync(b->par ? b->M1 : b->M0, save, sizeof(float) * b->mtotal, cudaMemcpyDeviceToDevice, b->stream);
    cudaMemsetAsync(b->flag, 0, sizeof(int), b->stream);
    cudaStreamSynchronize(b->stream);
    cudaFree(save);
    b->spec_valid = false;
    if (rc != MM_OK) return rc;
    if (choice) {
        choice[0] = b->r1;
        choice[1] = b->r3;
        choice[2] = b->threads;
        choice[3] = b->r2;
    }
    return MM_OK;
}
