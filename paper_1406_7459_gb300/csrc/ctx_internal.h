// ctx_internal.h -- the solver context behind the C ABI, shared by the
// translation units that implement include/mm.h (mm_api.cu, adaptive.cu,
// step_surrogate.cu).
#pragma once
#include <cuda_runtime.h>

#include "../../include/mm.h"
#include "mm_internal.h"

namespace mmk {

// Record a message for mm_last_error() and return `code`.
int set_error_fmt(int code, const char* fmt, ...);

}  // namespace mmk

#define CU(expr)                                                                               \
    do {                                                                                       \
        cudaError_t _e = (expr);                                                               \
        if (_e != cudaSuccess)                                                                 \
            return mmk::set_error_fmt(_e == cudaErrorMemoryAllocation ? MM_ENOMEM : MM_ECUDA,   \
                                      "%s: %s (%s:%d)", #expr, cudaGetErrorString(_e), __FILE__, \
                                      __LINE__);                                               \
    } while (0)

// internal header of the ABI translation units: the kernels' types unqualified
using namespace mmk;

struct mm_ctx {
    int grid[3];
    double cell[3];
    double Ms, A, Ku, alpha, gamma;
    double Hext[3];
    cudaStream_t stream;
    cudaStream_t cap;          // private stream used only for graph capture
    int device;
    Geom g;
    Geom gf;                   // geometry of the two-kernel step: g, or a ragged film's carrier lengths
    Launch l;
    float* Kt = nullptr;
    float* Kd = nullptr;       // 2-D spectrum per z offset, exchange folded in (two-kernel step)
    float* Kd0 = nullptr;      // the same without exchange (two-kernel demag evaluation)
    float2* S = nullptr;
    float* Mbuf[2] = {nullptr, nullptr};
    int cur = 0;
    float* H = nullptr;
    int* flag = nullptr;
    double* partials = nullptr;
    double* Edev = nullptr;
    double* Ehost = nullptr;   // page-locked copy
    float2* tw = nullptr;      // twiddles of x, y, z back to back
    // step graphs [kind][parity]: kind 0 one step, kind 1 kGraphSteps steps
    cudaGraphExec_t step_exec[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};
    double step_dt[2][2] = {{0, 0}, {0, 0}};
    unsigned long long step_ver[2][2] = {{0, 0}, {0, 0}};
    unsigned long long ver = 1;   // bumped when H_ext changes
    int warm = 0;                 // steps launched directly with warm_dt, warm_ver (mm_step)
    double warm_dt = 0;
    unsigned long long warm_ver = 0;
    bool use_graphs = true;
    int form = -1;                // mm_step_form of the last run of steps
    FastFns fast;              // compile-time kernels (when the grid has them)
    FastStepFns fs;            // two-kernel step (films on compile-time lengths)
    FastSplitFns fsplit;       // compile-time split pass 2 (thick samples)
    bool has_fs = false;
    bool rag = false;          // has_fs or has_ss through the ragged kernels; Kt is formed on demand
    bool has_ss = false;       // thick samples: compile-time split pass 2 + the x-step kernel
    bool has_gx = false;       // generic x passes: the step's pass 3 also forms the next x spectrum
    float* Kt_ex = nullptr;    // has_ss: tensor spectrum with the exchange stencil folded in (ragged: plain,
                               // on the carrier lengths)
    float2* Sh = nullptr;      // plane-kernel output of the two-kernel step (layout of S)
    int method = MM_INTEGRATOR_EULER;
    float* Mst = nullptr;      // Runge-Kutta stage state
    float* acc = nullptr;      // Runge-Kutta weighted slope sum
    float* sur = nullptr;      // surrogate stepper: M_ref, H_ref, x, y, H_d (5 x 3N)
    double* sur_r = nullptr;   // residual sums
    bool spec_valid = false;   // S holds the x half-spectrum of M[cur] (two-kernel step)
    float* dpk[7] = {};        // Dormand-Prince stage slopes (adaptive runs), 3*N each
    unsigned* dperr = nullptr; // error estimate of the last trial step (float bits)
    unsigned* hperr = nullptr; // its page-locked host copy
    PersistFns pf;             // persistent step (square power-of-two films it is built for)
    bool has_persist = false;  // the persistent step fits this grid and device
    int step_path = MM_STEP_AUTO;
    long long wait_limit = kGridWaitLimit;   // polls of a grid-barrier wait
    GridBar* gbar = nullptr;   // grid-barrier counters of the persistent step
};

namespace mmk {

// Field and LLG coefficients of the context for a step of size dt.
LlgCoef make_coef(const mm_ctx* c, double dt);
// x R2C, plane, x C2R (+ field / step per mode) of M into out on stream s;
// invalidates a pending step spectrum.
cudaError_t form_spectrum(mm_ctx* c, const float* M, cudaStream_t s, float* Mcopy = nullptr,
                          const XComb& comb = XComb{});
// Whether a Runge-Kutta stage of this context is the plane pass and one
// kernel (fused_stage) instead of a field evaluation and a stage update.
// On films up to kFusedCells: there a stage saves two launches and passes
// (us per RK4 step, fused against field evaluations and stage updates:
// 256x256x4 70 against 80, 600x400x1 115 against 127, 200x300x6 201 against
// 205); on larger ones the stage kernel's registers cost more than the passes
// (400x480x2 213 against 211, 620x640x1 198 against 193, 512x512x4 408 against
// 390, 1000x1000x1 513 against 408).  Not where the plane kernel runs more
// than 512 threads.  Thick samples gain throughout (100x80x20 145 against
// 148, 160x120x20 229 against 241, 256x256x16 369 against 375; 200x160x20 423
// against 417).
constexpr int kFusedCells = 370000;
inline bool fused_stages(const mm_ctx* c) {
    return c->has_fs ? c->g.N <= kFusedCells && (c->rag || c->fs.ta <= 512) : c->has_ss && (c->rag || c->l.fx);
}
// One stage at the state Y whose x spectrum is in S: the slope's use per st
// (mode kModeStage, which leaves the next state's spectrum in S, or kModeErr).
int fused_stage(mm_ctx* c, int mode, const float* Y, const StageArgs& st, const LlgCoef& cf, cudaStream_t s);
int run_passes(mm_ctx* c, int mode, const float* M, float* out, double dt, cudaStream_t s);

}  // namespace mmk
