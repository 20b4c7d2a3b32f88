// split_fast.cu -- instantiations of the compile-time split pass 2
// (split_fast.cuh) for power-of-two thick samples, and its launch.
#include "split_fast.cuh"

namespace mmk {

template <int NY> static void fill_y(FastSplitFns* f) {
    f->yf = k_yfwd_fast<NY>;
    f->yi = k_yinv_fast<NY>;
    f->ylpc = YLayout<NY>::LPC;
    f->ty = YLayout<NY>::THREADS;
    f->sy = YLayout<NY>::BYTES;
}
template <int NZ> static void fill_z(FastSplitFns* f) {
    f->zc = k_zconv_fast<NZ>;
    f->zw = ZLayout<NZ>::W;
    f->tz = ZLayout<NZ>::THREADS;
    f->sz = ZLayout<NZ>::BYTES;
}
template <int NZ> static void fill_zcol(FastSplitFns* f) {
    f->zc = k_zcol_fast<NZ>;
    f->zw = 0;                               // marks the one-position-per-thread kernel
    f->tz = kZcolThreads;
    f->sz = 0;
}

bool fast_split_lookup(int ny, int nz, FastSplitFns* f) {
    switch (ny) {
        case 16: fill_y<16>(f); break;
        case 32: fill_y<32>(f); break;
        case 64: fill_y<64>(f); break;
        case 128: fill_y<128>(f); break;
        case 256: fill_y<256>(f); break;
        case 512: fill_y<512>(f); break;
        case 1024: fill_y<1024>(f); break;
        default: return false;
    }
    switch (nz) {
        case 1: fill_zcol<1>(f); break;
        case 2: fill_zcol<2>(f); break;
        case 4: fill_zcol<4>(f); break;
        case 8: fill_zcol<8>(f); break;
        case 16: fill_z<16>(f); break;
        case 32: fill_z<32>(f); break;
        case 64: fill_z<64>(f); break;
        case 128: fill_z<128>(f); break;
        default: return false;
    }
    return true;
}

cudaError_t configure_fast_split(const FastSplitFns& f) {
    cudaError_t e = cudaFuncSetAttribute(f.yf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)f.sy);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f.yi, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)f.sy);
    if (e == cudaSuccess && f.sz) e = cudaFuncSetAttribute(f.zc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)f.sz);
    return e;
}

cudaError_t launch_fast_split(const Geom& g, const FastSplitFns& f, const float* Kt, float2* S, cudaStream_t s) {
    cudaLaunchAttribute attr[1];
    const int lines = g.Hx * 3 * g.nz;
    const int gy = (lines + f.ylpc - 1) / f.ylpc;
    cudaLaunchConfig_t cy = launch_config(dim3(gy), f.ty, f.sy, s, attr);
    cudaError_t e = cudaLaunchKernelEx(&cy, f.yf, g, S);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cz = f.zw ? launch_config(dim3(g.Hx * (g.Ly / f.zw)), f.tz, f.sz, s, attr)
                                 : launch_config(dim3(1), f.tz, 0, s, attr);
    if (!f.zw) cz.gridDim = dim3((g.Ly + f.tz - 1) / f.tz, g.Hx);
    e = cudaLaunchKernelEx(&cz, f.zc, g, Kt, S);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cy, f.yi, g, S);
}

// The x-step kernel in place on S: it reads its tile of S (all kx of R rows
// of a layer) into shared memory before it writes the same tile back.
cudaError_t launch_xstep(const Geom& g, const FastStepFns& fs, const LlgCoef& c, int mode, float2* S, const float* M,
                         float* out, int* flag, cudaStream_t s, float* Mcopy) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = launch_config(dim3(g.nz * (g.Jr / fs.rb)), fs.tb, fs.sb, s, attr);
    return cudaLaunchKernelEx(&cfg, fs.kb[mode], g, c, (const float2*)S, mode == kModeStep ? S : (float2*)nullptr,
                              M, out, mode == kModeStep ? flag : (int*)nullptr,
                              mode == kModeStep ? Mcopy : (float*)nullptr);
}

cudaError_t launch_split_xstep(const Geom& g, const FastSplitFns& f2, const FastStepFns& fs, const LlgCoef& c,
                               int mode, const float* Kt, float2* S, const float* M, float* out, int* flag,
                               cudaStream_t s, float* Mcopy) {
    cudaError_t e = launch_fast_split(g, f2, Kt, S, s);
    if (e != cudaSuccess) return e;
    return launch_xstep(g, fs, c, mode, S, M, out, flag, s, Mcopy);
}

}  // namespace mmk
