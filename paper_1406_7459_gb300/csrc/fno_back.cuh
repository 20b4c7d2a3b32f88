// fno_back.cuh -- backward kernels of the FNO surrogate (fno.cu) that pass
// over whole activations, one pass per layer.
//
// Bound by HBM: at width 32, batch 8 and 256 x 256 pixels an activation is
// 67 MB in FP32, more than a third of L2 with its neighbours.  A layer's
// backward pass reads the gradient, the pre-activation and the layer's input
// once and writes the BF16 gradient for the spectral path and W^T du once
// (0.3 GB); the activation's derivative, the BF16 copy, the weight gradient
// and the channel map as separate kernels moved 0.77 GB.  Measured there: a
// layer 97 us against 269 in the four kernels, the head 25 against 140, the
// lift's gradient 20 against 71, loss and gradients in all 2.87 -> 1.55 ms.
// A layer is bound by instruction issue (erf and exp of the derivative) next
// to HBM.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "mm_internal.h"

namespace mmk {

// a b + c per lane, two FP32 lanes per instruction
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_pack(a)), "l"(f2_pack(b)), "l"(f2_pack(c)));
    return f2_unpack(r);
}

// (sr, si) += (a + i c)(xr + i xi) with the roundings of k_mode_inv's sums over
// rows and over channels, spelled out: left to the compiler's contraction, an
// imaginary part of k_y_inverse differed in its last bit now and then, and a
// few values in 10^5 turned over in BF16 (62 x 86, width 16, 16 modes, batch 6:
// gradients 1.4e-5 apart, 8e-8 so; times unchanged).  Spelled out in
// k_mode_inv too, forward passes got up to 4 % slower (64 x 64, width 32,
// batch 4: 134.6 us and 140.6).
__device__ __forceinline__ void row_term(float a, float c, float xr, float xi, float& sr, float& si) {
    sr = __fadd_rn(sr, fmaf(a, xr, -__fmul_rn(c, xi)));
    si = __fadd_rn(si, fmaf(a, xi, __fmul_rn(c, xr)));
}
__device__ __forceinline__ void mode_term(float a, float c, float xr, float xi, float& sr, float& si) {
    sr = __fadd_rn(sr, fmaf(a, xr, -__fmul_rn(c, xi)));
    si = __fadd_rn(si, fmaf(c, xr, __fmul_rn(a, xi)));
}

__device__ __forceinline__ float gelu_grad_f(float x) {
    return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * expf(-0.5f * x * x) * 0.3989422804014327f;
}

// Pixels p .. p+3 of a channel row of np pixels (zero past it).
__device__ __forceinline__ float4 load_px4(const float* __restrict__ row, long long p, long long np, bool vec) {
    if (vec && p + 4 <= np) return *reinterpret_cast<const float4*>(row + p);
    float4 v;
    v.x = p < np ? row[p] : 0.f;
    v.y = p + 1 < np ? row[p + 1] : 0.f;
    v.z = p + 2 < np ? row[p + 2] : 0.f;
    v.w = p + 3 < np ? row[p + 3] : 0.f;
    return v;
}
__device__ __forceinline__ void store_px4(float* __restrict__ row, long long p, long long np, bool vec, float4 v) {
    if (vec && p + 4 <= np) {
        *reinterpret_cast<float4*>(row + p) = v;
        return;
    }
    if (p < np) row[p] = v.x;
    if (p + 1 < np) row[p + 1] = v.y;
    if (p + 2 < np) row[p + 2] = v.z;
    if (p + 3 < np) row[p + 3] = v.w;
}

// What the gradient of a layer's pre-activation is made of.
enum LayerBack { kBackAct = 0, kBackHead = 1 };   // dv gelu'(u); Q^T dy (the last layer)

// One layer: du = dv gelu'(u), or Q^T dy, in BF16 into db16; out = W^T du;
// per block the partial sums of gW[o][c] = sum_p du[o][p] v[c][p] and gb[o] =
// sum_p du[o][p] (CW CW + CW floats; k_back_reduce adds them: a block's atomic
// adds on the 33 cache lines of a layer's gradient queued for 20 us).
// A block walks tiles of TP pixels of one sample: du and v staged in shared
// memory (row stride TP + 4: the eight row groups of a warp start four banks
// apart), then 4 x 4 (o, c) tiles of the weight gradient per thread and
// pixel group, every operand a 16-byte read of four pixels, two pixels per
// FMA; and 4 pixels x OC channels of the channel map per thread.
template <int CW> struct LayerBackCfg {
    static constexpr int T = 256;
    static constexpr int TP = CW <= 16 ? 256 : (CW <= 32 ? 128 : 64);
    static constexpr int TS = TP + 4;
    static constexpr int NG = CW / 4;                     // row groups per operand
    static constexpr int GS = NG * NG, PG = T / GS;       // threads per (o, c) grid, pixel groups
    static constexpr int QUADS = TP / 4;
    static constexpr int OC = CW / (T / QUADS);           // channel-map outputs per thread
    static constexpr int TILE = CW * TS;
    static constexpr size_t BYTES = sizeof(float) * (2 * TILE > T * 16 ? 2 * TILE : T * 16);
};

template <int CW, int KIND>
__global__ void __launch_bounds__(256, CW <= 32 ? 3 : 2)
    k_layer_back(const float* __restrict__ dv, const float* __restrict__ u, const float* __restrict__ v,
                 const float* __restrict__ W, const float* __restrict__ Q, long long np, int B,
                 __nv_bfloat16* __restrict__ db16, float* __restrict__ out, float* __restrict__ part) {
    using Cfg = LayerBackCfg<CW>;
    constexpr int T = Cfg::T, TP = Cfg::TP, TS = Cfg::TS, NG = Cfg::NG, GS = Cfg::GS, PG = Cfg::PG;
    constexpr int QUADS = Cfg::QUADS, OC = Cfg::OC;
    static_assert(PG <= QUADS && T % QUADS == 0 && CW * QUADS % T == 0 && (OC == 4 || OC == 2), "tiling");
    extern __shared__ __align__(16) float lb_smem[];
    pdl_wait();
    pdl_trigger();
    __shared__ __align__(16) float Ws[CW * CW];
    __shared__ float Qs[3 * CW];
    __shared__ float bs[CW];
    float* as = lb_smem;                                  // du [o][TS]
    float* fs = lb_smem + Cfg::TILE;                      // v [c][TS]
    for (int i = threadIdx.x; i < CW * CW; i += T) Ws[i] = W[i];
    for (int i = threadIdx.x; i < CW; i += T) bs[i] = 0.f;
    if constexpr (KIND == kBackHead)
        for (int i = threadIdx.x; i < 3 * CW; i += T) Qs[i] = Q[i];
    const bool vec = (np & 3) == 0;
    const long long tpb = (np + TP - 1) / TP, ntiles = (long long)B * tpb;
    const int gi = threadIdx.x % GS, pg = threadIdx.x / GS;
    const int gc = gi % NG, go = gi / NG;
    const int qd = threadIdx.x % QUADS, c0 = (threadIdx.x / QUADS) * OC;
    float2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int b = (int)(tile / tpb);
        const long long p0 = (tile - (long long)b * tpb) * TP;
        __syncthreads();                                  // the previous tile's reads are done
        // each trip takes T / QUADS rows: row r0 + n (T / QUADS), quad qd
        const int r0 = threadIdx.x / QUADS;
        const long long p = p0 + 4 * qd, row0 = ((long long)b * CW + r0) * np;
        const bool whole = vec && p + 4 <= np;
        float4 y0, y1, y2;
        if constexpr (KIND == kBackHead) {
            const float* dy = dv + (long long)b * 3 * np;
            y0 = load_px4(dy, p, np, vec);
            y1 = load_px4(dy + np, p, np, vec);
            y2 = load_px4(dy + 2 * np, p, np, vec);
        }
        constexpr int TRIPS = CW * QUADS / T;
        const long long dr = (long long)(T / QUADS) * np;
        const float* dvp = dv + row0;                     // kBackAct only
        const float* up = u + row0;
        const float* vp = v + row0;
        __nv_bfloat16* hp = db16 + row0 + p;
#pragma unroll (TRIPS < 4 ? TRIPS : 4)
        for (int n = 0; n < TRIPS; ++n) {
            const int r = r0 + n * (T / QUADS);
            float4 dd, x, f;
            if (whole) {
                if constexpr (KIND == kBackAct) {
                    dd = *reinterpret_cast<const float4*>(dvp + p);
                    x = *reinterpret_cast<const float4*>(up + p);
                }
                f = *reinterpret_cast<const float4*>(vp + p);
            } else {
                if constexpr (KIND == kBackAct) {
                    dd = load_px4(dvp, p, np, false);
                    x = load_px4(up, p, np, false);
                }
                f = load_px4(vp, p, np, false);
            }
            if constexpr (KIND == kBackHead) {
                const float w0 = Qs[r], w1 = Qs[CW + r], w2 = Qs[2 * CW + r];
                dd.x = fmaf(w2, y2.x, fmaf(w1, y1.x, w0 * y0.x));
                dd.y = fmaf(w2, y2.y, fmaf(w1, y1.y, w0 * y0.y));
                dd.z = fmaf(w2, y2.z, fmaf(w1, y1.z, w0 * y0.z));
                dd.w = fmaf(w2, y2.w, fmaf(w1, y1.w, w0 * y0.w));
            } else {
                dd.x *= gelu_grad_f(x.x);
                dd.y *= gelu_grad_f(x.y);
                dd.z *= gelu_grad_f(x.z);
                dd.w *= gelu_grad_f(x.w);
            }
            *reinterpret_cast<float4*>(as + r * TS + 4 * qd) = dd;
            *reinterpret_cast<float4*>(fs + r * TS + 4 * qd) = f;
            if (whole) {
                __nv_bfloat162 h[2] = {__floats2bfloat162_rn(dd.x, dd.y), __floats2bfloat162_rn(dd.z, dd.w)};
                *reinterpret_cast<uint2*>(hp) = *reinterpret_cast<uint2*>(h);
            } else {
                if (p < np) hp[0] = __float2bfloat16(dd.x);
                if (p + 1 < np) hp[1] = __float2bfloat16(dd.y);
                if (p + 2 < np) hp[2] = __float2bfloat16(dd.z);
                if (p + 3 < np) hp[3] = __float2bfloat16(dd.w);
            }
            dvp += dr;
            up += dr;
            vp += dr;
            hp += dr;
        }
        __syncthreads();
        // weight gradient: rows o = go + NG i, c = gc + NG j of pixel quads
        // pg, pg + PG, ...
#pragma unroll 2
        for (int q = pg; q < QUADS; q += PG) {
            float4 a[4], f[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(as + (go + NG * i) * TS + 4 * q);
#pragma unroll
            for (int j = 0; j < 4; ++j) f[j] = *reinterpret_cast<const float4*>(fs + (gc + NG * j) * TS + 4 * q);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j] = fma2(make_float2(a[i].x, a[i].y), make_float2(f[j].x, f[j].y), acc[i][j]);
                    acc[i][j] = fma2(make_float2(a[i].z, a[i].w), make_float2(f[j].z, f[j].w), acc[i][j]);
                }
        }
        // channel map out[c][p] = sum_o W[o][c] du[o][p], o ascending
        {
            float2 lo[OC], hi[OC];
#pragma unroll
            for (int j = 0; j < OC; ++j) lo[j] = hi[j] = make_float2(0.f, 0.f);
#pragma unroll 8
            for (int o = 0; o < CW; ++o) {
                const float4 d = *reinterpret_cast<const float4*>(as + o * TS + 4 * qd);
                float w[OC];
                if constexpr (OC == 4) {
                    const float4 w4 = *reinterpret_cast<const float4*>(Ws + o * CW + c0);
                    w[0] = w4.x;
                    w[1] = w4.y;
                    w[2] = w4.z;
                    w[3] = w4.w;
                } else {
                    const float2 w2 = *reinterpret_cast<const float2*>(Ws + o * CW + c0);
                    w[0] = w2.x;
                    w[1] = w2.y;
                }
#pragma unroll
                for (int j = 0; j < OC; ++j) {
                    const float2 ww = make_float2(w[j], w[j]);
                    lo[j] = fma2(ww, make_float2(d.x, d.y), lo[j]);
                    hi[j] = fma2(ww, make_float2(d.z, d.w), hi[j]);
                }
            }
#pragma unroll
            for (int j = 0; j < OC; ++j)
                store_px4(out + ((long long)b * CW + c0 + j) * np, p, np, vec,
                          make_float4(lo[j].x, lo[j].y, hi[j].x, hi[j].y));
        }
        // bias: rows of the tile, eight threads each... one partial per thread
        for (int e = threadIdx.x; e < CW * 8; e += T) {
            const int r = e / 8, s = e % 8;
            float t = 0.f;
            for (int q = s; q < QUADS; q += 8) {
                const float4 d = *reinterpret_cast<const float4*>(as + r * TS + 4 * q);
                t += (d.x + d.y) + (d.z + d.w);
            }
            for (int o = 4; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o, 8);
            if (s == 0) bs[r] += t;                       // one thread per row
        }
    }
    // the pixel groups' sums through shared memory, this block's partial
    __syncthreads();
    part += (size_t)blockIdx.x * (CW * CW + CW);
    float* red = lb_smem;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) red[threadIdx.x * 16 + i * 4 + j] = acc[i][j].x + acc[i][j].y;
    __syncthreads();
    for (int e = threadIdx.x; e < CW * CW; e += T) {
        const int o = e / CW, c = e % CW;
        const int g = (o % NG) * NG + c % NG, k = (o / NG) * 4 + c / NG;
        float s = 0.f;
        for (int q = 0; q < PG; ++q) s += red[(q * GS + g) * 16 + k];
        part[e] = s;
    }
    for (int i = threadIdx.x; i < CW; i += T) part[CW * CW + i] = bs[i];
}

// The head: dy = 2 (y - t) / n into dy, the loss sum, and per block the
// partial sums of gQ[j][c] = sum_p dy[j][p] v[c][p] and gq[j] = sum_p dy[j][p]
// (3 CW + 3).  A block takes kHeadPx pixels
// of one sample (four per thread); a warp takes the channels w, w + 8, ... of
// them, lanes on pixel quads.
constexpr int kHeadPx = 1024;
template <int CW>
__global__ void __launch_bounds__(256, CW <= 32 ? 4 : 2) k_head_back(const float* __restrict__ y, const float* __restrict__ t,
                                                   const float* __restrict__ v, long long np, long long n,
                                                   float* __restrict__ dy, double* __restrict__ loss,
                                                   float* __restrict__ part) {
    constexpr int CH = (CW + 7) / 8;                      // channels per warp
    pdl_wait();
    pdl_trigger();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long cpb = (np + kHeadPx - 1) / kHeadPx;
    const int b = (int)(blockIdx.x / cpb);
    const long long p0 = (blockIdx.x - (long long)b * cpb) * kHeadPx;
    const bool vec = (np & 3) == 0;
    const bool vec_t = vec && (reinterpret_cast<uintptr_t>(t) & 15) == 0;   // the caller's buffer
    // dy of the chunk, formed once per block
    __shared__ __align__(16) float ds[3][kHeadPx];
    part += (size_t)blockIdx.x * (3 * CW + 3);
    const float fn = (float)n;
    float acc[CH][3];
#pragma unroll
    for (int k = 0; k < CH; ++k) acc[k][0] = acc[k][1] = acc[k][2] = 0.f;
    double ls = 0.0;
    float sq[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const long long row = ((long long)b * 3 + j) * np, p = p0 + 4 * threadIdx.x;
        const float4 a = load_px4(y + row, p, np, vec), c = load_px4(t + row, p, np, vec_t);
        const float4 e = make_float4(a.x - c.x, a.y - c.y, a.z - c.z, a.w - c.w);
        const float4 d = make_float4(2.f * e.x / fn, 2.f * e.y / fn, 2.f * e.z / fn, 2.f * e.w / fn);
        ls += (double)e.x * e.x + (double)e.y * e.y + (double)e.z * e.z + (double)e.w * e.w;
        sq[j] = (d.x + d.y) + (d.z + d.w);
        *reinterpret_cast<float4*>(&ds[j][4 * threadIdx.x]) = d;   // zero past np
        store_px4(dy + row, p, np, vec, d);
    }
    __syncthreads();
#pragma unroll 2
    for (int q = lane; q < kHeadPx / 4; q += 32) {
        const long long p = p0 + 4 * q;
        if (p >= np) break;
        float4 x[CH];
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            const int c = warp + 8 * k;
            if (c < CW) x[k] = load_px4(v + ((long long)b * CW + c) * np, p, np, vec);
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float4 d = *reinterpret_cast<const float4*>(&ds[j][4 * q]);
#pragma unroll
            for (int k = 0; k < CH; ++k)
                if (warp + 8 * k < CW)
                    acc[k][j] += (d.x * x[k].x + d.y * x[k].y) + (d.z * x[k].z + d.w * x[k].w);
        }
    }
#pragma unroll
    for (int k = 0; k < CH; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            float s = acc[k][j];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (lane == 0 && warp + 8 * k < CW) part[j * CW + warp + 8 * k] = s;
        }
    for (int o = 16; o > 0; o >>= 1) ls += __shfl_down_sync(0xffffffffu, ls, o);
    __shared__ double lsum[8];
    __shared__ float qsum[8][3];
#pragma unroll
    for (int j = 0; j < 3; ++j)
        for (int o = 16; o > 0; o >>= 1) sq[j] += __shfl_down_sync(0xffffffffu, sq[j], o);
    if (lane == 0) {
        lsum[warp] = ls;
        for (int j = 0; j < 3; ++j) qsum[warp][j] = sq[j];
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        float s = 0.f;
        for (int w = 0; w < 8; ++w) s += qsum[w][threadIdx.x];
        part[3 * CW + threadIdx.x] = s;
    }
    if (threadIdx.x == 32) {
        double s = 0.0;
        for (int w = 0; w < 8; ++w) s += lsum[w];
        atomicAdd(loss, s);
    }
}

// The lift: per block the partial sums of gP[o][f] = sum_p dv[o][p] x_f[p]
// over the features (three inputs, y / H, x / W) and gp[o] = sum_p dv[o][p]
// (6 CW); tiled like the head.
template <int CW>
__global__ void __launch_bounds__(256, CW <= 32 ? 4 : 2) k_lift_back(const float* __restrict__ dv, const float* __restrict__ x, int H,
                                                   int W, float* __restrict__ part) {
    constexpr int CH = (CW + 7) / 8;
    pdl_wait();
    pdl_trigger();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long np = (long long)H * W, cpb = (np + kHeadPx - 1) / kHeadPx;
    const int b = (int)(blockIdx.x / cpb);
    const long long p0 = (blockIdx.x - (long long)b * cpb) * kHeadPx;
    const bool vec = (np & 3) == 0;
    const bool vec_x = vec && (reinterpret_cast<uintptr_t>(x) & 15) == 0;   // the caller's buffer
    // the chunk's features, formed once per block
    __shared__ __align__(16) float fs[5][kHeadPx];
    part += (size_t)blockIdx.x * (6 * CW);
    {
        const long long p = p0 + 4 * threadIdx.x;
#pragma unroll
        for (int j = 0; j < 3; ++j)
            *reinterpret_cast<float4*>(&fs[j][4 * threadIdx.x]) =
                load_px4(x + ((long long)b * 3 + j) * np, p, np, vec_x);
        int yy = (int)(p / W), xx = (int)(p - (long long)yy * W);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            fs[3][4 * threadIdx.x + e] = (float)yy / (float)H;
            fs[4][4 * threadIdx.x + e] = (float)xx / (float)W;
            if (++xx == W) {
                xx = 0;
                ++yy;
            }
        }
    }
    float acc[CH][6];
#pragma unroll
    for (int k = 0; k < CH; ++k)
#pragma unroll
        for (int f = 0; f < 6; ++f) acc[k][f] = 0.f;
    __syncthreads();
#pragma unroll 2
    for (int q = lane; q < kHeadPx / 4; q += 32) {
        const long long p = p0 + 4 * q;
        if (p >= np) break;
        float4 a[CH];                                     // zero past np
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            const int c = warp + 8 * k;
            a[k] = c < CW ? load_px4(dv + ((long long)b * CW + c) * np, p, np, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
            acc[k][5] += (a[k].x + a[k].y) + (a[k].z + a[k].w);
        }
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            const float4 f = *reinterpret_cast<const float4*>(&fs[j][4 * q]);
#pragma unroll
            for (int k = 0; k < CH; ++k)
                acc[k][j] += (a[k].x * f.x + a[k].y * f.y) + (a[k].z * f.z + a[k].w * f.w);
        }
    }
#pragma unroll
    for (int k = 0; k < CH; ++k)
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            float s = acc[k][j];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            const int c = warp + 8 * k;
            if (lane == 0 && c < CW) part[j < 5 ? c * 5 + j : 5 * CW + c] = s;
        }
}

// Adds the blocks' partials into the gradient, in block order: job j < L is
// layer j, L the head, L + 1 the lift; 32 outputs per block, eight threads
// to each.
struct BackJobs {
    const float *layer, *head, *lift;          // partials: L x nl blocks, nh blocks, nh blocks
    float *gW, *gb, *gQ, *gq, *gP, *gp;
    int C, L, nl, nh;
    long long layer_stride;                    // floats between two layers' partials
};
__global__ void __launch_bounds__(256) k_back_reduce(BackJobs q) {
    pdl_wait();
    const int job = blockIdx.y, C = q.C;
    const int n = job < q.L ? C * C + C : (job == q.L ? 3 * C + 3 : 6 * C);
    const int nb = job < q.L ? q.nl : q.nh;
    const float* src = job < q.L ? q.layer + job * q.layer_stride : (job == q.L ? q.head : q.lift);
    const int e = blockIdx.x * 32 + (threadIdx.x & 31), seg = threadIdx.x >> 5;
    if (blockIdx.x * 32 >= n) return;
    __shared__ float red[8][32];
    float s = 0.f;
    if (e < n)
#pragma unroll 8
        for (int b = seg; b < nb; b += 8) s += src[(size_t)b * n + e];
    red[seg][threadIdx.x & 31] = s;
    __syncthreads();
    if (seg != 0 || e >= n) return;
    float t = 0.f;
    for (int k = 0; k < 8; ++k) t += red[k][threadIdx.x];
    if (job < q.L) {
        if (e < C * C) q.gW[(size_t)job * C * C + e] = t;
        else q.gb[(size_t)job * C + e - C * C] = t;
    } else if (job == q.L) {
        if (e < 3 * C) q.gQ[e] = t;
        else q.gq[e - 3 * C] = t;
    } else {
        if (e < 5 * C) q.gP[e] = t;
        else q.gp[e - 5 * C] = t;
    }
}

// Batches: the per-mode channel mix,
//   w[b][o][md] = sum_c R[c][o][md] vh[b][c][md]  (conjT: conj(R[o][c][md])),
// a block per (32 modes, o, kMixNB samples), the channels 2 w and 2 w + 1
// modulo 8 to warp w (C even), the samples in registers so that one read of R
// serves them all (loads past the batch are clamped, so that they all issue
// together).  The eight partial sums are added in k_mode_inv's order, for the
// same bits ahead of the BF16 rounding.  Bound by the latency of its loads from L2:
// loss and gradients at 256 x 256, width 32, 16 modes, batch 8 took 1733 us
// with all eight samples in one block and 1640 with four in each of two; then
// 1607 with a warp's channels one after the other and 1572 unrolled over
// them, so that its loads issue together (each pair from one run).
constexpr int kMixNB = 4;
__global__ void __launch_bounds__(128) k_mode_mix(const float* __restrict__ vr, const float* __restrict__ vi,
                                                  const float* __restrict__ Rre, const float* __restrict__ Rim, int C,
                                                  int nmode, int B, int conjT, float* __restrict__ wr,
                                                  float* __restrict__ wi) {
    __shared__ float red[4][2 * kMixNB][32];
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, o = blockIdx.y, b0 = blockIdx.z * kMixNB;
    const int md = blockIdx.x * 32 + lane, mc = min(md, nmode - 1);
    const float sgn = conjT ? -1.f : 1.f;
    const long long xs = (long long)C * nmode;            // one sample's modes
    float sr[2][kMixNB], si[2][kMixNB];
#pragma unroll
    for (int k = 0; k < kMixNB; ++k) sr[0][k] = sr[1][k] = si[0][k] = si[1][k] = 0.f;
    auto add = [&](int c, float (&ar)[kMixNB], float (&ai)[kMixNB]) {
        const long long ri = (conjT ? (long long)o * C + c : (long long)c * C + o) * nmode + mc;
        const float rr = __ldg(Rre + ri), rm = sgn * __ldg(Rim + ri);
#pragma unroll
        for (int k = 0; k < kMixNB; ++k) {
            const long long xi = min(b0 + k, B - 1) * xs + (long long)c * nmode + mc;
            const float xr = __ldg(vr + xi), xm = __ldg(vi + xi);
            mode_term(rr, rm, xr, xm, ar[k], ai[k]);
        }
    };
#pragma unroll 4
    for (int c = 2 * warp; c + 1 < C; c += 8) {
        add(c, sr[0], si[0]);
        add(c + 1, sr[1], si[1]);
    }
#pragma unroll
    for (int k = 0; k < kMixNB; ++k) {
        red[warp][2 * k][lane] = sr[0][k] + sr[1][k];
        red[warp][2 * k + 1][lane] = si[0][k] + si[1][k];
    }
    __syncthreads();
    for (int e = warp; e < 2 * kMixNB; e += 4) {
        const int k = e >> 1;
        if (b0 + k >= B || md >= nmode) continue;
        const float t = (red[0][e][lane] + red[1][e][lane]) + (red[2][e][lane] + red[3][e][lane]);
        (e & 1 ? wi : wr)[(b0 + k) * xs + (long long)o * nmode + md] = t;
    }
}

// and the inverse y transform: Zb[bo][y][kx] = sum_iy G[y][iy] w[bo][iy][kx]
// in BF16 (real parts at kx, imaginary parts at m + kx); m a multiple of 4.
// A block takes one (b, o) and H / gridDim.y rows y; a thread one y and four
// kx, its row of G in 16-byte reads.
__global__ void __launch_bounds__(256) k_y_inverse(const float* __restrict__ wr, const float* __restrict__ wi, int m,
                                                   const float* __restrict__ Gre, const float* __restrict__ Gim, int H,
                                                   __nv_bfloat16* __restrict__ Zb) {
    extern __shared__ __align__(16) float yi_smem[];
    pdl_wait();
    pdl_trigger();
    const int nmode = 2 * m * m, nky = 2 * m, mq = m / 4;
    float* sr_ = yi_smem;
    float* si_ = yi_smem + nmode;
    const size_t bo = blockIdx.x;
    for (int i = threadIdx.x; i < nmode / 4; i += blockDim.x) {
        reinterpret_cast<float4*>(sr_)[i] = __ldg(reinterpret_cast<const float4*>(wr + bo * nmode) + i);
        reinterpret_cast<float4*>(si_)[i] = __ldg(reinterpret_cast<const float4*>(wi + bo * nmode) + i);
    }
    __syncthreads();
    const int yr = (H + gridDim.y - 1) / gridDim.y, y0 = blockIdx.y * yr, y1 = min(H, y0 + yr);
    for (int it = threadIdx.x; it < (y1 - y0) * mq; it += blockDim.x) {
        const int y = y0 + it / mq, k0 = 4 * (it % mq);
        const float4* gr = reinterpret_cast<const float4*>(Gre + (size_t)y * nky);
        const float4* gi = reinterpret_cast<const float4*>(Gim + (size_t)y * nky);
        float4 sr = make_float4(0.f, 0.f, 0.f, 0.f), si = sr;
#pragma unroll 4
        for (int i4 = 0; i4 < nky / 4; ++i4) {
            const float4 a4 = __ldg(gr + i4), c4 = __ldg(gi + i4);
            const float av[4] = {a4.x, a4.y, a4.z, a4.w}, cv[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 xr = *reinterpret_cast<const float4*>(sr_ + (4 * i4 + e) * m + k0);
                const float4 xi = *reinterpret_cast<const float4*>(si_ + (4 * i4 + e) * m + k0);
                row_term(av[e], cv[e], xr.x, xi.x, sr.x, si.x);
                row_term(av[e], cv[e], xr.y, xi.y, sr.y, si.y);
                row_term(av[e], cv[e], xr.z, xi.z, sr.z, si.z);
                row_term(av[e], cv[e], xr.w, xi.w, sr.w, si.w);
            }
        }
        __nv_bfloat16* z = Zb + (bo * H + y) * nky + k0;
        __nv_bfloat162 hr[2] = {__floats2bfloat162_rn(sr.x, sr.y), __floats2bfloat162_rn(sr.z, sr.w)};
        __nv_bfloat162 hi[2] = {__floats2bfloat162_rn(si.x, si.y), __floats2bfloat162_rn(si.z, si.w)};
        *reinterpret_cast<uint2*>(z) = *reinterpret_cast<uint2*>(hr);
        *reinterpret_cast<uint2*>(z + m) = *reinterpret_cast<uint2*>(hi);
    }
}

// dR[c][o][mode] += sum_b dw[b][o][mode] conj(vh[b][c][mode]), four modes per
// thread (nmode a multiple of 4, 16-byte aligned rows), b ascending.
__global__ void __launch_bounds__(256) k_dR4(const float* __restrict__ dwr, const float* __restrict__ dwi,
                                             const float* __restrict__ vr, const float* __restrict__ vi, int C,
                                             int nmode, int B, float* __restrict__ gre, float* __restrict__ gim) {
    pdl_wait();
    pdl_trigger();
    const int m4 = nmode / 4;
    const int total = C * C * m4;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int md = t % m4, o = (t / m4) % C, c = t / (m4 * C);
        float4 sr = make_float4(0.f, 0.f, 0.f, 0.f), si = sr;
#pragma unroll 4
        for (int b = 0; b < B; ++b) {
            const long long io = ((long long)b * C + o) * nmode + 4 * md, ic = ((long long)b * C + c) * nmode + 4 * md;
            const float4 gr = __ldg(reinterpret_cast<const float4*>(dwr + io));
            const float4 gi = __ldg(reinterpret_cast<const float4*>(dwi + io));
            const float4 ar = __ldg(reinterpret_cast<const float4*>(vr + ic));
            const float4 ai = __ldg(reinterpret_cast<const float4*>(vi + ic));
            sr.x += gr.x * ar.x + gi.x * ai.x;
            sr.y += gr.y * ar.y + gi.y * ai.y;
            sr.z += gr.z * ar.z + gi.z * ai.z;
            sr.w += gr.w * ar.w + gi.w * ai.w;
            si.x += gi.x * ar.x - gr.x * ai.x;
            si.y += gi.y * ar.y - gr.y * ai.y;
            si.z += gi.z * ar.z - gr.z * ai.z;
            si.w += gi.w * ar.w - gr.w * ai.w;
        }
        const long long e = ((long long)c * C + o) * nmode + 4 * md;
        float4* r = reinterpret_cast<float4*>(gre + e);
        float4* m = reinterpret_cast<float4*>(gim + e);
        const float4 r0 = *r, m0 = *m;
        *r = make_float4(r0.x + sr.x, r0.y + sr.y, r0.z + sr.z, r0.w + sr.w);
        *m = make_float4(m0.x + si.x, m0.y + si.y, m0.z + si.z, m0.w + si.w);
    }
}

}  // namespace mmk
