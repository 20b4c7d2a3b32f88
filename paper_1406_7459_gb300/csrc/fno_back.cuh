// fno_back.cuh -- backward kernels of the FNO surrogate (fno.cu) that pass
// over whole activations, one pass per layer.
//
// Bound by HBM: at width 32, batch 8 and 256 x 256 pixels an activation is
// 67 MB in FP32, more than a third of L2 with its neighbours.  A layer's
// backward pass reads the gradient, the pre-activation and the layer's input
// once and writes the BF16 gradient for the spectral path and W^T du once
// (0.3 GB); the activation's derivative, the BF16 copy, the weight gradient
// and the channel map as separate kernels moved 0.77 GB.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "fft_device.cuh"

namespace mmk {

// a b + c per lane, two FP32 lanes per instruction
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_pack(a)), "l"(f2_pack(b)), "l"(f2_pack(c)));
    return f2_unpack(r);
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
// gW[o][c] += sum_p du[o][p] v[c][p]; gb[o] += sum_p du[o][p].
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
                 __nv_bfloat16* __restrict__ db16, float* __restrict__ out, float* __restrict__ gW,
                 float* __restrict__ gb) {
    using Cfg = LayerBackCfg<CW>;
    constexpr int T = Cfg::T, TP = Cfg::TP, TS = Cfg::TS, NG = Cfg::NG, GS = Cfg::GS, PG = Cfg::PG;
    constexpr int QUADS = Cfg::QUADS, OC = Cfg::OC;
    static_assert(PG <= QUADS && T % QUADS == 0 && (OC == 4 || OC == 2), "tiling");
    extern __shared__ __align__(16) float lb_smem[];
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
#pragma unroll 2
        for (int e = threadIdx.x; e < CW * QUADS; e += T) {
            const int r = e / QUADS, q = e % QUADS;
            const long long p = p0 + 4 * q, row = ((long long)b * CW + r) * np;
            float4 d;
            if constexpr (KIND == kBackHead) {
                const float* dy = dv + (long long)b * 3 * np;
                const float4 y0 = load_px4(dy, p, np, vec), y1 = load_px4(dy + np, p, np, vec),
                             y2 = load_px4(dy + 2 * np, p, np, vec);
                const float w0 = Qs[r], w1 = Qs[CW + r], w2 = Qs[2 * CW + r];
                d.x = fmaf(w2, y2.x, fmaf(w1, y1.x, w0 * y0.x));
                d.y = fmaf(w2, y2.y, fmaf(w1, y1.y, w0 * y0.y));
                d.z = fmaf(w2, y2.z, fmaf(w1, y1.z, w0 * y0.z));
                d.w = fmaf(w2, y2.w, fmaf(w1, y1.w, w0 * y0.w));
            } else {
                d = load_px4(dv + row, p, np, vec);
                const float4 x = load_px4(u + row, p, np, vec);
                d.x *= gelu_grad_f(x.x);
                d.y *= gelu_grad_f(x.y);
                d.z *= gelu_grad_f(x.z);
                d.w *= gelu_grad_f(x.w);
            }
            *reinterpret_cast<float4*>(as + r * TS + 4 * q) = d;
            *reinterpret_cast<float4*>(fs + r * TS + 4 * q) = load_px4(v + row, p, np, vec);
            __nv_bfloat16* o16 = db16 + row + p;
            if (vec && p + 4 <= np) {
                __nv_bfloat162 h[2] = {__floats2bfloat162_rn(d.x, d.y), __floats2bfloat162_rn(d.z, d.w)};
                *reinterpret_cast<uint2*>(o16) = *reinterpret_cast<uint2*>(h);
            } else {
                if (p < np) o16[0] = __float2bfloat16(d.x);
                if (p + 1 < np) o16[1] = __float2bfloat16(d.y);
                if (p + 2 < np) o16[2] = __float2bfloat16(d.z);
                if (p + 3 < np) o16[3] = __float2bfloat16(d.w);
            }
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
            const long long p = p0 + 4 * qd;
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
    // the pixel groups' sums through shared memory, one atomic per output
    __syncthreads();
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
        atomicAdd(gW + e, s);
    }
    for (int i = threadIdx.x; i < CW; i += T) atomicAdd(gb + i, bs[i]);
}

// The head: dy = 2 (y - t) / n into dy, the loss sum, gQ[j][c] += sum_p
// dy[j][p] v[c][p] and gq[j] += sum_p dy[j][p].  A block takes kHeadPx pixels
// of one sample; a warp takes the channels w, w + 8, ... of them, lanes on
// pixel quads.
constexpr int kHeadPx = 1024;
template <int CW>
__global__ void __launch_bounds__(256) k_head_back(const float* __restrict__ y, const float* __restrict__ t,
                                                   const float* __restrict__ v, long long np, long long n,
                                                   float* __restrict__ dy, double* __restrict__ loss,
                                                   float* __restrict__ gQ, float* __restrict__ gq) {
    constexpr int CH = (CW + 7) / 8;                      // channels per warp
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long cpb = (np + kHeadPx - 1) / kHeadPx;
    const int b = (int)(blockIdx.x / cpb);
    const long long p0 = (blockIdx.x - (long long)b * cpb) * kHeadPx;
    const bool vec = (np & 3) == 0;
    const bool vec_t = vec && (reinterpret_cast<uintptr_t>(t) & 15) == 0;   // the caller's buffer
    const float fn = (float)n;
    float acc[CH][3], sq[3] = {0.f, 0.f, 0.f};
    double ls = 0.0;
#pragma unroll
    for (int k = 0; k < CH; ++k) acc[k][0] = acc[k][1] = acc[k][2] = 0.f;
    for (int q = lane; q < kHeadPx / 4; q += 32) {
        const long long p = p0 + 4 * q;
        if (p >= np) break;
        float4 d[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const long long row = ((long long)b * 3 + j) * np;
            const float4 a = load_px4(y + row, p, np, vec), c = load_px4(t + row, p, np, vec_t);
            const float4 e = make_float4(a.x - c.x, a.y - c.y, a.z - c.z, a.w - c.w);
            d[j] = make_float4(2.f * e.x / fn, 2.f * e.y / fn, 2.f * e.z / fn, 2.f * e.w / fn);
            if (warp == 0) {
                ls += (double)e.x * e.x + (double)e.y * e.y + (double)e.z * e.z + (double)e.w * e.w;
                sq[j] += (d[j].x + d[j].y) + (d[j].z + d[j].w);
                store_px4(dy + row, p, np, vec, d[j]);
            }
        }
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            const int c = warp + 8 * k;
            if (c >= CW) break;
            const float4 x = load_px4(v + ((long long)b * CW + c) * np, p, np, vec);
#pragma unroll
            for (int j = 0; j < 3; ++j)
                acc[k][j] += (d[j].x * x.x + d[j].y * x.y) + (d[j].z * x.z + d[j].w * x.w);
        }
    }
#pragma unroll
    for (int k = 0; k < CH; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            float s = acc[k][j];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (lane == 0 && warp + 8 * k < CW) atomicAdd(gQ + j * CW + warp + 8 * k, s);
        }
    if (warp == 0) {
        for (int o = 16; o > 0; o >>= 1) ls += __shfl_down_sync(0xffffffffu, ls, o);
        if (lane == 0) atomicAdd(loss, ls);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            float s = sq[j];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (lane == 0) atomicAdd(gq + j, s);
        }
    }
}

// The lift: gP[o][f] += sum_p dv[o][p] x_f[p] over the features (three
// inputs, y / H, x / W), gp[o] += sum_p dv[o][p]; tiled like the head.
template <int CW>
__global__ void __launch_bounds__(256) k_lift_back(const float* __restrict__ dv, const float* __restrict__ x, int H,
                                                   int W, float* __restrict__ gP, float* __restrict__ gp) {
    constexpr int CH = (CW + 7) / 8;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long np = (long long)H * W, cpb = (np + kHeadPx - 1) / kHeadPx;
    const int b = (int)(blockIdx.x / cpb);
    const long long p0 = (blockIdx.x - (long long)b * cpb) * kHeadPx;
    const bool vec = (np & 3) == 0;
    const bool vec_x = vec && (reinterpret_cast<uintptr_t>(x) & 15) == 0;   // the caller's buffer
    float acc[CH][6];
#pragma unroll
    for (int k = 0; k < CH; ++k)
#pragma unroll
        for (int f = 0; f < 6; ++f) acc[k][f] = 0.f;
    for (int q = lane; q < kHeadPx / 4; q += 32) {
        const long long p = p0 + 4 * q;
        if (p >= np) break;
        float4 f[5];
#pragma unroll
        for (int j = 0; j < 3; ++j) f[j] = load_px4(x + ((long long)b * 3 + j) * np, p, np, vec_x);
        float cy[4], cx[4];
        int yy = (int)(p / W), xx = (int)(p - (long long)yy * W);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            cy[e] = (float)yy / (float)H;
            cx[e] = (float)xx / (float)W;
            if (++xx == W) {
                xx = 0;
                ++yy;
            }
        }
        f[3] = make_float4(cy[0], cy[1], cy[2], cy[3]);
        f[4] = make_float4(cx[0], cx[1], cx[2], cx[3]);
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            const int c = warp + 8 * k;
            if (c >= CW) break;
            const float4 a = load_px4(dv + ((long long)b * CW + c) * np, p, np, vec);   // zero past np
#pragma unroll
            for (int j = 0; j < 5; ++j)
                acc[k][j] += (a.x * f[j].x + a.y * f[j].y) + (a.z * f[j].z + a.w * f[j].w);
            acc[k][5] += (a.x + a.y) + (a.z + a.w);
        }
    }
#pragma unroll
    for (int k = 0; k < CH; ++k)
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            float s = acc[k][j];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            const int c = warp + 8 * k;
            if (lane == 0 && c < CW) atomicAdd(j < 5 ? gP + c * 5 + j : gp + c, s);
        }
}

// dR[c][o][mode] += sum_b dw[b][o][mode] conj(vh[b][c][mode]), four modes per
// thread (nmode a multiple of 4, 16-byte aligned rows), b ascending.
__global__ void __launch_bounds__(256) k_dR4(const float* __restrict__ dwr, const float* __restrict__ dwi,
                                             const float* __restrict__ vr, const float* __restrict__ vi, int C,
                                             int nmode, int B, float* __restrict__ gre, float* __restrict__ gim) {
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
