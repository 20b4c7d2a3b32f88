// energy.cu -- the energy of Eq. (1) summed in FP64.
//
// Per cell: exchange as the link sum |m_i - m_j|^2 / delta^2 over the +x,
// +y, +z neighbours that exist (each link once; the discrete form of
// A (grad m)^2 matching the free-boundary stencil of Eq. (4)), anisotropy
// (M_y^2 + M_z^2)/Ms^2, demag H_d . M and Zeeman H_ext . M.  Every block
// writes its partial sums and the last block to finish adds them in a fixed
// order, so the result is deterministic.
//
// FP64 instructions, conversions from FP32 among them, issue at about two
// per clock and SM here, so the kernel is bound by their count: a warp takes
// 31 cells of a row (the 32nd lane holds the right neighbour's values) and
// walks up kRows or kRowsLarge rows, so that a cell is converted once and
// serves its left and lower neighbours' links through a shuffle and a
// register, and the constant factors are applied to the sums: 35 FP64
// instructions per cell against 60 when every link converts its own pair.
// A call on 200x60x3 57 us with it, 82 with a thread per cell and a
// separate reduction and status read; on 512x512x8 405 against 480.
// Row and column come from the warp's index, without a division per cell.
#include "mm_internal.h"

namespace mmk {

constexpr int kEnergyThreads = 256;
constexpr int kEnergySums = 8;        // x, y, z links; M_y^2 + M_z^2; H . M; M_x, M_y, M_z
constexpr int kEnergyMaxBlocks = 1024;
constexpr int kRowsSmall = 4, kRowsLarge = 16;

// partial sums, then the count of finished blocks (zero between calls)
size_t energy_partials_elems(int) { return (size_t)kEnergyMaxBlocks * kEnergySums + 1; }

// v summed over the block; valid in thread 0.
__device__ inline double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < kEnergyThreads / 32; ++i) s += red[i];
    return s;
}

struct EnergyCoef {
    double ax, ay, az;         // A V / (Ms^2 delta^2) per axis
    double an, de;             // Ku V / Ms^2, -mu0 V / 2
    double zx, zy, zz;         // -mu0 V H_ext
};

template <int ROWS>
__global__ void __launch_bounds__(kEnergyThreads) k_energy(int nx, int ny, int nz, int wpr, int segs, int items,
                                                            const float* __restrict__ M, const float* __restrict__ H,
                                                            EnergyCoef cf, const int* __restrict__ flag,
                                                            double* __restrict__ part, double* __restrict__ out) {
    __shared__ double red[kEnergyThreads / 32];
    __shared__ bool last;
    const int lane = threadIdx.x & 31;
    const size_t N = (size_t)nx * ny * nz, sxy = (size_t)nx * ny;
    double s[kEnergySums] = {0, 0, 0, 0, 0, 0, 0, 0};
    // item: 31 columns from i0 of ROWS rows from j0 of layer k
    for (int it = blockIdx.x * (kEnergyThreads / 32) + (threadIdx.x >> 5); it < items;
         it += gridDim.x * (kEnergyThreads / 32)) {
        const int wi = it % wpr, rest = it / wpr;
        const int j0 = (rest % segs) * ROWS, k = rest / segs;
        const int i = wi * 31 + lane;
        const bool in = i < nx;                             // holds a cell's values
        const bool own = in && (lane < 31 || i + 1 == nx);  // and adds that cell's terms
        const bool right = own && i + 1 < nx;
        const size_t base = (in ? i : 0) + (size_t)nx * j0 + sxy * k;
        double m[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) m[c] = (double)M[c * N + base];
        for (int r = 0; r < ROWS && j0 + r < ny; ++r) {
            const size_t cell = base + (size_t)r * nx;
            const bool up = j0 + r + 1 < ny;
            double x[3], y[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                x[c] = __shfl_down_sync(0xffffffffu, m[c], 1);
                y[c] = up ? (double)M[c * N + cell + nx] : m[c];
            }
            if (right) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const double d = x[c] - m[c];
                    s[0] += d * d;
                }
            }
            if (own) {
                if (up) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const double d = y[c] - m[c];
                        s[1] += d * d;
                    }
                }
                if (k + 1 < nz) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const double d = (double)M[c * N + cell + sxy] - m[c];
                        s[2] += d * d;
                    }
                }
                s[3] += m[1] * m[1];
                s[3] += m[2] * m[2];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    s[4] += (double)H[c * N + cell] * m[c];
                    s[5 + c] += m[c];
                }
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) m[c] = y[c];
        }
    }
#pragma unroll
    for (int q = 0; q < kEnergySums; ++q) {
        const double t = block_sum(s[q], red);
        if (threadIdx.x == 0) part[(size_t)blockIdx.x * kEnergySums + q] = t;
    }
    unsigned long long* done = reinterpret_cast<unsigned long long*>(part + (size_t)kEnergyMaxBlocks * kEnergySums);
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(done, 1ull) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double t[kEnergySums];
#pragma unroll
    for (int q = 0; q < kEnergySums; ++q) {
        double v = 0.0;
        for (int b = threadIdx.x; b < (int)gridDim.x; b += kEnergyThreads)
            v += __ldcg(part + (size_t)b * kEnergySums + q);
        t[q] = block_sum(v, red);
    }
    if (threadIdx.x == 0) {
        const double ex = cf.ax * t[0] + cf.ay * t[1] + cf.az * t[2];
        const double an = cf.an * t[3], de = cf.de * t[4];
        const double ze = cf.zx * t[5] + cf.zy * t[6] + cf.zz * t[7];
        out[0] = ex + an + de + ze;
        out[1] = ex;
        out[2] = an;
        out[3] = de;
        out[4] = ze;
        out[5] = (double)*flag;                             // the status word, read by the same copy
        *done = 0;
    }
}

cudaError_t energy_reduce_full(const Geom& g, double Ms, const double Hext[3], const double cell[3], double A,
                               double Ku, const float* M, const float* Hd, const int* flag, double* partials,
                               double* out_dev, cudaStream_t s) {
    const double V = cell[0] * cell[1] * cell[2], w = A * V / (Ms * Ms), z = -kMu0 * V;
    EnergyCoef cf;
    cf.ax = w / (cell[0] * cell[0]);
    cf.ay = w / (cell[1] * cell[1]);
    cf.az = w / (cell[2] * cell[2]);
    cf.an = Ku * V / (Ms * Ms);
    cf.de = -0.5 * kMu0 * V;
    cf.zx = z * Hext[0];
    cf.zy = z * Hext[1];
    cf.zz = z * Hext[2];
    // 31 cells per warp; the last cell of a row needs no right neighbour
    const int wpr = g.nx > 1 ? (g.nx - 1 + 30) / 31 : 1;
    const int wpb = kEnergyThreads / 32;
    // few rows per warp while the items would not fill the SMs otherwise
    const bool large = (long long)wpr * g.nz * ((g.ny + kRowsLarge - 1) / kRowsLarge) >= 152LL * 2 * wpb;
    const int rows = large ? kRowsLarge : kRowsSmall;
    const int segs = (g.ny + rows - 1) / rows;
    const int items = wpr * segs * g.nz;
    int blocks = (items + wpb - 1) / wpb;
    if (blocks > kEnergyMaxBlocks) blocks = kEnergyMaxBlocks;
    if (large)
        k_energy<kRowsLarge><<<blocks, kEnergyThreads, 0, s>>>(g.nx, g.ny, g.nz, wpr, segs, items, M, Hd, cf, flag,
                                                               partials, out_dev);
    else
        k_energy<kRowsSmall><<<blocks, kEnergyThreads, 0, s>>>(g.nx, g.ny, g.nz, wpr, segs, items, M, Hd, cf, flag,
                                                               partials, out_dev);
    return cudaGetLastError();
}

}  // namespace mmk
