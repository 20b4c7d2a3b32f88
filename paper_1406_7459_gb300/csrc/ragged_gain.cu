// ragged_gain.cu -- gains of the transforms on carrier lengths.
//
// The butterflies' FP32 constants and the twiddle tables have moduli that are
// not one (0.70710677 for sqrt(1/2), and so on), and the nearest values of the
// few constants in the butterflies happen to lie below: forward and back, a
// wavenumber loses up to 1e-7 of itself, most of them 4e-8 to 9e-8, while 0 and
// 1, whose paths hold none of those constants, lose nothing.  The tensor
// spectrum is divided by these gains, so that H_demag keeps its scale (random
// states of 100x80x20: 1.5e-7 too small without, as large as all its other
// rounding).
//
// The gain of wavenumber k is the mean over the cells j < N of inverse[j][k]
// times forward[k][j].  Every entry of either is a product over the digits of
// k and j (Fft2: DFT_P, twiddle, DFT_Q, the odd half's factor), each factor its
// exact value times 1 + a small deviation, so the gain is one plus the sum of
// the factors' mean deviations, to 1e-14.  The constants are those of
// fft_device.cuh and fast_fft.cuh, rounded as there, the arithmetic is FP64.
#include <complex>
#include <map>
#include <mutex>
#include <vector>

#include "fast_fft.cuh"
#include "mm_internal.h"

namespace mmk {

typedef std::complex<double> Cd;

constexpr double kTwoPi = 6.28318530717958647692;

static Cd exact_w(long long k, int n) { return std::polar(1.0, -kTwoPi * (double)(k % n) / n); }
static Cd rounded_w(long long k, int n) {
    const Cd w = exact_w(k, n);
    return Cd((float)w.real(), (float)w.imag());
}
static double deviation(Cd value, Cd exact) { return (value * std::conj(exact)).real() - 1.0; }

// The butterflies of fft_device.cuh and fast_fft.cuh (dftp).
static void dft(std::vector<Cd>& a);
static void dft_split(std::vector<Cd>& a, int A, int B, Cd (*w)(int k, int n)) {   // n = A B: B DFT_A, twiddles, A DFT_B
    const int n = A * B;
    std::vector<std::vector<Cd>> c(B);
    for (int r = 0; r < B; ++r) {
        for (int i = 0; i < A; ++i) c[r].push_back(a[r + B * i]);
        dft(c[r]);
        for (int q = 1; q < A; ++q)
            if (r > 0) c[r][q] *= w(r * q, n);
    }
    for (int q = 0; q < A; ++q) {
        std::vector<Cd> t(B);
        for (int r = 0; r < B; ++r) t[r] = c[r][q];
        dft(t);
        for (int r = 0; r < B; ++r) a[q + A * r] = t[r];
    }
}
static Cd w_any(int k, int n) { return 4 * k == n ? Cd(0, -1) : rounded_w(k, n); }
static void dft(std::vector<Cd>& a) {
    const Cd i(0, 1);
    switch (a.size()) {
        case 2: a = {a[0] + a[1], a[0] - a[1]}; break;
        case 3: {
            const Cd t = a[1] + a[2], m = a[0] - 0.5 * t, u = -i * (double)kSqrt3Half * (a[1] - a[2]);
            a = {a[0] + t, m + u, m - u};
            break;
        }
        case 4: {
            const Cd t0 = a[0] + a[2], t1 = a[0] - a[2], t2 = a[1] + a[3], t3 = -i * (a[1] - a[3]);
            a = {t0 + t2, t1 + t3, t0 - t2, t1 - t3};
            break;
        }
        case 5: {
            const double c1 = kC51, c2 = kC52, s1 = kS51, s2 = kS52;
            const Cd t1 = a[1] + a[4], t2 = a[2] + a[3], u1 = a[1] - a[4], u2 = a[2] - a[3];
            const Cd m1 = a[0] + c1 * t1 + c2 * t2, m2 = a[0] + c2 * t1 + c1 * t2;
            const Cd n1 = s1 * u1 + s2 * u2, n2 = s2 * u1 - s1 * u2;
            a = {a[0] + t1 + t2, m1 - i * n1, m2 - i * n2, m2 + i * n2, m1 + i * n1};
            break;
        }
        case 6: dft_split(a, 2, 3, w_any); break;
        case 8: dft_split(a, 4, 2, w_any); break;
        case 12: dft_split(a, 4, 3, w_any); break;
        case 16: dft_split(a, 4, 4, w_any); break;
        case 20: dft_split(a, 4, 5, w_any); break;
        case 24: dft_split(a, 8, 3, w_any); break;
        case 32: dft_split(a, 16, 2, w_any); break;
        default: break;
    }
}

// Mean deviations of DFT_R's matrix by rows (out) and columns (in).
static void dft_deviations(int R, std::vector<double>* rows, std::vector<double>* cols) {
    rows->assign(R, 0.0);
    cols->assign(R, 0.0);
    for (int c = 0; c < R; ++c) {
        std::vector<Cd> e(R, 0.0);
        e[c] = 1.0;
        dft(e);
        for (int r = 0; r < R; ++r) {
            const double d = deviation(e[r], exact_w((long long)r * c, R)) / R;
            (*rows)[r] += d;
            (*cols)[c] += d;
        }
    }
}

template <int N> static bool split_of(int n, int* P, int* Q) {
    if (n != N) return false;
    *P = Split<N>::P;
    *Q = Split<N>::Q;
    return true;
}

// 1 / gain of k <= N (the mean of k and 2N - k, which share a tensor entry).
// z: the split pass's z columns, whose inverse runs the steps in reverse order
// (up to 8 layers: one DFT per half).
static std::vector<double> inverse_gains(int N, bool z) {
    int P = N, Q = 1;
    if (N > 8)
        (void)(split_of<16>(N, &P, &Q) || split_of<24>(N, &P, &Q) || split_of<32>(N, &P, &Q) ||
               split_of<48>(N, &P, &Q) || split_of<64>(N, &P, &Q) || split_of<96>(N, &P, &Q) ||
               split_of<128>(N, &P, &Q) || split_of<192>(N, &P, &Q) || split_of<256>(N, &P, &Q) ||
               split_of<320>(N, &P, &Q) || split_of<384>(N, &P, &Q) || split_of<512>(N, &P, &Q) ||
               split_of<640>(N, &P, &Q) || split_of<768>(N, &P, &Q) || split_of<1024>(N, &P, &Q));
    std::vector<double> rp, cp, rq, cq, ta(P, 0.0), tt(Q, 0.0), g(2 * N + 1);
    dft_deviations(P, &rp, &cp);
    dft_deviations(Q, &rq, &cq);
    for (int a = 1; a < P; ++a)
        for (int t = 1; t < Q; ++t) {
            const double d = deviation(rounded_w(2LL * t * a, 2 * N), exact_w(2LL * t * a, 2 * N));
            ta[a] += d / Q;
            tt[t] += d / P;
        }
    double odd = 0.0;
    for (int j = 1; j < N; ++j) odd += deviation(rounded_w(j, 2 * N), exact_w(j, 2 * N)) / N;
    for (int m = 0; m < N; ++m) {
        const int a = m % P, b = m / P;
        const double back = z || Q == 1 ? cp[a] + ta[a] + cq[b] : cp[m / Q] + tt[m % Q] + cq[m % Q];
        g[2 * m] = rp[a] + ta[a] + rq[b] + back;
        g[2 * m + 1] = g[2 * m] + 2.0 * odd;
    }
    g[2 * N] = g[0];
    std::vector<double> out(N + 1);
    for (int k = 0; k <= N; ++k) out[k] = 1.0 / (1.0 + 0.5 * (g[k] + g[2 * N - k]));
    return out;
}

void ragged_inverse_gains(int L, bool z, double* out) {
    const int N = L / 2;
    if (N < 1) {
        out[0] = 1.0;
        return;
    }
    // constants of the length alone, formed once
    static std::mutex mu;
    static std::map<int, std::vector<double>> known;
    std::lock_guard<std::mutex> lock(mu);
    std::vector<double>& v = known[2 * N + (z ? 1 : 0)];
    if (v.empty()) v = inverse_gains(N, z);
    for (int k = 0; k <= N; ++k) out[k] = v[k];
}

}  // namespace mmk
