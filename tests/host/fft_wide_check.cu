// Host check of the register FFT (fft_reg.cuh) where the transforms of dft.cu use it:
// FP64 at N = 8 .. 32 and FP32 at N = 48, both signs, plain and centred, against the
// dense sums in long double. Prints "N type S kind max|error| / max|y|". And of the
// symmetry that the forward transforms of N = 8 and 16 rely on: "N symmetry" and the number
// of k for which the transform of conj(x) is not bit for bit the mirrored
// conjugate of the transform of x.
#include <cmath>
#include <cstdio>
#include <random>

#include "../../paper_1211_0540_gb300/csrc/fft_reg.cuh"

using namespace bte::fftr;

template <int N, class V>
static void roots(V (&rt)[N]) {
    const double pi = 3.14159265358979323846;
    for (int t = 0; t < N; ++t) {
        rt[t].x = (decltype(rt[t].x))std::cos(2 * pi * t / N);
        rt[t].y = (decltype(rt[t].y))std::sin(2 * pi * t / N);
    }
}

template <int N, int S, bool CENTRED, class V>
static double check(std::mt19937 &g) {
    const long double pi = 3.141592653589793238462643383279502884L;
    V rt[N], x[N], y[N];
    roots<N>(rt);
    std::uniform_real_distribution<float> u(-1.f, 1.f);
    for (int j = 0; j < N; ++j) y[j] = x[j] = mk((decltype(x[0].x))u(g), (decltype(x[0].x))u(g));
    if (CENTRED) centred<N, S>(y, rt);
    else fft<N, S, N>(y, rt);
    const int h = CENTRED ? N / 2 : 0;
    long double err = 0, mag = 0;
    for (int k = 0; k < N; ++k) {
        long double re = 0, im = 0;
        for (int j = 0; j < N; ++j) {
            const long double a = 2 * pi * S * (long double)((k - h) * (j - h)) / N;
            re += x[j].x * std::cos(a) - x[j].y * std::sin(a);
            im += x[j].x * std::sin(a) + x[j].y * std::cos(a);
        }
        err = std::fmax(err, std::hypot(re - y[k].x, im - y[k].y));
        mag = std::fmax(mag, std::hypot(re, im));
    }
    return (double)(err / mag);
}

template <int N, class V>
static void all(std::mt19937 &g, const char *type) {
    std::printf("%d %s +1 plain %.3e\n", N, type, check<N, 1, false, V>(g));
    std::printf("%d %s -1 plain %.3e\n", N, type, check<N, -1, false, V>(g));
    std::printf("%d %s +1 centred %.3e\n", N, type, check<N, 1, true, V>(g));
    std::printf("%d %s -1 centred %.3e\n", N, type, check<N, -1, true, V>(g));
}

template <int N>
static void symmetry(std::mt19937 &g) {
    float2 rt[N], a[N], b[N];
    roots<N>(rt);
    std::uniform_real_distribution<float> u(-1.f, 1.f);
    int bad = 0;
    for (int rep = 0; rep < 200; ++rep) {
        for (int j = 0; j < N; ++j) {
            a[j] = make_float2(u(g), rep % 2 ? u(g) : 0.f);
            b[j] = make_float2(a[j].x, -a[j].y);
        }
        centred<N, -1>(a, rt);
        centred<N, -1>(b, rt);
        for (int k = 0; k < N; ++k) {
            const int m = k ? N - k : 0;
            bad += !(b[k].x == a[m].x && b[k].y == -a[m].y);
        }
    }
    std::printf("%d symmetry %d\n", N, bad);
}

int main() {
    std::mt19937 g(11);
    all<8, double2>(g, "f64");
    all<12, double2>(g, "f64");
    all<16, double2>(g, "f64");
    all<24, double2>(g, "f64");
    all<32, double2>(g, "f64");
    all<48, float2>(g, "f32");
    symmetry<8>(g);
    symmetry<16>(g);
    return 0;
}
