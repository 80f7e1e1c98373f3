// Mixed-radix FFT on a register array, all indices compile-time.
//
//   y_k = sum_j x_j w^(S j k),  w = exp(2 pi i / n),  S = +1 or -1,
//
// natural order in and out, for n = 2^a 3^b. Decimation in time (Cooley-Tukey):
// with n = R n2 (radix R = 4 if it divides n, else 3, else 2), j = n2 j1 + j2
// and k = k1 + R k2,
//   y_{k1 + R k2} = sum_{j2} w_{n2}^{S j2 k2} [ w_n^{S j2 k1} sum_{j1} x_{n2 j1 + j2} w_R^{S j1 k1} ],
// i.e. n2 transforms of size R, the twiddles w_n^{S j2 k1}, then R transforms
// of size n2. A transform of size 16 takes 160 real operations (128 additions
// in the eight radix-4 butterflies, 8 general twiddles of 4 each) instead of
// the 1024 FMAs of the dense matrix.
//
// Twiddles come from one table of the top-level size NT,
// root[t] = exp(2 pi i t / NT): w_n^t = root[(t NT / n) mod NT]. Indices 0,
// NT/4, NT/2 and 3NT/4 are +-1 and +-i and cost no multiplication; with the
// loops unrolled every index is a compile-time constant, so on the device the
// table (in constant memory) supplies FMA operands directly. FP32 and FP64,
// host and device: the same code is checked against the dense sum on the CPU.
#pragma once

#include <cuda_runtime.h>

namespace bte {
namespace fftr {

// The vector types: float2 or double2, by overloads.
__host__ __device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }
__host__ __device__ __forceinline__ double2 mk(double a, double b) { return make_double2(a, b); }
__host__ __device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__host__ __device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

template <class V>
__host__ __device__ __forceinline__ V cadd(V a, V b) { return mk(a.x + b.x, a.y + b.y); }
template <class V>
__host__ __device__ __forceinline__ V csub(V a, V b) { return mk(a.x - b.x, a.y - b.y); }
template <class V>
__host__ __device__ __forceinline__ V cneg(V a) { return mk(-a.x, -a.y); }
// i s a for s = +1 or -1
template <int S, class V>
__host__ __device__ __forceinline__ V cmul_i(V a) {
    return S > 0 ? mk(-a.y, a.x) : mk(a.y, -a.x);
}

// v w_NT^(S t), t >= 0 (compile-time after unrolling)
template <int NT, int S, class V>
__host__ __device__ __forceinline__ V twiddle(V v, int t, const V (&rt)[NT]) {
    const int u = ((S * t) % NT + NT) % NT;
    if (u == 0) return v;
    if (2 * u == NT) return cneg(v);
    if (4 * u == NT) return cmul_i<1>(v);
    if (4 * u == 3 * NT) return cmul_i<-1>(v);
    const V w = rt[u];
    return mk(fma_(v.x, w.x, -(v.y * w.y)), fma_(v.x, w.y, v.y * w.x));
}

// In place: x <- DFT_S(x) of size N inside a top-level transform of size NT.
template <int N, int S, int NT, class V>
__host__ __device__ __forceinline__ void fft(V (&x)[N], const V (&rt)[NT]) {
    static_assert(NT % N == 0, "sub-transform size");
    if constexpr (N == 1) {
    } else if constexpr (N == 2) {
        const V a = x[0], b = x[1];
        x[0] = cadd(a, b);
        x[1] = csub(a, b);
    } else if constexpr (N == 3) {
        // w_3^S = -1/2 + i S sin(2 pi / 3); sin(2 pi / 3) = Im root[NT / 3]
        const auto s3 = rt[NT / 3].y;
        const V a = x[0], t = cadd(x[1], x[2]), u = csub(x[1], x[2]);
        const decltype(a.x) half = -0.5f;
        const V m = mk(fma_(half, t.x, a.x), fma_(half, t.y, a.y));
        const V r = cmul_i<S>(mk(s3 * u.x, s3 * u.y));
        x[0] = cadd(a, t);
        x[1] = cadd(m, r);
        x[2] = csub(m, r);
    } else if constexpr (N == 4) {
        const V a = cadd(x[0], x[2]), b = csub(x[0], x[2]);
        const V c = cadd(x[1], x[3]), d = cmul_i<S>(csub(x[1], x[3]));
        x[0] = cadd(a, c);
        x[1] = cadd(b, d);
        x[2] = csub(a, c);
        x[3] = csub(b, d);
    } else {
        constexpr int R = N % 4 == 0 ? 4 : (N % 3 == 0 ? 3 : 2);
        constexpr int N2 = N / R;
        V A[R][N2];
#pragma unroll
        for (int j2 = 0; j2 < N2; ++j2) {
            V v[R];
#pragma unroll
            for (int j1 = 0; j1 < R; ++j1) v[j1] = x[N2 * j1 + j2];
            fft<R, S, NT>(v, rt);
#pragma unroll
            for (int k1 = 0; k1 < R; ++k1) A[k1][j2] = twiddle<NT, S>(v[k1], j2 * k1 * (NT / N), rt);
        }
#pragma unroll
        for (int k1 = 0; k1 < R; ++k1) {
            V u[N2];
#pragma unroll
            for (int j2 = 0; j2 < N2; ++j2) u[j2] = A[k1][j2];
            fft<N2, S, NT>(u, rt);
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) x[k1 + R * k2] = u[k2];
        }
    }
}

// Centred transform of one pencil (N/2 even):
//   y_k = sum_j x_j w^(S (k - N/2)(j - N/2)) = (-1)^k sum_j (-1)^j x_j w^(S j k),
// since w^(-N/2 k) = (-1)^k and w^((N/2)^2) = (-1)^(N/2) = 1.
template <int N, int S, class V>
__host__ __device__ __forceinline__ void centred(V (&y)[N], const V (&rt)[N]) {
    static_assert(N % 4 == 0, "N/2 must be even");
#pragma unroll
    for (int j = 1; j < N; j += 2) y[j] = cneg(y[j]);
    fft<N, S, N>(y, rt);
#pragma unroll
    for (int k = 1; k < N; k += 2) y[k] = cneg(y[k]);
}

}  // namespace fftr
}  // namespace bte
