// Centred discrete Fourier transforms of Sec. 3.2 on the grid of Eq. meshpoints
// for the FP64 operator, and for FP32 on the grid (N = 48) that the fused
// transforms do not hold, with the conservation projection of Sec. 3.3 and the
// Heun update behind the inverse:
//   fhat_k = (2 pi)^{-3/2} dv^3 sum_j f_j exp(-i zeta_k . v_j),
//   Qt_j   = Re (2 pi)^{-3/2} dz^3 sum_k Qhat_k exp(+i zeta_k . v_j).
// One thread per pencil, register FFTs (fft_reg.cuh). The passes along j3 and
// j2 of a plane j1 run in one warp (N <= 32; several planes of a small grid),
// the plane in shared memory; the pass along j1 goes through global memory,
// which holds any N and spreads one cell over N planes' CTAs. FP64 adds cost 16
// clocks a warp here, so the FFT's 10 operations a value and pass instead of
// the dense sum's 64 (N = 16) count: 128 cells N = 16, forward 307 -> 46 us,
// inverse with projection 256 -> 57 us; one cell 68 -> 26 and 83 -> 31 us (cold
// caches; bound there by the chain of FP64 operations).
//
// Layouts. f and Qt are the caller's FP64 cell arrays (per-slot element
// offsets, -1 for the padding slots of a 32-cell group, which come last and are skipped).
// T is cell-major [slot][M]. fhat and Qhat are in the group layout of the
// convolution, [group][m][lane] (a warp reads one grid point of 32 cells as one
// row), or cell-major where the convolution takes the cells one by one (CELL).
#include <cmath>
#include <map>
#include <mutex>

#include "fft_reg.cuh"
#include "fpconv.cuh"
#include "kernels.h"

namespace bte {

namespace {

__constant__ double2 c_r64_8[8], c_r64_12[12], c_r64_16[16], c_r64_24[24], c_r64_32[32];
__constant__ float2 c_r32_48[48];

template <int N, class V> struct Root;
template <> struct Root<8, double2> { static __device__ const double2 (&get())[8] { return c_r64_8; } };
template <> struct Root<12, double2> { static __device__ const double2 (&get())[12] { return c_r64_12; } };
template <> struct Root<16, double2> { static __device__ const double2 (&get())[16] { return c_r64_16; } };
template <> struct Root<24, double2> { static __device__ const double2 (&get())[24] { return c_r64_24; } };
template <> struct Root<32, double2> { static __device__ const double2 (&get())[32] { return c_r64_32; } };
template <> struct Root<48, float2> { static __device__ const float2 (&get())[48] { return c_r32_48; } };

template <class V> struct Real;
template <> struct Real<float2> {
    using T = float;
    static __device__ T of(double x) { return fpc::narrow(x); }
    static __device__ double wide(T x) { return fpc::widen(x); }
};
template <> struct Real<double2> {
    using T = double;
    static __device__ T of(double x) { return x; }
    static __device__ double wide(T x) { return x; }
};

template <int N>
struct Plane {
    static constexpr int P = N <= 32 ? 32 / N : 1;     // planes per CTA
    static constexpr int NT = N <= 32 ? 32 : 64;       // one thread per pencil
    static constexpr int G = (N + P - 1) / P;          // CTAs per cell
};
constexpr int kAxisWarps = 4;     // pencils per CTA of the group-layout passes
constexpr int kFinishThreads = 256, kFinishChunk = 1024;

}  // namespace

// Passes along j3 (real rows of f) and j2: T[slot][j1][k2][k3].
template <int N, class V>
__global__ void __launch_bounds__(Plane<N>::NT)
dft_fwd_planes_kernel(const double *__restrict__ f, const int64_t *__restrict__ slot_off, DftSeg s, V *__restrict__ T,
                      int *status) {
    constexpr int M = N * N * N, P = Plane<N>::P;
    __shared__ V sh[P][N][N + 1];
    const int64_t off = slot_off[s.s0 + blockIdx.y];
    if (off < 0) return;
    const V(&rt)[N] = Root<N, V>::get();
    const int p = threadIdx.x / N, r = threadIdx.x % N, j1 = blockIdx.x * P + p;
    const bool act = p < P && j1 < N;
    V y[N];
    if (act) {  // along j3, row j2 = r
        const double *x = f + off + (int64_t)(j1 * N + r) * N;
        bool bad = false;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const double d = x[j];
            bad |= !fpc::finite64(d);
            y[j] = fftr::mk(Real<V>::of(d), (typename Real<V>::T)0);
        }
        if (bad) atomicOr(status, ST_NONFINITE);
        fftr::centred<N, -1>(y, rt);
#pragma unroll
        for (int k = 0; k < N; ++k) sh[p][r][k] = y[k];
    }
    __syncthreads();
    if (act) {  // along j2, column k3 = r
#pragma unroll
        for (int j = 0; j < N; ++j) y[j] = sh[p][j][r];
        fftr::centred<N, -1>(y, rt);
        V *o = T + s.eoff + (int64_t)blockIdx.y * M + j1 * N * N + r;
#pragma unroll
        for (int k = 0; k < N; ++k) o[k * N] = y[k];
    }
}

// Pass along j1, pencil pk = k2 N + k3, with the forward scale into fhat. Group
// layout: the lanes of a warp are the group's cells (whole rows are stored; a
// padding lane is 0). CELL: the lanes are pencils of one cell.
template <int N, class V, bool CELL>
__global__ void __launch_bounds__(CELL ? 32 : 32 * kAxisWarps)
dft_fwd_axis_kernel(const V *__restrict__ T, const int64_t *__restrict__ slot_off, DftSeg s,
                    typename Real<V>::T scale, V *__restrict__ G) {
    constexpr int NN = N * N, M = NN * N;
    const int lane = threadIdx.x & 31;
    const int slot = CELL ? (int)blockIdx.y : (int)blockIdx.y * kLanes + lane;
    const int pk = CELL ? (int)blockIdx.x * 32 + lane : (int)blockIdx.x * kAxisWarps + (int)(threadIdx.x >> 5);
    if (pk >= NN) return;
    const bool valid = slot_off[s.s0 + slot] >= 0;
    if (CELL && !valid) return;
    V *g = CELL ? G + s.eoff + (int64_t)slot * M : G + s.eoff + (int64_t)blockIdx.y * M * kLanes + lane;
    constexpr int64_t step = CELL ? 1 : kLanes;
    V y[N];
    const V *a = T + s.eoff + (int64_t)slot * M + pk;
#pragma unroll
    for (int j = 0; j < N; ++j) y[j] = valid ? a[j * NN] : fftr::mk((typename Real<V>::T)0, (typename Real<V>::T)0);
    fftr::centred<N, -1>(y, Root<N, V>::get());
#pragma unroll
    for (int k = 0; k < N; ++k) g[(int64_t)(k * NN + pk) * step] = fftr::mk(scale * y[k].x, scale * y[k].y);
}

// fhat made conjugate symmetric, as the fused transforms do (symmetrise in
// dft_fused.cu, where the reason stands; the FFT of N = 8 and 16 needs none). FP64 operator's
// error against extended precision, one cell N = 24, lambda = 1: 4.6e-15 without.
template <int N, class V, bool CELL>
__global__ void __launch_bounds__(256) dft_symmetrise_kernel(DftSeg s, V *__restrict__ G) {
    constexpr int M = N * N * N;
    const int lane = threadIdx.x & 31;
    const int m = CELL ? (int)(blockIdx.x * 256 + threadIdx.x) : (int)(blockIdx.x * 8 + (threadIdx.x >> 5));
    if (m >= M) return;
    const int mm = (mode_mirror(m / (N * N), N) * N + mode_mirror(m / N % N, N)) * N + mode_mirror(m % N, N);
    if (mm < m) return;  // the other one's thread
    V *g = CELL ? G + s.eoff + (int64_t)blockIdx.y * M : G + s.eoff + (int64_t)blockIdx.y * M * kLanes + lane;
    constexpr int64_t step = CELL ? 1 : kLanes;
    const V a = g[m * step], b = g[mm * step];
    const typename Real<V>::T half = 0.5f, re = half * (a.x + b.x), im = half * (a.y - b.y);
    g[mm * step] = fftr::mk(re, -im);
    g[m * step] = fftr::mk(re, im);
}

// Inverse pass along k1 out of Qhat: T[slot][j1][k2][k3]. Only the stored
// pencils hold Qhat (half-spectrum convolution), the others are 0.
template <int N, class V, bool CELL>
__global__ void __launch_bounds__(CELL ? 32 : 32 * kAxisWarps)
dft_inv_axis_kernel(const V *__restrict__ G, const int64_t *__restrict__ slot_off, DftSeg s, V *__restrict__ T) {
    constexpr int NN = N * N, M = NN * N;
    const int lane = threadIdx.x & 31;
    const int slot = CELL ? (int)blockIdx.y : (int)blockIdx.y * kLanes + lane;
    const int pk = CELL ? (int)blockIdx.x * 32 + lane : (int)blockIdx.x * kAxisWarps + (int)(threadIdx.x >> 5);
    if (pk >= NN || slot_off[s.s0 + slot] < 0) return;
    const V *g = CELL ? G + s.eoff + (int64_t)slot * M : G + s.eoff + (int64_t)blockIdx.y * M * kLanes + lane;
    constexpr int64_t step = CELL ? 1 : kLanes;
    const int k2 = pk / N;
    V y[N];
#pragma unroll
    for (int k = 0; k < N; ++k)
        y[k] = pencil_stored(k, k2, N) ? g[(int64_t)(k * NN + pk) * step]
                                       : fftr::mk((typename Real<V>::T)0, (typename Real<V>::T)0);
    fftr::centred<N, 1>(y, Root<N, V>::get());
    V *o = T + s.eoff + (int64_t)slot * M + pk;
#pragma unroll
    for (int j = 0; j < N; ++j) o[j * NN] = y[j];
}

// Inverse passes along k2 and k3 (real part, scaled) into the caller's cells,
// and the plane's sums of (1, v1, v2, v3, |v|^2) Qt into mom[(slot N + j1) 5 + i].
template <int N, class V>
__global__ void __launch_bounds__(Plane<N>::NT)
dft_inv_planes_kernel(const V *__restrict__ T, const int64_t *__restrict__ slot_off, DftSeg s,
                      typename Real<V>::T scale, double dv, double *__restrict__ q, double *__restrict__ mom) {
    constexpr int M = N * N * N, P = Plane<N>::P, h = N / 2;
    __shared__ V sh[P][N][N + 1];
    __shared__ double red[P][5][N];
    const int64_t off = slot_off[s.s0 + blockIdx.y];
    if (off < 0) return;
    const V(&rt)[N] = Root<N, V>::get();
    const int p = threadIdx.x / N, r = threadIdx.x % N, j1 = blockIdx.x * P + p;
    const bool act = p < P && j1 < N;
    V y[N];
    if (act) {  // along k2, column k3 = r
        const V *a = T + s.eoff + (int64_t)blockIdx.y * M + j1 * N * N + r;
#pragma unroll
        for (int k = 0; k < N; ++k) y[k] = a[k * N];
        fftr::centred<N, 1>(y, rt);
#pragma unroll
        for (int j = 0; j < N; ++j) sh[p][j][r] = y[j];
    }
    __syncthreads();
    double *R = reinterpret_cast<double *>(&sh[act ? p : 0][0][0]);  // the plane's Qt, rows of N + 1
    if (act) {  // along k3, row j2 = r
#pragma unroll
        for (int k = 0; k < N; ++k) y[k] = sh[p][r][k];
        fftr::centred<N, 1>(y, rt);
    }
    __syncthreads();
    constexpr bool stage = sizeof(V) == sizeof(double2);  // FP32 planes have no room for FP64 rows
    if (act) {
        double s0 = 0.0, s1 = 0.0, s2 = 0.0;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const double x = Real<V>::wide(scale * y[j].x), v = dv * (double)(j - h);
            if (stage) R[r * (N + 1) + j] = x;
            else q[off + (int64_t)(j1 * N + r) * N + j] = x;
            s0 += x;
            s1 = fma(v, x, s1);
            s2 = fma(v * v, x, s2);
        }
        const double v1 = dv * (double)(j1 - h), v2 = dv * (double)(r - h);
        red[p][0][r] = s0;
        red[p][1][r] = v1 * s0;
        red[p][2][r] = v2 * s0;
        red[p][3][r] = s1;
        red[p][4][r] = fma(fma(v1, v1, v2 * v2), s0, s2);
    }
    __syncthreads();
    for (int o = threadIdx.x; o < P * 5; o += Plane<N>::NT) {
        const int pl = o / 5, i = o % 5, jj = blockIdx.x * P + pl;
        if (jj >= N) continue;
        double a = 0.0;
        for (int k = 0; k < N; ++k) a += red[pl][i][k];
        mom[((int64_t)blockIdx.y * N + jj) * 5 + i] = a;
    }
    if (stage)
        for (int o = threadIdx.x; o < P * N * N; o += Plane<N>::NT) {
            const int pl = o / (N * N), e = o % (N * N), jj = blockIdx.x * P + pl;
            if (jj < N)
                q[off + (int64_t)jj * N * N + e] =
                    reinterpret_cast<const double *>(&sh[pl][0][0])[(e / N) * (N + 1) + e % N];
        }
}

// The projection Q = Qt - C^T (C C^T)^{-1} C Qt (Sec. 3.3) from the planes' sums,
// with the Heun update (ProjArgs mode: 0 none, 1 y = x + a Q, 2 y += a (qp + Q)).
// Several CTAs per cell; each adds the N planes' sums in the same order.
template <int N>
__global__ void __launch_bounds__(kFinishThreads)
project_planes_kernel(double *__restrict__ q, const int64_t *__restrict__ slot_off, DftSeg s, ProjArgs pa,
                      const double *__restrict__ mom, int mode, const double *__restrict__ x, double *__restrict__ y,
                      const double *__restrict__ qp, double a) {
    constexpr int M = N * N * N, h = N / 2;
    const int64_t off = slot_off[s.s0 + blockIdx.y];
    if (off < 0) return;
    __shared__ double mu[5], lam[5], g[3][N];
    const int t = threadIdx.x;
    constexpr int IT = kFinishChunk / kFinishThreads;
    double qv[IT], u[IT], w[IT];  // the operands first: their latency overlaps the sums
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int e = blockIdx.x * kFinishChunk + t + i * kFinishThreads;
        qv[i] = e < M ? q[off + e] : 0.0;
        u[i] = mode == 0 || e >= M ? 0.0 : mode == 1 ? x[off + e] : y[off + e];
        w[i] = mode == 2 && e < M ? qp[off + e] : 0.0;
    }
    if (t < 5) {
        double m = 0.0;
#pragma unroll
        for (int j = 0; j < N; ++j) m += mom[((int64_t)blockIdx.y * N + j) * 5 + t];
        mu[t] = m;
    }
    __syncthreads();
    if (t < 5) {
        double l = 0.0;
#pragma unroll
        for (int k = 0; k < 5; ++k) l = fma(pa.ainv[t * 5 + k], mu[k], l);
        lam[t] = l;
    }
    __syncthreads();
    if (t < 3 * N) {
        const double v = pa.dv * (double)(t % N - h);
        g[t / N][t % N] = fma(lam[1 + t / N], v, lam[4] * v * v) + (t < N ? lam[0] : 0.0);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int e = blockIdx.x * kFinishChunk + t + i * kFinishThreads;
        if (e >= M) break;
        const double v = qv[i] - ((g[0][e / (N * N)] + g[1][(e / N) % N]) + g[2][e % N]);
        q[off + e] = v;
        if (mode == 1) y[off + e] = fma(a, v, u[i]);
        else if (mode == 2) y[off + e] = fma(a, w[i] + v, u[i]);
    }
}

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------
namespace {

template <int N, class V>
void upload_root(const V (&sym)[N]) {
    V r[N];
    for (int t = 0; t < N; ++t) {
        const double th = 2.0 * 3.14159265358979323846 * t / N;
        r[t].x = (decltype(r[t].x))std::cos(th);
        r[t].y = (decltype(r[t].y))std::sin(th);
    }
    upload_symbol(sym, r);
}

template <int N, class V>
int forward_n(const double *f, const int64_t *off, const DftSeg &s, double scale, V *T, V *G, bool cell, int *status,
              cudaStream_t st) {
    using R = typename Real<V>::T;
    dft_fwd_planes_kernel<N, V><<<dim3(Plane<N>::G, s.nvalid), Plane<N>::NT, 0, st>>>(f, off, s, T, status);
    if (cell)
        dft_fwd_axis_kernel<N, V, true><<<dim3((N * N + 31) / 32, s.nvalid), 32, 0, st>>>(T, off, s, (R)scale, G);
    else
        dft_fwd_axis_kernel<N, V, false><<<dim3((N * N + kAxisWarps - 1) / kAxisWarps, s.nslots / kLanes),
                                            32 * kAxisWarps, 0, st>>>(T, off, s, (R)scale, G);
    if constexpr (N == 8 || N == 16 || N > 32) return 2;  // FP32 at N = 48 is within the full spectrum's error
    constexpr int M = N * N * N;
    if (cell) dft_symmetrise_kernel<N, V, true><<<dim3((M + 255) / 256, s.nvalid), 256, 0, st>>>(s, G);
    else dft_symmetrise_kernel<N, V, false><<<dim3((M + 7) / 8, s.nslots / kLanes), 256, 0, st>>>(s, G);
    return 3;
}

template <int N, class V>
int inverse_n(const V *G, const int64_t *off, const DftSeg &s, double scale, V *T, double *mom, double *q, bool cell,
              const ProjArgs &pa, int mode, const double *x, double *y, const double *qp, double a, cudaStream_t st) {
    using R = typename Real<V>::T;
    if (cell)
        dft_inv_axis_kernel<N, V, true><<<dim3((N * N + 31) / 32, s.nvalid), 32, 0, st>>>(G, off, s, T);
    else
        dft_inv_axis_kernel<N, V, false><<<dim3((N * N + kAxisWarps - 1) / kAxisWarps, s.nslots / kLanes),
                                            32 * kAxisWarps, 0, st>>>(G, off, s, T);
    dft_inv_planes_kernel<N, V><<<dim3(Plane<N>::G, s.nvalid), Plane<N>::NT, 0, st>>>(T, off, s, (R)scale, pa.dv, q,
                                                                                     mom);
    if (mode < 0) return 2;
    project_planes_kernel<N><<<dim3((N * N * N + kFinishChunk - 1) / kFinishChunk, s.nvalid), kFinishThreads, 0, st>>>(
        q, off, s, pa, mom, mode, x, y, qp, a);
    return 3;
}

}  // namespace

void dft_prepare(int N) {
    // roots of unity (constant memory is per device); must happen outside stream capture
    static std::map<int, uint64_t> done;  // device -> bit N
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    int dev = 0;
    cudaGetDevice(&dev);
    if (N < 0 || N > 48 || (done[dev] >> N) & 1u) return;
    switch (N) {
        case 8: upload_root<8>(c_r64_8); break;
        case 12: upload_root<12>(c_r64_12); break;
        case 16: upload_root<16>(c_r64_16); break;
        case 24: upload_root<24>(c_r64_24); break;
        case 32: upload_root<32>(c_r64_32); break;
        case 48: upload_root<48>(c_r32_48); break;
        default: return;
    }
    done[dev] |= (uint64_t)1 << N;
}

int launch_dft_forward(const double *f, const int64_t *slot_off, const DftSeg &s, double scale, void *T, void *G,
                       bool cell, int *status, cudaStream_t st) {
    double2 *T64 = (double2 *)T, *G64 = (double2 *)G;
    switch (s.N) {
        case 8: return forward_n<8>(f, slot_off, s, scale, T64, G64, cell, status, st);
        case 12: return forward_n<12>(f, slot_off, s, scale, T64, G64, cell, status, st);
        case 16: return forward_n<16>(f, slot_off, s, scale, T64, G64, cell, status, st);
        case 24: return forward_n<24>(f, slot_off, s, scale, T64, G64, cell, status, st);
        case 32: return forward_n<32>(f, slot_off, s, scale, T64, G64, cell, status, st);
        case 48: return forward_n<48>(f, slot_off, s, scale, (float2 *)T, (float2 *)G, cell, status, st);
        default: return 0;
    }
}

int launch_dft_inverse(const void *G, const int64_t *slot_off, const DftSeg &s, double scale, void *T, double *mom,
                       double *q, bool cell, const ProjArgs &pa, int mode, const double *x, double *y,
                       const double *qp, double a, cudaStream_t st) {
    const double2 *G64 = (const double2 *)G;
    double2 *T64 = (double2 *)T;
    switch (s.N) {
        case 8: return inverse_n<8>(G64, slot_off, s, scale, T64, mom, q, cell, pa, mode, x, y, qp, a, st);
        case 12: return inverse_n<12>(G64, slot_off, s, scale, T64, mom, q, cell, pa, mode, x, y, qp, a, st);
        case 16: return inverse_n<16>(G64, slot_off, s, scale, T64, mom, q, cell, pa, mode, x, y, qp, a, st);
        case 24: return inverse_n<24>(G64, slot_off, s, scale, T64, mom, q, cell, pa, mode, x, y, qp, a, st);
        case 32: return inverse_n<32>(G64, slot_off, s, scale, T64, mom, q, cell, pa, mode, x, y, qp, a, st);
        case 48:
            return inverse_n<48>((const float2 *)G, slot_off, s, scale, (float2 *)T, mom, q, cell, pa, mode, x, y, qp,
                                 a, st);
        default: return 0;
    }
}

}  // namespace bte
