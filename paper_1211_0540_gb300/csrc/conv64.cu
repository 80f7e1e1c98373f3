// FP64 weighted convolution (Sec. 3.2), the comparator operator: the direct
// double sum with FP64 weights and FP64 arithmetic,
//   Qhat(zeta_k) = sum over unordered pairs {m, n} of [W(k, m) + W(k, n)] fhat_m fhat_n,
// at the modes of the stored pencils (half spectrum, bte_internal.h). The FP64
// units bound it (two FMAs per SM and clock against 128 in FP32), six
// operations a pair, so what counts is the number of pairs: 2.42 M per cell at
// N = 16 (0.08 M with weight 0) instead of the 7.08 M terms of the plain sum over m (128 cells: 10.09
// -> 3.2 ms; six warp instructions of 16 clocks a pair on 152 SMs are 2.95 ms).
// A zeta point's terms are listed block by block ((m1, m2) of its pencil), its
// m_count values of m3 from m_first on (mod N), with the weights in that order;
// zeta points are sorted by cost, the largest first, against a long tail.
#include "kernels.h"

namespace bte {

namespace {
constexpr int kWarps64 = 4;  // warps per CTA
// The terms go to kSums sums in turn: sums a quarter as large round less, and the chain
// of dependent FMAs is shorter (128 cells N = 16 3.44 -> 3.31 ms, 200 cells N = 12 1.30 -> 1.21).
constexpr int kSums = 4;
__device__ __forceinline__ double tree(const double (&s)[kSums]) { return (s[0] + s[1]) + (s[2] + s[3]); }
}  // namespace

// One warp per (zeta point, 32-cell group), one lane per cell: the weight is
// warp-uniform and the fhat rows of the group layout are read coalesced. The
// groups of one zeta point are neighbours, so they share its weights in L1.
__global__ void __launch_bounds__(32 * kWarps64) conv64_plain_kernel(const double2 *__restrict__ F,
                                                                     double2 *__restrict__ Qh,
                                                                     const double *__restrict__ W,
                                                                     const Zeta64 *__restrict__ Z, int nz,
                                                                     const uint32_t *__restrict__ D, int N,
                                                                     int64_t eoff, int ngroups) {
    const int lane = threadIdx.x & 31;
    const int64_t M = (int64_t)N * N * N;
    const int64_t id = (int64_t)blockIdx.x * kWarps64 + (threadIdx.x >> 5);
    if (id >= (int64_t)nz * ngroups) return;
    const int g = (int)(id % ngroups);
    const Zeta64 z = Z[id / ngroups];
    const double2 *Fg = F + eoff + (int64_t)g * M * kLanes + lane;
    const double *w = W + z.woff;
    const int k1 = z.k1, k2 = z.k2, cnt = z.m_count, n3_first = pair_partner(z.k3, z.m_first, N);
    double re[kSums] = {}, im[kSums] = {};
    for (int b = 0; b < z.nblocks; ++b) {
        const uint32_t d = D[z.desc_off + b];
        const int m1 = (int)(d & 0xffffu), m2 = (int)(d >> 16);
        const double2 *A = Fg + (int64_t)((m1 * N + m2) * N) * kLanes;
        const double2 *B = Fg + (int64_t)((pair_partner(k1, m1, N) * N + pair_partner(k2, m2, N)) * N) * kLanes;
        int m3 = z.m_first, n3 = n3_first, t = 0;
        const auto term = [&](double &sr, double &si) {
            const double g_ = w[t++];
            const double2 a = A[m3 * kLanes], c = B[n3 * kLanes];
            sr += g_ * (a.x * c.x - a.y * c.y);
            si += g_ * (a.x * c.y + a.y * c.x);
            m3 = m3 + 1 == N ? 0 : m3 + 1;
            n3 = n3 == 0 ? N - 1 : n3 - 1;
        };
        while (t + kSums <= cnt) {
#pragma unroll
            for (int i = 0; i < kSums; ++i) term(re[i], im[i]);
        }
        while (t < cnt) term(re[0], im[0]);
        w += cnt;
    }
    const int64_t k = (int64_t)(k1 * N + k2) * N + z.k3;
    Qh[eoff + (int64_t)g * M * kLanes + k * kLanes + lane] = make_double2(tree(re), tree(im));
}

// Few cells (a partly filled group): one warp per (cell, zeta point), the lanes
// split the list (term q = lane, lane + 32, ...) and the partial sums are added
// by a fixed shuffle tree. The same FP64 sum, with every lane doing useful work
// when the group is not full (one cell would otherwise cost as much as 32).
__global__ void __launch_bounds__(32 * kWarps64) conv64_cells_kernel(const double2 *__restrict__ F,
                                                                     double2 *__restrict__ Qh,
                                                                     const double *__restrict__ W,
                                                                     const Zeta64 *__restrict__ Z, int nz,
                                                                     const uint32_t *__restrict__ D, int N,
                                                                     int64_t eoff) {
    const int lane = threadIdx.x & 31;
    const int64_t M = (int64_t)N * N * N;
    const int zi = blockIdx.x * kWarps64 + (threadIdx.x >> 5);
    if (zi >= nz) return;
    const Zeta64 z = Z[zi];
    const int64_t cell = eoff + (int64_t)blockIdx.y * M;  // fhat and Qhat cell-major
    const double2 *Fg = F + cell;
    const double *w = W + z.woff;
    const uint32_t *Dz = D + z.desc_off;
    const int k1 = z.k1, k2 = z.k2, cnt = z.m_count, n3_first = pair_partner(z.k3, z.m_first, N);
    const int nt = z.nblocks * cnt, bstep = 32 / cnt, tstep = 32 % cnt;
    double re[kSums] = {}, im[kSums] = {};
    int b = lane / cnt, t = lane % cnt, q = lane;
    const auto term = [&](double &sr, double &si) {
        const uint32_t d = Dz[b];
        const int m1 = (int)(d & 0xffffu), m2 = (int)(d >> 16);
        int m3 = z.m_first + t, n3 = n3_first - t;
        m3 -= m3 >= N ? N : 0;
        n3 += n3 < 0 ? N : 0;
        const double g_ = w[q];
        const double2 a = Fg[(m1 * N + m2) * N + m3];
        const double2 c = Fg[(pair_partner(k1, m1, N) * N + pair_partner(k2, m2, N)) * N + n3];
        sr += g_ * (a.x * c.x - a.y * c.y);
        si += g_ * (a.x * c.y + a.y * c.x);
        q += 32;
        b += bstep;
        t += tstep;
        if (t >= cnt) {
            t -= cnt;
            ++b;
        }
    };
    while (q + 32 * (kSums - 1) < nt) {
#pragma unroll
        for (int i = 0; i < kSums; ++i) term(re[i], im[i]);
    }
    while (q < nt) term(re[0], im[0]);
    double sr = tree(re), si = tree(im);
    for (int o = 16; o > 0; o >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        si += __shfl_xor_sync(0xffffffffu, si, o);
    }
    if (lane == 0) Qh[cell + (k1 * N + k2) * N + z.k3] = make_double2(sr, si);
}

void launch_conv64_cells(const double2 *F, double2 *Qh, const Table &t, int nvalid, int64_t eoff, cudaStream_t st) {
    dim3 grid((t.n_zeta64 + kWarps64 - 1) / kWarps64, nvalid);
    conv64_cells_kernel<<<grid, 32 * kWarps64, 0, st>>>(F, Qh, t.d_w64, t.d_zeta64, t.n_zeta64, t.d_desc, t.N, eoff);
}

void launch_conv64(const double2 *F, double2 *Qh, const Table &t, int64_t eoff, int ngroups, cudaStream_t st) {
    const int64_t warps = (int64_t)t.n_zeta64 * ngroups;
    conv64_plain_kernel<<<(unsigned)((warps + kWarps64 - 1) / kWarps64), 32 * kWarps64, 0, st>>>(
        F, Qh, t.d_w64, t.d_zeta64, t.n_zeta64, t.d_desc, t.N, eoff, ngroups);
}

}  // namespace bte
