// Learned collision path (mode BTE_LEARNED): surrogate -> conservation
// projection -> residual indicator -> exact fallback.
//
// Indicator (per cell). The exact operator is evaluated on S sampled zeta
// pencils (k1, k2) (fixed, seeded, |k1'|, |k2'| <= N/4), all N modes k3 of each:
//   Qhat(k)  = sum_m Ghat(xi_m, zeta_k) dz^3 fhat_m fhat_{k-m+N/2}     (Sec. 3.2)
//   Qhat-(k) = the same sum with the loss term of Ghat only,
// and compared with the forward transform of the projected surrogate output:
//   ind = ||Fhat[P Q_nn](k) - Qhat(k)||_S / ||Qhat-(k)||_S,
// i.e. the parity metric of the fast path restricted to S N modes. Cells with
// ind > tol are recomputed with the FP32 operator. Cost of the check: S of the
// N^2 pencils of the convolution (4 / 256 = 1.6 % at N = 16).
#include <algorithm>
#include <cmath>
#include <vector>

#include "bulk.cuh"
#include "learned.h"
#include "fpconv.cuh"
#include "project.cuh"
#include "rng.h"

namespace bte {

namespace {

// One CTA of kIndWarps warps per (sampled pencil, group), lane = cell: the
// warps work in pairs, each pair takes the pencil's kept (m1, m2) blocks in
// turn (unordered pairs, weights
// Ghat(k,m) + Ghat(k,n)) and each warp of a pair half of the N outputs k3,
// with the full and the loss weights side by side. A block's a and b rows and
// its weights come by bulk copies into a two-deep ring of the pair, issued two
// blocks ahead (read straight from L2 the loads left the FMA pipe 34 % busy:
// 1024 cells, N = 16, 57 us, with the ring 50). Half the outputs per warp keep the kernel at
// two CTAs per SM. Partial sums are added across the pairs in a fixed order, then
// compared with the transform of the projected surrogate output.
constexpr int kIndWarps = 8;
constexpr int kIndPairs = kIndWarps / 2;
constexpr int kIndStages = 2;
constexpr int kIndBlocks = 16;  // blocks of a part

// Pairs of one block for the outputs of half jh, in groups of four weights.
template <int N>
__host__ __device__ constexpr int ind_groups(int jh) {
    int c = 0;
    for (int m = 0; m < N; ++m)
        for (int j = jh * N / 2; j < (jh + 1) * N / 2; ++j) c += pair_on_grid(j, m, N);
    return (c + 3) / 4;
}
// Floats of a block's weights: half 0, then half 1, four full and four loss weights in turn.
template <int N>
__host__ __device__ constexpr int ind_weights() {
    return 8 * (ind_groups<N>(0) + ind_groups<N>(1));
}
template <int N>
constexpr int ind_stage_bytes() {
    return 2 * N * kLanes * 8 + 4 * ind_weights<N>();
}
template <int N>
constexpr size_t ind_smem() {
    const size_t ring = (size_t)kIndPairs * kIndStages * ind_stage_bytes<N>(), red = sizeof(float) * kIndPairs * 4 * N * kLanes;
    return ring > red ? ring : red;
}

// The pair sums of one block for the outputs k3 in [JH N/2, (JH + 1) N/2):
// acc = full (re, im) per output, then loss (re, im). The weight of the pair
// (m3, k3) sits at its rank among the half's pairs (m3 major, k3 minor), a
// compile-time index after unrolling.
template <int N, int JH>
__device__ __forceinline__ void indicator_block(const float2 (&av)[N], const float2 (&bv)[N], const float4 *w,
                                                float (&acc)[2 * N]) {
    constexpr int H = N / 2, J0 = JH * H;
    int wi = 0;
#pragma unroll
    for (int m3 = 0; m3 < N; ++m3)
#pragma unroll
        for (int j = J0; j < J0 + H; ++j) {
            const int n3 = j - m3 + H;
            if (n3 < 0 || n3 >= N) continue;
            const float4 f4 = w[2 * (wi >> 2)], l4 = w[2 * (wi >> 2) + 1];
            const int q = wi & 3;
            const float wF = q == 0 ? f4.x : q == 1 ? f4.y : q == 2 ? f4.z : f4.w;
            const float wL = q == 0 ? l4.x : q == 1 ? l4.y : q == 2 ? l4.z : l4.w;
            const float pr = av[m3].x * bv[n3].x - av[m3].y * bv[n3].y;
            const float pi = av[m3].x * bv[n3].y + av[m3].y * bv[n3].x;
            const int o = j - J0;
            acc[2 * o] = fmaf(wF, pr, acc[2 * o]);
            acc[2 * o + 1] = fmaf(wF, pi, acc[2 * o + 1]);
            acc[N + 2 * o] = fmaf(wL, pr, acc[N + 2 * o]);
            acc[N + 2 * o + 1] = fmaf(wL, pi, acc[N + 2 * o + 1]);
            ++wi;
        }
}

// A pencil has between N^2/8 and N^2/2 blocks: it is cut into parts of
// kIndBlocks blocks, one CTA each (blockIdx.z), so that the S x groups items
// fill the GPU and no SM is left with a whole long pencil. Each part reduces
// its pairs in a fixed order into part[], and the part that finishes last (an
// atomic count, no waiting) adds the parts in their order and forms the errors.
// 1024 cells, N = 16, 8 / 16 / 24 / 32 blocks a part: 59.7 / 51.0 / 48.2 / 57.6 us;
// 16 leaves a small batch with more CTAs (the indicator of a few cells 67 -> 47 us).
template <int N>
__global__ void __launch_bounds__(32 * kIndWarps, 2)
indicator_kernel(const float2 *__restrict__ F, const float2 *__restrict__ QN, const float *__restrict__ W,
                 const uint32_t *__restrict__ desc, const IndPencil *__restrict__ pens, int parts,
                 int64_t eoff, int nslots, float *err2, float *den2, float *part, unsigned *cnt, int *status) {
    constexpr int M = N * N * N, H = N / 2, ROW = N * kLanes * 8, STAGE = ind_stage_bytes<N>();
    extern __shared__ __align__(128) char ind_raw[];
    __shared__ __align__(8) uint64_t s_full[kIndPairs][kIndStages];
    __shared__ bool s_last;
    float *red = reinterpret_cast<float *>(ind_raw);  // [kIndPairs][4 N][32], after the ring's last use
    const int p = blockIdx.x, g = blockIdx.y, z = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int pair = warp >> 1, jh = warp & 1;
    const IndPencil pen = pens[p];
    const int nz = (pen.nblocks + kIndBlocks - 1) / kIndBlocks;
    if (z >= nz) return;
    const int k1 = pen.kk / N, k2 = pen.kk % N;
    const float2 *Fg = F + eoff + (int64_t)g * M * kLanes;  // fhat in the sector order of the group
    char *ring = ind_raw + (size_t)pair * kIndStages * STAGE;
    const bool producer = jh == 0 && lane == 0;
    if (producer) {
        for (int s = 0; s < kIndStages; ++s) mbar_init(smem_u32(&s_full[pair][s]), 1);
        fence_mbar_init();
    }
    __syncthreads();
    float acc[2 * N];  // this warp's outputs: full (re, im) per k3, then loss (re, im)
#pragma unroll
    for (int i = 0; i < 2 * N; ++i) acc[i] = 0.f;
    const int b0 = z * kIndBlocks + pair, bend = min((z + 1) * kIndBlocks, pen.nblocks);
    const int n = b0 < bend ? (bend - b0 + kIndPairs - 1) / kIndPairs : 0;
    auto issue = [&](int i) {  // rows of a group are N * 256 bytes, whole sectors
        const int b = b0 + i * kIndPairs, s = i % kIndStages;
        const uint32_t d = desc[pen.desc_off + b], bar = smem_u32(&s_full[pair][s]), dst = smem_u32(ring + s * STAGE);
        const int m1 = (int)(d & 0xffffu), m2 = (int)(d >> 16), n1 = k1 - m1 + H, n2 = k2 - m2 + H;
        mbar_expect_tx(bar, STAGE);
        bulk_g2s(dst, Fg + (int64_t)((m1 * N + m2) * N) * kLanes, ROW, bar);
        bulk_g2s(dst + ROW, Fg + (int64_t)((n1 * N + n2) * N) * kLanes, ROW, bar);
        bulk_g2s(dst + 2 * ROW, W + pen.wofs + (size_t)b * ind_weights<N>(), 4 * ind_weights<N>(), bar);
    };
    if (producer)
        for (int i = 0; i < kIndStages && i < n; ++i) issue(i);
    bool live = true;  // until a wait runs out: then the pair only keeps its barriers
    for (int i = 0; i < n; ++i) {
        const int s = i % kIndStages;
        if (live) live = __all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&s_full[pair][s]), (i / kIndStages) & 1));
        if (live) {
            const char *st = ring + s * STAGE;
            float2 av[N], bv[N];
#pragma unroll
            for (int e = 0; e < N; e += 2) {  // two modes of the lane per 16-byte load (rows start on a sector)
                const float4 a2 = *reinterpret_cast<const float4 *>(st + 8 * sector_index(e, lane));
                const float4 b2 = *reinterpret_cast<const float4 *>(st + ROW + 8 * sector_index(e, lane));
                av[e] = make_float2(a2.x, a2.y);
                av[e + 1] = make_float2(a2.z, a2.w);
                bv[e] = make_float2(b2.x, b2.y);
                bv[e + 1] = make_float2(b2.z, b2.w);
            }
            const float4 *w = reinterpret_cast<const float4 *>(st + 2 * ROW);
            if (jh == 0) indicator_block<N, 0>(av, bv, w, acc);
            else indicator_block<N, 1>(av, bv, w + 2 * ind_groups<N>(0), acc);
        }
        asm volatile("bar.sync %0, 64;" ::"r"(pair + 1) : "memory");  // both warps have read the stage
        if (producer && live && i + kIndStages < n) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue(i + kIndStages);
        }
        if (!live && lane == 0) atomicOr(status, ST_TIMEOUT);
    }
    if (producer && !live)  // no copy stays in flight (bounded again)
        for (int s = 0; s < kIndStages; ++s)
            for (uint32_t ph = 0; ph < 2; ++ph) mbar_wait_bounded(smem_u32(&s_full[pair][s]), ph);
    __syncthreads();  // the ring becomes the reduction's buffer
    // the pair's 4 N sums: full (re, im) of output k3 at 2 k3, loss at 2 N + 2 k3
#pragma unroll
    for (int o = 0; o < H; ++o) {
        const int k3 = jh * H + o;
        red[(pair * 4 * N + 2 * k3) * kLanes + lane] = acc[2 * o];
        red[(pair * 4 * N + 2 * k3 + 1) * kLanes + lane] = acc[2 * o + 1];
        red[(pair * 4 * N + 2 * N + 2 * k3) * kLanes + lane] = acc[N + 2 * o];
        red[(pair * 4 * N + 2 * N + 2 * k3 + 1) * kLanes + lane] = acc[N + 2 * o + 1];
    }
    __syncthreads();
    const size_t item = (size_t)p * gridDim.y + g;
    float *mine = part + (item * parts + z) * (4 * N * kLanes);
    for (int i = threadIdx.x; i < 4 * N * kLanes; i += 32 * kIndWarps) {
        float v = 0.f;
        for (int w = 0; w < kIndPairs; ++w) v += red[(size_t)w * 4 * N * kLanes + i];
        mine[i] = v;
    }
    __threadfence();  // this part's sums before the count
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(cnt + item, 1u) == (unsigned)nz - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();  // the other parts' sums after the count
    const float *h = part + item * parts * (4 * N * kLanes) + lane;
    float e = 0.f, dn = 0.f;
    const float2 *qn = QN + eoff + (int64_t)g * M * kLanes + (int64_t)pen.kk * N * kLanes + lane;
    for (int j = warp; j < N; j += kIndWarps) {
        float v[4] = {};
        for (int i = 0; i < nz; ++i)
#pragma unroll
            for (int o = 0; o < 4; ++o)
                v[o] += __ldcg(h + (i * 4 * N + (o >> 1) * 2 * N + 2 * j + (o & 1)) * kLanes);
        const float2 q = qn[(int64_t)j * kLanes];
        const float dr = q.x - v[0], di = q.y - v[1];
        e += dr * dr + di * di;
        dn += v[2] * v[2] + v[3] * v[3];
    }
    red[warp * kLanes + lane] = e;  // the pairs' sums were read before the count
    red[(kIndWarps + warp) * kLanes + lane] = dn;
    __syncthreads();
    if (warp != 0) return;
    e = dn = 0.f;
    for (int w = 0; w < kIndWarps; ++w) {
        e += red[w * kLanes + lane];
        dn += red[(kIndWarps + w) * kLanes + lane];
    }
    const int slot = g * kLanes + lane;
    err2[(size_t)p * nslots + slot] = e;
    den2[(size_t)p * nslots + slot] = dn;
}

__global__ void indicator_reduce_kernel(const float *__restrict__ err2, const float *__restrict__ den2, int S,
                                        int nslots, int nvalid, float *ind, double *ind64) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nslots) return;
    float e = 0.f, d = 0.f;
    for (int s = 0; s < S; ++s) {
        e += err2[(size_t)s * nslots + c];
        d += den2[(size_t)s * nslots + c];
    }
    const float v = c < nvalid ? sqrtf(e) / fmaxf(sqrtf(d), 1e-30f) : 0.f;
    ind[c] = v;
    if (ind64 && c < nvalid) ind64[c] = (double)v;  // the caller's array (slot = cell)
}

// Surrogate output to the caller's cells with the conservation projection of
// Sec. 3.3 fused in: Q = P_N(c Y), c = rho^2 / s_out per cell. One CTA per
// cell, one thread per pencil (j1, j2): the moments of Y are accumulated in
// double-float FP32 (the values are FP32), mu(Q) = c mu(Y) and lambda are
// formed in FP64, and Q_j = c Y_j - C_j^T lambda is written in FP64 on a
// coalesced mapping (one FP64 operation per value). Instructions bound it: 1024
// cells, N = 16, 34.6 us with five warp trees, the correction's polynomial per
// pencil and two renormalised additions a value, 21.7 us as it stands.
template <int N>
__global__ void __launch_bounds__((N * N + 31) / 32 * 32)
post_project_kernel(const float *__restrict__ Y, const double *__restrict__ rho, float s_out, ProjArgs pa,
                    double *__restrict__ Q) {
    constexpr int M = N * N * N, NN = N * N, H = N / 2, NT = (NN + 31) / 32 * 32, NW = NT / 32;
    const int r = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const float *y = Y + (size_t)r * M;
    double *q = Q + (size_t)r * M;
    __shared__ float red[NW][10];
    __shared__ float2 base[NN];
    __shared__ __align__(16) float2 sg[N];
    __shared__ double lam[5], tab[3][N], c_s;
    __shared__ float2 c_hl;
    if (t == 0) {  // the output scale, once per cell (an FP64 division), and its double-float split
        const double c = rho[r] * rho[r] / (double)s_out;
        const float hi = fpc::narrow(c);
        c_s = c;
        c_hl = make_float2(hi, fpc::narrow(c - fpc::widen(hi)));
    }
    Df mom[5];
    if (t < NN) {
        Df s0{0.f, 0.f}, s1{0.f, 0.f}, s2{0.f, 0.f};
        const float4 *yp = reinterpret_cast<const float4 *>(y + t * N);
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            const float4 v4 = yp[i];
            const float v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const int w = 4 * i + o - H;
                df_add(s0, v[o]);
                df_add_prod(s1, (float)w, v[o]);
                df_add_prod(s2, (float)(w * w), v[o]);
            }
        }
        const int w1 = t / N - H, w2 = t % N - H;
        mom[0] = s0;
        mom[1] = df_mul_int(s0, (float)w1);
        mom[2] = df_mul_int(s0, (float)w2);
        mom[3] = s1;
        mom[4] = df_add(df_mul_int(s0, (float)(w1 * w1 + w2 * w2)), s2);
    } else {
#pragma unroll
        for (int i = 0; i < 5; ++i) mom[i] = Df{0.f, 0.f};
    }
    Df sum;
    const int mi = df_warp_sum5(mom, sum);
    if (mi >= 0) {
        red[warp][2 * mi] = sum.hi;
        red[warp][2 * mi + 1] = sum.lo;
    }
    __syncthreads();
    if (warp == 0) {
        double mu = 0.0;
        if (lane < 5) {
            Df m{red[0][2 * lane], red[0][2 * lane + 1]};
#pragma unroll
            for (int w = 1; w < NW; ++w) m = df_add(m, Df{red[w][2 * lane], red[w][2 * lane + 1]});
            mu = (fpc::widen(m.hi) + fpc::widen(m.lo)) * c_s;
            mu *= lane == 0 ? 1.0 : (lane == 4 ? pa.dv * pa.dv : pa.dv);
        }
        double m5[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) m5[i] = __shfl_sync(0xffffffffu, mu, i);
        if (lane < 5) {
            double l = 0.0;
#pragma unroll
            for (int k = 0; k < 5; ++k) l = fma(pa.ainv[lane * 5 + k], m5[k], l);
            lam[lane] = l;
        }
        __syncwarp();
        correction_tables<N>(lam, pa.dv, tab);
    }
    __syncthreads();
    // The correction C^T lambda = base(j1, j2) + g(j3) is formed in FP64 per
    // pencil and per j3, then kept as double-float pairs (hi, lo): per value
    // Q = c Y - base - g is then FP32 work (an exact TwoProduct for c Y, an
    // exact TwoSum of the leading parts each and the sum of what they leave,
    // relative error ~2^-48) and one FP64 addition hi + lo, instead of three
    // FP64-unit operations.
    const auto split = [](double v) {
        const float hi = fpc::narrow(v);
        return make_float2(-hi, -fpc::narrow(v - fpc::widen(hi)));
    };
    if (t < NN) base[t] = split(tab[0][t / N] + tab[1][t % N]);
    if (t < N) sg[t] = split(tab[2][t]);
    __syncthreads();
    const float c_hi = c_hl.x, c_lo = c_hl.y;
    const bool wide = (reinterpret_cast<uintptr_t>(q) & 15u) == 0;
    const auto value = [&](float yv, float2 b, float2 g) {
        const float p = __fmul_rn(c_hi, yv), pe = fmaf(c_lo, yv, fmaf(c_hi, yv, -p));
        float s1, e1, s2, e2;
        two_sum_f(b.x, g.x, s1, e1);
        two_sum_f(p, s1, s2, e2);
        const float lo = __fadd_rn(__fadd_rn(pe, __fadd_rn(b.y, g.y)), __fadd_rn(e1, e2));
        return fpc::widen(s2) + fpc::widen(lo);
    };
    for (int e = 2 * t; e < M; e += 2 * NT) {  // two values of a pencil: 8-byte loads, 16-byte stores where q allows
        const float2 yv = *reinterpret_cast<const float2 *>(y + e);
        const float2 b = base[e / N];
        const float4 g = *reinterpret_cast<const float4 *>(&sg[e % N]);
        const double q0 = value(yv.x, b, make_float2(g.x, g.y)), q1 = value(yv.y, b, make_float2(g.z, g.w));
        if (wide) {
            *reinterpret_cast<double2 *>(q + e) = make_double2(q0, q1);
        } else {
            q[e] = q0;
            q[e + 1] = q1;
        }
    }
}

// The fallback of the learned mode, laid out on the device (one CTA): cells
// whose indicator is not <= tol are listed in increasing order, and the FP32
// operator's batch for them is written for up to nslots_cap slots: offsets
// (redo[s] M for the listed cells, -1 for the padding lanes of the last
// 32-cell group, -2 for the groups that hold no cell: the transforms skip
// them), the convolution's work list (the one-group template repeated for the
// groups in use, all groups of the costliest pencil first), its length and a
// zeroed queue counter. The statistics (cells seen, cells recomputed, the
// largest indicator as FP32 bits) accumulate in stats. No host round trip.
constexpr int kSetupThreads = 1024;
__global__ void __launch_bounds__(kSetupThreads)
fallback_setup_kernel(const float *__restrict__ ind, int ncells, double tol, int64_t M,
                      const ConvItem *__restrict__ tmpl, int ntmpl, int nslots_cap, int64_t *__restrict__ off,
                      ConvItem *__restrict__ items, int *__restrict__ nitems, unsigned *__restrict__ counter,
                      unsigned long long *__restrict__ stats) {
    __shared__ int warp_tot[kSetupThreads / 32];
    __shared__ int s_base;
    __shared__ unsigned s_max;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) {
        s_base = 0;
        s_max = 0u;
    }
    __syncthreads();
    for (int c0 = 0; c0 < ncells; c0 += kSetupThreads) {
        const int c = c0 + t;
        const float v = c < ncells ? ind[c] : 0.f;
        const int flag = (c < ncells && !((double)v <= tol)) ? 1 : 0;
        // the largest indicator (non-negative floats order as their bit patterns; NaN is left out)
        const unsigned vmax = __reduce_max_sync(0xffffffffu, (c < ncells && v >= 0.f) ? __float_as_uint(v) : 0u);
        if (lane == 0 && vmax) atomicMax(&s_max, vmax);
        // block-wide exclusive prefix sum of the flags (in cell order)
        const unsigned bal = __ballot_sync(0xffffffffu, flag);
        const int before = __popc(bal & ((1u << lane) - 1u));
        if (lane == 0) warp_tot[warp] = __popc(bal);
        __syncthreads();
        int wbase = 0;
        for (int w = 0; w < warp; ++w) wbase += warp_tot[w];
        const int base = s_base;
        if (flag) off[base + wbase + before] = (int64_t)c * M;
        __syncthreads();
        if (t == kSetupThreads - 1) s_base = base + wbase + before + flag;
        __syncthreads();
    }
    const int nredo = s_base, ngu = (nredo + kLanes - 1) / kLanes;
    for (int sl = nredo + t; sl < nslots_cap; sl += kSetupThreads) off[sl] = sl < ngu * kLanes ? -1 : -2;
    for (int i = t; i < ngu * ntmpl; i += kSetupThreads) {
        ConvItem it = tmpl[i / ngu];
        it.fofs = (uint64_t)((int64_t)(i % ngu) * M * kLanes);
        items[i] = it;
    }
    if (t == 0) {
        *nitems = ngu * ntmpl;
        *counter = 0u;
        atomicAdd(stats + 0, (unsigned long long)ncells);
        atomicAdd(stats + 1, (unsigned long long)nredo);
        atomicMax(stats + 2, (unsigned long long)s_max);
    }
}

// y = x + a Q (mode 1) or y += a (qp + Q) (mode 2) on n values: the time update
// of a Heun stage when Q comes from the learned mode.
__global__ void stage_update_kernel(const double *__restrict__ Q, const double *__restrict__ x, double *__restrict__ y,
                                    const double *__restrict__ qp, double a, int64_t n, int mode) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = mode == 1 ? fma(a, Q[i], x[i]) : fma(a, qp[i] + Q[i], y[i]);
}

}  // namespace

void launch_fallback_setup(const float *ind, int ncells, double tol, int64_t M, const ConvItem *tmpl, int ntmpl,
                           int nslots_cap, int64_t *off, ConvItem *items, int *nitems, unsigned *counter,
                           unsigned long long *stats, cudaStream_t st) {
    fallback_setup_kernel<<<1, kSetupThreads, 0, st>>>(ind, ncells, tol, M, tmpl, ntmpl, nslots_cap, off, items,
                                                        nitems, counter, stats);
}

void launch_stage_update(const double *Q, const double *x, double *y, const double *qp, double a, int64_t n,
                         int mode, cudaStream_t st) {
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, 4096);
    stage_update_kernel<<<(unsigned)blocks, 256, 0, st>>>(Q, x, y, qp, a, n, mode);
}

int build_indicator_table(const Table &t, int modes, uint64_t seed, IndicatorTable &out) {
    const int N = t.N, h = N / 2, q = N / 4;
    const int S = std::max(1, modes / N);
    const double dz3 = t.dz * t.dz * t.dz;
    const double c = std::sqrt(2.0 / 3.14159265358979323846);
    // SplitMix64 from `seed`; each pencil offset is (next mod (2q + 1)) - q,
    // k1' first; repeated pencils are skipped. Integer arithmetic only, so
    // every platform draws the same sample.
    SplitMix64 rng(seed);
    const uint64_t span = (uint64_t)(2 * q + 1);
    std::vector<int> kks;
    while ((int)kks.size() < S) {
        const int k1 = (int)(rng.next() % span) - q;
        const int k2 = (int)(rng.next() % span) - q;
        const int kk = (k1 + h) * N + (k2 + h);
        if (std::find(kks.begin(), kks.end(), kk) == kks.end()) kks.push_back(kk);
    }
    // the sampled pencils' own blocks: the modes are compared one by one, so the
    // sums run over the pencil's box with the plain pair weights Ghat(k, m) +
    // Ghat(k, n) (blocks (m1, m2) <= (n1, n2); a block that pairs with itself
    // keeps Ghat(k, m)), the full ones and those of the loss term, for the
    // outputs k3 < N/2 and then the others, each m3 ascending, then k3, in groups
    // of four full and four loss weights
    std::vector<float> w;
    std::vector<IndPencil> pens;
    std::vector<uint32_t> desc;
    int parts = 1;
    for (int kk : kks) {
        const int k1 = kk / N, k2 = kk % N;
        IndPencil pn{};
        pn.kk = kk;
        pn.desc_off = (int)desc.size();
        pn.wofs = w.size();
        for (int m1 = 0; m1 < N; ++m1)
            for (int m2 = 0; m2 < N; ++m2) {
                const int n1 = k1 - m1 + h, n2 = k2 - m2 + h;
                if (n1 < 0 || n1 >= N || n2 < 0 || n2 >= N || m1 > n1 || (m1 == n1 && m2 > n2)) continue;
                desc.push_back((uint32_t)m1 | ((uint32_t)m2 << 16));
            }
        pn.nblocks = (int)desc.size() - pn.desc_off;
        parts = std::max(parts, (pn.nblocks + kIndBlocks - 1) / kIndBlocks);
        for (int b = 0; b < pn.nblocks; ++b) {
            const uint32_t dd = desc[pn.desc_off + b];
            const int m1 = (int)(dd & 0xffffu), m2 = (int)(dd >> 16), n1 = k1 - m1 + h, n2 = k2 - m2 + h;
            const bool pair = !(m1 == n1 && m2 == n2);
            for (int jh = 0; jh < 2; ++jh) {
                size_t wi = 0;
                const size_t base = w.size();
                for (int m3 = 0; m3 < N; ++m3)
                    for (int k3 = jh * h; k3 < (jh + 1) * h; ++k3) {
                        const int n3 = k3 - m3 + h;
                        if (n3 < 0 || n3 >= N) continue;
                        double full = t.ghat(k1, k2, k3, m1, m2, m3);
                        const int sm = (m1 - h) * (m1 - h) + (m2 - h) * (m2 - h) + (m3 - h) * (m3 - h);
                        double g = -c * t.J[sm];
                        if (pair) {
                            const int sn = (n1 - h) * (n1 - h) + (n2 - h) * (n2 - h) + (n3 - h) * (n3 - h);
                            full += t.ghat(k1, k2, k3, n1, n2, n3);
                            g += -c * t.J[sn];
                        }
                        if (wi % 4 == 0) w.resize(w.size() + 8, 0.0f);
                        float *const e = &w[base + 8 * (wi / 4) + wi % 4];
                        ++wi;
                        e[0] = (float)(full * dz3);
                        e[4] = (float)(g * dz3);
                    }
            }
        }
        pens.push_back(pn);
    }
    out.S = S;
    out.parts = parts;
    out.kks = kks;
    cudaError_t e = cudaMalloc(&out.d_w, sizeof(float) * std::max<size_t>(w.size(), 4));
    if (e == cudaSuccess) e = cudaMalloc(&out.d_desc, sizeof(uint32_t) * std::max<size_t>(desc.size(), 1));
    if (e == cudaSuccess)
        e = upload(out.d_desc, desc.data(), sizeof(uint32_t) * desc.size());
    if (e == cudaSuccess) e = cudaMalloc(&out.d_pen, sizeof(IndPencil) * S);
    if (e == cudaSuccess) e = upload(out.d_w, w.data(), sizeof(float) * w.size());
    if (e == cudaSuccess) e = upload(out.d_pen, pens.data(), sizeof(IndPencil) * S);
    if (e == cudaSuccess) e = cudaMalloc(&out.d_kk, sizeof(int) * S);
    if (e == cudaSuccess) e = upload(out.d_kk, kks.data(), sizeof(int) * S);
    // shared memory of the cross-warp reduction (set outside any stream capture)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(indicator_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ind_smem<8>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(indicator_kernel<12>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ind_smem<12>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(indicator_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ind_smem<16>());
    if (e != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    return 0;
}

void free_indicator_table(IndicatorTable &t) {
    cudaFree(t.d_w);
    cudaFree(t.d_desc);
    cudaFree(t.d_pen);
    t.d_w = nullptr;
    t.d_desc = nullptr;
    cudaFree(t.d_kk);
    t.d_pen = nullptr;
    t.d_kk = nullptr;
}

void launch_post_project(const float *Y, const double *rho, int B, int N, float s_out, const ProjArgs &pa, double *Q,
                         cudaStream_t st) {
    switch (N) {
        case 8: post_project_kernel<8><<<B, 64, 0, st>>>(Y, rho, s_out, pa, Q); break;
        case 12: post_project_kernel<12><<<B, 160, 0, st>>>(Y, rho, s_out, pa, Q); break;
        case 16: post_project_kernel<16><<<B, 256, 0, st>>>(Y, rho, s_out, pa, Q); break;
        default: break;
    }
}

size_t indicator_scratch_floats(const IndicatorTable &it, int N, int nslots) {
    const size_t items = (size_t)it.S * (nslots / kLanes);
    return 2 * (size_t)it.S * nslots + nslots + items * it.parts * 4 * N * kLanes + items;
}

void launch_indicator(const IndicatorTable &it, const Table &t, const float2 *F, const float2 *QN, int64_t eoff,
                      int nslots, int nvalid, float *err2, float *den2, float *ind, double *ind64,
                      int *status, cudaStream_t st) {
    dim3 grid(it.S, nslots / kLanes, it.parts);
    // after err2, den2 and ind: the parts' sums, then the per-item counts
    const size_t items = (size_t)it.S * (nslots / kLanes);
    float *part = ind + nslots;
    unsigned *cnt = reinterpret_cast<unsigned *>(part + items * it.parts * 4 * t.N * kLanes);
    cudaMemsetAsync(cnt, 0, sizeof(unsigned) * items, st);
#define BTE_INDICATOR(n) \
    indicator_kernel<n><<<grid, 32 * kIndWarps, ind_smem<n>(), st>>>(F, QN, it.d_w, it.d_desc, it.d_pen, it.parts, \
                                                                     eoff, nslots, err2, den2, part, cnt, status)
    switch (t.N) {
        case 8: BTE_INDICATOR(8); break;
        case 12: BTE_INDICATOR(12); break;
        default: BTE_INDICATOR(16); break;
    }
#undef BTE_INDICATOR
    indicator_reduce_kernel<<<(nslots + 255) / 256, 256, 0, st>>>(err2, den2, it.S, nslots, nvalid, ind, ind64);
}

}  // namespace bte
