// FP32 weighted convolution (Sec. 3.2) for few cells: the lanes of a warp run
// over the pairs of a block instead of over cells.
//
// The kernels of conv32_device.cuh give every cell a lane, so one cell costs as
// much as 32 (a collide at N = 16: 55 us for 1 to 32 cells, 26 us for one cell here:
// 130 pencils of up to 128 blocks for 456 CTAs). Here one CTA takes a (cell, pencil, k3 tile): its warps take the
// pencil's (m1, m2) blocks in turn, and lane l the pairs l, l + 32, ... of a
// block in the order of the weight table (for_pairs), so that weights are read
// coalesced and a lane's pair t belongs to the same (m3, k3) in every block: it
// sums its pairs in registers, over the warp's few blocks, and the pencil's
// outputs are added once at the end (warps, then the pairs of each k3, in a fixed
// order, compensated). fhat is cell-major; a block's two rows go through the
// warp's shared memory (gathers from L1: 4.1 us a cell at N = 16), those and the
// weights of the next block are loaded during the current one.
// The loads bound it (a weight and two 8-byte modes per lane for six FMA-pipe
// operations): 2.8 us a cell at N = 16 once the chip is full, against 0.6 us with
// 32 cells in lanes, so those kernels take over as the batch grows
// (conv32_cells_limit).
#include "kernels.h"

namespace bte {

namespace {

// W warps per CTA; NE: pairs per lane, cpad <= 32 NE.
template <int N_, int T_, int NE_, int W_>
struct CellsShape {
    static constexpr int N = N_, T = T_, NE = NE_, W = W_, V = pair_visits(N_, T_);
    static constexpr int E = NE * 32;
    static constexpr int PT = 8;  // threads per output in the last sum
};

__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float x) {
    const float s = __fadd_rn(hi, x), bb = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb)));
    hi = s;
}

template <class S>
__global__ void __launch_bounds__(32 * S::W)
conv32_cells_kernel(const float2 *__restrict__ F, float2 *__restrict__ Qh, const float *__restrict__ Wt,
                    const uint32_t *__restrict__ D, const ConvItem *__restrict__ items,
                    const uint16_t *__restrict__ ent, const int16_t *__restrict__ rk, int kind0, int cpad0, int cpad1,
                    int64_t eoff) {
    constexpr int N = S::N, T = S::T, NE = S::NE, W = S::W, E = S::E;
    constexpr int64_t M = (int64_t)N * N * N;
    constexpr int RL = (2 * N + 31) / 32;
    __shared__ float2 red[W][E];
    __shared__ float2 srows[W][2][2 * N];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const ConvItem it = items[blockIdx.x];
    const int tile = (int)it.kind - kind0, cpad = tile ? cpad1 : cpad0, nb = (int)it.nblocks;
    const float2 *Fc = F + eoff + (int64_t)blockIdx.y * M;
    const float *w0 = Wt + it.wofs;
    int ma[NE], mb[NE];
    bool in[NE];
#pragma unroll
    for (int t = 0; t < NE; ++t) {
        const int e = lane + 32 * t;
        in[t] = e < cpad;
        const uint16_t c = in[t] ? ent[tile * E + e] : (uint16_t)0;
        ma[t] = c & 0xff;
        mb[t] = N + (c >> 8);
    }
    float re[NE], im[NE];
#pragma unroll
    for (int t = 0; t < NE; ++t) re[t] = im[t] = 0.f;
    // rows of block b: a in rows[0 .. N), b in rows[N .. 2N), RL values a lane
    float2(*rows)[2 * N] = srows[warp];
    float2 rv[RL];
    float wv[NE];
    auto load = [&](int b, uint32_t d) {
        const int m1 = (int)(d & 0xffffu), m2 = (int)(d >> 16);
        const float2 *A = Fc + (m1 * N + m2) * N;
        const float2 *B = Fc + (pair_partner((int)it.k1, m1, N) * N + pair_partner((int)it.k2, m2, N)) * N;
        const float *w = w0 + (size_t)b * cpad + lane;
#pragma unroll
        for (int q = 0; q < RL; ++q) {
            const int i = lane + 32 * q;
            rv[q] = i < N ? A[i] : i < 2 * N ? B[i - N] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int t = 0; t < NE; ++t) wv[t] = in[t] ? w[32 * t] : 0.f;
    };
    // the warp's blocks: warp, warp + W, ...; descriptors of up to 32 of them, one per lane
    for (int b0 = warp; b0 < nb; b0 += 32 * W) {
        const int mine = min(32, (nb - b0 + W - 1) / W);
        const uint32_t dl = lane < mine ? D[it.desc_off + b0 + lane * W] : 0u;
        load(b0, __shfl_sync(0xffffffffu, dl, 0));
        for (int i = 0; i < mine; ++i) {
            float2 *row = rows[i & 1];
#pragma unroll
            for (int q = 0; q < RL; ++q)
                if (lane + 32 * q < 2 * N) row[lane + 32 * q] = rv[q];
            float w[NE];
#pragma unroll
            for (int t = 0; t < NE; ++t) w[t] = wv[t];
            __syncwarp();  // the other buffer's readers passed the barrier before it
            if (i + 1 < mine) load(b0 + (i + 1) * W, __shfl_sync(0xffffffffu, dl, i + 1));
#pragma unroll
            for (int t = 0; t < NE; ++t) {
                const float2 a = row[ma[t]], b = row[mb[t]];
                const float tr = w[t] * a.x, ti = w[t] * a.y;
                re[t] = fmaf(tr, b.x, fmaf(-ti, b.y, re[t]));
                im[t] = fmaf(tr, b.y, fmaf(ti, b.x, im[t]));
            }
        }
        __syncwarp();
    }
#pragma unroll
    for (int t = 0; t < NE; ++t) red[warp][lane + 32 * t] = make_float2(re[t], im[t]);
    __syncthreads();
    // the warps' sums of each pair, then the pairs of each output by PT threads
    for (int e = threadIdx.x; e < E; e += 32 * W) {
        float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
#pragma unroll
        for (int q = 0; q < W; ++q) {
            const float2 v = red[q][e];
            two_sum_acc(rh, rl, v.x);
            two_sum_acc(ih, il, v.y);
        }
        red[0][e] = make_float2(rh, ih);  // this thread alone reads and writes column e
        red[1][e] = make_float2(rl, il);
    }
    __syncthreads();
    if (threadIdx.x >= T * S::PT) return;
    const int j = threadIdx.x / S::PT, part = threadIdx.x % S::PT;
    float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
    for (int i = part; i < S::V; i += S::PT) {
        const int e = rk[(tile * S::V + i) * T + j];
        if (e < 0) continue;
        const float2 h = red[0][e], l = red[1][e];
        two_sum_acc(rh, rl, h.x);
        two_sum_acc(ih, il, h.y);
        rl += l.x;
        il += l.y;
    }
    static_assert(T * S::PT % 32 == 0, "whole warps");
    constexpr unsigned mask = 0xffffffffu;
#pragma unroll
    for (int o = S::PT / 2; o > 0; o >>= 1) {
        const float a = __shfl_down_sync(mask, rh, o, S::PT), b = __shfl_down_sync(mask, rl, o, S::PT);
        const float c = __shfl_down_sync(mask, ih, o, S::PT), d = __shfl_down_sync(mask, il, o, S::PT);
        two_sum_acc(rh, rl, a);
        two_sum_acc(ih, il, c);
        rl += b;
        il += d;
    }
    if (part == 0)
        Qh[eoff + (int64_t)blockIdx.y * M + ((int)it.k1 * N + (int)it.k2) * N + tile * T + j] =
            make_float2(rh + rl, ih + il);
}

using C8 = CellsShape<8, 8, 2, 4>;
using C12 = CellsShape<12, 12, 4, 8>;
using C16 = CellsShape<16, 16, 7, 16>;
using C24 = CellsShape<24, 12, 8, 8>;
using C32 = CellsShape<32, 16, 13, 8>;

template <class S>
void launch(const float2 *F, float2 *Qh, const Table &t, int nvalid, int64_t eoff, cudaStream_t st) {
    conv32_cells_kernel<S><<<dim3(t.n_tmpl, nvalid), 32 * S::W, 0, st>>>(
        F, Qh, t.d_w32, t.d_desc, t.d_tmpl, t.d_ent, t.d_rk, t.kind0, t.cpad[0], t.cpad[1], eoff);
}

}  // namespace

int conv32_cells_entries(int N) {
    switch (N) {
        case 8: return C8::E;
        case 12: return C12::E;
        case 16: return C16::E;
        case 24: return C24::E;
        case 32: return C32::E;
        default: return 0;
    }
}

// Up to this many cells no call is slower with pairs in lanes than with cells in lanes and
// the items cut by their plan (us, pairs / cells in lanes, a collide and a Heun step:
// N = 8, 56 cells 24.6 / 26.5 and 36.3 / 43.0, 64 cells 26.6 / 26.6 and 38.3 / 43.1; N = 12, 20
// cells 33.8 / 36.0 and 57.4 / 61.7, 24 cells 36.0 / 36.3 and 63.6 / 61.5; N = 16, 1 cell 26 / 55,
// 8 cells 47.1 / 55.5, 11 cells 55.3 / 55.5 and 100.3 / 104.8, 12 cells 59.3 / 55.2 and 105.7 /
// 105.6; N = 24, 9 cells 246 / 266 and 501 / 549, 10 cells 269 / 266 and 547 / 547; N = 32, 10 cells
// 1168 / 1234 and 2349 / 2474, 12 cells 1390 / 1226 and 2793 / 2473).
int conv32_cells_limit(int N) {
    switch (N) {
        case 8: return 56;
        case 12: return 22;
        case 16: return 11;
        case 24: return 9;
        case 32: return 10;
        default: return 0;
    }
}

void launch_conv32_cells(const float2 *F, float2 *Qh, const Table &t, int nvalid, int64_t eoff, cudaStream_t st) {
    switch (t.N) {
        case 8: launch<C8>(F, Qh, t, nvalid, eoff, st); break;
        case 12: launch<C12>(F, Qh, t, nvalid, eoff, st); break;
        case 16: launch<C16>(F, Qh, t, nvalid, eoff, st); break;
        case 24: launch<C24>(F, Qh, t, nvalid, eoff, st); break;
        case 32: launch<C32>(F, Qh, t, nvalid, eoff, st); break;
        default: break;
    }
}

}  // namespace bte
