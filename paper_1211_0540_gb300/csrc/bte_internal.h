// Internal declarations of libbte (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <map>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/bte.h"
#include "radial.h"

namespace bte {

// Device status bits (atomicOr'ed by kernels, read by bte_sync_status).
enum : int { ST_TIMEOUT = 1, ST_NONFINITE = 2, ST_BADDESC = 4 };

constexpr int kLanes = 32;  // cells per group: one warp lane per cell

// ----------------------------------------------------------------------------
// Convolution kernel variants: N, k3-tile size T and tile origin K0.
// ----------------------------------------------------------------------------
struct ConvKind {
    int N, T, K0;
};
constexpr int kNumKinds = 10;
// kind ids: 0:(8,8,0) 1:(12,12,0) 2:(16,16,0) 3:(24,12,0) 4:(24,12,12) 5:(32,16,0) 6:(32,16,16)
//           7:(48,16,0) 8:(48,16,16) 9:(48,16,32)
inline ConvKind conv_kind(int id) {
    static const ConvKind k[kNumKinds] = {{8, 8, 0},    {12, 12, 0},  {16, 16, 0}, {24, 12, 0},  {24, 12, 12},
                                          {32, 16, 0},  {32, 16, 16}, {48, 16, 0}, {48, 16, 16}, {48, 16, 32}};
    return k[id];
}
// ----------------------------------------------------------------------------
// Half-spectrum convolution. f is real and only the real part of the inverse
// transform is kept, so the modes k and k* (index (N - k) mod N per dimension,
// k*' = -k') count only through Qhat_k + conj(Qhat_k*), and conj(fhat_m) =
// fhat_m* turns the second sum into one over the same products:
//   Qhat_k + conj(Qhat_k*) = sum_m [Gv(k, m) + Gv(k*, m*)] fhat_m fhat_n,
// n = k - m + N/2 taken mod N, Gv = Ghat where k - m + N/2 lies on the grid and
// 0 elsewhere (the zero extension; it differs between the two only in the
// modes of index 0, whose mirror is themselves). The convolutions evaluate
// one pencil (k1, k2) of each mirror pair with these weights; the inverse
// transforms take the other pencil as 0. Pencils that are their own mirror
// carry half the weight at every k3. At N = 16: 130 of 256 pencils, 2.34 instead
// of 3.55 million pairs per cell (and 0.08 million entries of weight 0, of blocks
// that only one of the two sums holds).
// ----------------------------------------------------------------------------
constexpr int mode_mirror(int i, int N) { return i == 0 ? 0 : N - i; }
// n = k - m + N/2 on the grid, and its index mod N
constexpr bool pair_on_grid(int k, int m, int N) { return k - m + N / 2 >= 0 && k - m + N / 2 < N; }
constexpr int pair_partner(int k, int m, int N) { return (k - m + N / 2 + N) % N; }
constexpr bool pair_on_grid_mirrored(int k, int m, int N) {
    return pair_on_grid(mode_mirror(k, N), mode_mirror(m, N), N);
}
// (k3, m3) has a weight in some block of a stored pencil
constexpr bool pair_kept(int k, int m, int N) { return pair_on_grid(k, m, N) || pair_on_grid_mirrored(k, m, N); }
// The order in which a block visits its pairs (k3, m3) of a tile of T outputs.
// T = N: m3 = i for i = 0 .. N - 1. T < N: i = 0 .. N stands for m' = -N/2 .. N/2
// (m3 = i mod N), so that for every k3 the partners are visited in one
// descending run: index 0 comes first for the pairs on the grid (m' = -N/2) and
// last for those that only the mirrored sum holds (m' = +N/2).
constexpr int pair_visits(int N, int T) { return T < N ? N + 1 : N; }
constexpr bool pair_visit(int k, int i, int N, int T) {
    if (T == N) return pair_kept(k, i, N);
    return i == 0 ? pair_on_grid(k, 0, N) : i == N ? pair_kept(k, 0, N) && !pair_on_grid(k, 0, N) : pair_kept(k, i, N);
}
// the pencil of the mirror pair that the convolutions evaluate
constexpr bool pencil_stored(int k1, int k2, int N) {
    return k1 > N / 2 || ((k1 == 0 || k1 == N / 2) && (k2 == 0 || k2 >= N / 2));
}
constexpr bool pencil_self_mirrored(int k1, int k2, int N) {
    return (k1 == 0 || k1 == N / 2) && (k2 == 0 || k2 == N / 2);
}

// Host to device, complete on return: cudaMemcpy from pageable memory may return while
// its last part is still on the way, in the legacy stream, for which callers'
// (non-blocking) streams do not wait.
inline cudaError_t upload(void *dst, const void *src, size_t bytes) {
    const cudaError_t e = cudaMemcpy(dst, src, bytes, cudaMemcpyHostToDevice);
    return e == cudaSuccess ? cudaStreamSynchronize(cudaStreamLegacy) : e;
}

int first_kind_for_N(int N);  // -1 if unsupported
int tiles_for_N(int N);
constexpr int kMaxTiles = 3;

// One warp-sized unit of convolution work: cell group g (32 lanes), pencil
// (k1, k2), k3 tile. Sorted by cost (descending) before upload.
struct ConvItem {
    uint64_t fofs;       // float2 offset of the group's fhat ([m][lane]) == qhat offset
    uint64_t wofs;       // float offset of the first weight block
    uint32_t desc_off;   // first (m1, m2) descriptor of the pencil
    uint32_t nblocks;    // kept (m1, m2) blocks of the pencil
    uint16_t k1, k2;
    uint16_t kind;       // ConvKind id
    uint16_t table;      // weight table index
};
static_assert(sizeof(ConvItem) == 32, "ConvItem layout");

// One zeta point of the FP64 convolution: for each of its pencil's blocks
// (desc_off ..) the m_count values of m3 from m_first on, mod N, with one
// weight each from woff on.
struct Zeta64 {
    uint64_t woff;
    uint32_t desc_off;
    uint16_t nblocks, k1, k2, k3, m_first, m_count;
};
static_assert(sizeof(Zeta64) == 24, "Zeta64 layout");

// Per-grid weight table and constants.
struct Table {
    int N = 0;
    double L = 0, lam = 0;
    double beta = 1.0;  // restitution parameter of the collision rule (1: elastic)
    int ntiles = 0;
    int kind0 = 0;
    double dv = 0, dz = 0;
    // FP32 half-spectrum pair weights (times dz^3): [tile][k1][k2][block][cpad]
    std::vector<uint64_t> wofs;          // per (tile, k1, k2)
    std::vector<uint32_t> desc_off;      // per (k1, k2)
    std::vector<uint32_t> nblocks;       // per (k1, k2)
    int cpad[kMaxTiles] = {0, 0, 0};
    size_t n_w32 = 0, n_desc = 0;
    float *d_w32 = nullptr;
    uint32_t *d_desc = nullptr;          // m1 | (m2 << 16)
    // FP64 pair weights (times dz^3), zeta-major, and the zeta points of the stored
    // pencils, costliest first; built lazily.
    double *d_w64 = nullptr;
    Zeta64 *d_zeta64 = nullptr;
    int n_zeta64 = 0;
    size_t n_w64 = 0;
    // On-the-fly weights (beta = 1): I and J in FP32 times sqrt(2/pi) dz^3, and
    // per k3 tile and block entry (kernel order) the third components of the
    // weight invariants as four 16-bit fields (estride entries per tile)
    float *d_I32 = nullptr, *d_J32 = nullptr;
    uint16_t *d_etab = nullptr;
    int estride = 0;
    // Work items of one 32-cell group (fofs 0, table 0), every k3 tile and
    // pencil with kept blocks, costliest first: the set-up-time template from
    // which bte_collide_noalloc expands its work list on the device.
    ConvItem *d_tmpl = nullptr;
    int n_tmpl = 0;
    // The convolution with pairs in lanes (N <= 32): per tile the entries of a block
    // (m3 | n3 << 8, conv32_cells_entries(N) a tile), and the entry of each (visit,
    // output j), [tile][pair_visits][T], -1 if none
    uint16_t *d_ent = nullptr;
    int16_t *d_rk = nullptr;
    // Projection: (C C^T)^{-1}, row-major 5x5 (C without the dv^3 factor folded in)
    double ainv[25];
    // Host FP64 radial tables on integer invariants (kept for the lazy FP64 table)
    std::vector<double> I, J;            // I[p * nq + q], J[s]
    int np = 0, nq = 0, ns = 0;
    // the convolution kinds of this table's k3 tiles (bit kind0 + tile)
    unsigned kinds_mask() const {
        unsigned m = 0;
        for (int i = 0; i < ntiles; ++i) m |= 1u << (kind0 + i);
        return m;
    }
    std::vector<uint32_t> desc_host;     // block descriptors (host copy, for the lazy FP32 table)
    double ghat(int k1, int k2, int k3, int m1, int m2, int m3) const;  // FP64, no dz^3
    // Gv(k, m) + Gv(k*, m*), halved on self-mirrored pencils (half-spectrum convolution); no dz^3
    double half_weight(int k1, int k2, int k3, int m1, int m2, int m3) const;
    double gain_inelastic(radial::Dd s, radial::Dd t) const;            // I(hz s, hz t) off the lattice
};

struct GraphKey {
    int64_t ninst;
    int table, mode, transport;
    double dt, eps;
    const void *f;
    void *stream;
    bool operator<(const GraphKey &o) const;
};

// How a convolution ran: pairs in lanes, items whole, in halves, in more parts.
enum ConvPath { CONV_NONE = 0, CONV_FEW, CONV_WHOLE, CONV_HALVES, CONV_PARTS };

// One configuration of the FP32 path (convolution variant and launch shape,
// compensated-merge interval, CTAs per cell of the fused transforms).
struct ConvCfg {
    int impl = 4, warps = 4, stages = 0, merge = 16, split = 0;
    int csplit = 1;   // variant 4: run the batch's split item list, or the few-cells kernel
    double ms = 0.0;  // measured time of one collide of the batch when tuned
};

struct Batch;  // device-side description of one instance layout (defined in api.cu)
struct Mlp;    // learned surrogate (mlp.h)
struct IndicatorTable;

enum ProfKernel { PK_CONV32 = 0, PK_CONV64 = 1, PK_COLLIDE = 2, PK_FORWARD = 3, PK_INVERSE = 4, PK_TRANSPORT = 5 };
struct ProfEntry {
    int kernel;
    cudaEvent_t a, b;
};
struct WallTable {
    double *d = nullptr;       // device M_w per velocity
    std::vector<double> host;  // same values on the host
};
struct GraphRec {
    cudaGraphExec_t exec = nullptr;
    uint64_t last_use = 0;        // context tick of the latest replay (least recently used is evicted first)
    std::vector<ProfEntry> prof;  // events baked into the graph
    int64_t launches = 0;         // kernels per replay
    std::vector<bte_instance> inst;  // the instance list the graph was captured for (the key holds a hash)
    std::vector<double> trdesc;      // the slab it was captured for (walls, temperatures, widths; hashed in the key)
};

}  // namespace bte

struct bte_ctx {
    int device = 0;
    int num_sms = 0;
    std::string err;
    std::vector<bte::Table *> tables;
    int *d_status = nullptr;
    unsigned *d_counter = nullptr;
    // grow-only scratch
    static constexpr int kScratch = 16;
    void *scratch[kScratch] = {nullptr};
    size_t scratch_bytes[kScratch] = {0};
    std::map<std::string, bte::Batch *> batches;  // per instance layout, at most batch_cache_max
    int batch_cache_max = 64;
    uint64_t batch_tick = 0;
    std::map<bte::GraphKey, bte::GraphRec> graphs;  // at most graph_cache_max
    int graph_cache_max = 32;
    uint64_t graph_tick = 0;
    // Per stream the context has enqueued work on: an event recorded after that
    // work. Waiting on these (instead of the whole device) lets the context free
    // or rebuild what its own kernels may still read.
    std::map<cudaStream_t, cudaEvent_t> fence;
    // profiling / launch accounting
    bool prof = false;
    int prof_mask = 63;        // bit k: record events around ProfKernel k
    bool capturing = false;
    std::vector<bte::ProfEntry> pending;       // direct launches and replays not yet read
    std::vector<bte::ProfEntry> cap_prof;      // entries of the graph being captured
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev_free;
    int64_t launches = 0, cap_launches = 0;
    double *d_wall = nullptr;  // unused scratch word pair
    std::map<std::tuple<int, double, double>, bte::WallTable> walls;  // (N, dv, T_w) -> M_w
    // transport coefficients of slabs with cells of unequal width, per width list:
    // device array [alpha (nx + 2) | gamma (nx + 2) | 1/dx (nx)]
    std::map<std::vector<double>, double *> grids;
    int conv_warps = 4;        // warps per CTA of the convolution kernel
    int conv_stages = 0;       // pipeline depth (blocks in flight per warp); 0 = automatic
    int conv_merge = 16;       // blocks per compensated (TwoSum) merge
    int conv_impl = 4;         // 0 warp items, 1 CTA-cooperative, 2 cooperative + packed f32x2,
                               // 3 as 2 at 2 CTAs/SM, 4 as 2 with the compensated sums in shared memory
    int dft_split = 0;         // CTAs per cell of the fused transforms (N <= 16), 0: by the number of cells
    int conv_split = 1;        // variant 4: split items, few-cells kernel
    int dft_fuse_stages = 1;   // FP32 Heun step: stage 1's inverse transform also forms stage 2's forward
    int debug_conv_stall = 0;  // testing only: make the convolution's waits run out
    int debug_conv_parts = 0;  // testing only: blocks a warp at which every item is cut (0: by the plan)
    int conv_path = 0;         // how the last FP32 collide's convolution ran (ConvPath)
    std::string gpu_name;      // device name (key of saved tuning caches)
    std::map<std::string, bte::ConvCfg> tuned;  // autotuned configuration per batch shape
    bte::Mlp *mlp = nullptr;   // learned surrogate (bte_mlp_init)
    bte::IndicatorTable *ind = nullptr;  // sampled modes of the fallback indicator
    int learned_tol_ppm = 10000;         // fallback when the indicator exceeds 1e-6 * this
    int learned_samples = 64;
    // learned-mode statistics, accumulated on the device by every call and
    // step: cells seen, cells recomputed, the largest indicator (FP32 bits)
    unsigned long long *d_lstats = nullptr;
};

namespace bte {

// conv32_cells.cu: entries per k3 tile, padded to whole warps (0: N unsupported)
int conv32_cells_entries(int N);

// tables.cpp
int build_table(Table &t, std::string &err);
int build_table_fp32(Table &t, std::string &err);  // the stored FP32 weights (built by build_table for N <= 32)
int build_table_fp64(Table &t, std::string &err);
void free_table(Table &t);

}  // namespace bte
