// Shift-free FMM with charges at Lagrange nodes (arXiv 2009.00767, Appendix STEP1-STEP5, Eq. 1-2;
// the summation scheme of Sec. 2.2.1), 2D log and 3D Coulomb kernels, on sm_103a.
//
// Data layout in device memory:
//   * the charges sorted by finest cell in Morton order, so that the charges of any cell at any
//     level are one contiguous range: FP32 forms keep (x, y, z, q) as a float4 "hi" and the
//     residues x - hi and the input index as a float4 "lo"; FP64 forms keep (x, y, z, q) as a Pos64;
//   * per level k, the cells in Morton order with d = 4^D node values each (node index
//     i + 4j + 16k): node charges Q_k and node potentials psi_k (node forms; psi_k in FP64), or
//     the vectors v_k and dual vectors u_k (literal form);
//   * node forms: per level a 7^D table of d x d node-to-node matrices, indexed by the offset
//     between source and target cell, laid out [offset][source node i][target node j];
//   * literal form: per level the interaction-list pairs in CSR order by target cell, and one
//     d x d FP64 matrix B = M_{m_i}^T M_b M_m per pair (row a: the root-node coordinate of the
//     source's vector, column l: that of the target's).
//
// Work items of the particle kernels are chunks of consecutive sorted charges within one finest
// cell (up to kChunk, or the near field's kWarpChunk), so crowded cells are split over warps and any
// distribution keeps every SM busy.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <vector>

#include "fmm.h"
#include "fmm_lagrange.h"
#include "p2p64.cuh"
#include "p2p_block.cuh"

namespace {

constexpr int kChunk = 128;      // charges per work item
constexpr int kWarpChunk = 24;     // targets per near-field warp work item, FP32
constexpr int kPairSlots = 64;     // the near field's pair counter is spread over this many words
constexpr int kWarpChunk64 = 32;   // and FP64
constexpr int kMaxLevels = 8;
constexpr double kLn2 = 0.69314718055994530942;

__host__ __device__ constexpr int nodes_of(int D) { return D == 2 ? 16 : 64; }
__host__ __device__ constexpr int offsets_of(int D) { return D == 2 ? 49 : 343; }   // 7^D table

// Eq. 1 on the nodes {-2, -1, 1, 2}: f_i(x) = prod_{j != i} (x - a_j) / (a_i - a_j), written as
// products of the two node pairs' quadratics.
template <typename T>
__host__ __device__ __forceinline__ void lag_basis(T x, T* w) {
    const T a = (x + T(1)) * (x - T(1));   // (x + 1)(x - 1)
    const T b = (x + T(2)) * (x - T(2));   // (x + 2)(x - 2)
    w[0] = a * (x - T(2)) * T(-1.0 / 12.0);
    w[1] = b * (x - T(1)) * T(1.0 / 6.0);
    w[2] = b * (x + T(1)) * T(-1.0 / 6.0);
    w[3] = a * (x + T(2)) * T(1.0 / 12.0);
}

// Morton order of coordinates below 2^10: bit b of axis a is bit b D + a, by shifts and masks (fmm_spread2 in 2D).
__host__ __device__ __forceinline__ uint32_t spread_bits(int D, uint32_t v) {
    if (D == 2) return fmm_spread2(v);
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    return (v | (v << 2)) & 0x09249249u;
}
__host__ __device__ __forceinline__ uint32_t compact_bits(int D, uint32_t v) {
    if (D == 2) return fmm_compact2(v);
    v &= 0x09249249u;
    v = (v | (v >> 2)) & 0x030c30c3u;
    v = (v | (v >> 4)) & 0x0300f00fu;
    v = (v | (v >> 8)) & 0x030000ffu;
    return (v | (v >> 16)) & 0x000003ffu;
}
__host__ __device__ __forceinline__ uint32_t morton_enc(int D, const int* c) {
    uint32_t m = spread_bits(D, (uint32_t)c[0]) | spread_bits(D, (uint32_t)c[1]) << 1;
    if (D == 3) m |= spread_bits(D, (uint32_t)c[2]) << 2;
    return m;
}
__host__ __device__ __forceinline__ void morton_dec(int D, uint32_t m, int* c) {
    c[0] = (int)compact_bits(D, m);
    c[1] = (int)compact_bits(D, m >> 1);
    c[2] = D == 3 ? (int)compact_bits(D, m >> 2) : 0;
}

// The pairwise interaction of a unit charge seen at distance vector r (0 for r = 0).
__host__ __device__ inline double kernel64(int D, double r2) {
    if (r2 == 0.0) return 0.0;
    return D == 2 ? 0.5 * log(r2) : 1.0 / sqrt(r2);
}

constexpr unsigned kFlagOutOfBox = 1u, kFlagNonFinite = 2u;

// The MUFU reciprocal square root, which takes a subnormal input for zero: no r^2 that counts is subnormal (the
// own cell's mask drops those, a forward pair has its tiny), so rsqrtf's handling of them is not needed.
__device__ __forceinline__ float mufu_rsqrt(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
}  // namespace

// A sorted charge of the FP64 forms: position and charge, one 32-byte load.
struct __align__(32) Pos64 {
    double x, y, z, w;
};

// Sums over finest cells: charges, particle-kernel chunks, near-field chunks.
struct Scan3 {
    int n, c, w;
};

struct fmm_lag_plan_s {
    int dev = 0, dim = 2, levels = 0, form = 0, d = 16;
    double box = 5.0;
    int64_t n_max = 0, nleaf = 1, last_n = 0;
    cudaStream_t st = nullptr, st2 = nullptr;
    cudaEvent_t ev[9] = {};   // 0 start, 1 far field start, 2 up done, 3 down done, 4 end, 5/6 p2p, 7 sorted
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    uint32_t* key = nullptr;       // [n_max] finest Morton key, input order
    uint32_t* rank = nullptr;      // [n_max] rank within the cell
    uint32_t* skey = nullptr;      // [n_max] key, sorted order
    int* count = nullptr;          // [nleaf]
    int* start = nullptr;          // [nleaf + 1]
    int* chunk_start = nullptr;    // [nleaf + 1]
    int* wchunk_start = nullptr;   // [nleaf + 1] near-field warp chunks
    int* wchunk_cell = nullptr;    // and the cell of each
    int* order = nullptr;          // [n_max] sorted -> input index, FP64 forms (FP32: lo.w)
    Scan3* scan = nullptr;  // per tile of the scan
    float4* hi = nullptr;          // FP32 forms
    float4* lo = nullptr;
    Pos64* p64 = nullptr;        // FP64 forms
    double* nearf = nullptr;       // [n_max] near field, sorted order
    unsigned* status = nullptr;
    unsigned* h_status = nullptr;  // pinned
    unsigned long long* pairs = nullptr;   // near-field pair counter
    int* next_item = nullptr;              // near-field work counter
    void* node[kMaxLevels + 1] = {};       // Q_k (node) or v_k (literal), d values per cell
    void* pot[kMaxLevels + 1] = {};        // psi_k (node) or u_k (literal), one allocation at pot[2]
    size_t pot_bytes = 0;
    double* psi0 = nullptr;                // FP32 form: the finest cells' potentials as one FP64 value a cell
    float* dpsi = nullptr;                 // and FP32 differences from it
    void* K = nullptr;                     // node forms: operators of levels 2..levels
    int* pair_start[kMaxLevels + 1] = {};  // literal: CSR by target cell
    int* pair_src[kMaxLevels + 1] = {};
    double* B[kMaxLevels + 1] = {};
    int64_t npairs[kMaxLevels + 1] = {};
    int64_t m2l_pairs = 0;
    uint64_t bytes = 0;
    int launches = 0;
    int grid_particles = 0;
    int sms = 0;
    cudaStream_t last_st = nullptr;   // the stream of the last call, for comparison only
    bool serial = false;   // every kernel in turn on the plan's stream (per-kernel timing)
    int grid_p2p = 0;      // resident blocks of the FP64 near-field kernel, all SMs
    double2* logtab = nullptr;   // 2D FP64 forms: the logarithm's table (fp64_math.cuh)
};

namespace {

// ------------------------------------------------------------------------------ binning

// Finest cell of charge i with the FP64 floor/clamp rule (finest_coord): its Morton key; plus the input checks.
template <int D>
__device__ __forceinline__ uint32_t bin_key(const double* __restrict__ pos, const double* __restrict__ q, int64_t i, int L,
                                            double box, float side_over_box, unsigned* __restrict__ status) {
    const int side = 1 << L;
    const long long bb = __double_as_longlong(box);
    int c[3] = {0, 0, 0};
    unsigned bad = finite_bits(q[i]) ? 0u : kFlagNonFinite;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const double x = pos[i * D + a];
        if (!finite_bits(x)) {
            bad |= kFlagNonFinite;
        } else {
            if (!in_box_bits(x, bb)) bad |= kFlagOutOfBox;
            c[a] = finest_coord(x, (double)side, side_over_box, box, side);
        }
    }
    if (bad) atomicOr(status, bad);
    return morton_enc(D, c);
}

// Every charge's key and its rank within the cell (atomic).
template <int D>
__global__ void k_bin(const double* __restrict__ pos, const double* __restrict__ q, int64_t n, int L,
                      double box, float side_over_box, uint32_t* __restrict__ key, uint32_t* __restrict__ rank,
                      int* __restrict__ count, unsigned* __restrict__ status) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t k = bin_key<D>(pos, q, i, L, box, side_over_box, status);
    key[i] = k;
    rank[i] = (uint32_t)atomicAdd(count + k, 1);
}

// The same with few cells for the charges: a block ranks its share in shared memory and takes each cell's
// places at once.
// What bounds k_bin there: 512 populations are 16 cache lines, whose atomics queue up.
constexpr int kBinFewCells = 4096, kBinFewThreads = 1024;
// With fewer charges a block meets most cells once and saves nothing.  The whole sort, k_bin against k_bin_few:
// 512 cells (3D) 20,000 charges 31.4 and 32.2 us, 40,000 36.2 and 32.5, 160,000 52.9 and 38.8; 4,096 cells
// 60,000 35.7 and 37.3, 262,144 44.7 and 41.3, 2^20 80.3 and 62.0; 64 cells 5,000 29.3 and 30.4, 9,728 31.0 and
// 30.1.
inline bool bin_few(int64_t nleaf, int64_t n) { return nleaf <= kBinFewCells && n >= 64 * nleaf && n >= 8192; }

template <int D>
__global__ void __launch_bounds__(kBinFewThreads)
k_bin_few(const double* __restrict__ pos, const double* __restrict__ q, int64_t n, int L, double box, float side_over_box,
          uint32_t* __restrict__ key, uint32_t* __restrict__ rank, int* __restrict__ count, int nleaf,
          unsigned* __restrict__ status) {
    __shared__ int cells[kBinFewCells];
    for (int c = threadIdx.x; c < nleaf; c += kBinFewThreads) cells[c] = 0;
    __syncthreads();
    const int64_t share = (n + gridDim.x - 1) / gridDim.x, i1 = min(n, (blockIdx.x + 1) * share);
    const int64_t i0 = blockIdx.x * share + threadIdx.x;
    for (int64_t i = i0; i < i1; i += kBinFewThreads) {
        const uint32_t k = bin_key<D>(pos, q, i, L, box, side_over_box, status);
        key[i] = k;
        rank[i] = (uint32_t)atomicAdd(cells + k, 1);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < nleaf; c += kBinFewThreads)
        if (cells[c]) cells[c] = atomicAdd(count + c, cells[c]);
    __syncthreads();
    for (int64_t i = i0; i < i1; i += kBinFewThreads) rank[i] += (uint32_t)cells[key[i]];
}

// Exclusive scans of the populations and of the chunk counts (chunks of kChunk, and of wchunk for the near
// field's warps, whose cells are listed) over the finest cells, in tiles of kScanTile cells: each tile's sums, then each tile's scan
// behind the sums of the tiles before it (at most 65,536 cells, 128 tiles).
constexpr int kScanTile = 512;

__device__ __forceinline__ Scan3 scan_add(Scan3 a, Scan3 b) { return Scan3{a.n + b.n, a.c + b.c, a.w + b.w}; }
__device__ __forceinline__ Scan3 scan_cell(const int* __restrict__ count, int b, int nleaf, int wchunk) {
    const int n = b < nleaf ? count[b] : 0;
    return Scan3{n, (n + kChunk - 1) / kChunk, (n + wchunk - 1) / wchunk};
}
// exclusive scan of one value a thread over the block; *total receives the block's sum
__device__ __forceinline__ Scan3 scan_block(Scan3 v, Scan3* total) {
    __shared__ Scan3 warps[kScanTile / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Scan3 inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const Scan3 y = Scan3{__shfl_up_sync(0xffffffffu, inc.n, o), __shfl_up_sync(0xffffffffu, inc.c, o),
                              __shfl_up_sync(0xffffffffu, inc.w, o)};
        if (lane >= o) inc = scan_add(inc, y);
    }
    __syncthreads();
    if (lane == 31) warps[warp] = inc;
    __syncthreads();
    Scan3 before = {0, 0, 0}, all = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < kScanTile / 32; ++i) {
        if (i < warp) before = scan_add(before, warps[i]);
        all = scan_add(all, warps[i]);
    }
    *total = all;
    return Scan3{before.n + inc.n - v.n, before.c + inc.c - v.c, before.w + inc.w - v.w};
}

__global__ void __launch_bounds__(kScanTile) k_scan_sums(const int* __restrict__ count, int nleaf, int wchunk,
                                                         Scan3* __restrict__ sums) {
    Scan3 total;
    scan_block(scan_cell(count, blockIdx.x * kScanTile + threadIdx.x, nleaf, wchunk), &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanTile) k_scan(const int* __restrict__ count, int nleaf, int wchunk,
                                                    const Scan3* __restrict__ sums, int* __restrict__ start,
                                                    int* __restrict__ chunk_start, int* __restrict__ wchunk_start,
                                                    int* __restrict__ wchunk_cell) {
    Scan3 before = {0, 0, 0}, total;
    for (int t = threadIdx.x; t < (int)blockIdx.x; t += kScanTile) before = scan_add(before, sums[t]);
    scan_block(before, &before);
    const int b = blockIdx.x * kScanTile + threadIdx.x;
    const Scan3 v = scan_add(before, scan_block(scan_cell(count, b, nleaf, wchunk), &total));
    if (b < nleaf) {
        start[b] = v.n;
        chunk_start[b] = v.c;
        wchunk_start[b] = v.w;
        for (int i = (count[b] + wchunk - 1) / wchunk; i-- > 0;) wchunk_cell[v.w + i] = b;
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        start[nleaf] = before.n + total.n;
        chunk_start[nleaf] = before.c + total.c;
        wchunk_start[nleaf] = before.w + total.w;
    }
}

// Charges into sorted order.  FP32 forms: the input index rides in lo.w, so that a charge is two scattered
// 16-byte writes; the sorted keys are written by k_p2m, whose warps know their cell.
// 2^20 charges in 2D: the call 406 -> 385 us against four scattered writes, input index and key among them.
template <int D, bool k64>
__global__ void k_scatter(const double* __restrict__ pos, const double* __restrict__ q, int64_t n,
                          const uint32_t* __restrict__ key, const uint32_t* __restrict__ rank,
                          const int* __restrict__ start, int* __restrict__ order, float4* __restrict__ hi,
                          float4* __restrict__ lo, Pos64* __restrict__ p64) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t s = (int64_t)start[key[i]] + rank[i];
    const double x = pos[i * D], y = pos[i * D + 1], z = D == 3 ? pos[i * D + 2] : 0.0;
    if constexpr (k64) {
        order[s] = (int)i;
        p64[s] = Pos64{x, y, z, q[i]};
    } else {
        const float hx = (float)x, hy = (float)y, hz = (float)z;
        hi[s] = make_float4(hx, hy, hz, (float)q[i]);
        lo[s] = make_float4((float)(x - (double)hx), (float)(y - (double)hy), (float)(z - (double)hz), __int_as_float((int)i));
    }
}

// The finest cell of chunk work item w: the last b with chunk_start[b] <= w.
__device__ __forceinline__ int chunk_leaf(const int* __restrict__ chunk_start, int nleaf, int w) {
    int lo = 0, hi = nleaf;   // chunk_start[lo] <= w < chunk_start[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(chunk_start + mid) <= w) lo = mid;
        else hi = mid;
    }
    return lo;
}

// ------------------------------------------------------------------------------ near field

// Sec. 2.1 E-2 in FP32, each pair of the own and adjacent cells once for both sides.  A work item of a warp
// is a chunk of up to kWarpChunk targets of a finest cell A and a group of A's "forward" cells: A itself
// and the neighbours whose offset is positive in (z, y, x) order (13 in 3D, 4 in 2D), so that every
// unordered pair of adjacent cells is met once.  Lanes over sources, registers over targets: the group's
// later sources (A's charges after the chunk, then the forward cells') are walked 64 at a time, two a
// lane; the targets' coordinates and charges are shared-memory broadcasts, and two targets' arithmetic
// runs in packed FP32x2.  A pair's 1/r (or log r) feeds a register partial of the target and the sum of the
// source, which stays in its lane and goes out with one FP64 atomic.  The chunk
// against itself is one-sided.  Differences come from two-word coordinates, (hi_t - hi_s) + (lo_t - lo_s), so a
// close pair's distance keeps about 48 bits.  Pairs inside A below r^2 = 2^-126, FP32's smallest normal number,
// count as coincident and give 0.  Two charges either side of a cell's edge may share one two-word point: the
// pairs with the forward cells add tiny = (2^-50 box)^2 to r^2, which moves no pair that the words tell apart
// by more than their own rounding (1.4% of 200,000 charges' call in 3D; a maximum with tiny instead 5%).
// After kP2PRun chunks the lanes' partials of a target are summed across the warp (warp_reduce_scatter) and
// added in FP64.
// What bounds it: the FMA pipe, 14 packed instructions (two cycles each) for two targets in 3D, 9 of them
// the two-word differences.  A lane holds two sources, so that the targets' shared-memory broadcasts (8
// wavefronts for two targets) serve four pairs.  200,000 charges in 3D, levels 3: 468 us against 739 us for
// 64 targets over the lanes and a butterfly over the lanes per source tile (31 shuffles, 62 selects) for the
// source's side, and 486 us with one source a lane; 2^20 in 2D, levels 7: 238, 368 and 256 us, and 200 with
// the two changes below.
// In 2D, with a few chunks an item, the warps of an SM are at many places of the unrolled code and wait for
// instructions, so the code is kept small: the chunk itself and a last half chunk share a body, and whole
// chunks are masked in every cell (the call 384 -> 366 us; in 3D, where one body runs for long, the call would
// grow by 0.8% and 6%).
constexpr int kP2PWarps = 4;     // warps per block, each on its own work items
template <int D>
__host__ __device__ constexpr int fwd_group() { return D == 3 ? 4 : 5; }   // forward cells per work item

// Forward cell f of a cell: f = 0 the cell itself, then the offsets o > 0 in (z, y, x) order.
template <int D>
__device__ __forceinline__ void fwd_offset(int f, int* o) {
    o[0] = o[1] = o[2] = 0;
    if (f == 0) return;
    const int e = f - 1;
    if constexpr (D == 3) {
        if (e < 9) { o[0] = e % 3 - 1; o[1] = e / 3 - 1; o[2] = 1; }
        else if (e < 12) { o[0] = e - 10; o[1] = 1; }
        else { o[0] = 1; }
    } else {
        if (e < 3) { o[0] = e - 1; o[1] = 1; }
        else { o[0] = 1; }
    }
}

// The later sources of a chunk [t0, t0 + T) of cell b and group g: slot s of range i (end[i - 1] <= s <
// end[i]) is the sorted charge s + first[i].  Returns the ordered pairs the item covers, both directions
// of the later pairs and, with the own cell, the chunk's own T^2.
template <int D>
__device__ __forceinline__ unsigned long long later_sources(const int* __restrict__ start, int b, int b1, int t0, int T,
                                                            int g, int side, uint32_t (&first)[5], uint32_t (&end)[5]) {
    constexpr int F = D == 3 ? 14 : 5, FG = fwd_group<D>();
    int c[3];
    morton_dec(D, (uint32_t)b, c);
    uint32_t slots = 0;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int f = g * FG + i;
        uint32_t from = 0, count = 0;
        if (i < FG && f < F) {
            int o[3];
            fwd_offset<D>(f, o);
            const int nc[3] = {c[0] + o[0], c[1] + o[1], c[2] + o[2]};
            bool in = nc[0] >= 0 && nc[0] < side && nc[1] >= 0 && nc[1] < side;
            if (D == 3) in = in && nc[2] >= 0 && nc[2] < side;
            if (f == 0) {
                from = (uint32_t)(t0 + T);
                count = (uint32_t)(b1 - t0 - T);
            } else if (in) {
                const uint32_t nb = morton_enc(D, nc);
                from = (uint32_t)start[nb];
                count = (uint32_t)start[nb + 1] - from;
            }
        }
        first[i] = from - slots;
        slots += count;
        end[i] = slots;
    }
    return 2ull * slots * (unsigned long long)T + (g == 0 ? (unsigned long long)T * (unsigned long long)T : 0ull);
}

// FP32 to FP64 by integer operations, off the narrow FP64 pipe (subnormals flush to zero; infinities and
// NaN stay what they are)
__device__ __forceinline__ double f2d(float f) {
    const uint32_t u = __float_as_uint(f), e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
    const uint32_t x = e == 0xffu ? 0x7ffu : e + 896u;
    return e == 0u ? 0.0 : __hiloint2double((int)((u & 0x80000000u) | (x << 20) | (m >> 3)), (int)((m & 7u) << 29));
}

// a chunk's targets in pairs: {x, x, y, y}, {z, z, q, q} (high words), {x, x, y, y} and {z, z} (low words)
template <int D>
struct LagTargets {
    float4 xy[kWarpChunk / 2], zq[kWarpChunk / 2], lxy[kWarpChunk / 2];
    float2 lz[D == 3 ? kWarpChunk / 2 : 1];
};

// A lane's source, its coordinates negated and duplicated: {-x, -x} (high and low words), {q, q}, {tiny, tiny}.
template <int D>
struct LagSource {
    float2 x[D], l[D], q, tiny;
    __device__ LagSource(float4 h, float4 lo, float2 t) {
        x[0] = make_float2(-h.x, -h.x);
        x[1] = make_float2(-h.y, -h.y);
        l[0] = make_float2(-lo.x, -lo.x);
        l[1] = make_float2(-lo.y, -lo.y);
        if constexpr (D == 3) {
            x[2] = make_float2(-h.z, -h.z);
            l[2] = make_float2(-lo.z, -lo.z);
        }
        q = make_float2(h.w, h.w);
        tiny = t;
    }
};

// 1 / r (3D) or log2 r^2 (2D) of the lane's source and target pair t; kMask: 0 for a coincident pair (tiny = 0)
template <int D, bool kMask>
__device__ __forceinline__ float2 p2p_lag_pair(const LagSource<D>& s, float4 A, float4 B, float4 C, float2 lz) {
    const float2 dx = __fadd2_rn(__fadd2_rn(make_float2(A.x, A.y), s.x[0]), __fadd2_rn(make_float2(C.x, C.y), s.l[0]));
    const float2 dy = __fadd2_rn(__fadd2_rn(make_float2(A.z, A.w), s.x[1]), __fadd2_rn(make_float2(C.z, C.w), s.l[1]));
    float2 r2 = __ffma2_rn(dy, dy, __ffma2_rn(dx, dx, s.tiny));
    if constexpr (D == 3) {
        const float2 dz = __fadd2_rn(__fadd2_rn(make_float2(B.x, B.y), s.x[2]), __fadd2_rn(lz, s.l[2]));
        r2 = __ffma2_rn(dz, dz, r2);
    }
    float2 k = D == 3 ? make_float2(mufu_rsqrt(r2.x), mufu_rsqrt(r2.y)) : make_float2(mufu_lg2(r2.x), mufu_lg2(r2.y));
    if constexpr (kMask) {
        k.x = r2.x >= 0x1p-126f ? k.x : 0.f;
        k.y = r2.y >= 0x1p-126f ? k.y : 0.f;
    }
    return k;
}

// the lane's kS sources (1 or 2) against the chunk's 2 NP targets; returns the sources' sums
template <int D, bool kMask, int NP, int kS>
__device__ __forceinline__ float2 p2p_lag_chunk(float2 (&part)[NP], const LagTargets<D>& tg, float4 ha, float4 la,
                                                float4 hb, float4 lb, float2 ta, float2 tb) {
    const LagSource<D> a(ha, la, ta), b(hb, lb, tb);
    float2 sa = make_float2(0.f, 0.f), sb = make_float2(0.f, 0.f);
#pragma unroll
    for (int t = 0; t < NP; ++t) {
        const float4 A = tg.xy[t], B = tg.zq[t], C = tg.lxy[t];
        const float2 lz = D == 3 ? tg.lz[t] : make_float2(0.f, 0.f), q = make_float2(B.z, B.w);
        const float2 ka = p2p_lag_pair<D, kMask>(a, A, B, C, lz);
        part[t] = __ffma2_rn(a.q, ka, part[t]);
        sa = __ffma2_rn(q, ka, sa);
        if constexpr (kS == 2) {
            const float2 kb = p2p_lag_pair<D, kMask>(b, A, B, C, lz);
            part[t] = __ffma2_rn(b.q, kb, part[t]);
            sb = __ffma2_rn(q, kb, sb);
        }
    }
    return make_float2(sa.x + sa.y, sb.x + sb.y);
}

// one work item: the sum of target `lane` (units of 1 / r or log2 r^2), the later sources' added to nearf
template <int D, int NP>
__device__ __forceinline__ double p2p_lag_item(const float4* __restrict__ hi, const float4* __restrict__ lo, int t0,
                                               int T, bool self, const uint32_t (&first)[5], const uint32_t (&end)[5],
                                               uint32_t n_own, const LagTargets<D>& tg, float far, float2 tiny,
                                               int lane, double* __restrict__ nearf) {
    constexpr int W = NP <= 2 ? 4 : (NP <= 4 ? 8 : (NP <= 8 ? 16 : 32));
    const float4 far4 = make_float4(far, far, far, 0.f), zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const float2 none = make_float2(0.f, 0.f);
    float2 part[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) part[i] = make_float2(0.f, 0.f);
    double acc = 0.0;
    const uint32_t nsrc = end[4];
    auto load = [&](uint32_t slot, float4& h, float4& l, uint32_t& idx) {
        h = far4;
        l = zero4;
        idx = 0xffffffffu;
        if (slot < nsrc) {
            uint32_t f = first[0];
#pragma unroll
            for (int i = 0; i < 4; ++i) f = slot >= end[i] ? first[i + 1] : f;
            idx = slot + f;
            h = hi[idx];
            l = lo[idx];
        }
    };
    // the chunk's own charges, one-sided: in 2D the loop's first pass
    auto own = [](int c) { return D == 2 && c < 0; };
    auto load_own = [&](float4& h, float4& l) {
        h = lane < T ? hi[t0 + lane] : far4;
        l = lane < T ? lo[t0 + lane] : zero4;
    };
    if (D == 3 && self) {
        float4 h, l;
        load_own(h, l);
        p2p_lag_chunk<D, true, NP, 1>(part, tg, h, l, far4, zero4, none, none);
    }
    int run = 0;
#pragma unroll 1
    for (int c = D == 2 && self ? -1 : 0; c < (int)nsrc; c = own(c) ? 0 : c + 64) {
        float4 ha = far4, la = zero4, hb = far4, lb = zero4;
        uint32_t ia = 0xffffffffu, ib = 0xffffffffu;
        if (own(c)) {
            load_own(ha, la);
        } else {
            load((uint32_t)(c + lane), ha, la, ia);
            load((uint32_t)(c + 32 + lane), hb, lb, ib);
        }
        // a masked chunk may hold sources of the own cell and of forward ones
        const float ta = own(c) || (uint32_t)(c + lane) < n_own ? 0.f : tiny.x, tb = (uint32_t)(c + 32 + lane) < n_own ? 0.f : tiny.x;
        const float2 v = own(c) || c + 32 >= (int)nsrc   // a last half chunk
                             ? p2p_lag_chunk<D, true, NP, 1>(part, tg, ha, la, hb, lb, make_float2(ta, ta), make_float2(tb, tb))
                         : D == 2 || (uint32_t)c < n_own
                             ? p2p_lag_chunk<D, true, NP, 2>(part, tg, ha, la, hb, lb, make_float2(ta, ta), make_float2(tb, tb))
                             : p2p_lag_chunk<D, false, NP, 2>(part, tg, ha, la, hb, lb, tiny, tiny);
        if (ia != 0xffffffffu) atomicAdd(nearf + ia, f2d(v.x));
        if (ib != 0xffffffffu) atomicAdd(nearf + ib, f2d(v.y));
        run += 2;
        if (run >= kP2PRun) {
            acc += f2d(warp_reduce_scatter<W, NP>(part, lane));
#pragma unroll
            for (int i = 0; i < NP; ++i) part[i] = make_float2(0.f, 0.f);
            run = 0;
        }
    }
    return acc + f2d(warp_reduce_scatter<W, NP>(part, lane));
}

// A warp per work item (the grid is the bound on their number; wchunk_cell spares each a search for its cell,
// and Morton codes are shifts and masks: 2^20 charges in 2D 366 -> 350 us, 200,000 in 3D 590 -> 583): beside the far field, whose kernels have the
// higher priority, a resident grid would hold every SM until its last item.
template <int D>
__global__ void __launch_bounds__(kP2PWarps * 32, 5)
k_p2p32(const float4* __restrict__ hi, const float4* __restrict__ lo, const int* __restrict__ start,
        const int* __restrict__ wchunk_start, const int* __restrict__ wchunk_cell, int nleaf, int L, float box,
        float2 tiny, double* __restrict__ nearf, unsigned long long* __restrict__ pairs) {
    constexpr int F = D == 3 ? 14 : 5, FG = fwd_group<D>(), G = (F + FG - 1) / FG;
    __shared__ LagTargets<D> tgts[kP2PWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    LagTargets<D>& tg = tgts[wid];
    const int side = 1 << L;
    // empty source and target slots are zero charges outside the box, away from every charge and each other
    const float src_far = -0.25f * box, tgt_far = 1.25f * box;
    // from the constant bank where registers are short (3D); in 2D a register: 352 us for 2^20 charges against 355
    const float2 term = D == 2 ? make_float2(fmaxf((0x1p-50f * box) * (0x1p-50f * box), 0x1p-126f), 0.f) : tiny;
    const int64_t w = (int64_t)blockIdx.x * kP2PWarps + wid;
    if (w >= (int64_t)wchunk_start[nleaf] * G) return;
    const int cidx = (int)(w / G), g = (int)(w % G);
    const int b = wchunk_cell[cidx];
    const int b1 = start[b + 1], t0 = start[b] + (cidx - wchunk_start[b]) * kWarpChunk, T = min(kWarpChunk, b1 - t0);
    uint32_t first[5], end[5];
    const unsigned long long my_pairs = later_sources<D>(start, b, b1, t0, T, g, side, first, end);
    if (lane == 0 && my_pairs) atomicAdd(pairs + (w & (kPairSlots - 1)), my_pairs);
    const uint32_t n_own = g == 0 ? end[0] : 0u;
    if (lane < kWarpChunk) {
        const bool have = lane < T;
        const float4 h = have ? hi[t0 + lane] : make_float4(tgt_far, tgt_far, tgt_far, 0.f);
        const float4 l = have ? lo[t0 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
        const int o = lane & 1;
        float* A = reinterpret_cast<float*>(&tg.xy[lane >> 1]);
        float* B = reinterpret_cast<float*>(&tg.zq[lane >> 1]);
        float* C = reinterpret_cast<float*>(&tg.lxy[lane >> 1]);
        A[o] = h.x;
        A[2 + o] = h.y;
        B[o] = h.z;
        B[2 + o] = h.w;
        C[o] = l.x;
        C[2 + o] = l.y;
        if constexpr (D == 3) reinterpret_cast<float*>(&tg.lz[lane >> 1])[o] = l.z;
    }
    __syncwarp();
    double acc;
    const bool self = g == 0;
    switch ((T + 7) >> 3) {   // the chunk's target pairs, rounded up to a multiple of four
        case 1: acc = p2p_lag_item<D, 4>(hi, lo, t0, T, self, first, end, n_own, tg, src_far, term, lane, nearf); break;
        case 2: acc = p2p_lag_item<D, 8>(hi, lo, t0, T, self, first, end, n_own, tg, src_far, term, lane, nearf); break;
        default: acc = p2p_lag_item<D, 12>(hi, lo, t0, T, self, first, end, n_own, tg, src_far, term, lane, nearf); break;
    }
    if (lane < T) atomicAdd(nearf + t0 + lane, acc);
}

// The near field in FP64 (node and literal FP64 forms): p2p64.cuh's warp per chunk of up to kWarpChunk64
// targets and group of forward cells.  Resident warps take the items from a counter.
// 80,000 charges in 3D, levels 3: 3.40 ms against 19.7 ms for a kernel that took every ordered pair with FP64
// sqrt and divide (260M ordered pairs, 13 FP64 instructions for two of them: 3.2 ms at the pipe's rate).
constexpr int kP2PWarps64 = 4;

template <int D>
__global__ void __launch_bounds__(kP2PWarps64 * 32)
k_p2p64(const Pos64* __restrict__ p, const int* __restrict__ start, const int* __restrict__ wchunk_start,
        const int* __restrict__ wchunk_cell, int nleaf, int L, const double2* __restrict__ logtab, double* __restrict__ nearf, unsigned long long* __restrict__ pairs,
        int* __restrict__ next_item) {
    constexpr int F = D == 3 ? 14 : 5, FG = fwd_group<D>(), G = (F + FG - 1) / FG;
    static_assert(FG <= 5, "p2p64_block takes five ranges");
    __shared__ double2 tab[D == 2 ? kFmmLogEntries : 1];
    __shared__ P64Shared<D, false, kWarpChunk64> sh[kP2PWarps64];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if constexpr (D == 2) {
        for (int i = threadIdx.x; i < kFmmLogEntries; i += blockDim.x) tab[i] = logtab[i];
        __syncthreads();
    }
    constexpr double scale = D == 2 ? 0.5 : 1.0;   // log r = log(r^2) / 2
    const int side = 1 << L;
    const int64_t total = (int64_t)wchunk_start[nleaf] * G;
    unsigned long long my_pairs = 0;
    for (;;) {
        int64_t w = 0;
        if (lane == 0) w = atomicAdd(next_item, 1);
        w = __shfl_sync(0xffffffffu, w, 0);
        if (w >= total) break;
        const int cidx = (int)(w / G), g = (int)(w % G);
        const int b = wchunk_cell[cidx];
        const int b1 = start[b + 1], t0 = start[b] + (cidx - wchunk_start[b]) * kWarpChunk64;
        const int T = min(kWarpChunk64, b1 - t0);
        uint32_t first[5], end[5];
        my_pairs += later_sources<D>(start, b, b1, t0, T, g, side, first, end);
        auto load = [&](uint32_t i) {
            const Pos64 v = p[i];
            return P64{v.x, v.y, v.z, v.w};
        };
        p2p64_block<D, false, kWarpChunk64>(
            lane, T, g == 0, load((uint32_t)(t0 + min(lane, T - 1))), first, end, sh[wid], tab, load,
            [&](uint32_t i, const P64Acc<false>& a) { atomicAdd(nearf + i, scale * a.phi); },
            [&](const P64Acc<false>& a) { atomicAdd(nearf + t0 + lane, scale * a.phi); });
    }
    if (lane == 0 && my_pairs) atomicAdd(pairs + (blockIdx.x & (kPairSlots - 1)), my_pairs);
}

// ------------------------------------------------------------------------------ node charges

template <typename T>
__device__ __forceinline__ void atomic_add(T* a, T v) {
    atomicAdd(a, v);
}

// Sorted charges as seen from cells of side s: centre of cell c along an axis, and the local coordinate
// (position - centre) / (s/5) of charge i on axis a.  FP32: two-word positions, side and centre.
template <typename T>
struct PosReader;
template <>
struct PosReader<float> {
    const float4* hi;
    const float4* lo;
    float2 s;
    float inv;
    __device__ float2 centre(int c) const { return scatter_mul((float)c + 0.5f, s); }
    __device__ float local(int i, int a, float2 c) const {
        const float4 h = hi[i], l = lo[i];
        const float hv = a == 0 ? h.x : (a == 1 ? h.y : h.z), lv = a == 0 ? l.x : (a == 1 ? l.y : l.z);
        return ((hv - c.x) + (lv - c.y)) * inv;
    }
    __device__ float charge(int i) const { return hi[i].w; }
    __device__ int input(int i) const { return __float_as_int(lo[i].w); }
};
template <>
struct PosReader<double> {
    const Pos64* p;
    const int* order;
    double s, inv;
    __device__ double centre(int c) const { return ((double)c + 0.5) * s; }
    __device__ double local(int i, int a, double c) const {
        const Pos64 v = p[i];
        return ((a == 0 ? v.x : (a == 1 ? v.y : v.z)) - c) * inv;
    }
    __device__ double charge(int i) const { return p[i].w; }
    __device__ int input(int i) const { return order[i]; }
};

struct LevelPtrs {
    void* p[kMaxLevels + 1];
};

// Sum of v[i] over the warp's lanes, scattered: afterwards lane l holds entries [l V / 32, (l + 1) V / 32)
// (V >= 32) or, for V = 16, entry l / 2.
template <int V, typename T>
__device__ __forceinline__ void warp_reduce_nodes(T (&v)[V], int lane) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) {
        constexpr int W = V < 32 ? V : 32;
        const int live = V < 32 ? (m * V) / 32 : m * (V / W);   // entries kept at this step
        if (live == 0) {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], m);
        } else {
            const bool up = (lane & m) != 0;
#pragma unroll
            for (int i = 0; i < live; ++i) {
                const T send = up ? v[i] : v[i + live], keep = up ? v[i + live] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, m);
            }
        }
    }
}

// STEP2 summed per finest cell: sum_c q_c h(c) over the cell's charges.  Node forms: weights of the cell's
// own nodes; the coarser cells' node charges follow by k_up.  Literal U-bar-1: weights of the root box's
// nodes (root).  Also the sorted charges' keys.  A warp per chunk of up to kChunk charges of one cell, the charges over the lanes and the
// nodes' sums in registers; the lanes' sums are combined by a shuffle reduce-scatter, one atomic per node.
// 2^20 charges in 2D, levels 7: 45 us with the upward pass against 409 us for the charges' weights at each of six
// levels, staged in shared memory.
template <int D, typename T>
__global__ void __launch_bounds__(kChunk) k_p2m(PosReader<T> rd, const int* __restrict__ start,
                                                const int* __restrict__ chunk_start, int nleaf, bool root,
                                                T* __restrict__ out, uint32_t* __restrict__ skey) {
    constexpr int d = nodes_of(D);
    const int total = chunk_start[nleaf];
    const int lane = threadIdx.x & 31;
    for (int w = blockIdx.x * (kChunk / 32) + (threadIdx.x >> 5); w < total; w += gridDim.x * (kChunk / 32)) {
        const int b = chunk_leaf(chunk_start, nleaf, w);
        const int t0 = start[b] + (w - chunk_start[b]) * kChunk, t1 = min(t0 + kChunk, start[b + 1]);
        int cc[3] = {0, 0, 0};
        if (!root) morton_dec(D, (uint32_t)b, cc);
        decltype(rd.centre(0)) centre[D];
#pragma unroll
        for (int a = 0; a < D; ++a) centre[a] = rd.centre(cc[a]);
        T acc[d];
#pragma unroll
        for (int j = 0; j < d; ++j) acc[j] = T(0);
        for (int i = t0 + lane; i < t1; i += 32) {
            skey[i] = (uint32_t)b;
            T f[D][4];
#pragma unroll
            for (int a = 0; a < D; ++a) lag_basis<T>(rd.local(i, a, centre[a]), f[a]);
            const T q = rd.charge(i);
#pragma unroll
            for (int jz = 0; jz < (D == 3 ? 4 : 1); ++jz) {
                const T qz = D == 3 ? q * f[D - 1][jz] : q;
#pragma unroll
                for (int jy = 0; jy < 4; ++jy) {
                    const T qy = qz * f[1][jy];
#pragma unroll
                    for (int jx = 0; jx < 4; ++jx) acc[jx + 4 * jy + 16 * jz] += qy * f[0][jx];
                }
            }
        }
        warp_reduce_nodes<d, T>(acc, lane);
        T* o = out + (size_t)b * d;
        if constexpr (d < 32) {
            if ((lane & 1) == 0) atomic_add(o + (lane >> 1), acc[0]);
        } else {
#pragma unroll
            for (int i = 0; i < d / 32; ++i) atomic_add(o + lane * (d / 32) + i, acc[i]);
        }
    }
}

// Between levels (STEP4 for a cell and its child): per axis a cell's basis at the nodes of its two halves,
// E[4 h + i][j] = f_j(x_{h,i}) with x_{h,i} = (2.5 h - 1.25) + a_i / 2 in units where the cell's side is 5.
// A cubic is its own interpolant, so sums over charges and evaluations at charges pass through it exactly:
// a cell's node charges are E^T applied along each axis to its children's (U-bar-2), and a child's node
// potentials receive E applied to the cell's (D-bar-2).
// Both run in FP64 (they are a few percent of the particles' work), so that the FP32 form's node charges are
// rounded once per level and its node potentials, kept in FP64, not at all on the way down.
struct Halves {
    double e[8][4];
};
Halves make_halves() {
    const double a[4] = {-2.0, -1.0, 1.0, 2.0};
    Halves H;
    for (int h = 0; h < 2; ++h)
        for (int i = 0; i < 4; ++i) lag_basis<double>(2.5 * h - 1.25 + 0.5 * a[i], H.e[4 * h + i]);
    return H;
}

constexpr int kShiftWarps = 4;   // a warp per cell

// the 8^D values of a cell's children, x fastest: index (4 h + i) per axis -> (child, node)
template <int D>
__device__ __forceinline__ int child_value(int v) {
    int ch = 0, node = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const int c = (v >> (3 * a)) & 7;
        ch |= (c >> 2) << a;
        node |= (c & 3) << (2 * a);
    }
    return ch * nodes_of(D) + node;
}

template <int D, typename T>
__global__ void __launch_bounds__(kShiftWarps * 32) k_up(const T* __restrict__ child, T* __restrict__ parent, int ncell,
                                                         Halves H) {
    constexpr int N = D == 2 ? 64 : 512;
    __shared__ double buf[kShiftWarps][N + N / 2];
    __shared__ double E[8][4];
    if (threadIdx.x < 32) E[threadIdx.x >> 2][threadIdx.x & 3] = H.e[threadIdx.x >> 2][threadIdx.x & 3];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int m = blockIdx.x * kShiftWarps + warp;
    if (m >= ncell) return;
    double* in = buf[warp];
    double* out = in + N;
    const T* c = child + (size_t)m * (1 << D) * nodes_of(D);
    for (int v = lane; v < N; v += 32) in[v] = (double)c[child_value<D>(v)];
    __syncwarp();
    // along x (8 -> 4), then y, then z: the contracted axis has stride st, the ones before it 4 values
    int n = N, st = 1;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        n >>= 1;
        for (int v = lane; v < n; v += 32) {
            const int lowi = v % st, j = (v / st) & 3, high = v / (4 * st);
            const double* x = in + high * 8 * st + lowi;
            double t = 0.0;
#pragma unroll
            for (int i = 0; i < 8; ++i) t += E[i][j] * x[i * st];
            out[v] = t;
        }
        __syncwarp();
        double* swap = in;
        in = out;
        out = swap;
        st *= 4;
    }
    for (int v = lane; v < n; v += 32) parent[(size_t)m * nodes_of(D) + v] = (T)in[v];
}

template <int D>
__global__ void __launch_bounds__(kShiftWarps * 32) k_down(const double* __restrict__ parent, double* __restrict__ child, int ncell,
                                                           Halves H) {
    constexpr int N = D == 2 ? 64 : 512;
    __shared__ double buf[kShiftWarps][N + N / 2];
    __shared__ double E[8][4];
    if (threadIdx.x < 32) E[threadIdx.x >> 2][threadIdx.x & 3] = H.e[threadIdx.x >> 2][threadIdx.x & 3];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int m = blockIdx.x * kShiftWarps + warp;
    if (m >= ncell) return;
    // the last axis's values land in the full-size half of the buffer
    double* in = D == 2 ? buf[warp] : buf[warp] + N;
    double* out = D == 2 ? buf[warp] + N : buf[warp];
    for (int v = lane; v < nodes_of(D); v += 32) in[v] = parent[(size_t)m * nodes_of(D) + v];
    __syncwarp();
    // along x (4 -> 8), then y, then z: the axes before the expanded one have 8 values
    int n = nodes_of(D), st = 1;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        n <<= 1;
        for (int v = lane; v < n; v += 32) {
            const int lowi = v % st, i = (v / st) & 7, high = v / (8 * st);
            const double* x = in + high * 4 * st + lowi;
            double t = 0.0;
#pragma unroll
            for (int j = 0; j < 4; ++j) t += E[i][j] * x[j * st];
            out[v] = t;
        }
        __syncwarp();
        double* swap = in;
        in = out;
        out = swap;
        st *= 8;
    }
    double* c = child + (size_t)m * (1 << D) * nodes_of(D);
    for (int v = lane; v < N; v += 32) c[child_value<D>(v)] += in[v];
}

// The finest cells' node potentials for the FP32 evaluation: each cell's first node value in FP64 and the
// others' differences from it in FP32.  The weights of a charge sum to one, so phi = psi_0 + sum_j w_j
// (psi_j - psi_0), and FP32 rounds only the potential's variation over a cell.
template <int D>
__global__ void k_split_psi(const double* __restrict__ psi, int64_t nval, double* __restrict__ psi0,
                            float* __restrict__ delta) {
    constexpr int d = nodes_of(D);
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= nval) return;
    const double first = psi[v / d * d];
    delta[v] = (float)(psi[v] - first);
    if (v % d == 0) psi0[v / d] = first;
}

// ------------------------------------------------------------------------------ node potentials

// psi_m[j] += sum_{o in IL} sum_i K_k[o][i][j] Q_{m+o}[i].  Targets are grouped by
// the parity of their coordinates: within a parity class the interaction list is the same set of
// offsets (o_a in [-2 - p_a, 3 - p_a], Chebyshev distance >= 2), so a block takes a tile of targets of
// one class and a group of offsets, and applies each offset's d x d matrix to the tile's source columns,
// a small dense product from shared memory.  The next offset's matrix and columns arrive by cp.async
// beside the current product.
// What bounds it: FP32 at 4 x 4 sums a thread, where 64 FMAs take 12 wavefronts of shared memory; a thread
// per node and eight targets took nine loads for eight FMAs.  200,000 charges in 3D, levels 3: 124 -> 40 us
// alone; 2^20 in 2D, levels 7: 66 -> 20 us.  FP64 (0.82 ms for 80,000 in 3D, levels 3) is bound by its pipe.
constexpr int kM2LThreads = 128;
template <int D>
__host__ __device__ constexpr int m2l_tile() { return D == 2 ? 128 : 32; }   // targets a block
template <int D, typename T>
__host__ __device__ constexpr int m2l_stride() { return nodes_of(D) + 16 / (int)sizeof(T); }   // of a source column
template <int D, typename T>
__host__ __device__ constexpr int m2l_buf() { return nodes_of(D) * nodes_of(D) + m2l_tile<D>() * m2l_stride<D, T>(); }
template <int D, typename T>
constexpr size_t m2l_smem_bytes() { return 2 * (size_t)m2l_buf<D, T>() * sizeof(T); }

// All levels in one launch: level k's blocks begin at base[k].
struct M2LLevels {
    const void* K[kMaxLevels + 1];
    LevelPtrs Q, psi;
    int base[kMaxLevels + 2];
};

template <typename T>
struct alignas(16) Vec4 {
    T v[4];
};

// 16 bytes to shared memory, or 16 zero bytes
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool have) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                 ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(have ? 16 : 0) : "memory");
}

// sums of targets tg + r NTG (r < R) at nodes 4 jg .. 4 jg + 3 over one offset, added to acc.  FP32: with
// Kahan's compensation, as a plain running sum over a group's offsets (up to 7 x 64 terms in 3D) would leave
// about 1e-6 of the far field in rounding.
template <int D, typename T, int R, int RT>
__device__ __forceinline__ void m2l_product(const T* __restrict__ sK, const T* __restrict__ sQ, int jg, int tg,
                                            T (&acc)[RT][4], T (&comp)[RT][4]) {
    constexpr int d = nodes_of(D), S = m2l_stride<D, T>(), NTG = m2l_tile<D>() / RT;
    T t[R][4];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) t[r][j] = T(0);
#pragma unroll 2
    for (int i = 0; i < d; i += 4) {
        Vec4<T> kv[4], qv[R];
#pragma unroll
        for (int ii = 0; ii < 4; ++ii) kv[ii] = *reinterpret_cast<const Vec4<T>*>(sK + (i + ii) * d + 4 * jg);
#pragma unroll
        for (int r = 0; r < R; ++r) qv[r] = *reinterpret_cast<const Vec4<T>*>(sQ + (tg + r * NTG) * S + i);
#pragma unroll
        for (int ii = 0; ii < 4; ++ii)
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int j = 0; j < 4; ++j) t[r][j] += kv[ii].v[j] * qv[r].v[ii];
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if constexpr (sizeof(T) == 4) {
                const T y = t[r][j] - comp[r][j];
                const T sum = acc[r][j] + y;
                comp[r][j] = (sum - acc[r][j]) - y;
                acc[r][j] = sum;
            } else {
                acc[r][j] += t[r][j];
            }
        }
}

template <int D, typename T>
__global__ void __launch_bounds__(kM2LThreads) k_m2l(M2LLevels lv, int ngroups) {
    constexpr int d = nodes_of(D), TT = m2l_tile<D>(), S = m2l_stride<D, T>(), JG = d / 4, NTG = kM2LThreads / JG,
                  RT = TT / NTG;
    constexpr int NOFF = D == 2 ? 27 : 189, RAW = D == 2 ? 36 : 216;
    constexpr int PER16 = 16 / (int)sizeof(T), CH = d / PER16, NQ = CH * TT / kM2LThreads;   // 16-byte pieces of a column
    static_assert(RT == 4 && NQ * kM2LThreads == CH * TT, "whole tiles");
    extern __shared__ __align__(16) unsigned char m2l_smem[];
    __shared__ int s_off[NOFF];   // the group's offsets as base-6 digits
    T* buf = reinterpret_cast<T*>(m2l_smem);
    int k = 2;
    while ((int)blockIdx.x >= lv.base[k + 1]) ++k;
    const T* K = static_cast<const T*>(lv.K[k]);
    const T* Q = static_cast<const T*>(lv.Q.p[k]);
    double* psi = static_cast<double*>(lv.psi.p[k]);   // FP64 sums in every form
    const int side = 1 << k, pside = side >> 1;
    const int nparent = D == 2 ? pside * pside : pside * pside * pside;
    const int ntiles = (nparent + TT - 1) / TT;
    int blk = blockIdx.x - lv.base[k];
    const int g = blk % ngroups;
    blk /= ngroups;
    const int tile = blk % ntiles, par = blk / ntiles;
    const int p[3] = {par & 1, (par >> 1) & 1, (par >> 2) & 1};
    const int tid = threadIdx.x, jg = tid % JG, tg = tid / JG;
    const int per = (NOFF + ngroups - 1) / ngroups, e0 = g * per, cnt = min(NOFF, e0 + per) - e0;
    auto offset = [&](int raw, int a) { return (a == 0 ? raw : (a == 1 ? raw / 6 : raw / 36)) % 6 - 2 - p[a]; };
    if (tid < 32) {   // offsets e0 .. e0 + cnt - 1 of the class, x fastest
        int before = 0;
        for (int r0 = 0; r0 < RAW; r0 += 32) {
            const int raw = r0 + tid;
            int cheb = max(abs(offset(raw, 0)), abs(offset(raw, 1)));
            if (D == 3) cheb = max(cheb, abs(offset(raw, 2)));
            const bool valid = raw < RAW && cheb >= 2;
            const unsigned m = __ballot_sync(0xffffffffu, valid);
            const int e = before + __popc(m & ((1u << tid) - 1u)) - e0;
            if (valid && e >= 0 && e < cnt) s_off[e] = raw;
            before += __popc(m);
        }
    }
    // the targets whose source columns this thread loads pieces of, and the tile's end
    int tc[NQ][D];
    const int rows = min(TT, nparent - tile * TT);
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
        const int P = tile * TT + (tid + m * kM2LThreads) / CH;
        tc[m][0] = 2 * (P % pside) + p[0];
        tc[m][1] = 2 * ((P / pside) % pside) + p[1];
        if constexpr (D == 3) tc[m][2] = 2 * (P / (pside * pside)) + p[2];   // outside the grid past the last target
    }
    __syncthreads();
    auto stage = [&](int e) {
        const int raw = s_off[e];
        int o[D], oidx = 0;
#pragma unroll
        for (int a = D - 1; a >= 0; --a) {
            o[a] = offset(raw, a);
            oidx = 7 * oidx + o[a] + 3;
        }
        T* sK = buf + (e & 1) * m2l_buf<D, T>();
        T* sQ = sK + d * d;
        const T* Ko = K + (size_t)oidx * d * d;
        for (int x = tid; x < d * d / PER16; x += kM2LThreads) cp_async16(sK + x * PER16, Ko + x * PER16, true);
#pragma unroll
        for (int m = 0; m < NQ; ++m) {
            const int x = tid + m * kM2LThreads, tt = x / CH, c = x % CH;
            bool in = tt < rows;
            uint32_t cell = 0;
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const int v = tc[m][a] + o[a];
                in = in && v >= 0 && v < side;
                cell |= spread_bits(D, (uint32_t)v & 0xffu) << a;
            }
            cp_async16(sQ + tt * S + c * PER16, in ? Q + (size_t)cell * d + c * PER16 : Q, in);
        }
    };
    T acc[RT][4], comp[RT][4];
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[r][j] = comp[r][j] = T(0);
    stage(0);
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int e = 0; e < cnt; ++e) {
        if (e + 1 < cnt) stage(e + 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        const T* sK = buf + (e & 1) * m2l_buf<D, T>();
        // level 2 has few targets of a class: one row of sums holds them
        if (rows <= NTG) m2l_product<D, T, 1, RT>(sK, sK + d * d, jg, tg, acc, comp);
        else m2l_product<D, T, RT, RT>(sK, sK + d * d, jg, tg, acc, comp);
        __syncthreads();
    }
    // out by way of shared memory, so that a warp's atomics fall on consecutive nodes
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        Vec4<T> v;
#pragma unroll
        for (int j = 0; j < 4; ++j) v.v[j] = acc[r][j];
        *reinterpret_cast<Vec4<T>*>(buf + (tg + r * NTG) * d + 4 * jg) = v;
    }
    __syncthreads();
    for (int x = tid; x < rows * d; x += kM2LThreads) {
        const int P = tile * TT + x / d;
        uint32_t cell = spread_bits(D, (uint32_t)(2 * (P % pside) + p[0])) |
                        spread_bits(D, (uint32_t)(2 * ((P / pside) % pside) + p[1])) << 1;
        if constexpr (D == 3) cell |= spread_bits(D, (uint32_t)(2 * (P / (pside * pside)) + p[2])) << 2;
        atomicAdd(psi + (size_t)cell * d + x % d, (double)buf[x]);
    }
}

// ------------------------------------------------------------------------------ evaluation

// Node forms: phi_far(c) = h_m(c) . psi_m of the charge's finest cell (which k_down has left with the sum
// of all levels), the tensor-product contraction done axis by axis; phi in input order = far + near (nearf
// in units of near_unit), written only if the inputs passed.  psi is null without a far field; psi0 (FP32)
// is what k_split_psi took off it.
// 2^20 charges in 2D, levels 7: 54 us with the downward pass against 332 us for an interpolation at each of six
// levels with its FP64 centre and division.
template <int D, typename T>
__global__ void k_l2p(PosReader<T> rd, const uint32_t* __restrict__ skey, int64_t n, const T* __restrict__ psi,
                      const double* __restrict__ psi0, const double* __restrict__ nearf, double near_unit,
                      const unsigned* __restrict__ status, double* __restrict__ phi) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    T v = T(0);
    double base = 0.0;
    if (psi != nullptr) {
        const uint32_t cell = skey[i];
        if (psi0 != nullptr) base = psi0[cell];
        int cc[3];
        morton_dec(D, cell, cc);
        T f[D][4];
#pragma unroll
        for (int a = 0; a < D; ++a) lag_basis<T>(rd.local((int)i, a, rd.centre(cc[a])), f[a]);
        const T* ps = psi + (size_t)cell * nodes_of(D);
#pragma unroll
        for (int iz = 0; iz < (D == 3 ? 4 : 1); ++iz) {
            T u = T(0);
#pragma unroll
            for (int iy = 0; iy < 4; ++iy) {
                T r = T(0);
#pragma unroll
                for (int ix = 0; ix < 4; ++ix) r += f[0][ix] * __ldg(ps + ix + 4 * iy + 16 * iz);
                u += f[1][iy] * r;
            }
            if constexpr (D == 3) v += f[2][iz] * u;
            else v = u;
        }
    }
    if (*(volatile const unsigned*)status != 0u) return;
    phi[rd.input((int)i)] = fma(near_unit, nearf[i], base + (double)v);
}

// ------------------------------------------------------------------------------ literal form

// U-bar-2: v_k of a cell = sum of its 2^D children's (contiguous in Morton order), no shift.
template <int D>
__global__ void k_lit_up(const double* __restrict__ child, double* __restrict__ parent, int64_t ncell) {
    constexpr int d = nodes_of(D);
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= ncell * d) return;
    const int64_t c = x / d, j = x % d;
    double s = 0.0;
    for (int ch = 0; ch < (1 << D); ++ch) s += child[((c << D) + ch) * d + j];
    parent[x] = s;
}

// D-bar-1 and D-bar-2 of one level: u_m = sum_{pairs (m_i, m)} B^T v_{m_i} + u_parent(m).
// Threads: d target coordinates l x (256 / d) pair lanes; B rows are read coalesced over l.
template <int D>
__global__ void __launch_bounds__(256) k_lit_down(const int* __restrict__ pstart, const int* __restrict__ psrc,
                                                  const double* __restrict__ B, const double* __restrict__ v,
                                                  const double* __restrict__ uparent, double* __restrict__ u,
                                                  int64_t ncell) {
    constexpr int d = nodes_of(D), PG = 256 / d;
    __shared__ double s_red[256];
    const int64_t m = blockIdx.x;
    if (m >= ncell) return;
    const int l = threadIdx.x % d, g = threadIdx.x / d;
    double acc = 0.0;
    for (int e = pstart[m] + g; e < pstart[m + 1]; e += PG) {
        const double* vs = v + (size_t)psrc[e] * d;
        const double* Be = B + (size_t)e * d * d;
        for (int a = 0; a < d; ++a) acc += __ldg(vs + a) * Be[(size_t)a * d + l];
    }
    s_red[threadIdx.x] = acc;
    __syncthreads();
    if (g == 0) {
        for (int r = 1; r < PG; ++r) acc += s_red[r * d + l];
        if (uparent) acc += uparent[(size_t)(m >> D) * d + l];
        u[(size_t)m * d + l] = acc;
    }
}

// F(v) = L_{m^l}(v) for each charge's own v (unit charge at the root box's nodes) + near field.
template <int D>
__global__ void k_lit_eval(const Pos64* __restrict__ p, const uint32_t* __restrict__ skey, int64_t n, double box,
                           const double* __restrict__ u, const double* __restrict__ nearf,
                           const int* __restrict__ order, const unsigned* __restrict__ status,
                           double* __restrict__ phi) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Pos64 c = p[i];
    const double inv = 5.0 / box, centre = 0.5 * box;
    double f[3][4];
    lag_basis<double>((c.x - centre) * inv, f[0]);
    lag_basis<double>((c.y - centre) * inv, f[1]);
    if (D == 3) lag_basis<double>((c.z - centre) * inv, f[2]);
    const double* ul = u + (size_t)skey[i] * nodes_of(D);
    double far = 0.0;
    for (int j = 0; j < nodes_of(D); ++j) {
        double w = f[0][j & 3] * f[1][(j >> 2) & 3];
        if (D == 3) w *= f[2][j >> 4];
        far += ul[j] * w;
    }
    if (*(volatile const unsigned*)status != 0u) return;
    phi[order[i]] = far + nearf[i];
}

// STEP3-STEP5 for one pair per block: M_m and M_{m_i} (columns h_m(p_l) of the root nodes),
// M_b[i][j] = K(node j of m - node i of m_i), T = M_b M_m, B = M_{m_i}^T T, all FP64.
template <int D>
__global__ void __launch_bounds__(256) k_lit_build(const int* __restrict__ ptgt, const int* __restrict__ psrc,
                                                   int64_t npairs, int k, double box, double* __restrict__ B) {
    constexpr int d = nodes_of(D);
    extern __shared__ double smem[];
    double* Mm = smem;             // [d][d]
    double* Mi = Mm + d * d;       // [d][d]
    double* T = Mi + d * d;        // [d][d], first M_b then M_b M_m
    double* Mb = T + d * d;        // [d][d]
    const int64_t e = blockIdx.x;
    if (e >= npairs) return;
    const double s = box / (double)(1 << k), h = s / 5.0;
    const double a_node[4] = {-2.0, -1.0, 1.0, 2.0};
    int cm[3], ci[3];
    morton_dec(D, (uint32_t)ptgt[e], cm);
    morton_dec(D, (uint32_t)psrc[e], ci);
    for (int x = threadIdx.x; x < d * d; x += blockDim.x) {
        const int row = x / d, col = x % d;   // row: cell node, col: root node
        const int rn[3] = {row & 3, (row >> 2) & 3, row >> 4};
        const int cn[3] = {col & 3, (col >> 2) & 3, col >> 4};
        double wm = 1.0, wi = 1.0;
        for (int a = 0; a < D; ++a) {
            const double pr = 0.5 * box + (box / 5.0) * a_node[cn[a]];   // root node coordinate
            double f[4];
            lag_basis<double>((pr - ((double)cm[a] + 0.5) * s) / h, f);
            wm *= f[rn[a]];
            lag_basis<double>((pr - ((double)ci[a] + 0.5) * s) / h, f);
            wi *= f[rn[a]];
        }
        Mm[x] = wm;
        Mi[x] = wi;
        // M_b[i = row][j = col]: source node i of m_i, target node j of m
        double r2 = 0.0;
        for (int a = 0; a < D; ++a) {
            const double pt = ((double)cm[a] + 0.5) * s + h * a_node[cn[a]];
            const double ps = ((double)ci[a] + 0.5) * s + h * a_node[rn[a]];
            r2 += (pt - ps) * (pt - ps);
        }
        Mb[x] = kernel64(D, r2);
    }
    __syncthreads();
    for (int x = threadIdx.x; x < d * d; x += blockDim.x) {
        const int i = x / d, l = x % d;
        double acc = 0.0;
        for (int j = 0; j < d; ++j) acc += Mb[i * d + j] * Mm[j * d + l];
        T[x] = acc;
    }
    __syncthreads();
    double* Be = B + (size_t)e * d * d;
    for (int x = threadIdx.x; x < d * d; x += blockDim.x) {
        const int a = x / d, l = x % d;
        double acc = 0.0;
        for (int i = 0; i < d; ++i) acc += Mi[i * d + a] * T[i * d + l];
        Be[x] = acc;
    }
}

// ------------------------------------------------------------------------------ direct sum

template <int D>
__global__ void k_direct_targets(const double* __restrict__ pos, const double* __restrict__ q, int64_t n,
                                 const int64_t* __restrict__ tgt, int64_t nt, double* __restrict__ phi) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    const int64_t i = tgt[t];
    const double x = pos[i * D], y = pos[i * D + 1], z = D == 3 ? pos[i * D + 2] : 0.0;
    double acc = 0.0;
    for (int64_t j = 0; j < n; ++j) {
        if (j == i) continue;
        const double dx = x - pos[j * D], dy = y - pos[j * D + 1], dz = D == 3 ? z - pos[j * D + 2] : 0.0;
        acc += q[j] * kernel64(D, dx * dx + dy * dy + dz * dz);
    }
    phi[t] = acc;
}

// ------------------------------------------------------------------------------ host helpers

int64_t ipow(int64_t b, int e) {
    int64_t r = 1;
    while (e-- > 0) r *= b;
    return r;
}

// The interaction list of cell m (coords) at level k, as Morton indices.
int il_cells(int D, int k, const int* m, std::vector<uint32_t>& out) {
    const int side = 1 << k;
    out.clear();
    int lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
    for (int a = 0; a < D; ++a) {
        const int p = m[a] >> 1;
        lo[a] = std::max(0, 2 * (p - 1));
        hi[a] = std::min(side - 1, 2 * (p + 1) + 1);
    }
    int c[3] = {0, 0, 0};
    for (c[2] = (D == 3 ? lo[2] : 0); c[2] <= (D == 3 ? hi[2] : 0); ++c[2])
        for (c[1] = lo[1]; c[1] <= hi[1]; ++c[1])
            for (c[0] = lo[0]; c[0] <= hi[0]; ++c[0]) {
                int cheb = 0;
                for (int a = 0; a < D; ++a) cheb = std::max(cheb, std::abs(c[a] - m[a]));
                if (cheb >= 2) out.push_back(morton_enc(D, c));
            }
    return (int)out.size();
}

bool valid_form(int f) { return f == FMM_LAG_NODE_F32 || f == FMM_LAG_NODE_F64 || f == FMM_LAG_LITERAL_F64; }

fmm_status cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return FMM_OK;
    return e == cudaErrorMemoryAllocation ? FMM_ERR_OOM : FMM_ERR_CUDA;
}

template <typename T>
fmm_status alloc(fmm_lag_plan_s* pl, T** p, size_t count) {
    const size_t bytes = std::max<size_t>(count, 1) * sizeof(T);
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), bytes);
    if (e != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        return cuda_status(e);
    }
    pl->bytes += bytes;
    return FMM_OK;
}

void plan_free(fmm_lag_plan_s* pl) {
    if (!pl) return;
    cudaFree(pl->key); cudaFree(pl->rank); cudaFree(pl->skey); cudaFree(pl->count); cudaFree(pl->start);
    cudaFree(pl->chunk_start); cudaFree(pl->wchunk_start); cudaFree(pl->wchunk_cell); cudaFree(pl->order); cudaFree(pl->hi); cudaFree(pl->lo); cudaFree(pl->p64);
    cudaFree(pl->nearf); cudaFree(pl->status); cudaFree(pl->pairs); cudaFree(pl->next_item); cudaFree(pl->K); cudaFree(pl->logtab);
    cudaFree(pl->scan); cudaFree(pl->pot[2]); cudaFree(pl->psi0); cudaFree(pl->dpsi);
    for (int k = 0; k <= kMaxLevels; ++k) {
        cudaFree(pl->node[k]); cudaFree(pl->pair_start[k]); cudaFree(pl->pair_src[k]);
        cudaFree(pl->B[k]);
    }
    for (auto& e : pl->ev) if (e) cudaEventDestroy(e);
    if (pl->ev_fork) cudaEventDestroy(pl->ev_fork);
    if (pl->ev_join) cudaEventDestroy(pl->ev_join);
    if (pl->st2) cudaStreamDestroy(pl->st2);
    if (pl->h_status) cudaFreeHost(pl->h_status);
    delete pl;
}

// Node-to-node operators of levels 2..L, FP64 on the host: K_k[o][i][j] = K(node j of the target
// - node i of the source at offset o), o over the 7^D table (the near offsets stay zero).
std::vector<double> build_operators(int D, int L, double box) {
    const int d = nodes_of(D), no = offsets_of(D);
    const double a_node[4] = {-2.0, -1.0, 1.0, 2.0};
    std::vector<double> K((size_t)std::max(0, L - 1) * no * d * d, 0.0);
    for (int k = 2; k <= L; ++k) {
        const double s = box / (double)(1 << k), h = s / 5.0;
        double* Kk = K.data() + (size_t)(k - 2) * no * d * d;
        for (int oi = 0; oi < no; ++oi) {
            const int o[3] = {oi % 7 - 3, (oi / 7) % 7 - 3, D == 3 ? oi / 49 - 3 : 0};
            if (std::max(std::abs(o[0]), std::max(std::abs(o[1]), std::abs(o[2]))) < 2) continue;
            for (int i = 0; i < d; ++i)
                for (int j = 0; j < d; ++j) {
                    const int ni[3] = {i & 3, (i >> 2) & 3, i >> 4}, nj[3] = {j & 3, (j >> 2) & 3, j >> 4};
                    double r2 = 0.0;
                    for (int a = 0; a < D; ++a) {
                        const double r = h * (a_node[nj[a]] - a_node[ni[a]]) - o[a] * s;
                        r2 += r * r;
                    }
                    Kk[((size_t)oi * d + i) * d + j] = kernel64(D, r2);
                }
        }
    }
    return K;
}

// the plan's stream behind the far field's
void lag_join(fmm_lag_plan_s* pl, cudaStream_t far_st) {
    if (far_st == pl->st) return;
    cudaEventRecord(pl->ev_join, far_st);
    cudaStreamWaitEvent(pl->st, pl->ev_join, 0);
}

// The far field of the node forms on its stream, joined with the near field: node charges of the
// finest cells, up the tree, over the interaction lists, down the tree, evaluation.
template <int D, typename T>
int enqueue_nodes(fmm_lag_plan_s* pl, const PosReader<T>& rd, int64_t n, unsigned gp, unsigned gb, double near_unit,
                  double* phi) {
    constexpr int d = nodes_of(D);
    const int L = pl->levels;
    cudaStream_t st = pl->serial ? pl->st : pl->st2;
    int launches = 0;
    static const Halves H = make_halves();
    const auto shift_blocks = [](int64_t cells) { return (unsigned)((cells + kShiftWarps - 1) / kShiftWarps); };
    if (L >= 2) {
        k_p2m<D, T><<<gp, kChunk, 0, st>>>(rd, pl->start, pl->chunk_start, (int)pl->nleaf, false,
                                           static_cast<T*>(pl->node[L]), pl->skey);
        ++launches;
        for (int k = L - 1; k >= 2; --k) {
            const int64_t cells = ipow(1 << k, D);
            k_up<D, T><<<shift_blocks(cells), kShiftWarps * 32, 0, st>>>(
                static_cast<const T*>(pl->node[k + 1]), static_cast<T*>(pl->node[k]), (int)cells, H);
            ++launches;
        }
    }
    cudaEventRecord(pl->ev[2], st);
    if (L >= 2) {
        const int ngroups = D == 2 ? 3 : 27;
        M2LLevels lv{};
        int blocks = 0;
        for (int k = 2; k <= L; ++k) {
            lv.K[k] = static_cast<const T*>(pl->K) + (size_t)(k - 2) * offsets_of(D) * d * d;
            lv.Q.p[k] = pl->node[k];
            lv.psi.p[k] = pl->pot[k];
            lv.base[k] = blocks;
            blocks += (int)(((ipow(1 << (k - 1), D) + m2l_tile<D>() - 1) / m2l_tile<D>()) * (1 << D) * ngroups);
        }
        lv.base[L + 1] = blocks;
        k_m2l<D, T><<<(unsigned)blocks, kM2LThreads, m2l_smem_bytes<D, T>(), st>>>(lv, ngroups);
        ++launches;
    }
    cudaEventRecord(pl->ev[3], st);
    for (int k = 2; k < L; ++k) {
        const int64_t cells = ipow(1 << k, D);
        k_down<D><<<shift_blocks(cells), kShiftWarps * 32, 0, st>>>(
            static_cast<const double*>(pl->pot[k]), static_cast<double*>(pl->pot[k + 1]), (int)cells, H);
        ++launches;
    }
    const T* psi = L >= 2 ? static_cast<const T*>(pl->pot[L]) : nullptr;
    const double* psi0 = nullptr;
    if constexpr (sizeof(T) == 4) {
        if (L >= 2) {
            const int64_t nval = pl->nleaf * d;
            k_split_psi<D><<<(unsigned)((nval + 255) / 256), 256, 0, st>>>(static_cast<const double*>(pl->pot[L]), nval,
                                                                          pl->psi0, pl->dpsi);
            ++launches;
            psi = pl->dpsi;
            psi0 = pl->psi0;
        }
    }
    lag_join(pl, st);
    k_l2p<D, T><<<gb, 256, 0, pl->st>>>(rd, pl->skey, n, psi, psi0, pl->nearf, near_unit, pl->status, phi);
    return launches + 1;
}

template <int D>
fmm_status enqueue(fmm_lag_plan_s* pl, const double* pos, const double* q, int64_t n, double* phi) {
    constexpr int d = nodes_of(D);
    const int L = pl->levels;
    const bool f64 = pl->form != FMM_LAG_NODE_F32, lit = pl->form == FMM_LAG_LITERAL_F64;
    cudaStream_t st = pl->st;
    int launches = 0;
    cudaEventRecord(pl->ev[0], st);
    cudaMemsetAsync(pl->count, 0, sizeof(int) * (size_t)pl->nleaf, st);
    cudaMemsetAsync(pl->pairs, 0, kPairSlots * sizeof(unsigned long long), st);
    if (L >= 2) {   // sums that start at zero: the finest cells' node values, every level's potentials
        cudaMemsetAsync(pl->node[L], 0, (size_t)pl->nleaf * d * (f64 ? 8 : 4), st);
        if (!lit) cudaMemsetAsync(pl->pot[2], 0, pl->pot_bytes, st);
    }
    const unsigned gb = (unsigned)((n + 255) / 256);
    const float side_over_box = (float)((double)(1 << L) / pl->box);
    if (bin_few(pl->nleaf, n))
        k_bin_few<D><<<(unsigned)pl->sms, kBinFewThreads, 0, st>>>(pos, q, n, L, pl->box, side_over_box, pl->key, pl->rank,
                                                                   pl->count, (int)pl->nleaf, pl->status);
    else
        k_bin<D><<<gb, 256, 0, st>>>(pos, q, n, L, pl->box, side_over_box, pl->key, pl->rank, pl->count, pl->status);
    const unsigned tiles = (unsigned)((pl->nleaf + kScanTile - 1) / kScanTile);
    const int wchunk = f64 ? kWarpChunk64 : kWarpChunk;
    k_scan_sums<<<tiles, kScanTile, 0, st>>>(pl->count, (int)pl->nleaf, wchunk, pl->scan);
    k_scan<<<tiles, kScanTile, 0, st>>>(pl->count, (int)pl->nleaf, wchunk, pl->scan, pl->start, pl->chunk_start,
                                        pl->wchunk_start, pl->wchunk_cell);
    if (f64)
        k_scatter<D, true><<<gb, 256, 0, st>>>(pos, q, n, pl->key, pl->rank, pl->start, pl->order, nullptr, nullptr,
                                               pl->p64);
    else
        k_scatter<D, false><<<gb, 256, 0, st>>>(pos, q, n, pl->key, pl->rank, pl->start, nullptr, pl->hi, pl->lo,
                                                nullptr);
    launches += 4;
    cudaEventRecord(pl->ev[7], st);
    cudaEventRecord(pl->ev[1], st);
    // The far field on the second stream, which has the device's highest priority, beside the near field on
    // the plan's stream (in serial mode everything in turn on the plan's stream).
    cudaStream_t far_st = pl->serial ? st : pl->st2;
    if (!pl->serial) {
        cudaEventRecord(pl->ev_fork, st);
        cudaStreamWaitEvent(pl->st2, pl->ev_fork, 0);
    }
    const unsigned gp = (unsigned)pl->grid_particles;
    cudaMemsetAsync(pl->nearf, 0, sizeof(double) * (size_t)n, st);
    if (f64) cudaMemsetAsync(pl->next_item, 0, sizeof(int), st);
    cudaEventRecord(pl->ev[5], st);
    if (f64) {
        k_p2p64<D><<<(unsigned)pl->grid_p2p, kP2PWarps64 * 32, 0, st>>>(
            pl->p64, pl->start, pl->wchunk_start, pl->wchunk_cell, (int)pl->nleaf, L, pl->logtab, pl->nearf, pl->pairs, pl->next_item);
    } else {
        // a chunk per kWarpChunk charges and a partial one per occupied cell at most
        constexpr int F = D == 3 ? 14 : 5, G = (F + fwd_group<D>() - 1) / fwd_group<D>();
        const int64_t items = (std::min<int64_t>(pl->nleaf, n) + n / kWarpChunk) * G;
        const float apart = 0x1p-50f * (float)pl->box, tiny = std::max(apart * apart, 0x1p-126f);
        k_p2p32<D><<<(unsigned)((items + kP2PWarps - 1) / kP2PWarps), kP2PWarps * 32, 0, st>>>(
            pl->hi, pl->lo, pl->start, pl->wchunk_start, pl->wchunk_cell, (int)pl->nleaf, L, (float)pl->box,
            make_float2(tiny, tiny), pl->nearf, pl->pairs);
    }
    ++launches;
    cudaEventRecord(pl->ev[6], st);
    if (pl->serial) cudaEventRecord(pl->ev[1], st);   // the far-field stages start after the near field

    // the finest cells' side and the scale of their local coordinates
    const double cs = pl->box / (double)(1 << L);
    const float cs_hi = (float)cs;
    const PosReader<float> rd32{pl->hi, pl->lo, make_float2(cs_hi, (float)(cs - (double)cs_hi)), (float)(5.0 / cs)};
    const PosReader<double> rd64{pl->p64, pl->order, cs, 5.0 / cs};
    const double near_unit = !f64 && D == 2 ? 0.5 * kLn2 : 1.0;   // the 2D FP32 near field is in log2 r^2
    if (lit && L < 2) {
        // no interaction lists: phi is the near field
        cudaEventRecord(pl->ev[2], far_st);
        cudaEventRecord(pl->ev[3], far_st);
        lag_join(pl, far_st);
        k_l2p<D, double><<<gb, 256, 0, st>>>(rd64, pl->skey, n, nullptr, nullptr, pl->nearf, near_unit, pl->status,
                                             phi);
        ++launches;
    } else if (!lit) {
        if (f64) launches += enqueue_nodes<D, double>(pl, rd64, n, gp, gb, near_unit, phi);
        else launches += enqueue_nodes<D, float>(pl, rd32, n, gp, gb, near_unit, phi);
    } else {
        // U-bar-1: v of every finest cell from the charges' root-node images
        k_p2m<D, double><<<gp, kChunk, 0, far_st>>>(PosReader<double>{pl->p64, pl->order, pl->box, 5.0 / pl->box}, pl->start,
                                                pl->chunk_start, (int)pl->nleaf, true, static_cast<double*>(pl->node[L]), pl->skey);
        ++launches;
        // U-bar-2: sums up the tree (levels below 2 are never read)
        for (int k = L - 1; k >= 2; --k) {
            const int64_t ncell = ipow(1 << k, D);
            k_lit_up<D><<<(unsigned)((ncell * d + 255) / 256), 256, 0, far_st>>>(
                static_cast<const double*>(pl->node[k + 1]), static_cast<double*>(pl->node[k]), ncell);
            ++launches;
        }
        cudaEventRecord(pl->ev[2], far_st);
        // D-bar-1 and D-bar-2 level by level, top down
        for (int k = 2; k <= L; ++k) {
            const int64_t ncell = ipow(1 << k, D);
            k_lit_down<D><<<(unsigned)ncell, 256, 0, far_st>>>(pl->pair_start[k], pl->pair_src[k], pl->B[k],
                                                           static_cast<const double*>(pl->node[k]),
                                                           k >= 3 ? static_cast<const double*>(pl->pot[k - 1]) : nullptr,
                                                           static_cast<double*>(pl->pot[k]), ncell);
            ++launches;
        }
        cudaEventRecord(pl->ev[3], far_st);
        lag_join(pl, far_st);
        k_lit_eval<D><<<gb, 256, 0, st>>>(pl->p64, pl->skey, n, pl->box, static_cast<const double*>(pl->pot[L]),
                                          pl->nearf, pl->order, pl->status, phi);
        ++launches;
    }
    cudaEventRecord(pl->ev[4], st);
    pl->launches = launches;
    pl->last_n = n;
    pl->last_st = st;
    return cuda_status(cudaGetLastError());
}

}  // namespace

extern "C" {

fmm_status fmm_lag_plan(fmm_lag_plan_t* out, int dim, int64_t n_max, int levels, double box, int form,
                        void* stream) {
    if (!out || (dim != 2 && dim != 3) || n_max < 1 || n_max > (int64_t(1) << 30) || !valid_form(form) ||
        !(box > 0.0) || !std::isfinite(box) || levels < 0)
        return FMM_ERR_INVALID_ARG;
    const bool lit = form == FMM_LAG_LITERAL_F64;
    const int lmax = dim == 2 ? (lit ? 7 : 8) : (lit ? 3 : 5);
    if (levels > lmax) return FMM_ERR_INVALID_ARG;
    auto* pl = new (std::nothrow) fmm_lag_plan_s;
    if (!pl) return FMM_ERR_OOM;
    pl->dim = dim; pl->levels = levels; pl->form = form; pl->box = box; pl->n_max = n_max;
    pl->d = nodes_of(dim);
    pl->st = static_cast<cudaStream_t>(stream);
    pl->nleaf = ipow(1 << levels, dim);
    const int d = pl->d;
    const bool f64 = form != FMM_LAG_NODE_F32;
    fmm_status rc = cuda_status(cudaGetDevice(&pl->dev));
    int sms = 0;
    if (rc == FMM_OK) rc = cuda_status(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, pl->dev));
    pl->sms = std::max(1, sms);
    pl->grid_particles = std::max(1, sms) * 8;
    int per_sm = 0;
    if (rc == FMM_OK)
        rc = cuda_status(
            dim == 2 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_p2p64<2>, kP2PWarps64 * 32, 0)
                     : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_p2p64<3>, kP2PWarps64 * 32, 0));
    pl->grid_p2p = std::max(1, sms) * std::max(1, per_sm);
    int least = 0, greatest = 0;
    if (rc == FMM_OK) rc = cuda_status(cudaDeviceGetStreamPriorityRange(&least, &greatest));
    if (rc == FMM_OK) rc = cuda_status(cudaStreamCreateWithPriority(&pl->st2, cudaStreamNonBlocking, greatest));
    for (auto& e : pl->ev)
        if (rc == FMM_OK) rc = cuda_status(cudaEventCreate(&e));
    if (rc == FMM_OK) rc = cuda_status(cudaEventCreateWithFlags(&pl->ev_fork, cudaEventDisableTiming));
    if (rc == FMM_OK) rc = cuda_status(cudaEventCreateWithFlags(&pl->ev_join, cudaEventDisableTiming));
    const size_t n = (size_t)n_max;
    if (rc == FMM_OK) rc = alloc(pl, &pl->key, n);
    if (rc == FMM_OK) rc = alloc(pl, &pl->rank, n);
    if (rc == FMM_OK) rc = alloc(pl, &pl->skey, n);
    if (rc == FMM_OK && f64) rc = alloc(pl, &pl->order, n);
    if (rc == FMM_OK) rc = alloc(pl, &pl->nearf, n);
    if (rc == FMM_OK) rc = alloc(pl, &pl->count, (size_t)pl->nleaf);
    if (rc == FMM_OK) rc = alloc(pl, &pl->start, (size_t)pl->nleaf + 1);
    if (rc == FMM_OK) rc = alloc(pl, &pl->chunk_start, (size_t)pl->nleaf + 1);
    if (rc == FMM_OK) rc = alloc(pl, &pl->wchunk_start, (size_t)pl->nleaf + 1);
    // a chunk per kWarpChunk charges and a partial one per occupied cell at most
    if (rc == FMM_OK) rc = alloc(pl, &pl->wchunk_cell, std::min((size_t)pl->nleaf, n) + n / (f64 ? kWarpChunk64 : kWarpChunk));
    if (rc == FMM_OK) rc = alloc(pl, &pl->status, 1);
    if (rc == FMM_OK) rc = alloc(pl, &pl->pairs, kPairSlots);
    if (rc == FMM_OK) rc = alloc(pl, &pl->next_item, 1);
    if (rc == FMM_OK && f64) rc = alloc(pl, &pl->p64, n);
    if (rc == FMM_OK && f64 && dim == 2) {
        std::vector<double2> tab(kFmmLogEntries);
        for (int j = 0; j < kFmmLogEntries; ++j) tab[j] = fmm_log_entry(j);
        rc = alloc(pl, &pl->logtab, tab.size());
        if (rc == FMM_OK)
            rc = cuda_status(cudaMemcpy(pl->logtab, tab.data(), sizeof(double2) * tab.size(), cudaMemcpyHostToDevice));
    }
    if (rc == FMM_OK && !f64) rc = alloc(pl, &pl->hi, n);
    if (rc == FMM_OK && !f64) rc = alloc(pl, &pl->lo, n);
    const size_t vb = f64 ? 8 : 4;
    if (rc == FMM_OK) rc = alloc(pl, &pl->scan, (size_t)((pl->nleaf + kScanTile - 1) / kScanTile));
    for (int k = 2; k <= levels && rc == FMM_OK; ++k) {
        const size_t bytes = (size_t)ipow(1 << k, dim) * d * vb;
        rc = alloc(pl, reinterpret_cast<char**>(&pl->node[k]), bytes);
        pl->pot_bytes += bytes / vb * 8;   // FP64 in every form
    }
    if (rc == FMM_OK && levels >= 2) {
        char* pot = nullptr;
        rc = alloc(pl, &pot, pl->pot_bytes);
        for (int k = 2; k <= levels && rc == FMM_OK; ++k) {
            pl->pot[k] = pot;
            pot += (size_t)ipow(1 << k, dim) * d * 8;
        }
        if (rc == FMM_OK && !f64) rc = alloc(pl, &pl->psi0, (size_t)pl->nleaf);
        if (rc == FMM_OK && !f64) rc = alloc(pl, &pl->dpsi, (size_t)pl->nleaf * d);
    }
    if (rc == FMM_OK) rc = cuda_status(cudaMemset(pl->status, 0, sizeof(unsigned)));
    if (rc == FMM_OK) rc = cuda_status(cudaMallocHost(reinterpret_cast<void**>(&pl->h_status), sizeof(unsigned)));
    if (rc == FMM_OK && dim == 3 && !lit)
        rc = cuda_status(f64 ? cudaFuncSetAttribute(k_m2l<3, double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                    (int)m2l_smem_bytes<3, double>())
                             : cudaFuncSetAttribute(k_m2l<3, float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                    (int)m2l_smem_bytes<3, float>()));
    if (rc == FMM_OK && !lit && levels >= 2) {
        const std::vector<double> K = build_operators(dim, levels, box);
        if (f64) {
            double* Kd = nullptr;
            rc = alloc(pl, &Kd, K.size());
            pl->K = Kd;
            if (rc == FMM_OK) rc = cuda_status(cudaMemcpy(Kd, K.data(), K.size() * 8, cudaMemcpyHostToDevice));
        } else {
            std::vector<float> Kf(K.begin(), K.end());
            float* Kd = nullptr;
            rc = alloc(pl, &Kd, Kf.size());
            pl->K = Kd;
            if (rc == FMM_OK) rc = cuda_status(cudaMemcpy(Kd, Kf.data(), Kf.size() * 4, cudaMemcpyHostToDevice));
        }
        for (int k = 2; k <= levels; ++k) {
            std::vector<uint32_t> il;
            for (int64_t c = 0; c < ipow(1 << k, dim); ++c) {
                int cc[3];
                morton_dec(dim, (uint32_t)c, cc);
                pl->m2l_pairs += il_cells(dim, k, cc, il);
            }
        }
    }
    if (rc == FMM_OK && lit && levels >= 2) {
        const size_t smem = 4 * (size_t)d * d * sizeof(double);
        cudaError_t e = dim == 2 ? cudaFuncSetAttribute(k_lit_build<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                                 : cudaFuncSetAttribute(k_lit_build<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        rc = cuda_status(e);
        for (int k = 2; k <= levels && rc == FMM_OK; ++k) {
            const int64_t ncell = ipow(1 << k, dim);
            std::vector<int> ps((size_t)ncell + 1, 0), src, tgt;
            std::vector<uint32_t> il;
            for (int64_t c = 0; c < ncell; ++c) {
                int cc[3];
                morton_dec(dim, (uint32_t)c, cc);
                il_cells(dim, k, cc, il);
                for (uint32_t s : il) {
                    src.push_back((int)s);
                    tgt.push_back((int)c);
                }
                ps[(size_t)c + 1] = (int)src.size();
            }
            pl->npairs[k] = (int64_t)src.size();
            pl->m2l_pairs += pl->npairs[k];
            int* dtgt = nullptr;
            rc = alloc(pl, &pl->pair_start[k], ps.size());
            if (rc == FMM_OK) rc = alloc(pl, &pl->pair_src[k], src.size());
            if (rc == FMM_OK) rc = alloc(pl, &pl->B[k], src.size() * (size_t)d * d);
            if (rc == FMM_OK) rc = cuda_status(cudaMalloc(&dtgt, std::max<size_t>(1, tgt.size()) * sizeof(int)));
            if (rc == FMM_OK)
                rc = cuda_status(cudaMemcpy(pl->pair_start[k], ps.data(), ps.size() * 4, cudaMemcpyHostToDevice));
            if (rc == FMM_OK && !src.empty())
                rc = cuda_status(cudaMemcpy(pl->pair_src[k], src.data(), src.size() * 4, cudaMemcpyHostToDevice));
            if (rc == FMM_OK && !tgt.empty())
                rc = cuda_status(cudaMemcpy(dtgt, tgt.data(), tgt.size() * 4, cudaMemcpyHostToDevice));
            if (rc == FMM_OK && !src.empty()) {
                if (dim == 2)
                    k_lit_build<2><<<(unsigned)src.size(), 256, smem>>>(dtgt, pl->pair_src[k], (int64_t)src.size(), k,
                                                                       box, pl->B[k]);
                else
                    k_lit_build<3><<<(unsigned)src.size(), 256, smem>>>(dtgt, pl->pair_src[k], (int64_t)src.size(), k,
                                                                       box, pl->B[k]);
                rc = cuda_status(cudaGetLastError());
                if (rc == FMM_OK) rc = cuda_status(cudaDeviceSynchronize());
            }
            if (dtgt) cudaFree(dtgt);
        }
    }
    if (rc != FMM_OK) {
        plan_free(pl);
        return rc;
    }
    *out = pl;
    return FMM_OK;
}

fmm_status fmm_lag_potential(fmm_lag_plan_t pl, const double* pos, const double* q, int64_t n, double* phi) {
    if (!pl || n < 0 || n > pl->n_max || (n > 0 && (!pos || !q || !phi))) return FMM_ERR_INVALID_ARG;
    if (n == 0) {
        pl->last_n = 0;
        return FMM_OK;
    }
    return pl->dim == 2 ? enqueue<2>(pl, pos, q, n, phi) : enqueue<3>(pl, pos, q, n, phi);
}

fmm_status fmm_lag_sync(fmm_lag_plan_t pl) {
    if (!pl) return FMM_ERR_INVALID_ARG;
    // a call joins its far field's stream back before the evaluation, so its stream is all there is to wait
    // for; after a change of stream the last call's is waited for as well
    fmm_status rc = FMM_OK;
    if (pl->st != pl->last_st) rc = cuda_status(cudaEventSynchronize(pl->ev[4]));
    if (rc == FMM_OK) rc = cuda_status(cudaMemcpyAsync(pl->h_status, pl->status, sizeof(unsigned), cudaMemcpyDeviceToHost, pl->st));
    if (rc == FMM_OK) rc = cuda_status(cudaStreamSynchronize(pl->st));
    if (rc != FMM_OK) return rc;
    const unsigned flags = *pl->h_status;
    if (flags) {
        cudaMemset(pl->status, 0, sizeof(unsigned));
        return (flags & kFlagNonFinite) ? FMM_ERR_NONFINITE : FMM_ERR_OUT_OF_BOX;
    }
    return FMM_OK;
}

fmm_status fmm_lag_stats_get(fmm_lag_plan_t pl, fmm_lag_stats* out) {
    if (!pl || !out) return FMM_ERR_INVALID_ARG;
    std::memset(out, 0, sizeof(*out));
    out->n = pl->last_n;
    out->dim = pl->dim;
    out->levels = pl->levels;
    out->form = pl->form;
    out->workspace_bytes = pl->bytes;
    out->m2l_pairs = pl->m2l_pairs;
    if (pl->last_n == 0) return FMM_OK;
    auto span = [&](int a, int b) {
        float ms = 0.f;
        return cudaEventElapsedTime(&ms, pl->ev[a], pl->ev[b]) == cudaSuccess ? (double)ms : 0.0;
    };
    out->ms_total = span(0, 4);
    out->ms_sort = span(0, 7);
    out->ms_up = span(1, 2);
    out->ms_down = span(2, 3);
    out->ms_eval = span(3, 4);
    out->ms_p2p = span(5, 6);
    unsigned long long pairs[kPairSlots];
    if (cudaMemcpy(pairs, pl->pairs, sizeof(pairs), cudaMemcpyDeviceToHost) != cudaSuccess) return FMM_ERR_CUDA;
    for (unsigned long long v : pairs) out->p2p_pairs += (int64_t)v;
    out->kernel_launches = pl->launches;
    return FMM_OK;
}

fmm_status fmm_lag_set_concurrency(fmm_lag_plan_t pl, int streams) {
    if (!pl || (streams != 1 && streams != 2)) return FMM_ERR_INVALID_ARG;
    pl->serial = streams == 1;
    return FMM_OK;
}

fmm_status fmm_lag_set_stream(fmm_lag_plan_t pl, void* stream) {
    if (!pl) return FMM_ERR_INVALID_ARG;
    pl->st = static_cast<cudaStream_t>(stream);
    return FMM_OK;
}

}  // extern "C"

namespace {
template <int D>
__global__ void k_cells(const uint32_t* __restrict__ key, int64_t n, int32_t* __restrict__ cells) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int c[3];
    morton_dec(D, key[i], c);
    for (int a = 0; a < D; ++a) cells[i * D + a] = c[a];
}
}  // namespace

extern "C" {

fmm_status fmm_lag_cells(fmm_lag_plan_t pl, int32_t* cells) {
    if (!pl || (!cells && pl->last_n > 0)) return FMM_ERR_INVALID_ARG;
    if (pl->last_n == 0) return FMM_OK;
    const unsigned g = (unsigned)((pl->last_n + 255) / 256);
    if (pl->dim == 2) k_cells<2><<<g, 256, 0, pl->st>>>(pl->key, pl->last_n, cells);
    else k_cells<3><<<g, 256, 0, pl->st>>>(pl->key, pl->last_n, cells);
    return cuda_status(cudaGetLastError());
}

fmm_status fmm_lag_direct_targets(int dim, int64_t n, const double* pos, const double* q, int64_t nt,
                                  const int64_t* tgt, double* phi, void* stream) {
    if ((dim != 2 && dim != 3) || n < 0 || nt < 0 || (nt > 0 && (!pos || !q || !tgt || !phi))) return FMM_ERR_INVALID_ARG;
    if (nt == 0) return FMM_OK;
    const unsigned g = (unsigned)((nt + 127) / 128);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (dim == 2) k_direct_targets<2><<<g, 128, 0, st>>>(pos, q, n, tgt, nt, phi);
    else k_direct_targets<3><<<g, 128, 0, st>>>(pos, q, n, tgt, nt, phi);
    return cuda_status(cudaGetLastError());
}

void fmm_lag_plan_destroy(fmm_lag_plan_t pl) {
    if (!pl) return;
    cudaStreamSynchronize(pl->st);
    cudaStreamSynchronize(pl->st2);
    plan_free(pl);
}

}  // extern "C"
