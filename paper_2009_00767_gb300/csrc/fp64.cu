// fp64.cu -- the plain FP64 path of the shift-free FMM on the CUDA cores.
//
// Scaled, box-centred form (w = (z - c) / s for a square of side s and centre c):
//   P2M (U-bar of Sec. 2.2.1, every level straight from the particles, no M2M):
//       M_0 = sum q,   M_m = sum q w^m  (m = 1..p)           -- pure power sums
//   M2L (D-bar-1): b'[t] = sum_{d in IL offsets} T_d M[t + d]  (+ M_0 ln s on b'_0), where the
//       40 scale-free operators T_d fold in Greengard's 2D conversion and the -1/m of the
//       moments, built once per plan in FP64
//   L2P (D-bar-2 by linearity, no L2L): phi_far += Re sum_l b'_l w^l for every level
//   P2P (E-2 of Sec. 2.1): own + eight adjacent finest squares, j != i, r > 0
// Everything is FP64; GB300's FP64 pipe is narrow, so these kernels are DFMA-bound.
#include "fmm_internal.cuh"
#include "fp64_math.cuh"

namespace {

constexpr int kWarpsPerBlock = 4;

// -------------------------------------------------------------------------------- P2M
// One warp per 32 consecutive box-sorted particles; for each level the per-particle power
// sums are written to shared memory and reduced column-wise over runs of equal square key
// (a segmented reduction); each run head adds its sums into the level's grid atomically.
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
k_p2m_f64(const fmm_p64* __restrict__ sp, const uint32_t* __restrict__ skey, int64_t n, int levels, int p,
          double box, FmmLevelPtrs g) {
    extern __shared__ double smem[];
    __shared__ uint32_t bid[kWarpsPerBlock][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ncol = 2 * (p + 1), stride = ncol + 1;
    double* rows = smem + (size_t)warp * 32 * stride;
    const int64_t i = ((int64_t)blockIdx.x * kWarpsPerBlock + warp) * 32 + lane;
    if (((int64_t)blockIdx.x * kWarpsPerBlock + warp) * 32 >= n) return;   // whole warp idle
    const bool valid = i < n;
    fmm_p64 P = valid ? sp[i] : fmm_p64{0.0, 0.0, 0.0, 0.0};
    uint32_t key = valid ? skey[i] : 0u;
    for (int k = 2; k <= levels; ++k) {
        const uint32_t kk = key >> (2 * (levels - k));
        const double s = box / (double)(1 << k);
        const double inv_s = (double)(1 << k) / box;
        const uint32_t bx = fmm_compact2(kk), by = fmm_compact2(kk >> 1);
        const double wx = (P.x - ((double)bx + 0.5) * s) * inv_s;
        const double wy = (P.y - ((double)by + 0.5) * s) * inv_s;
        double* r = rows + lane * stride;
        double pr = P.q, pi = 0.0;   // q w^m
        r[0] = pr;
        r[1] = 0.0;
        for (int m = 1; m <= p; ++m) {
            double nr = pr * wx - pi * wy;
            double ni = pr * wy + pi * wx;
            pr = nr;
            pi = ni;
            r[2 * m] = pr;
            r[2 * m + 1] = pi;
        }
        bid[warp][lane] = valid ? kk : 0xffffffffu;
        __syncwarp();
        const int W = fmm_grid_width(k);
        double* A = reinterpret_cast<double*>(g.A[k]);
        for (int col = lane; col < ncol; col += 32) {
            uint32_t cur = bid[warp][0];
            double run = 0.0;
            for (int rr = 0; rr < 32; ++rr) {
                uint32_t b = bid[warp][rr];
                if (b == 0xffffffffu) break;
                if (b != cur) {
                    size_t cell = (size_t)(fmm_compact2(cur >> 1) + FMM_HALO) * W + fmm_compact2(cur) + FMM_HALO;
                    atomicAdd(A + cell * ncol + col, run);
                    run = 0.0;
                    cur = b;
                }
                run += rows[rr * stride + col];
            }
            size_t cell = (size_t)(fmm_compact2(cur >> 1) + FMM_HALO) * W + fmm_compact2(cur) + FMM_HALO;
            atomicAdd(A + cell * ncol + col, run);
        }
        __syncwarp();
    }
}

// -------------------------------------------------------------------------------- M2L
struct M2LArgs {
    FmmLevelPtrs g;
    const double2* T;              // [49][p+1][p+1], [d][k][l]
    int64_t base[FMM_MAX_LEVELS + 2];   // first flattened target of each level (levels 2..L)
    double ln_s[FMM_MAX_LEVELS + 1];
    int levels, p;
};

// One warp per target square of any level 2..L; lane l accumulates output coefficient l
// (and l + 32 when p >= 32) over the square's interaction list.
__global__ void __launch_bounds__(kWarpsPerBlock * 32) k_m2l_f64(M2LArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t gt = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
    if (gt >= a.base[a.levels + 1]) return;
    int k = 2;
    while (gt >= a.base[k + 1]) ++k;
    const int64_t t = gt - a.base[k];
    const int side = 1 << k;
    const int tx = (int)(t % side), ty = (int)(t / side);
    const int px = tx & 1, py = ty & 1;
    const int p1 = a.p + 1, W = fmm_grid_width(k);
    const double2* A = reinterpret_cast<const double2*>(a.g.A[k]);
    double2* B = reinterpret_cast<double2*>(a.g.B[k]);
    for (int l0 = 0; l0 < p1; l0 += 32) {
        const int l = l0 + lane;
        double accr = 0.0, acci = 0.0;
        for (int dy = -2 - py; dy <= 3 - py; ++dy) {
            const int sy = ty + dy;
            if (sy < 0 || sy >= side) continue;
            for (int dx = -2 - px; dx <= 3 - px; ++dx) {
                const int sx = tx + dx;
                if (sx < 0 || sx >= side) continue;
                if (dx >= -1 && dx <= 1 && dy >= -1 && dy <= 1) continue;
                const double2* src = A + ((size_t)(sy + FMM_HALO) * W + (sx + FMM_HALO)) * p1;
                const double2* Td = a.T + (size_t)((dx + 3) + 7 * (dy + 3)) * p1 * p1;
                if (l < p1) {
                    for (int kk = 0; kk < p1; ++kk) {
                        const double2 m = src[kk];
                        const double2 tt = Td[(size_t)kk * p1 + l];
                        accr = fma(tt.x, m.x, accr);
                        accr = fma(-tt.y, m.y, accr);
                        acci = fma(tt.x, m.y, acci);
                        acci = fma(tt.y, m.x, acci);
                    }
                    if (l == 0) accr = fma(a.ln_s[k], src[0].x, accr);
                }
            }
        }
        if (l < p1) B[(size_t)t * p1 + l] = make_double2(accr, acci);
    }
}

// -------------------------------------------------------------------------------- L2P
// kField: also the far field's gradient, grad phi = (Re f', -Im f') with f'(z) = sum_l l b_l w^(l-1) / s
// (one Horner pass for the expansion and its derivative), per sorted particle into grad_far.
template <bool kField>
__global__ void k_l2p_f64(const fmm_p64* __restrict__ sp, const uint32_t* __restrict__ skey, int64_t n,
                          int levels, int p, double box, FmmLevelPtrs g, double* __restrict__ phi_far,
                          double2* __restrict__ grad_far) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const fmm_p64 P = sp[i];
    const uint32_t key = skey[i];
    const int p1 = p + 1;
    double far = 0.0, gx = 0.0, gy = 0.0;
    for (int k = 2; k <= levels; ++k) {
        const uint32_t kk = key >> (2 * (levels - k));
        const double s = box / (double)(1 << k);
        const double inv_s = (double)(1 << k) / box;
        const uint32_t bx = fmm_compact2(kk), by = fmm_compact2(kk >> 1);
        const double wx = (P.x - ((double)bx + 0.5) * s) * inv_s;
        const double wy = (P.y - ((double)by + 0.5) * s) * inv_s;
        const double2* Bt = reinterpret_cast<const double2*>(g.B[k]) + ((size_t)by * (1u << k) + bx) * p1;
        double2 acc = Bt[p], d = make_double2(0.0, 0.0);
        for (int l = p - 1; l >= 0; --l) {
            const double2 b = Bt[l];
            if (kField) {   // d <- d w + acc before acc moves on: d ends as the derivative
                const double dr = fma(d.x, wx, fma(-d.y, wy, acc.x));
                const double di = fma(d.x, wy, fma(d.y, wx, acc.y));
                d.x = dr;
                d.y = di;
            }
            const double r = fma(acc.x, wx, fma(-acc.y, wy, b.x));
            const double im = fma(acc.x, wy, fma(acc.y, wx, b.y));
            acc.x = r;
            acc.y = im;
        }
        far += acc.x;
        if (kField) {
            gx += d.x * inv_s;
            gy -= d.y * inv_s;
        }
    }
    phi_far[i] = far;
    if (kField) grad_far[i] = make_double2(gx, gy);
}

// -------------------------------------------------------------------------------- P2P + final phi
// The near field by pair symmetry: log r^2 is the same for both particles of a pair, so each pair of
// the own and adjacent squares is evaluated once.  One warp per block of up to FMM_P2P_BLOCK targets of
// a finest square (blk_map, from the sort's scan).  Its pairs are
//   * the block against itself: lane l (a target) meets target (l + s) mod T at step s = 1 .. T / 2;
//   * the block against its "later" sources, 32 at a time, one a lane: the rest of the own square after
//     the block, then the forward neighbours E, NE, N, NW.  At step s lane l meets target (l + s) mod T,
//     so the lanes' targets differ and their sums can live in shared memory (one row of T sums per T
//     lanes) while the source's sum stays in a register.
// A last chunk of at most 16 sources gives each source two lanes that share the steps.  Every result is
// added to the far field with an FP64 atomic; k_finish_f64 then writes phi in input order.
//
// What bounds it: FP64 issue (fp64_math.cuh), 11 instructions a pair: 2 + 2 for r^2, 5 for the logarithm
// and one FMA for each side.  The rolled loop keeps the code small and needs no sums in registers, so
// the pipe always has a warp ready.  2^20 uniform particles, levels 8: 1.93 ms against 15.0 ms for a
// kernel that took every ordered pair with the library's log.
// kField: also grad phi, q (dx, dy) / r^2 to the target and the opposite to the source.
constexpr int kP2PWarps64 = 8;
// With fewer blocks than this, CTAs of two warps instead of eight: 152 SMs x 4 schedulers x 8 warps
// are not filled either way, and the smaller CTAs reach more SMs.
constexpr int64_t kP2PSmall = 4096;
// sums per target of a block of T: 32 / T rows of T for whole chunks (at most 31 + T), and for the
// second lanes of a split chunk 16 / T rows more (at most 15 + T)
constexpr int kP2PRows = 31 + FMM_P2P_BLOCK + 1, kP2PRows2 = 15 + FMM_P2P_BLOCK + 1;

template <bool kField>
struct P2PAcc {
    double phi, gx, gy;
};

template <bool kField>
__device__ __forceinline__ void p2p64_pair(P2PAcc<kField>& a, double (*__restrict__ row)[kField ? 3 : 1], double sx,
                                           double sy, double sq, double tx, double ty, double tq,
                                           const double2* __restrict__ tab) {
    const double dx = tx - sx, dy = ty - sy;
    const double r2 = fma(dx, dx, dy * dy);
    const double lg = fmm_log(r2, tab);
    (*row)[0] = fma(sq, lg, (*row)[0]);
    a.phi = fma(tq, lg, a.phi);
    if constexpr (kField) {
        const bool normal = (unsigned)__double2hiint(r2) - 0x00100000u < 0x7fe00000u;
        const double iv = normal ? fmm_rcp(r2) : (r2 > 0.0 ? 1.0 / r2 : 0.0);
        const double wx = dx * iv, wy = dy * iv;
        (*row)[1] = fma(sq, wx, (*row)[1]);
        (*row)[2] = fma(sq, wy, (*row)[2]);
        a.gx = fma(-tq, wx, a.gx);
        a.gy = fma(-tq, wy, a.gy);
    }
}

template <bool kField>
__device__ __forceinline__ void p2p64_add(double* __restrict__ phi, double2* __restrict__ grad, int64_t i,
                                          const P2PAcc<kField>& a) {
    atomicAdd(phi + i, 0.5 * a.phi);   // log r = log(r^2) / 2
    if constexpr (kField) {
        atomicAdd(&grad[i].x, a.gx);
        atomicAdd(&grad[i].y, a.gy);
    }
}

template <bool kField>
__global__ void __launch_bounds__(kP2PWarps64 * 32)
k_p2p_f64(const fmm_p64* __restrict__ sp, const uint32_t* __restrict__ leaf_start,
          const uint32_t* __restrict__ bstart, const uint2* __restrict__ bmap, uint32_t nleaf, int levels,
          const double2* __restrict__ logtab, double* __restrict__ phi, double2* __restrict__ grad,
          const unsigned int* __restrict__ status, unsigned long long* __restrict__ counters) {
    constexpr int V = kField ? 3 : 1;
    __shared__ double2 tab[kFmmLogEntries];
    __shared__ double tgt[kP2PWarps64][3][FMM_P2P_BLOCK];
    __shared__ double rows[kP2PWarps64][kP2PRows + kP2PRows2][V];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kFmmLogEntries; i += blockDim.x) tab[i] = logtab[i];
    __syncthreads();
    const uint32_t w = blockIdx.x * (blockDim.x >> 5) + warp;
    if (w >= bstart[nleaf]) return;
    if (*(volatile const unsigned int*)status != 0u) return;   // inputs failed the device checks
    const uint2 lt = bmap[w];
    const uint32_t leaf = lt.x, t0 = leaf_start[leaf], t1 = leaf_start[leaf + 1];
    const uint32_t b0 = t0 + (uint32_t)FMM_P2P_BLOCK * lt.y;
    const int T = (int)min((uint32_t)FMM_P2P_BLOCK, t1 - b0);
    // later sources: [b0 + T, t1) of the own square, then the forward neighbours
    const uint2 nb = fmm_forward_neighbour(leaf_start, leaf, levels, lane);
    const uint32_t n_own = t1 - b0 - (uint32_t)T;
    uint32_t end[5], first[5];
    end[0] = n_own;
    first[0] = b0 + (uint32_t)T;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        first[i + 1] = __shfl_sync(0xffffffffu, nb.x, i) - end[i];   // sorted index minus slot
        end[i + 1] = end[i] + __shfl_sync(0xffffffffu, nb.y, i);
    }
    const uint32_t nsrc = end[4];
    if (lane == 0) {
        const unsigned slot = leaf % FMM_COUNTER_SLOTS;
        atomicAdd(&counters[slot], (unsigned long long)T * ((t1 - t0) + 2ull * (nsrc - n_own)) - (unsigned long long)T);
        atomicMax(&counters[FMM_COUNTER_SLOTS + slot], (unsigned long long)(t1 - t0));
    }
    double* const X = tgt[warp][0];
    double* const Y = tgt[warp][1];
    double* const Q = tgt[warp][2];
    auto row = rows[warp];
    fmm_p64 own = fmm_p64{0.0, 0.0, 0.0, 0.0};
    if (lane < T) {
        own = sp[b0 + lane];
        X[lane] = own.x;
        Y[lane] = own.y;
        Q[lane] = own.q;
    }
    for (int i = lane; i < kP2PRows + kP2PRows2; i += 32)
#pragma unroll
        for (int v = 0; v < V; ++v) row[i][v] = 0.0;
    __syncwarp();
    // the block against itself: at the last step of an even T the lanes of the lower half cover all pairs
    P2PAcc<kField> mine = {};
    for (int s = 1; 2 * s <= T; ++s) {
        const int lim = 2 * s == T ? s : T;
        if (lane < lim) {
            const int t = lane + s < T ? lane + s : lane + s - T;
            p2p64_pair<kField>(mine, row + t, own.x, own.y, own.q, X[t], Y[t], Q[t], tab);
        }
        __syncwarp();
    }
    const int lt_row = lane / T;
    for (uint32_t c = 0; c < nsrc; c += 32u) {
        const bool split = nsrc - c <= 16u;   // two lanes a source, half of the targets each
        const int sl = split ? lane & 15 : lane;
        const int half = (T + 1) >> 1;
        const int s0 = split && lane >= 16 ? half : 0, s1 = split && lane < 16 ? half : T;
        const int base = split ? (lane < 16 ? 0 : kP2PRows) + (sl / T) * T : lt_row * T;
        const uint32_t slot = c + (uint32_t)sl;
        const bool has = slot < nsrc;
        P2PAcc<kField> a = {};
        uint32_t idx = 0;
        fmm_p64 S = fmm_p64{0.0, 0.0, 0.0, 0.0};
        if (has) {
            uint32_t f = first[0];
#pragma unroll
            for (int i = 0; i < 4; ++i) f = slot >= end[i] ? first[i + 1] : f;
            idx = slot + f;
            S = sp[idx];
        }
        int t = (sl + s0) % T;
        for (int s = 0; s < (split ? half : T); ++s) {
            if (has && s0 + s < s1) p2p64_pair<kField>(a, row + base + t, S.x, S.y, S.q, X[t], Y[t], Q[t], tab);
            t = t + 1 == T ? 0 : t + 1;
            __syncwarp();
        }
        if (split) {
            a.phi += __shfl_xor_sync(0xffffffffu, a.phi, 16);
            if constexpr (kField) {
                a.gx += __shfl_xor_sync(0xffffffffu, a.gx, 16);
                a.gy += __shfl_xor_sync(0xffffffffu, a.gy, 16);
            }
        }
        if (has && (!split || lane < 16)) p2p64_add<kField>(phi, grad, idx, a);
    }
    if (lane < T) {
        auto sum = [&](int i0, int i1) {
            for (int i = i0 + lane; i < i1; i += T) {
                mine.phi += row[i][0];
                if constexpr (kField) {
                    mine.gx += row[i][1];
                    mine.gy += row[i][2];
                }
            }
        };
        sum(0, kP2PRows);
        sum(kP2PRows, kP2PRows + kP2PRows2);
        p2p64_add<kField>(phi, grad, b0 + lane, mine);
    }
}

// phi (and E = -grad phi) in input order
template <bool kField>
__global__ void k_finish_f64(const fmm_p64* __restrict__ sp, int64_t n, const double* __restrict__ acc,
                             const double2* __restrict__ grad, const unsigned int* __restrict__ status,
                             double* __restrict__ phi, double* __restrict__ field) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (*(volatile const unsigned int*)status != 0u) return;   // inputs failed the device checks
    const int64_t o = (int64_t)sp[i].w;
    phi[o] = acc[i];
    if (kField) {
        field[2 * o] = -grad[i].x;
        field[2 * o + 1] = -grad[i].y;
    }
}

// -------------------------------------------------------------------------------- FP64 direct sum
__global__ void k_direct_f64(int64_t n, const double2* __restrict__ xy, const double* __restrict__ q,
                             const int64_t* __restrict__ targets, double* __restrict__ out) {
    __shared__ double red[32];
    const int64_t it = targets[blockIdx.x];
    const double2 zi = xy[it];
    double acc = 0.0;
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
        const double2 zj = xy[j];
        const double dx = zi.x - zj.x, dy = zi.y - zj.y;
        const double r2 = fma(dx, dx, dy * dy);
        if (j != it && r2 > 0.0) acc = fma(q[j], 0.5 * log(r2), acc);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) out[blockIdx.x] = v;
    }
}

}  // namespace

int fmm_launch_fp64(fmm_plan_s* pl, double* phi, double* field) {
    cudaStream_t st = pl->stream;
    const int64_t n = pl->n;
    const int L = pl->levels, p = pl->p;
    int launches = 0;
    // P2M
    cudaEventRecord(pl->ev[1], st);
    if (L >= 2) {
        for (int k = 2; k <= L; ++k)
            if (cudaMemsetAsync(pl->grids.A[k], 0, pl->a_bytes[k], st) != cudaSuccess) return -1;
        const int64_t warps = (n + 31) / 32;
        const unsigned blocks = (unsigned)((warps + kWarpsPerBlock - 1) / kWarpsPerBlock);
        const size_t shm = sizeof(double) * kWarpsPerBlock * 32 * (2 * (p + 1) + 1);
        if (shm > 48 * 1024 &&
            cudaFuncSetAttribute(k_p2m_f64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm) != cudaSuccess)
            return -1;
        k_p2m_f64<<<blocks, kWarpsPerBlock * 32, shm, st>>>(pl->sorted64, pl->sorted_key, n, L, p, pl->box,
                                                            pl->grids);
        ++launches;
    }
    cudaEventRecord(pl->ev[2], st);
    // M2L
    if (L >= 2) {
        M2LArgs a;
        a.g = pl->grids;
        a.T = pl->T64;
        a.levels = L;
        a.p = p;
        int64_t acc = 0;
        for (int k = 0; k <= FMM_MAX_LEVELS + 1; ++k) a.base[k] = 0;
        for (int k = 2; k <= L; ++k) {
            a.base[k] = acc;
            acc += (int64_t)1 << (2 * k);
        }
        a.base[L + 1] = acc;
        for (int k = 0; k <= FMM_MAX_LEVELS; ++k) a.ln_s[k] = log(pl->box / (double)(1 << k));
        const unsigned blocks = (unsigned)((acc + kWarpsPerBlock - 1) / kWarpsPerBlock);
        k_m2l_f64<<<blocks, kWarpsPerBlock * 32, 0, st>>>(a);
        ++launches;
    }
    cudaEventRecord(pl->ev[3], st);
    // L2P
    {
        const unsigned blocks = (unsigned)((n + 127) / 128);
        if (field)
            k_l2p_f64<true><<<blocks, 128, 0, st>>>(pl->sorted64, pl->sorted_key, n, L, p, pl->box, pl->grids,
                                                    pl->phi_far, pl->near_grad);
        else
            k_l2p_f64<false><<<blocks, 128, 0, st>>>(pl->sorted64, pl->sorted_key, n, L, p, pl->box, pl->grids,
                                                     pl->phi_far, nullptr);
        ++launches;
    }
    cudaEventRecord(pl->ev[4], st);
    // P2P, then phi in input order
    {
        const uint32_t nleaf = 1u << (2 * L);
        const int64_t wmax = (int64_t)nleaf + n / FMM_P2P_BLOCK + 1;
        // few blocks: two warps a CTA, so that they reach more SMs
        const int warps = wmax < kP2PSmall ? 2 : kP2PWarps64;
        const unsigned blocks = (unsigned)((wmax + warps - 1) / warps), nblk = (unsigned)((n + 255) / 256);
        if (field) {
            k_p2p_f64<true><<<blocks, warps * 32, 0, st>>>(pl->sorted64, pl->leaf_start, pl->leaf_bstart, pl->blk_map,
                                                           nleaf, L, pl->logtab, pl->phi_far, pl->near_grad,
                                                           pl->d_status, pl->d_counters);
            k_finish_f64<true><<<nblk, 256, 0, st>>>(pl->sorted64, n, pl->phi_far, pl->near_grad, pl->d_status, phi,
                                                     field);
        } else {
            k_p2p_f64<false><<<blocks, warps * 32, 0, st>>>(pl->sorted64, pl->leaf_start, pl->leaf_bstart,
                                                            pl->blk_map, nleaf, L, pl->logtab, pl->phi_far, nullptr,
                                                            pl->d_status, pl->d_counters);
            k_finish_f64<false><<<nblk, 256, 0, st>>>(pl->sorted64, n, pl->phi_far, nullptr, pl->d_status, phi,
                                                      nullptr);
        }
        launches += 2;
    }
    cudaEventRecord(pl->ev[5], st);
    if (cudaGetLastError() != cudaSuccess) return -1;
    return launches;
}

int fmm_launch_direct_f64(int64_t n, const double* xy, const double* q, int64_t nt, const int64_t* targets,
                          double* phi_t, cudaStream_t stream) {
    if (nt == 0) return 0;
    k_direct_f64<<<(unsigned)nt, 256, 0, stream>>>(n, reinterpret_cast<const double2*>(xy), q, targets, phi_t);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}
