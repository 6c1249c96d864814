// p2p64.cuh -- the FP64 near field of one block of targets, each pair evaluated once for both sides;
// shared by the FP64 path of the complex form (fp64.cu) and the FP64 Lagrange-node forms (lagrange.cu).
//
// One warp takes a block of up to MT targets of a finest cell.  Its pairs are
//   * the block against itself: lane l (a target) meets target (l + s) mod T at step s = 1 .. T / 2;
//   * the block against its "later" sources, 32 at a time, one a lane: up to five ranges of sorted
//     particles (the rest of the own cell after the block, forward neighbours).  At step s lane l meets
//     target (l + s) mod T, so the lanes' targets differ and their sums can live in shared memory (one
//     row of T sums per T lanes) while the source's sum stays in a register.
// A last chunk of at most 16 sources gives each source two lanes that share the steps.
//
// What bounds it: FP64 issue (fp64_math.cuh).  2D: 11 instructions a pair, 4 for r^2, 5 for the
// logarithm, an FMA for each side; 3D: 13.  The rolled loop keeps the code small and needs no sums in
// registers, so the pipe always has a warp ready.
#pragma once

#include "fp64_math.cuh"

// a charge: position and charge (z unused in 2D)
struct P64 {
    double x, y, z, q;
};

template <bool kField>
struct P64Acc {
    double phi, gx, gy;   // 2D phi in units of log r^2; the gradient with kField only
};

// the warp's shared memory: the block's targets, and the sums per target of a block of T: 32 / T rows of T
// for whole chunks (at most 31 + T), for the second lanes of a split chunk 16 / T rows more (at most 15 + T)
template <int D, bool kField, int MT>
struct P64Shared {
    static constexpr int V = kField ? 3 : 1, kRows = 32 + MT, kRows2 = 16 + MT;
    double tgt[D + 1][MT];
    double rows[kRows + kRows2][V];
};

template <int D, bool kField, int MT>
__device__ __forceinline__ void p2p64_pair(P64Acc<kField>& a, P64Shared<D, kField, MT>& sh, int row, int t, P64 s,
                                           const double2* __restrict__ tab) {
    const double dx = sh.tgt[0][t] - s.x, dy = sh.tgt[1][t] - s.y;
    double r2 = fma(dx, dx, dy * dy);
    if constexpr (D == 3) {
        const double dz = sh.tgt[2][t] - s.z;
        r2 = fma(dz, dz, r2);
    }
    double k;   // a coincident pair gives 0
    if constexpr (D == 2) {
        k = fmm_log(r2, tab);
    } else {
        const bool normal = (unsigned)__double2hiint(r2) - 0x00100000u < 0x7fe00000u;
        k = normal ? fmm_rsqrt(r2) : (r2 > 0.0 ? 1.0 / sqrt(r2) : 0.0);
    }
    double* v = sh.rows[row + t];
    v[0] = fma(s.q, k, v[0]);
    const double tq = sh.tgt[D][t];
    a.phi = fma(tq, k, a.phi);
    if constexpr (kField) {
        const double iv = fmm_rcp_range(r2) ? fmm_rcp(r2) : (r2 > 0.0 ? 1.0 / r2 : 0.0);
        const double wx = dx * iv, wy = dy * iv;
        v[1] = fma(s.q, wx, v[1]);
        v[2] = fma(s.q, wy, v[2]);
        a.gx = fma(-tq, wx, a.gx);
        a.gy = fma(-tq, wy, a.gy);
    }
}

// The block's T targets (own: lane's target) against itself (`self`) and the nsrc = end[4] later sources
// (source slot s of range i is the sorted particle s + first[i], end[i] the slots up to range i).
// load(i): the sorted particle i; add(i, acc): its share, called once per later source, and
// add_target(acc) by the lanes below T.
template <int D, bool kField, int MT, class Load, class Add, class AddTarget>
__device__ __forceinline__ void p2p64_block(int lane, int T, bool self, P64 own, const uint32_t (&first)[5],
                                            const uint32_t (&end)[5], P64Shared<D, kField, MT>& sh,
                                            const double2* __restrict__ tab, Load load, Add add, AddTarget add_target) {
    using S = P64Shared<D, kField, MT>;
    __syncwarp();
    if (lane < T) {
        sh.tgt[0][lane] = own.x;
        sh.tgt[1][lane] = own.y;
        if constexpr (D == 3) sh.tgt[2][lane] = own.z;
        sh.tgt[D][lane] = own.q;
    }
    for (int i = lane; i < S::kRows + S::kRows2; i += 32)
#pragma unroll
        for (int v = 0; v < S::V; ++v) sh.rows[i][v] = 0.0;
    __syncwarp();
    P64Acc<kField> mine = {};
    if (self) {   // at the last step of an even T the lanes of the lower half cover all pairs
        for (int s = 1; 2 * s <= T; ++s) {
            if (lane < (2 * s == T ? s : T))
                p2p64_pair<D, kField, MT>(mine, sh, 0, lane + s < T ? lane + s : lane + s - T, own, tab);
            __syncwarp();
        }
    }
    const uint32_t nsrc = end[4];
    for (uint32_t c = 0; c < nsrc; c += 32u) {
        const bool split = nsrc - c <= 16u;   // two lanes a source, half of the targets each
        const int sl = split ? lane & 15 : lane, half = (T + 1) >> 1;
        const int s0 = split && lane >= 16 ? half : 0, s1 = split && lane < 16 ? half : T;
        const int base = (split && lane >= 16 ? S::kRows : 0) + (sl / T) * T;
        const uint32_t slot = c + (uint32_t)sl;
        const bool has = slot < nsrc;
        P64Acc<kField> a = {};
        uint32_t idx = 0;
        P64 src = P64{0.0, 0.0, 0.0, 0.0};
        if (has) {
            uint32_t f = first[0];
#pragma unroll
            for (int i = 0; i < 4; ++i) f = slot >= end[i] ? first[i + 1] : f;
            idx = slot + f;
            src = load(idx);
        }
        int t = (sl + s0) % T;
        for (int s = 0; s < (split ? half : T); ++s) {
            if (has && s0 + s < s1) p2p64_pair<D, kField, MT>(a, sh, base, t, src, tab);
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
        if (has && (!split || lane < 16)) add(idx, a);
    }
    if (lane < T) {
        auto sum = [&](int i0, int i1) {
            for (int i = i0 + lane; i < i1; i += T) {
                mine.phi += sh.rows[i][0];
                if constexpr (kField) {
                    mine.gx += sh.rows[i][1];
                    mine.gy += sh.rows[i][2];
                }
            }
        };
        sum(0, S::kRows);
        sum(S::kRows, S::kRows + S::kRows2);
        add_target(mine);
    }
}
