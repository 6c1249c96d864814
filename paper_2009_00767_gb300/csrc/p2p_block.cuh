// p2p_block.cuh -- the near field (E-2 of Sec. 2.1) of one block of targets, shared by the
// single-system kernel (mixed.cu) and the batched one (batch.cu).
#pragma once

#include "mixed_common.cuh"

namespace {

// Near field (E-2 of Sec. 2.1): every particle of a finest square against the particles of that
// square and its (up to) eight neighbours, in FP32 on square-local coordinates.
//
// One warp takes a block of up to 24 targets of one finest square.  The lanes walk the sources 32 at a
// time (the own square's first, then the four forward neighbours', whose pairs serve both sides, see
// below), each lane holding one source moved into the target square's frame, and keep one FP32 partial
// sum per target in registers; the targets' coordinates are shared-memory broadcasts, two targets per
// load.  The arithmetic of two targets runs in packed FP32x2 instructions, so a pair costs one lg2 on
// the MUFU unit and two to three FP32 slots.
// Coincidence (r^2 = 0: the target itself, duplicate points) only arises within the own square,
// whose chunks test r^2 > 0; a forward neighbour's pair adds 2^-100 to r^2 instead, which keeps the
// logarithm finite should two particles of adjacent squares round to the same FP32 point and
// changes no other pair.  After each run of kP2PRun chunks the partials of each target are
// combined across the warp by a shuffle reduce-scatter (lane t ends with target t's sum) and
// added in float-float, so crowded squares keep their accuracy.
constexpr int kP2PRun = 16;   // chunks of 32 sources summed in FP32 before the float-float add

__device__ __forceinline__ float mufu_lg2(float x) {
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// 1 / x on the MUFU unit (within one ulp)
__device__ __forceinline__ float mufu_rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Sum of v[l & (W - 1)] over the warp's lanes, returned in lane l (v[t] = p[t / 2].x or .y for
// t < 2 NP, 0 beyond).  The low log2(W) lane bits scatter (at the step with mask m a lane keeps
// the half of its live entries whose bit m matches its own and sends the other half to its
// partner), the remaining bits add by butterfly.
template <int W, int NP>
__device__ __forceinline__ float warp_reduce_scatter(const float2 (&p)[NP], int lane) {
    float v[W];
#pragma unroll
    for (int i = 0; i < W; ++i) v[i] = i < 2 * NP ? ((i & 1) ? p[i >> 1].y : p[i >> 1].x) : 0.f;
#pragma unroll
    for (int m = W / 2; m >= 1; m >>= 1) {
        const bool up = (lane & m) != 0;
#pragma unroll
        for (int i = 0; i < m; ++i) {
            const float send = up ? v[i] : v[i + m];
            const float keep = up ? v[i + m] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
    }
    float s = v[0];
#pragma unroll
    for (int m = W; m < 32; m <<= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
    return s;
}

// one own-square chunk: the lane's source (sx, sy, q) against the NP target pairs of the block (the
// coordinates of targets past the block's end are zero and their sums are dropped)
template <int NP>
__device__ __forceinline__ void p2p_chunk(float2 (&part)[NP], const float4* __restrict__ tg, float4 src) {
    const float2 nsx = make_float2(-src.x, -src.x), nsy = make_float2(-src.y, -src.y);
    const float2 q2 = make_float2(src.z, src.z);
#pragma unroll
    for (int tp = 0; tp < NP; ++tp) {
        const float4 t = tg[tp];   // {x of target 2tp, x of 2tp + 1, y of 2tp, y of 2tp + 1}
        const float2 dx = __fadd2_rn(make_float2(t.x, t.y), nsx);
        const float2 dy = __fadd2_rn(make_float2(t.z, t.w), nsy);
        const float2 r2 = __ffma2_rn(dx, dx, __fmul2_rn(dy, dy));
        float2 lg = make_float2(mufu_lg2(r2.x), mufu_lg2(r2.y));
        lg.x = r2.x > 0.f ? lg.x : 0.f;
        lg.y = r2.y > 0.f ? lg.y : 0.f;
        part[tp] = __ffma2_rn(q2, lg, part[tp]);
    }
}

// ---------------------------------------------------------------- symmetric near field
// The pair term log r^2 is symmetric, so each pair of adjacent squares is evaluated once: the
// block's targets take their own square in full (both orders, as above) and only the four
// "forward" neighbours E (+1, 0), NE (+1, +1), N (0, +1) and NW (-1, +1); the other four
// neighbours are covered by the squares that have this one as their forward neighbour.  For a
// forward pair the logarithm serves both sides: q_s L goes to the target (register partials, as
// above) and q_t L to the source, summed over the block's targets in the lane that holds the
// source and added to the source's accumulator with one FP64 atomic per lane and chunk.

// The block's sources: the own square's particles [t0, t0 + n_own) in nch_own chunks, then the
// four forward neighbours' in lane order (seg[b]: sorted index minus slot, frame shift; thr:
// first slot of forward neighbours 1..3).
struct P2PSymSources {
    const float4* sp;
    const int4* seg;
    uint32_t thr[3];
    uint32_t t0, n_own, nch_own, n_fw;

    // source of chunk c for this lane in the target square's frame, and for a forward chunk its
    // sorted index (0xffffffff past the end, where q = 0)
    __device__ __forceinline__ float4 load(uint32_t c, int lane, uint32_t* idx) const {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        *idx = 0xffffffffu;
        if (c < nch_own) {
            const uint32_t s = 32u * c + (uint32_t)lane;
            if (s < n_own) v = sp[t0 + s];
        } else {
            const uint32_t s = 32u * (c - nch_own) + (uint32_t)lane;
            if (s < n_fw) {
                const int b = (s >= thr[0] ? 1 : 0) + (s >= thr[1] ? 1 : 0) + (s >= thr[2] ? 1 : 0);
                const int4 g = seg[b];
                *idx = s + (uint32_t)g.x;
                v = sp[*idx];
                v.x += __int_as_float(g.y);
                v.y += __int_as_float(g.z);
            }
        }
        return v;
    }
};

// one forward chunk: the lane's source against the NP target pairs, both sides; returns the
// source's sum over the block's targets (targets past the block's end have q = 0)
template <int NP>
__device__ __forceinline__ float p2p_chunk_sym(float2 (&part)[NP], const float4* __restrict__ tg,
                                               const float2* __restrict__ tq, float4 src) {
    const float2 nsx = make_float2(-src.x, -src.x), nsy = make_float2(-src.y, -src.y);
    const float2 q2 = make_float2(src.z, src.z);
    const float2 tiny = make_float2(0x1p-100f, 0x1p-100f);
    float2 sacc = make_float2(0.f, 0.f);
#pragma unroll
    for (int tp = 0; tp < NP; ++tp) {
        const float4 t = tg[tp];
        const float2 dx = __fadd2_rn(make_float2(t.x, t.y), nsx);
        const float2 dy = __fadd2_rn(make_float2(t.z, t.w), nsy);
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, tiny));
        const float2 lg = make_float2(mufu_lg2(r2.x), mufu_lg2(r2.y));
        part[tp] = __ffma2_rn(q2, lg, part[tp]);
        sacc = __ffma2_rn(tq[tp], lg, sacc);
    }
    return sacc.x + sacc.y;
}

// the block's own-square and forward-neighbour sums: returns target `lane`'s sum (log2 r^2 units,
// float-float) and adds each forward source's sum to acc[its sorted index]
template <int NP>
__device__ __forceinline__ float2 p2p_block_sym(const P2PSymSources& S, const float4* __restrict__ tg,
                                                const float2* __restrict__ tq, int lane, double* __restrict__ acc) {
    constexpr int W = NP <= 2 ? 4 : (NP <= 4 ? 8 : (NP <= 8 ? 16 : 32));
    const uint32_t nch = S.nch_own + (S.n_fw + 31u) / 32u;
    float2 near = make_float2(0.f, 0.f);
    for (uint32_t r0 = 0; r0 < nch; r0 += kP2PRun) {
        const uint32_t r1 = min(nch, r0 + (uint32_t)kP2PRun);
        float2 part[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) part[i] = make_float2(0.f, 0.f);
        uint32_t idx;
        float4 cur = S.load(r0, lane, &idx);
        for (uint32_t c = r0; c < r1; ++c) {
            uint32_t nidx = idx;
            const float4 nxt = (c + 1 < r1) ? S.load(c + 1, lane, &nidx) : cur;
            if (c < S.nch_own) {
                p2p_chunk<NP>(part, tg, cur);
            } else {
                const float ssum = p2p_chunk_sym<NP>(part, tg, tq, cur);
                if (idx != 0xffffffffu) atomicAdd(acc + idx, fmm_f2d_bits(ssum));
            }
            cur = nxt;
            idx = nidx;
        }
        near = ff_add_f(near, warp_reduce_scatter<W, NP>(part, lane));
    }
    return near;
}

// Symmetric near field of the targets [b0, b0 + T) (T <= 24) of finest square `leaf` with
// particles [t0, t1): target `lane`'s own-square and forward sum (log2 r^2 units, float-float) is
// returned, the forward sources' shares go to acc.  *pairs receives the ordered pairs covered
// (both directions of every forward pair).  tgt (16 float4), tq (16 float2) and seg (4 int4) are
// the warp's shared memory.
__device__ __forceinline__ float2 p2p_near_sym(const float4* __restrict__ sp, const uint32_t* __restrict__ ls,
                                               uint32_t leaf, uint32_t t0, uint32_t t1, uint32_t b0, int T,
                                               int levels, float s_leaf, float4* tgt, float2* tq, int4* seg,
                                               int lane, double* __restrict__ acc, uint32_t* pairs) {
    const uint2 nb = fmm_forward_neighbour(ls, leaf, levels, lane);
    const uint32_t n_own = t1 - t0;
    uint32_t incl = nb.y;
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    const uint32_t excl = incl - nb.y;
    const uint32_t n_fw = __shfl_sync(0xffffffffu, incl, 3);
    if (lane < 4) {
        const float ox = (float)(lane == 3 ? -1 : (lane == 2 ? 0 : 1)) * s_leaf;
        const float oy = (float)(lane == 0 ? 0 : 1) * s_leaf;
        seg[lane] = make_int4((int)(nb.x - excl), __float_as_int(ox), __float_as_int(oy), 0);
    }
    P2PSymSources S;
    S.sp = sp;
    S.seg = seg;
#pragma unroll
    for (int i = 0; i < 3; ++i) S.thr[i] = __shfl_sync(0xffffffffu, excl, i + 1);
    S.t0 = t0;
    S.n_own = n_own;
    S.nch_own = (n_own + 31u) / 32u;
    S.n_fw = n_fw;
    *pairs = (uint32_t)T * (n_own + 2u * n_fw) - (uint32_t)T;
    {
        float x = 0.f, y = 0.f, q = 0.f;
        if (lane < T) {
            const float4 P = sp[b0 + lane];
            x = P.x;
            y = P.y;
            q = P.z;
        }
        float* t = reinterpret_cast<float*>(&tgt[lane >> 1]);
        t[lane & 1] = x;
        t[2 + (lane & 1)] = y;
        reinterpret_cast<float*>(&tq[lane >> 1])[lane & 1] = q;
    }
    __syncwarp();
    switch ((T + 3) >> 2) {
        case 1: return p2p_block_sym<2>(S, tgt, tq, lane, acc);
        case 2: return p2p_block_sym<4>(S, tgt, tq, lane, acc);
        case 3: return p2p_block_sym<6>(S, tgt, tq, lane, acc);
        case 4: return p2p_block_sym<8>(S, tgt, tq, lane, acc);
        case 5: return p2p_block_sym<10>(S, tgt, tq, lane, acc);
        default: return p2p_block_sym<12>(S, tgt, tq, lane, acc);
    }
}

// ---------------------------------------------------------------- crowded squares
// The symmetric near field of squares above FMM_CROWD_POP particles (listed by the sort).  Each lane holds
// two sources, so that a target pair read from shared memory serves four pairs and the independent work
// covers the latencies of the MUFU and of the source loads; and the own square is taken once for both sides
// too: a block of up to kCrowdTargets targets against itself one-sided, then its "later" sources -- the rest
// of the own square after the block, masked at r^2 = 0, and the forward neighbours, whose pairs at r^2 = 0
// count as r^2 = 2^-100 as above.  Own and forward sources share a chunk, so there the term is a source's
// own: 0.5 ms of the call below, where one body masked them all alike (and gave 0 for such a forward pair).
// The sources of a large square's blocks are split into up to kCrowdParts work items, so that a square of
// ten thousand particles does not end as one long tail.
// What bounds it: the MUFU, one lg2 a pair (16 a clock and SM), with the FMA pipe (6 packed instructions
// of two cycles for two pairs) and issue close behind.
// 2^24 clustered particles (32 Gaussians, levels 10, 2.1e11 ordered pairs): 28.5 ms against 33.5 ms for blocks
// of 24 targets, one source a lane and the own square in full; of the difference 3 ms are the own square's
// second half.  24 targets 30.7 ms, 48 targets with one source a lane 29.0 ms, the targets in registers
// instead of shared memory (one source a lane, 16 warps an SM) 41.7 ms, waiting for source loads.
constexpr int kCrowdBlocksPerSm = 4;
struct P2PCrowdShared {
    float4 tg[kCrowdTargets / 2];
    float2 tq[kCrowdTargets / 2];
    int4 seg[5];   // ranges of later sources: {sorted index minus slot, frame shift x, y, first slot past it}
};

// two sources of the lane against the NP target pairs, both sides.  kMask: a source of the own square has
// tiny = 0, so that a pair at r^2 = 0 gives 0; else every tiny is 2^-100.  Returns the sources' sums.
template <bool kMask, int NP>
__device__ __forceinline__ float2 p2p_chunk_sym2(float2 (&part)[NP], const float4* __restrict__ tg,
                                                 const float2* __restrict__ tq, float4 a, float4 b, float tiny_a,
                                                 float tiny_b) {
    const float2 ax = make_float2(-a.x, -a.x), ay = make_float2(-a.y, -a.y), aq = make_float2(a.z, a.z);
    const float2 bx = make_float2(-b.x, -b.x), by = make_float2(-b.y, -b.y), bq = make_float2(b.z, b.z);
    float2 sa = make_float2(0.f, 0.f), sb = make_float2(0.f, 0.f);
    auto log2_r2 = [&](float2 dx, float2 dy, float tiny) {
        if (!kMask) tiny = 0x1p-100f;
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, make_float2(tiny, tiny)));
        float2 lg = make_float2(mufu_lg2(r2.x), mufu_lg2(r2.y));
        if (kMask) {
            lg.x = r2.x > 0.f ? lg.x : 0.f;
            lg.y = r2.y > 0.f ? lg.y : 0.f;
        }
        return lg;
    };
#pragma unroll
    for (int tp = 0; tp < NP; ++tp) {
        const float4 t = tg[tp];
        const float2 q = tq[tp], tx = make_float2(t.x, t.y), ty = make_float2(t.z, t.w);
        const float2 la = log2_r2(__fadd2_rn(tx, ax), __fadd2_rn(ty, ay), tiny_a);
        const float2 lb = log2_r2(__fadd2_rn(tx, bx), __fadd2_rn(ty, by), tiny_b);
        part[tp] = __ffma2_rn(bq, lb, __ffma2_rn(aq, la, part[tp]));
        sa = __ffma2_rn(q, la, sa);
        sb = __ffma2_rn(q, lb, sb);
    }
    return make_float2(sa.x + sa.y, sb.x + sb.y);
}

// The block's targets [b0, b0 + T) against the slots [c0, c1) of its later sources and, with part 0,
// against themselves; slots below n_own belong to the own square.
__device__ __forceinline__ void p2p_crowd_item(const float4* __restrict__ sp, uint32_t b0, int T, bool self,
                                               uint32_t c0, uint32_t c1, uint32_t n_own, const P2PCrowdShared& sh,
                                               int lane, double* __restrict__ acc) {
    constexpr int NP = kCrowdTargets / 2;
    float2 part[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) part[i] = make_float2(0.f, 0.f);
    if (self) p2p_chunk<NP>(part, sh.tg, lane < T ? sp[b0 + lane] : make_float4(0.f, 0.f, 0.f, 0.f));
    const uint32_t e0 = (uint32_t)sh.seg[0].w, e1 = (uint32_t)sh.seg[1].w, e2 = (uint32_t)sh.seg[2].w,
                   e3 = (uint32_t)sh.seg[3].w;
    auto load = [&](uint32_t s, uint32_t* idx) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        *idx = 0xffffffffu;
        if (s < c1) {
            const int4 g = sh.seg[(s >= e0 ? 1 : 0) + (s >= e1 ? 1 : 0) + (s >= e2 ? 1 : 0) + (s >= e3 ? 1 : 0)];
            *idx = s + (uint32_t)g.x;
            v = sp[*idx];
            v.x += __int_as_float(g.y);
            v.y += __int_as_float(g.z);
        }
        return v;
    };
    float2 near = make_float2(0.f, 0.f);
    uint32_t ia, ib;
    float4 a = load(c0 + (uint32_t)lane, &ia), b = load(c0 + 32u + (uint32_t)lane, &ib);
    int run = 1;
#pragma unroll 1
    for (uint32_t c = c0; c < c1; c += 64u) {
        uint32_t na, nb;   // the next sources' loads are in flight meanwhile
        const float4 xa = load(c + 64u + (uint32_t)lane, &na), xb = load(c + 96u + (uint32_t)lane, &nb);
        // a chunk may hold the last of the own square and the first of the forward ones
        const float ta = c + (uint32_t)lane < n_own ? 0.f : 0x1p-100f, tb = c + 32u + (uint32_t)lane < n_own ? 0.f : 0x1p-100f;
        const float2 v = c < n_own ? p2p_chunk_sym2<true, NP>(part, sh.tg, sh.tq, a, b, ta, tb)
                                   : p2p_chunk_sym2<false, NP>(part, sh.tg, sh.tq, a, b, ta, tb);
        if (ia != 0xffffffffu) atomicAdd(acc + ia, fmm_f2d_bits(v.x));
        if (ib != 0xffffffffu) atomicAdd(acc + ib, fmm_f2d_bits(v.y));
        a = xa;
        b = xb;
        ia = na;
        ib = nb;
        run += 2;
        if (run >= kP2PRun) {
            near = ff_add_f(near, warp_reduce_scatter<32>(part, lane));
#pragma unroll
            for (int i = 0; i < NP; ++i) part[i] = make_float2(0.f, 0.f);
            run = 0;
        }
    }
    near = ff_add_f(near, warp_reduce_scatter<32>(part, lane));
    if (lane < T) atomicAdd(acc + b0 + lane, fmm_f2d_bits(near.x) + fmm_f2d_bits(near.y));
}

// Item `item` of the crowded square `leaf` with particles [t0, t1).  Returns the ordered pairs covered (both
// directions of every later pair); sh is the warp's shared memory.
__device__ __forceinline__ unsigned long long p2p_near_crowd(const float4* __restrict__ sp,
                                                             const uint32_t* __restrict__ ls, uint32_t leaf,
                                                             uint32_t t0, uint32_t t1, uint32_t item, int levels,
                                                             float s_leaf, P2PCrowdShared& sh, int lane,
                                                             double* __restrict__ acc) {
    const uint2 nb = fmm_forward_neighbour(ls, leaf, levels, lane);
    uint32_t n_fw = nb.y;
    n_fw += __shfl_xor_sync(0xffffffffu, n_fw, 1);
    n_fw += __shfl_xor_sync(0xffffffffu, n_fw, 2);
    n_fw = __shfl_sync(0xffffffffu, n_fw, 0);
    const uint32_t n = t1 - t0, nblk = fmm_crowd_blocks(n), parts = fmm_crowd_parts(n);
    const uint32_t blk = item / parts, prt = item % parts;
    const uint32_t b0 = t0 + (uint32_t)((unsigned long long)n * blk / nblk);
    const int T = (int)(t0 + (uint32_t)((unsigned long long)n * (blk + 1) / nblk) - b0);
    const uint32_t n_own = t1 - b0 - (uint32_t)T, n_src = n_own + n_fw;
    // parts of whole 64-source chunks
    const uint32_t chunks = (n_src + 63u) / 64u;
    const uint32_t c0 = 64u * (uint32_t)((unsigned long long)chunks * prt / parts);
    const uint32_t c1 = min(n_src, 64u * (uint32_t)((unsigned long long)chunks * (prt + 1) / parts));
    __syncwarp();
    uint32_t slots = n_own;
    if (lane == 0) sh.seg[0] = make_int4((int)(b0 + (uint32_t)T), 0, 0, (int)n_own);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t first = __shfl_sync(0xffffffffu, nb.x, i), cnt = __shfl_sync(0xffffffffu, nb.y, i);
        const float ox = (float)(i == 3 ? -1 : (i == 2 ? 0 : 1)) * s_leaf, oy = (float)(i == 0 ? 0 : 1) * s_leaf;
        if (lane == i)
            sh.seg[1 + i] = make_int4((int)(first - slots), __float_as_int(ox), __float_as_int(oy), (int)(slots + cnt));
        slots += cnt;
    }
    for (int i = lane; i < kCrowdTargets; i += 32) {
        const float4 own = i < T ? sp[b0 + i] : make_float4(0.f, 0.f, 0.f, 0.f);
        float* t = reinterpret_cast<float*>(&sh.tg[i >> 1]);
        t[i & 1] = own.x;
        t[2 + (i & 1)] = own.y;
        reinterpret_cast<float*>(&sh.tq[i >> 1])[i & 1] = own.z;
    }
    __syncwarp();
    const bool self = prt == 0u;
    p2p_crowd_item(sp, b0, T, self, c0, c1, n_own, sh, lane, acc);
    return 2ull * (unsigned long long)T * (c1 > c0 ? c1 - c0 : 0u) + (self ? (unsigned long long)T * (T - 1) : 0ull);
}

// ---------------------------------------------------------------- near field with the field
// The same symmetric scheme with grad phi beside phi: a pair adds q_s log2 r^2 to the target's
// phi and q_s (dx, dy) / r^2 to its gradient (dx, dy = target - source), and for a forward pair q_t
// log2 r^2 and -q_t (dx, dy) / r^2 to the source's; 1 / r^2 comes from the MUFU reciprocal.  A
// coincident own-square pair (r^2 = 0) gives 0 to both.  The field of a close pair goes as 1 / r,
// so FP32 square-local coordinates alone (about 1e-9 of the box) would limit it; each coordinate
// also carries its FP32 rounding residue (written by the sort for field calls), and a pair's
// difference takes the high words (exact for close pairs) plus the residues' difference.
// What bounds it: instruction fetch first.  The loop over the target pairs is unrolled, so each instance for a
// number of pairs is up to 7 kB; one body for both kinds of chunk and four instances instead of six of two
// bodies each keep the warps of an SM in the same code.  200,003 particles in a ring (levels 7): 62 us against 91,
// where a warp waited six issue slots for an instruction (0.1 now); then the waits on registers' latencies, with
// 16 warps an SM.  Uniform particles at level 8, the kernel alone: 56 us at one a square (56 with the six
// instances), 72 at two (72), 85 at four (84), 113 at eight (129), 202 at 16 (353), 528 at 31 (817).
struct NearField {
    float2 phi, gx, gy;   // float-float sums of target `lane`
};

// One chunk: the lane's source against the NP target pairs, the targets' side and, with kSource, the source's (an
// own-square chunk's is dropped).  tiny is 0 in the own square, where a coincident pair gives 0, and 2^-100
// elsewhere.
template <bool kSource, int NP>
__device__ __forceinline__ float3 p2p_chunk_field(float2 (&pp)[NP], float2 (&px)[NP], float2 (&py)[NP],
                                                  const float4* __restrict__ tg, const float4* __restrict__ tl,
                                                  const float2* __restrict__ tq, float4 src, float2 slo, float tiny) {
    const float2 nsx = make_float2(-src.x, -src.x), nsy = make_float2(-src.y, -src.y);
    const float2 nlx = make_float2(-slo.x, -slo.x), nly = make_float2(-slo.y, -slo.y);
    const float2 q2 = make_float2(src.z, src.z), tiny2 = make_float2(tiny, tiny);
    float2 sp = make_float2(0.f, 0.f), sx = make_float2(0.f, 0.f), sy = make_float2(0.f, 0.f);
#pragma unroll
    for (int tp = 0; tp < NP; ++tp) {
        const float4 t = tg[tp], u = tl[tp];
        // the coordinates' high words differ exactly for close pairs; the low words carry the rest
        const float2 dx = __fadd2_rn(__fadd2_rn(make_float2(t.x, t.y), nsx), __fadd2_rn(make_float2(u.x, u.y), nlx));
        const float2 dy = __fadd2_rn(__fadd2_rn(make_float2(t.z, t.w), nsy), __fadd2_rn(make_float2(u.z, u.w), nly));
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, tiny2));
        const bool ax = r2.x > 0.f, ay = r2.y > 0.f;
        const float2 lg = make_float2(ax ? mufu_lg2(r2.x) : 0.f, ay ? mufu_lg2(r2.y) : 0.f);
        const float2 iv = make_float2(ax ? mufu_rcp(r2.x) : 0.f, ay ? mufu_rcp(r2.y) : 0.f);
        const float2 wx = __fmul2_rn(dx, iv), wy = __fmul2_rn(dy, iv);   // (dx, dy) / r^2
        const float2 qt = tq[tp];
        pp[tp] = __ffma2_rn(q2, lg, pp[tp]);
        px[tp] = __ffma2_rn(q2, wx, px[tp]);
        py[tp] = __ffma2_rn(q2, wy, py[tp]);
        if constexpr (!kSource) continue;
        sp = __ffma2_rn(qt, lg, sp);
        sx = __ffma2_rn(qt, wx, sx);
        sy = __ffma2_rn(qt, wy, sy);
    }
    return make_float3(sp.x + sp.y, -(sx.x + sx.y), -(sy.x + sy.y));   // the source's phi and gradient
}

// the source of chunk c with its coordinates' low words (frame shift by TwoSum), for the field
__device__ __forceinline__ float4 load_lo(const P2PSymSources& S, const float2* __restrict__ lo, uint32_t c, int lane,
                                          uint32_t* idx, float2* vlo) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    *vlo = make_float2(0.f, 0.f);
    *idx = 0xffffffffu;
    if (c < S.nch_own) {
        const uint32_t s = 32u * c + (uint32_t)lane;
        if (s < S.n_own) {
            v = S.sp[S.t0 + s];
            *vlo = lo[S.t0 + s];
        }
    } else {
        const uint32_t s = 32u * (c - S.nch_own) + (uint32_t)lane;
        if (s < S.n_fw) {
            const int b = (s >= S.thr[0] ? 1 : 0) + (s >= S.thr[1] ? 1 : 0) + (s >= S.thr[2] ? 1 : 0);
            const int4 g = S.seg[b];
            *idx = s + (uint32_t)g.x;
            v = S.sp[*idx];
            float2 l = lo[*idx];
            const float ox = __int_as_float(g.y), oy = __int_as_float(g.z);
            const float sx = v.x + ox, sy = v.y + oy;
            l.x += two_sum_err(v.x, ox, sx);
            l.y += two_sum_err(v.y, oy, sy);
            v.x = sx;
            v.y = sy;
            *vlo = l;
        }
    }
    return v;
}

// kCrowded: own-square chunks have a body of their own, which leaves out the source's side
template <int NP, bool kCrowded = false>
__device__ __forceinline__ NearField p2p_block_sym_field(const P2PSymSources& S, const float2* __restrict__ lo,
                                                         const float4* __restrict__ tg, const float4* __restrict__ tl,
                                                         const float2* __restrict__ tq, int lane,
                                                         double* __restrict__ acc, double2* __restrict__ accg) {
    constexpr int W = NP <= 2 ? 4 : (NP <= 4 ? 8 : (NP <= 8 ? 16 : 32));
    const uint32_t nch = S.nch_own + (S.n_fw + 31u) / 32u;
    NearField out;
    out.phi = out.gx = out.gy = make_float2(0.f, 0.f);
    for (uint32_t r0 = 0; r0 < nch; r0 += kP2PRun) {
        const uint32_t r1 = min(nch, r0 + (uint32_t)kP2PRun);
        float2 pp[NP], px[NP], py[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) pp[i] = px[i] = py[i] = make_float2(0.f, 0.f);
        uint32_t idx;
        float2 clo;
        float4 cur = load_lo(S, lo, r0, lane, &idx, &clo);
        for (uint32_t c = r0; c < r1; ++c) {
            uint32_t nidx = idx;
            float2 nlo = clo;
            const float4 nxt = (c + 1 < r1) ? load_lo(S, lo, c + 1, lane, &nidx, &nlo) : cur;
            const bool own = c < S.nch_own;
            const float3 sv =
                kCrowded && own ? p2p_chunk_field<false, NP>(pp, px, py, tg, tl, tq, cur, clo, 0.f)
                                : p2p_chunk_field<true, NP>(pp, px, py, tg, tl, tq, cur, clo, own ? 0.f : 0x1p-100f);
            if (idx != 0xffffffffu) {   // a forward source
                atomicAdd(acc + idx, fmm_f2d_bits(sv.x));
                atomicAdd(&accg[idx].x, fmm_f2d_bits(sv.y));
                atomicAdd(&accg[idx].y, fmm_f2d_bits(sv.z));
            }
            cur = nxt;
            idx = nidx;
            clo = nlo;
        }
        out.phi = ff_add_f(out.phi, warp_reduce_scatter<W, NP>(pp, lane));
        out.gx = ff_add_f(out.gx, warp_reduce_scatter<W, NP>(px, lane));
        out.gy = ff_add_f(out.gy, warp_reduce_scatter<W, NP>(py, lane));
    }
    return out;
}

// p2p_near_sym with the gradient: target `lane`'s phi (log2 r^2 units) and grad phi sums; the
// forward sources' shares go to acc and accg.
__device__ __forceinline__ NearField p2p_near_sym_field(const float4* __restrict__ sp, const float2* __restrict__ lo,
                                                        const uint32_t* __restrict__ ls, uint32_t leaf, uint32_t t0,
                                                        uint32_t t1, uint32_t b0, int T, int levels, float s_leaf,
                                                        float4* tgt, float4* tlo, float2* tq, int4* seg, int lane,
                                                        double* __restrict__ acc, double2* __restrict__ accg,
                                                        uint32_t* pairs) {
    const uint2 nb = fmm_forward_neighbour(ls, leaf, levels, lane);
    const uint32_t n_own = t1 - t0;
    uint32_t incl = nb.y;
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    const uint32_t excl = incl - nb.y;
    const uint32_t n_fw = __shfl_sync(0xffffffffu, incl, 3);
    if (lane < 4) {
        const float ox = (float)(lane == 3 ? -1 : (lane == 2 ? 0 : 1)) * s_leaf;
        const float oy = (float)(lane == 0 ? 0 : 1) * s_leaf;
        seg[lane] = make_int4((int)(nb.x - excl), __float_as_int(ox), __float_as_int(oy), 0);
    }
    P2PSymSources S;
    S.sp = sp;
    S.seg = seg;
#pragma unroll
    for (int i = 0; i < 3; ++i) S.thr[i] = __shfl_sync(0xffffffffu, excl, i + 1);
    S.t0 = t0;
    S.n_own = n_own;
    S.nch_own = (n_own + 31u) / 32u;
    S.n_fw = n_fw;
    *pairs = (uint32_t)T * (n_own + 2u * n_fw) - (uint32_t)T;
    {
        float x = 0.f, y = 0.f, q = 0.f;
        float2 l = make_float2(0.f, 0.f);
        if (lane < T) {
            const float4 P = sp[b0 + lane];
            x = P.x;
            y = P.y;
            q = P.z;
            l = lo[b0 + lane];
        }
        float* t = reinterpret_cast<float*>(&tgt[lane >> 1]);
        t[lane & 1] = x;
        t[2 + (lane & 1)] = y;
        float* u = reinterpret_cast<float*>(&tlo[lane >> 1]);
        u[lane & 1] = l.x;
        u[2 + (lane & 1)] = l.y;
        reinterpret_cast<float*>(&tq[lane >> 1])[lane & 1] = q;
    }
    __syncwarp();
    // squares of a few particles fill only the smallest instance: 2^18 particles at one a square of level 9, 206 us
    // against 228 us without it; instances for 12 and 20 targets too would cost 344 us against 202 at 16 a square
    switch ((T + 3) >> 2) {
        case 1: return p2p_block_sym_field<2>(S, lo, tgt, tlo, tq, lane, acc, accg);
        case 2: return p2p_block_sym_field<4>(S, lo, tgt, tlo, tq, lane, acc, accg);
        case 3:
        case 4: return p2p_block_sym_field<8>(S, lo, tgt, tlo, tq, lane, acc, accg);
        default: break;
    }
    // the second body pays where most chunks are the own square's: the call on 60,000 particles in one square
    // 3.32 against 4.49 ms, half of them in it 1.21 against 1.32 ms
    return n_own > (uint32_t)FMM_CROWD_POP ? p2p_block_sym_field<12, true>(S, lo, tgt, tlo, tq, lane, acc, accg)
                                           : p2p_block_sym_field<12>(S, lo, tgt, tlo, tq, lane, acc, accg);
}

// phi = far + near x ln2 / 2 (the float-float factor turns sum q log2 r^2 into sum q ln r)
__device__ __forceinline__ double p2p_phi(float2 far, float2 near) {
    const float2 v = ff_add(far, ff_mul(near, make_float2(0.3465736f, -9.523271e-10f)));
    return fmm_f2d_bits(v.x) + fmm_f2d_bits(v.y);
}

}  // namespace
