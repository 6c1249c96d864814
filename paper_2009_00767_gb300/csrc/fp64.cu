// fp64.cu -- the plain FP64 path of the shift-free FMM on the CUDA cores.
//
// Scaled, box-centred form (w = (z - c) / s for a square of side s and centre c):
//   P2M (U-bar-1 of Sec. 2.2.1): the finest squares' moments from the particles,
//       M_0 = sum q,   M_m = sum q w^m  (m = 1..p)           -- pure power sums
//   M2M (U-bar-2): each coarser square's from its four children, re-expanded about its centre
//   M2L (D-bar-1): b'[t] = sum_{d in IL offsets} T_d M[t + d]  (+ M_0 (log|d| + ln s) on b'_0), where
//       T_d folds in Greengard's 2D conversion and the -1/m of the moments
//   L2L (D-bar-2): each square's local expansion re-expanded about its children's centres and added
//       to theirs, so that the finest squares hold the sum of all levels
//   L2P: phi_far = Re sum_l b'_l w^l of the particle's finest square
//   P2P (E-2 of Sec. 2.1): own + eight adjacent finest squares, r > 0
// M2M and L2L are finite sums, exact for truncated expansions.  Everything is FP64; GB300's FP64 pipe is
// narrow (one warp instruction per SM in about 19 clocks), so each kernel is bound by its FP64
// instructions and is written to need few of them.
//
// The translations factor into diagonal powers and one real matrix, T_d[k][l] = d^-l R[k][l] d^-k, and a
// quarter turn of d only multiplies by powers of i.  So the squares at d, i d, -d and -i d need one product
// with the real matrix between them: with G_s[k] = d^-k sum_r i^(-r s) M_k(square at i^r d),
//     b'_l += d^-l sum_k R[k][l] G_((k + l) mod 4)[k],
// 2 instead of 16 FP64 instructions per (k, l) for four squares.  M2M and L2L, whose four children sit a
// quarter turn apart, have the same form with binomials for R.
#include "fmm_internal.cuh"
#include "p2p64.cuh"

namespace {

constexpr int kWarpsPerBlock = 4;

// -------------------------------------------------------------------------------- P2M
// One warp per 32 consecutive box-sorted particles: the particles' powers are written to shared memory
// and reduced column-wise over runs of equal square key (a segmented reduction); each run head adds its
// sums into the finest level's grid atomically.
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
k_p2m_f64(const fmm_p64* __restrict__ sp, const uint32_t* __restrict__ skey, int64_t n, int levels, int p,
          double s, double inv_s, double* __restrict__ A) {
    extern __shared__ double smem[];
    __shared__ uint32_t bid[kWarpsPerBlock][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ncol = 2 * (p + 1), stride = ncol + 1;
    double* rows = smem + (size_t)warp * 32 * stride;
    const int64_t i = ((int64_t)blockIdx.x * kWarpsPerBlock + warp) * 32 + lane;
    if (((int64_t)blockIdx.x * kWarpsPerBlock + warp) * 32 >= n) return;   // whole warp idle
    const bool valid = i < n;
    fmm_p64 P = valid ? sp[i] : fmm_p64{0.0, 0.0, 0.0, 0.0};
    const uint32_t key = valid ? skey[i] : 0u;
    const double wx = (P.x - ((double)fmm_compact2(key) + 0.5) * s) * inv_s;
    const double wy = (P.y - ((double)fmm_compact2(key >> 1) + 0.5) * s) * inv_s;
    double* r = rows + lane * stride;
    double pr = P.q, pi = 0.0;   // q w^m
    r[0] = pr;
    r[1] = 0.0;
    for (int m = 1; m <= p; ++m) {
        const double nr = fma(pr, wx, -(pi * wy));
        const double ni = fma(pr, wy, pi * wx);
        pr = nr;
        pi = ni;
        r[2 * m] = pr;
        r[2 * m + 1] = pi;
    }
    bid[warp][lane] = valid ? key : 0xffffffffu;
    __syncwarp();
    const int W = fmm_grid_width(levels);
    for (int col = lane; col < ncol; col += 32) {
        uint32_t cur = bid[warp][0];
        double run = 0.0;
        for (int rr = 0; rr < 32; ++rr) {
            const uint32_t b = bid[warp][rr];
            if (b == 0xffffffffu) break;
            if (b != cur) {
                const size_t cell = (size_t)(fmm_compact2(cur >> 1) + FMM_HALO) * W + fmm_compact2(cur) + FMM_HALO;
                atomicAdd(A + cell * ncol + col, run);
                run = 0.0;
                cur = b;
            }
            run += rows[rr * stride + col];
        }
        const size_t cell = (size_t)(fmm_compact2(cur >> 1) + FMM_HALO) * W + fmm_compact2(cur) + FMM_HALO;
        atomicAdd(A + cell * ncol + col, run);
    }
}

// -------------------------------------------------------------------------------- M2M, M2L, L2L
// Work split of the three: a CTA takes as many squares as its threads hold whole coefficient rows
// (blockDim.x / (p + 1)); a thread is one (square, coefficient), first of the input, then of the output.
// At p = 20 that fills 126 of 128 threads, where a warp a square would fill 21 of 32.
constexpr int kFarThreads = 128, kFarThreadsSmall = 64;

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
// a i^r
__device__ __forceinline__ double2 crot(double2 a, int r) {
    const double2 b = (r & 1) ? make_double2(-a.y, a.x) : a;
    return (r & 2) ? make_double2(-b.x, -b.y) : b;
}
// (1 - i)^j and ((1 + i) / 4)^m, exact
__device__ __forceinline__ double2 pow_1mi(int j) {
    const int h = j >> 1;   // (1 - i)^2 = -2 i
    const double v = ldexp(1.0, h);
    return crot((j & 1) ? make_double2(v, -v) : make_double2(v, 0.0), -h);
}
__device__ __forceinline__ double2 pow_delta(int m) {
    const int h = m >> 1;   // (1 + i)^2 = 2 i
    const double v = ldexp(1.0, h - 2 * m);
    return crot((m & 1) ? make_double2(v, v) : make_double2(v, 0.0), h);
}
// grid position of the child r quarter turns from the (+, +) one: its centre is at i^r (1 + i) / 4
__device__ __forceinline__ int child_x(int r) { return r == 0 || r == 3; }
__device__ __forceinline__ int child_y(int r) { return r < 2; }

// sum_k Rm[k][l] G[(l + sgn k) mod 4][k] over k, G as [4][p1]; k in runs of four, so that the row of G
// is known within a run
__device__ __forceinline__ double2 far_matvec(const double* __restrict__ col, int stride, const double2* __restrict__ G,
                                              int p1, int l, int sgn) {
    double2 u = make_double2(0.0, 0.0), v = make_double2(0.0, 0.0);
    const double2* g0 = G + (l & 3) * p1;
    const double2* g1 = G + ((l + sgn) & 3) * p1;
    const double2* g2 = G + ((l + 2) & 3) * p1;
    const double2* g3 = G + ((l - sgn) & 3) * p1;
    int k = 0;
    for (; k + 3 < p1; k += 4) {
        const double r0 = col[k * stride], r1 = col[(k + 1) * stride], r2 = col[(k + 2) * stride],
                     r3 = col[(k + 3) * stride];
        const double2 a = g0[k], b = g1[k + 1], c = g2[k + 2], d = g3[k + 3];
        u.x = fma(r0, a.x, u.x);
        u.y = fma(r0, a.y, u.y);
        v.x = fma(r1, b.x, v.x);
        v.y = fma(r1, b.y, v.y);
        u.x = fma(r2, c.x, u.x);
        u.y = fma(r2, c.y, u.y);
        v.x = fma(r3, d.x, v.x);
        v.y = fma(r3, d.y, v.y);
    }
    for (; k < p1; ++k) {
        const double r = col[k * stride];
        const double2 a = G[((l + sgn * k) & 3) * p1 + k];
        u.x = fma(r, a.x, u.x);
        u.y = fma(r, a.y, u.y);
    }
    return cadd(u, v);
}

// Upward pass: level k's moments from level k + 1's (w = w' / 2 + i^r (1 + i) / 4),
//     M_m = ((1+i)/4)^m sum_{j <= m} C(m, j) G_((m - j) mod 4)[j],   G_s[j] = (1-i)^j sum_r i^(r s) M_j(child r).
__global__ void __launch_bounds__(kFarThreads)
k_m2m_f64(const double2* __restrict__ child, double2* __restrict__ parent, const double* __restrict__ binom, int k,
          int p1) {
    extern __shared__ __align__(16) double smem[];
    double* C = smem;                                                  // [m][j] = C(m, j)
    double2* G = reinterpret_cast<double2*>(smem + ((p1 * p1 + 1) & ~1));   // [square][4][p1]
    const int per = blockDim.x / p1, tl = threadIdx.x / p1, c = threadIdx.x % p1;
    const uint32_t side = 1u << k, par = blockIdx.x * per + tl;
    const bool live = tl < per && par < side * side;
    const uint32_t px = par % side, py = par / side;
    for (int i = threadIdx.x; i < p1 * p1; i += blockDim.x) C[i] = binom[i];
    if (live) {
        const int W = fmm_grid_width(k + 1);
        double2 z[4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
            z[r] = child[((size_t)(2 * py + child_y(r) + FMM_HALO) * W + 2 * px + child_x(r) + FMM_HALO) * p1 + c];
        const double2 a0 = cadd(z[0], z[2]), a1 = csub(z[0], z[2]), b0 = cadd(z[1], z[3]), b1 = csub(z[1], z[3]);
        const double2 f = pow_1mi(c);
        double2* g = G + (size_t)tl * 4 * p1 + c;
        g[0] = cmul(f, cadd(a0, b0));
        g[p1] = cmul(f, cadd(a1, crot(b1, 1)));
        g[2 * p1] = cmul(f, csub(a0, b0));
        g[3 * p1] = cmul(f, csub(a1, crot(b1, 1)));
    }
    __syncthreads();
    if (!live) return;
    const double2 u = far_matvec(C + c * p1, 1, G + (size_t)tl * 4 * p1, p1, c, -1);
    parent[((size_t)(py + FMM_HALO) * fmm_grid_width(k) + px + FMM_HALO) * p1 + c] = cmul(pow_delta(c), u);
}

// Downward pass: level k's local expansions added to its children's,
//     b'_l(child r) += (1-i)^l i^(-r l) sum_q i^(r q) sum_{m = q mod 4} C(m, l) ((1+i)/4)^m b_m.
__global__ void __launch_bounds__(kFarThreads)
k_l2l_f64(const double2* __restrict__ parent, double2* __restrict__ child, const double* __restrict__ binom, int k,
          int p1) {
    extern __shared__ __align__(16) double smem[];
    double* C = smem;
    double2* H = reinterpret_cast<double2*>(smem + ((p1 * p1 + 1) & ~1));   // [square][p1]
    const int per = blockDim.x / p1, tl = threadIdx.x / p1, c = threadIdx.x % p1;
    const uint32_t side = 1u << k, par = blockIdx.x * per + tl;
    const bool live = tl < per && par < side * side;
    const uint32_t px = par % side, py = par / side;
    for (int i = threadIdx.x; i < p1 * p1; i += blockDim.x) C[i] = binom[i];
    if (live) H[tl * p1 + c] = cmul(pow_delta(c), parent[(size_t)par * p1 + c]);
    __syncthreads();
    if (!live) return;
    const double2* h = H + tl * p1;
    double2 S[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) S[q] = make_double2(0.0, 0.0);
    for (int m0 = 0; m0 < p1; m0 += 4)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (m0 + q < p1) {
                const double r = C[(m0 + q) * p1 + c];   // 0 for m < l
                S[q].x = fma(r, h[m0 + q].x, S[q].x);
                S[q].y = fma(r, h[m0 + q].y, S[q].y);
            }
    const double2 a0 = cadd(S[0], S[2]), a1 = csub(S[0], S[2]), b0 = cadd(S[1], S[3]), b1 = csub(S[1], S[3]);
    const double2 v[4] = {cadd(a0, b0), cadd(a1, crot(b1, 1)), csub(a0, b0), csub(a1, crot(b1, 1))};
    const double2 f = pow_1mi(c);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        double2* b = child + ((size_t)(2 * py + child_y(r)) * (2 * side) + 2 * px + child_x(r)) * p1 + c;
        *b = cadd(*b, crot(cmul(f, v[r]), -r * c));
    }
}

struct M2LArgs {
    FmmLevelPtrs g;
    const double* R;               // [k][l]
    const double2* dpow;           // [orbit][k]: d^-k
    int64_t base[FMM_MAX_LEVELS + 2];   // first CTA of each level (levels 2..L)
    double ln_s[FMM_MAX_LEVELS + 1];
    double ln_d[kFmmOrbits];
    int levels, p;
};

// The offsets of every interaction list as orbits of quarter turns.  Orbits 0..3 are whole in every list.
// Orbits 4..8 (3, b) have two members in a list, which depend on the target's parity: x = +-3 at r = 2 px,
// y = +-3 at r = 1 + 2 py.  Orbit 9 (3, 3) has one.  Ten products with R stand for 27 squares.
// A CTA's targets share the parity class.  The next orbit's moments are loaded before the products of
// the current one; G has two buffers, so an orbit costs one barrier.
// 2^20 uniform particles, levels 8, p = 20: 2.44 ms against 10.14 ms for a product per square with the
// complex operator, lanes over l.
__global__ void __launch_bounds__(kFarThreads) k_m2l_f64(M2LArgs a) {
    extern __shared__ __align__(16) double smem[];
    const int p1 = a.p + 1, per = blockDim.x / p1, tl = threadIdx.x / p1, c = threadIdx.x % p1;
    double* R = smem;
    double2* D = reinterpret_cast<double2*>(smem + ((p1 * p1 + 1) & ~1));   // [orbit][p1]
    double2* Gb = D + kFmmOrbits * p1;                                     // [2][square][4][p1]
    for (int i = threadIdx.x; i < p1 * p1; i += blockDim.x) R[i] = a.R[i];
    for (int i = threadIdx.x; i < kFmmOrbits * p1; i += blockDim.x) D[i] = a.dpow[i];
    int k = 2;
    while ((int64_t)blockIdx.x >= a.base[k + 1]) ++k;
    const int w2 = 1 << (k - 1), W = fmm_grid_width(k);
    const int groups = (w2 * w2 + per - 1) / per;
    const int rel = (int)((int64_t)blockIdx.x - a.base[k]);
    const int cls = rel / groups, u = (rel % groups) * per + tl;
    const int px = cls & 1, py = cls >> 1;
    const bool live = tl < per && u < w2 * w2;
    const int tx = 2 * (live ? u % w2 : 0) + px, ty = 2 * (live ? u / w2 : 0) + py;
    // squares outside the domain are the grid's zero halo
    const double2* src = reinterpret_cast<const double2*>(a.g.A[k]) +
                         ((size_t)(ty + FMM_HALO) * W + tx + FMM_HALO) * p1 + c;
    auto at = [&](int dx, int dy) { return src[(dy * W + dx) * p1]; };
    double2 z[4];
    auto load = [&](int o) {
        const int dx = fmm_orbit_x(o), dy = fmm_orbit_y(o);
        if (o < 4) {
            z[0] = at(dx, dy);
            z[1] = at(-dy, dx);
            z[2] = at(-dx, -dy);
            z[3] = at(dy, -dx);
        } else if (o < 9) {
            z[0] = px ? at(-dx, -dy) : at(dx, dy);
            z[1] = py ? at(dy, -dx) : at(-dy, dx);
        } else {
            z[0] = at(px ? -3 : 3, py ? -3 : 3);
        }
    };
    double2 b = make_double2(0.0, 0.0);
    double mono = 0.0;
    if (live) load(0);
    __syncthreads();
#pragma unroll 1
    for (int o = 0; o < kFmmOrbits; ++o) {
        double2* G = Gb + ((size_t)(o & 1) * per + tl) * 4 * p1;
        double2 f = make_double2(0.0, 0.0);
        if (live) {
            f = D[o * p1 + c];
            double2* g = G + c;
            double m0;   // the orbit's charge (thread c = 0)
            if (o < 4) {
                const double2 a0 = cadd(z[0], z[2]), a1 = csub(z[0], z[2]), b0 = cadd(z[1], z[3]),
                              b1 = crot(csub(z[1], z[3]), 1);
                const double2 t = cadd(a0, b0);
                m0 = t.x;
                g[0] = cmul(f, t);
                g[p1] = cmul(f, csub(a1, b1));
                g[2 * p1] = cmul(f, csub(a0, b0));
                g[3 * p1] = cmul(f, cadd(a1, b1));
            } else if (o < 9) {
                m0 = z[0].x + z[1].x;
                const double2 x = cmul(f, z[0]), y = cmul(f, z[1]);
                const double2 xs = px ? make_double2(-x.x, -x.y) : x, yi = crot(y, py ? 3 : 1);
                g[0] = cadd(x, y);
                g[p1] = csub(xs, yi);
                g[2 * p1] = csub(x, y);
                g[3 * p1] = cadd(xs, yi);
            } else {
                m0 = z[0].x;
                const int r = px ? (py ? 2 : 1) : (py ? 3 : 0);
                const double2 x = cmul(f, z[0]);
                g[0] = x;
                g[p1] = crot(x, -r);
                g[2 * p1] = crot(x, -2 * r);
                g[3 * p1] = crot(x, -3 * r);
            }
            if (c == 0) mono = fma(m0, a.ln_d[o] + a.ln_s[k], mono);
            if (o + 1 < kFmmOrbits) load(o + 1);
        }
        __syncthreads();
        if (live) b = cadd(b, cmul(f, far_matvec(R + c, p1, G, p1, c, 1)));
    }
    if (!live) return;
    if (c == 0) b.x += mono;
    reinterpret_cast<double2*>(a.g.B[k])[((size_t)ty * (1u << k) + tx) * p1 + c] = b;
}

// -------------------------------------------------------------------------------- L2P
// The finest square's local expansion at each particle by Horner's rule, added to the near field (near, grad)
// and written in input order, unless the inputs failed the device checks.
// kField: also the far field's gradient, grad phi = (Re f', -Im f') with f'(z) = sum_l l b_l w^(l-1) / s
// (one Horner pass for the expansion and its derivative), and E = -grad phi.
template <bool kField>
__global__ void k_l2p_f64(const fmm_p64* __restrict__ sp, const uint32_t* __restrict__ skey, int64_t n,
                          int levels, int p, double s, double inv_s, const double2* __restrict__ B,
                          const double* __restrict__ near, const double2* __restrict__ grad,
                          const unsigned int* __restrict__ status, double* __restrict__ phi, double* __restrict__ field) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (*(volatile const unsigned int*)status != 0u) return;
    const fmm_p64 P = sp[i];
    double2 acc = make_double2(0.0, 0.0), d = make_double2(0.0, 0.0);
    if (levels >= 2) {   // else no far field
        const uint32_t key = skey[i];
        const uint32_t bx = fmm_compact2(key), by = fmm_compact2(key >> 1);
        const double wx = (P.x - ((double)bx + 0.5) * s) * inv_s;
        const double wy = (P.y - ((double)by + 0.5) * s) * inv_s;
        const double2* Bt = B + ((size_t)by * (1u << levels) + bx) * (p + 1);
        acc = Bt[p];
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
    }
    const int64_t o = (int64_t)P.w;
    phi[o] = acc.x + near[i];
    if (kField) {
        const double2 g = grad[i];
        field[2 * o] = -(d.x * inv_s + g.x);
        field[2 * o + 1] = d.y * inv_s - g.y;
    }
}

// -------------------------------------------------------------------------------- P2P
// The near field, each pair of the own and adjacent squares once (p2p64.cuh): one warp per block of up to
// FMM_P2P_BLOCK targets of a finest square (blk_map, from the sort's scan), whose later sources are the
// rest of the own square and the forward neighbours E, NE, N, NW.  Every result is added to the particle's
// sum with an FP64 atomic.
// 2^20 uniform particles, levels 8: 1.93 ms against 15.0 ms for a kernel that took every ordered pair with
// the library's log.
// kField: also grad phi, q (dx, dy) / r^2 to the target and the opposite to the source.
constexpr int kP2PWarps64 = 8;
// With fewer blocks than this, CTAs of two warps instead of eight: 152 SMs x 4 schedulers x 8 warps
// are not filled either way, and the smaller CTAs reach more SMs.  The kernel alone, two against eight warps:
// 427 blocks (4,096 particles, levels 4) 47 and 53 us, 898 (20,000, levels 3) 737 and 917, 2,757 (60,000, levels
// 4) 1.48 and 1.87 ms; above the line the gain fades: 6,827 (65,536, levels 6) 154 and 168 us, 27,307 (2^18,
// levels 7) 494 and 520.
constexpr int64_t kP2PSmall = 4096;

template <bool kField>
__device__ __forceinline__ void p2p64_add(double* __restrict__ phi, double2* __restrict__ grad, int64_t i,
                                          const P64Acc<kField>& a) {
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
    __shared__ double2 tab[kFmmLogEntries];
    __shared__ P64Shared<2, kField, FMM_P2P_BLOCK> sh[kP2PWarps64];
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
    const uint2 nb = fmm_forward_neighbour(leaf_start, leaf, levels, lane);
    uint32_t end[5], first[5];   // later sources: sorted index minus slot, slots up to the range's end
    first[0] = b0 + (uint32_t)T;
    end[0] = t1 - first[0];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        first[i + 1] = __shfl_sync(0xffffffffu, nb.x, i) - end[i];
        end[i + 1] = end[i] + __shfl_sync(0xffffffffu, nb.y, i);
    }
    if (lane == 0) {
        const unsigned slot = leaf % FMM_COUNTER_SLOTS;
        atomicAdd(&counters[slot], (unsigned long long)T * ((t1 - t0) + 2ull * (end[4] - end[0])) - (unsigned long long)T);
        atomicMax(&counters[FMM_COUNTER_SLOTS + slot], (unsigned long long)(t1 - t0));
    }
    auto load = [&](uint32_t i) {
        const fmm_p64 v = sp[i];
        return P64{v.x, v.y, 0.0, v.q};
    };
    p2p64_block<2, kField, FMM_P2P_BLOCK>(
        lane, T, true, load(b0 + min(lane, T - 1)), first, end, sh[warp], tab, load,
        [&](uint32_t i, const P64Acc<kField>& a) { p2p64_add<kField>(phi, grad, i, a); },
        [&](const P64Acc<kField>& a) { p2p64_add<kField>(phi, grad, b0 + lane, a); });
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
    // The far field runs on the plan's own stream, at the device's highest priority, beside the near field on
    // the caller's.  Both are bound by the FP64 pipe; what overlaps is the chain of small launches of the
    // coarse levels, which leaves most of the chip idle, and with few particles all of it: 4,096 particles
    // (levels 4, p = 16) 174 -> 135 us, 2^20 (levels 8, p = 20) 5.17 -> 5.05 ms.
    // In turn on the caller's stream with fmm_set_concurrency(plan, 1) and without a plan (no stream2).
    const bool owned = pl->stream2 != nullptr, two = owned && !pl->serial;
    cudaStream_t near_st = pl->stream, st = two ? pl->stream2 : pl->stream;
    const int64_t n = pl->n;
    const int L = pl->levels, p = pl->p, p1 = p + 1;
    const double s = pl->box / (double)(1 << L), inv_s = (double)(1 << L) / pl->box;
    // a grid of (2^k)^2 squares in CTAs of whole rows: few squares take smaller CTAs, to reach more SMs.  M2L with
    // 64 and 128 threads: levels 4, p = 16 34.3 and 35.0 us, levels 5, p = 12 39.1 and 47.0; levels 6, p = 16 158
    // and 145, levels 7 557 and 487 (the real matrix is copied to shared memory for fewer squares).
    const int threads = L <= 5 ? kFarThreadsSmall : kFarThreads, per = threads / p1;
    const int tab = (p1 * p1 + 1) & ~1;   // doubles of a real matrix in shared memory, 16-byte aligned
    const double* R = pl->ftab;
    const double* binom = R + tab;
    const double2* dpow = reinterpret_cast<const double2*>(binom + tab);
    const size_t shm_up = sizeof(double) * tab + sizeof(double2) * 4 * p1 * per;
    const size_t shm_down = sizeof(double) * tab + sizeof(double2) * p1 * per;
    const size_t shm_m2l = sizeof(double) * tab + sizeof(double2) * (kFmmOrbits * p1 + 2 * 4 * p1 * per);
    int launches = 0;
    // P2M of the finest level (its grid starts at zero), then the upward pass
    cudaEventRecord(pl->ev[1], near_st);
    // the finest grid is free from the call's start on (the previous call's L2P ended there)
    if (two && cudaStreamWaitEvent(st, pl->ev[0], 0) != cudaSuccess) return -1;
    if (L >= 2 && cudaMemsetAsync(pl->grids.A[L], 0, pl->a_bytes[L], st) != cudaSuccess) return -1;
    if (two && cudaStreamWaitEvent(st, pl->ev[1], 0) != cudaSuccess) return -1;
    if (L >= 2) {
        const int64_t warps = (n + 31) / 32;
        const unsigned blocks = (unsigned)((warps + kWarpsPerBlock - 1) / kWarpsPerBlock);
        const size_t shm = sizeof(double) * kWarpsPerBlock * 32 * (2 * p1 + 1);
        if (shm > 48 * 1024 &&
            cudaFuncSetAttribute(k_p2m_f64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm) != cudaSuccess)
            return -1;
        k_p2m_f64<<<blocks, kWarpsPerBlock * 32, shm, st>>>(pl->sorted64, pl->sorted_key, n, L, p, s, inv_s,
                                                            static_cast<double*>(pl->grids.A[L]));
        ++launches;
        for (int k = L - 1; k >= 2; --k) {
            k_m2m_f64<<<((1 << (2 * k)) + per - 1) / per, threads, shm_up, st>>>(
                static_cast<const double2*>(pl->grids.A[k + 1]), static_cast<double2*>(pl->grids.A[k]), binom, k, p1);
            ++launches;
        }
    }
    cudaEventRecord(pl->ev[2], st);
    // M2L of every level
    if (L >= 2) {
        M2LArgs a;
        a.g = pl->grids;
        a.R = R;
        a.dpow = dpow;
        a.levels = L;
        a.p = p;
        int64_t acc = 0;
        for (int k = 0; k <= FMM_MAX_LEVELS + 1; ++k) a.base[k] = 0;
        for (int k = 2; k <= L; ++k) {
            a.base[k] = acc;
            acc += 4 * ((((int64_t)1 << (2 * (k - 1))) + per - 1) / per);
        }
        a.base[L + 1] = acc;
        for (int k = 0; k <= FMM_MAX_LEVELS; ++k) a.ln_s[k] = log(pl->box / (double)(1 << k));
        for (int o = 0; o < kFmmOrbits; ++o) {
            const double x = fmm_orbit_x(o), y = fmm_orbit_y(o);
            a.ln_d[o] = 0.5 * log(x * x + y * y);
        }
        k_m2l_f64<<<(unsigned)acc, threads, shm_m2l, st>>>(a);
        ++launches;
    }
    cudaEventRecord(pl->ev[3], st);
    // the downward pass
    for (int k = 2; k < L; ++k) {
        k_l2l_f64<<<((1 << (2 * k)) + per - 1) / per, threads, shm_down, st>>>(
            static_cast<const double2*>(pl->grids.B[k]), static_cast<double2*>(pl->grids.B[k + 1]), binom, k, p1);
        ++launches;
    }
    if (owned) cudaEventRecord(pl->ev[15], st);
    // the near field, on the caller's stream
    if (cudaMemsetAsync(pl->phi_far, 0, sizeof(double) * (size_t)n, near_st) != cudaSuccess ||
        (field && cudaMemsetAsync(pl->near_grad, 0, sizeof(double2) * (size_t)n, near_st) != cudaSuccess))
        return -1;
    if (owned) cudaEventRecord(pl->ev[8], near_st);
    {
        const uint32_t nleaf = 1u << (2 * L);
        const int64_t wmax = (int64_t)nleaf + n / FMM_P2P_BLOCK + 1;
        // few blocks: two warps a CTA, so that they reach more SMs
        const int warps = wmax < kP2PSmall ? 2 : kP2PWarps64;
        const unsigned blocks = (unsigned)((wmax + warps - 1) / warps);
        if (field)
            k_p2p_f64<true><<<blocks, warps * 32, 0, near_st>>>(pl->sorted64, pl->leaf_start, pl->leaf_bstart,
                                                                pl->blk_map, nleaf, L, pl->logtab, pl->phi_far,
                                                                pl->near_grad, pl->d_status, pl->d_counters);
        else
            k_p2p_f64<false><<<blocks, warps * 32, 0, near_st>>>(pl->sorted64, pl->leaf_start, pl->leaf_bstart,
                                                                 pl->blk_map, nleaf, L, pl->logtab, pl->phi_far, nullptr,
                                                                 pl->d_status, pl->d_counters);
        ++launches;
    }
    if (owned) cudaEventRecord(pl->ev[9], near_st);
    if (two && cudaStreamWaitEvent(near_st, pl->ev[15], 0) != cudaSuccess) return -1;
    cudaEventRecord(pl->ev[4], near_st);
    // L2P at the finest level, with the near field and in input order
    {
        const unsigned blocks = (unsigned)((n + 127) / 128);
        const double2* B = static_cast<const double2*>(pl->grids.B[L]);
        if (field)
            k_l2p_f64<true><<<blocks, 128, 0, near_st>>>(pl->sorted64, pl->sorted_key, n, L, p, s, inv_s, B, pl->phi_far,
                                                         pl->near_grad, pl->d_status, phi, field);
        else
            k_l2p_f64<false><<<blocks, 128, 0, near_st>>>(pl->sorted64, pl->sorted_key, n, L, p, s, inv_s, B, pl->phi_far,
                                                          nullptr, pl->d_status, phi, nullptr);
        ++launches;
    }
    cudaEventRecord(pl->ev[5], near_st);
    if (cudaGetLastError() != cudaSuccess) return -1;
    return launches;
}

int fmm_launch_direct_f64(int64_t n, const double* xy, const double* q, int64_t nt, const int64_t* targets,
                          double* phi_t, cudaStream_t stream) {
    if (nt == 0) return 0;
    k_direct_f64<<<(unsigned)nt, 256, 0, stream>>>(n, reinterpret_cast<const double2*>(xy), q, targets, phi_t);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}
