// noalloc.cu -- fmm_potential_noalloc: the FP64 path with every workspace in a fixed,
// file-scope device array, for callers that must not allocate device memory.
//
// Some callers cannot call cudaMalloc: code that runs after an application has fixed its
// memory budget (a real-time or embedded loop that forbids allocation after start-up), code
// that shares a device with an allocator that owns all free memory (a framework's caching
// pool), or a plugin that may not create allocations of its own.  fmm_potential needs a plan,
// and fmm_plan allocates; this entry point needs none.  Its scratch is the static array below,
// which the CUDA runtime reserves on a device when the library's module is loaded there and
// keeps until the process exits.  With lazy module loading (the CUDA default) that happens at
// the first use of the library on the device -- this entry point's first call, or the first
// library kernel -- so a caller whose allocator claims the free memory later should make one
// call first.
//
// Host code sees `g_noalloc_scratch` only as a host-side stand-in symbol, not as a device
// address: a kernel handed that name faults or, where the GPU can reach host memory, uses the
// wrong memory.  The device address is therefore looked up once per device, with that device
// current, by cudaGetSymbolAddress, and passed to the kernels.
#include <mutex>

#include "fmm_internal.cuh"
#include "fp64_math.cuh"

namespace {

// Limits of the no-allocation path and the scratch they need (each sub-buffer 256-byte aligned):
// particles <= 65536, levels <= 6, p <= 20.  Worst case about 7.8 MB; the array holds 8.5 MB.
constexpr int64_t kMaxN = 65536;
constexpr int kMaxLevels = 6;
constexpr int kMaxP = 20;
constexpr size_t kScratchBytes = (size_t)8704 * 1024;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
void* g_scratch_ptr[kMaxDevices] = {};
cudaEvent_t g_events[kMaxDevices][6] = {};

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

// The FP64 path's tables (the plan's host-side build_far_tables), built on the device so that the call
// needs neither a host buffer nor a host-to-device copy: R[k][l] = (-1)^(k+1) C(l+k-1, k-1) / k with
// R[0][l] = -1 / l, then C(m, j), then d^-k of the interaction lists' orbits.
__global__ void k_build_far_tables(int p1, double* __restrict__ tab) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const int pad = (p1 * p1 + 1) & ~1;
    const int k = e / p1, l = e % p1;
    if (e < p1 * p1) {
        double r = 0.0;
        if (k == 0) {
            r = l ? -1.0 / (double)l : 0.0;
        } else {
            double b = 1.0;   // C(l+k-1, k-1) by the multiplicative formula (exact for these sizes)
            for (int i = 1; i <= k - 1; ++i) b = b * (double)(l + i) / (double)i;
            r = ((k & 1) ? 1.0 : -1.0) / (double)k * b;
        }
        tab[e] = r;
        double c = l <= k ? 1.0 : 0.0;   // C(k, l)
        for (int i = 1; i <= l && l <= k; ++i) c = c * (double)(k - l + i) / (double)i;
        tab[pad + e] = c;
    }
    if (e < kFmmOrbits * p1) {
        const double x = fmm_orbit_x(k), y = fmm_orbit_y(k), r2 = x * x + y * y;
        double2 v = make_double2(1.0, 0.0);
        const double ix = x / r2, iy = -y / r2;
        for (int i = 0; i < l; ++i) v = make_double2(v.x * ix - v.y * iy, v.x * iy + v.y * ix);
        reinterpret_cast<double2*>(tab + 2 * pad)[e] = v;
    }
}

__global__ void k_build_logtab(double2* __restrict__ tab) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < kFmmLogEntries) tab[j] = fmm_log_entry(j);
}

// Carve the plan's workspaces out of the scratch block; returns the bytes used.
size_t carve(fmm_plan_s* pl, unsigned char* base) {
    const int64_t n = pl->n;
    const int L = pl->levels, p1 = pl->p + 1;
    const int64_t m = (int64_t)1 << (2 * L);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        unsigned char* ptr = base ? base + off : nullptr;
        off = align256(off + bytes);
        return ptr;
    };
    pl->keys = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * n));
    pl->rank = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * n));
    pl->counts = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * m));
    pl->leaf_start = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * (m + 1)));
    pl->scan_blocks = fmm_scan_blocks(m);
    pl->block_sums = reinterpret_cast<uint32_t*>(take(sizeof(unsigned long long) * (pl->scan_blocks + 1)));
    pl->leaf_bstart = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * (m + 1)));
    pl->blk_map = reinterpret_cast<uint2*>(take(sizeof(uint2) * (m + n / FMM_P2P_BLOCK + 1)));
    pl->sorted_key = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * n));
    pl->sorted64 = reinterpret_cast<fmm_p64*>(take(sizeof(fmm_p64) * n));
    pl->phi_far = reinterpret_cast<double*>(take(sizeof(double) * n));
    for (int k = 2; k <= L; ++k) {
        const size_t W = (size_t)fmm_grid_width(k);
        pl->a_bytes[k] = W * W * p1 * sizeof(double2);
        pl->grids.A[k] = take(pl->a_bytes[k]);
        pl->grids.B[k] = take(((size_t)1 << (2 * k)) * p1 * sizeof(double2));
    }
    pl->ftab = reinterpret_cast<double*>(take(sizeof(double) * fmm_far_table_doubles(p1)));
    pl->logtab = reinterpret_cast<double2*>(take(sizeof(double2) * kFmmLogEntries));
    pl->d_status = reinterpret_cast<unsigned int*>(take(sizeof(unsigned int)));
    pl->d_counters = reinterpret_cast<unsigned long long*>(take(FMM_COUNTERS * sizeof(unsigned long long)));
    return off;
}

// Once per device, with that device current: the scratch block's device address and the
// (memory-free) events the stage launchers record.
fmm_status setup(int dev, void** scratch, cudaEvent_t** events) {
    if (dev < 0 || dev >= kMaxDevices) return FMM_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_ptr[dev]) {
        void* ptr = nullptr;
        const cudaError_t r = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
        if (r != cudaSuccess || !ptr) {
            // the module (and with it the array) could not be loaded on this device
            return r == cudaErrorMemoryAllocation ? FMM_ERR_OOM : FMM_ERR_CUDA;
        }
        for (int e = 0; e < 6; ++e)
            if (cudaEventCreate(&g_events[dev][e]) != cudaSuccess) {
                for (int f = 0; f < e; ++f) {   // a later call starts the set-up again
                    cudaEventDestroy(g_events[dev][f]);
                    g_events[dev][f] = nullptr;
                }
                return FMM_ERR_CUDA;
            }
        g_scratch_ptr[dev] = ptr;
    }
    *scratch = g_scratch_ptr[dev];
    *events = g_events[dev];
    return FMM_OK;
}

}  // namespace

extern "C" fmm_status fmm_potential_noalloc(int64_t n, int levels, int p, double box, const double* xy,
                                            const double* q, double* phi, void* stream) {
    if (n < 1 || n > kMaxN || levels < 0 || levels > kMaxLevels || p < 1 || p > kMaxP || !(box > 0.0) ||
        !(box < 1e300) || !xy || !q || !phi)
        return FMM_ERR_INVALID_ARG;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return FMM_ERR_CUDA;
    void* scratch = nullptr;
    cudaEvent_t* events = nullptr;
    fmm_status s = setup(dev, &scratch, &events);
    if (s != FMM_OK) return s;

    fmm_plan_s pl{};
    pl.device = dev;
    pl.n = n;
    pl.levels = levels;
    pl.p = p;
    pl.box = box;
    pl.precision = FMM_FP64;
    pl.stream = static_cast<cudaStream_t>(stream);
    if (carve(&pl, nullptr) > kScratchBytes) return FMM_ERR_INVALID_ARG;   // cannot happen within the limits
    carve(&pl, static_cast<unsigned char*>(scratch));
    pl.ev = events;   // the FP64 stages record the first six

    // The array keeps the previous call's contents: clear what must start at zero.
    cudaStream_t st = pl.stream;
    if (cudaMemsetAsync(pl.d_status, 0, sizeof(unsigned int), st) != cudaSuccess ||
        cudaMemsetAsync(pl.d_counters, 0, FMM_COUNTERS * sizeof(unsigned long long), st) != cudaSuccess)
        return FMM_ERR_CUDA;
    for (int k = 2; k <= levels; ++k)   // the halos of the moment grids read as zero
        if (cudaMemsetAsync(pl.grids.A[k], 0, pl.a_bytes[k], st) != cudaSuccess) return FMM_ERR_CUDA;
    const int ntab = (p + 1) * (p + 1 > kFmmOrbits ? p + 1 : kFmmOrbits);
    // an error left pending by the caller's own earlier work is not this call's to report or clear
    if (cudaPeekAtLastError() != cudaSuccess) return FMM_ERR_CUDA;
    k_build_far_tables<<<(ntab + 255) / 256, 256, 0, st>>>(p + 1, pl.ftab);
    k_build_logtab<<<(kFmmLogEntries + 127) / 128, 128, 0, st>>>(pl.logtab);
    if (cudaPeekAtLastError() != cudaSuccess) return FMM_ERR_CUDA;
    cudaEventRecord(pl.ev[0], st);
    if (fmm_launch_sort(&pl, xy, q) < 0 || fmm_launch_fp64(&pl, phi) < 0) return FMM_ERR_CUDA;

    // Wait for the stream and report what the device checks found (phi is unwritten then).
    unsigned int flags = 0;
    if (cudaMemcpyAsync(&flags, pl.d_status, sizeof(unsigned int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return FMM_ERR_CUDA;
    if (flags & FMM_FLAG_NONFINITE) return FMM_ERR_NONFINITE;
    if (flags & FMM_FLAG_OUT_OF_BOX) return FMM_ERR_OUT_OF_BOX;
    return FMM_OK;
}
