// Block statistics (Sec. 2.1 transform range, Eq. 2 per block) of a field in
// device memory, computed without allocating any memory.
//
// Some callers cannot allocate device memory when they call us: a service
// that reserves all device memory at start-up and hands it to its own pool,
// code on a latency-critical path that must not pay for cudaFree's implicit
// device-wide synchronisation, or code that runs while the process is short
// of memory and must not fail for that reason. mpr_create allocates its
// context; this entry point instead works in a fixed scratch array that the
// library holds on every device that loads it, and writes only into buffers
// the caller passes.
#include <cuda_runtime.h>

#include <cstdint>

#include "mpr.h"
#include "mpr_internal.h"
#include "mpr_launch.h"
#include "mpr_ptrcheck.h"
#include "mpr_stats.cuh"

using namespace mpr;

namespace {

constexpr int kMaxBlocks = MPR_NOALLOC_MAX_BLOCKS;
constexpr size_t kHeader = 256;
constexpr size_t kScratchBytes = kHeader + (size_t)kMaxBlocks * (sizeof(double) + 3 * sizeof(int32_t));

// The scratch array: [0, 8) z-range in order-preserving uint32 form, [8, 12)
// CTAs of the statistics kernel that have finished,
// [256, ...) per-block sample sums (double), sample counts and gap counts per
// colour (int32). Every call overwrites what it reads; nothing survives a call
// in a form the next one depends on.
static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

struct Scratch {
    uint32_t* mm;
    double* ssum;
    int32_t* nsamp;
    int32_t* ng0;
    int32_t* ng1;
};

Scratch carve(unsigned char* base) {
    Scratch s;
    s.mm = reinterpret_cast<uint32_t*>(base);
    s.ssum = reinterpret_cast<double*>(base + kHeader);
    s.nsamp = reinterpret_cast<int32_t*>(base + kHeader + (size_t)kMaxBlocks * sizeof(double));
    s.ng0 = s.nsamp + kMaxBlocks;
    s.ng1 = s.ng0 + kMaxBlocks;
    return s;
}

// Device address of the scratch array on the current device (the host-side
// symbol is only a stand-in, not a device address). It is looked up on every
// call: the lookup allocates nothing, and an address kept from an earlier call
// would dangle after the device was reset (cudaDeviceReset) and its context
// re-created.
cudaError_t scratch_address(unsigned char** out) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
    if (e != cudaSuccess) return e;
    *out = static_cast<unsigned char*>(p);
    return cudaSuccess;
}

__device__ __forceinline__ float ord_to_float(uint32_t u) {
    const uint32_t v = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
    return __uint_as_float(v);
}

// The min/max reduction accumulates into the scratch; start it from the
// identity of min and max.
__global__ void k_na_reset(uint32_t* mm) {
    mm[0] = 0xffffffffu;
    mm[1] = 0u;
    mm[2] = 0u;   // finished CTAs
}

// z_min / z_max as doubles (both 0 when there is no sample).
__device__ __forceinline__ double2 sample_range(const uint32_t* __restrict__ mm) {
    if (mm[0] == 0xffffffffu) return make_double2(0.0, 0.0);
    return make_double2((double)ord_to_float(mm[0]), (double)ord_to_float(mm[1]));
}

// The closing part, by one CTA: the range, the global sample mean (fallback of
// blocks without samples, Sec. 3.3.3), then each block's mean sample angle and
// gap count.
__device__ void na_finalize(int nblk, const Scratch& sc, double2 range, double* __restrict__ zrange,
                            float* __restrict__ mean_angle, int32_t* __restrict__ n_gap) {
    __shared__ double s_sum[32 * kStatsMaxWarps];
    __shared__ long long s_cnt[32 * kStatsMaxWarps];
    double sum = 0.0;
    long long cnt = 0;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) {
        sum += sc.ssum[b];
        cnt += sc.nsamp[b];
    }
    s_sum[threadIdx.x] = sum;
    s_cnt[threadIdx.x] = cnt;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            s_sum[threadIdx.x] += s_sum[threadIdx.x + w];
            s_cnt[threadIdx.x] += s_cnt[threadIdx.x + w];
        }
        __syncthreads();
    }
    const double gmean = s_cnt[0] > 0 ? s_sum[0] / (double)s_cnt[0] : 0.0;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) {
        const int ns = sc.nsamp[b];
        mean_angle[b] = (float)(ns > 0 ? sc.ssum[b] / (double)ns : gmean);
        n_gap[b] = sc.ng0[b] + sc.ng1[b];
    }
    if (threadIdx.x == 0) {
        zrange[0] = range.x;
        zrange[1] = range.y;
    }
}

// Eq. 2 per block with the range read from device memory: one CTA per block,
// owned bonds (right and down), FP64 sums. The CTA that finishes last runs the
// closing part (with launches of their own for the range and the closing part
// a 256^2 field took 25.7 us, with them here 22.4; 53.9 with a warp per block and
// a general cosine per bond).
__global__ void __launch_bounds__(32 * kStatsMaxWarps)
k_na_block_stats(Geom g, const float* __restrict__ values, const uint8_t* __restrict__ mask,
                 double q, double J, double* __restrict__ Es, int32_t* __restrict__ Nsp,
                 int32_t* __restrict__ Nb, Scratch sc, float* __restrict__ mean_angle,
                 int32_t* __restrict__ n_gap, double* __restrict__ zrange) {
    __shared__ StatsShared sh;
    __shared__ bool last;
    const int b = blockIdx.x;
    const double2 range = sample_range(sc.mm);
    const bool degenerate = !(range.y > range.x);
    const int by = b / g.nbx, bx = b % g.nbx;
    const int y0 = by * g.lb, x0 = bx * g.lb;
    const int y1 = min(g.H, y0 + g.lb), x1 = min(g.W, x0 + g.lb);
    const double scale = degenerate ? 0.0 : 6.283185307179586476925 / (range.y - range.x);
    // (no absent sites: a bond crosses the block's right / lower edge unless
    // that edge is the grid's)
    const BlockSums r = block_sums<false>(values, mask, g.W, y0, x0, y1, x1, x1 < g.W, y1 < g.H,
                                          range.x, range.y, scale, q, J, true, nullptr, 0, 0, sh);
    if (threadIdx.x == 0) {
        Es[b] = r.es;
        Nsp[b] = r.nsp;
        Nb[b] = r.nb;
        sc.ssum[b] = r.sm;
        sc.nsamp[b] = r.ns;
        sc.ng0[b] = r.g0;
        sc.ng1[b] = r.g1;
        __threadfence();
        last = atomicAdd(&sc.mm[2], 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    na_finalize(g.nblk, sc, range, zrange, mean_angle, n_gap);
}

// The pointer is device memory of `device` (the current one) or managed memory.
bool on_device(const void* p, int device) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return noalloc_pointer_ok(at.type, at.device, device);
}

}  // namespace

extern "C" mpr_status mpr_block_stats_noalloc(const mpr_grid* grid, const uint8_t* mask,
                                              const float* values, double q, double J,
                                              double* Es, int32_t* Nsp, int32_t* Nb,
                                              float* mean_angle, int32_t* n_gap, double* zrange,
                                              void* cuda_stream) {
    if (!grid || !mask || !values || !Es || !Nsp || !Nb || !mean_angle || !n_gap || !zrange)
        return MPR_EINVAL;
    const int H = grid->height, W = grid->width, lb = grid->block;
    if (H < 1 || W < 1 || H > MAX_SIDE || W > MAX_SIDE || lb < 1) return MPR_EINVAL;
    if (!(q > 0.0 && q <= 0.5) || !(J > 0.0)) return MPR_EINVAL;
    Geom g;
    g.H = H;
    g.W = W;
    g.Wh = (W + 1) / 2;
    g.lb = lb;
    g.nbx = (W + lb - 1) / lb;
    g.nby = (H + lb - 1) / lb;
    if ((int64_t)g.nbx * g.nby > kMaxBlocks) return MPR_EINVAL;  // beyond the scratch array
    g.nblk = g.nbx * g.nby;
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess) {
        cudaGetLastError();
        return MPR_ECUDA;
    }
    const void* ptrs[] = {mask, values, Es, Nsp, Nb, mean_angle, n_gap, zrange};
    for (const void* p : ptrs)
        if (!on_device(p, device)) return MPR_EINVAL;
    unsigned char* base = nullptr;
    if (scratch_address(&base) != cudaSuccess) return MPR_ECUDA;
    const Scratch sc = carve(base);
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const int64_t n = (int64_t)H * W;
    k_na_reset<<<1, 1, 0, s>>>(sc.mm);
    launch_minmax_field(values, mask, n, sc.mm, s);
    k_na_block_stats<<<g.nblk, stats_threads(g.nblk), 0, s>>>(g, values, mask, q, J, Es, Nsp, Nb,
                                                              sc, mean_angle, n_gap, zrange);
    return cudaPeekAtLastError() == cudaSuccess ? MPR_OK : MPR_ECUDA;
}
