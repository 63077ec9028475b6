// One calibration iteration of a small field as one launch: a thread-block
// cluster per realization pair runs the pair's start, all n_eq + n_meas sweeps
// and the energy averages of the measured ones.
//
// A small field's half-step is a launch with a handful of CTAs whose time is
// launch and latency (2.9 us for the 2.7 k gap sites per colour of a 128^2
// field with a third of its sites missing; an iteration has 90 of them). Here
// it is 1.1 us, the latency of one site's update and the cluster barrier. (With
// the angles exchanged through L2 instead of shared memory: 1.7 us.) Chains of different pairs never
// interact, so a pair's half-steps need no grid-wide order: 16 CTAs of one
// cluster, ordered by the hardware cluster barrier, hold up to 8192 gap sites
// per colour, one per thread, which keeps its site's angles, temperatures and
// energy sums in registers. What neighbours read, cos and sin of q times the
// angle, lies in a shared-memory cell of the owner's CTA, read through the
// cluster's distributed shared memory: no trip to L2 in a half-step, and every
// cosine is taken once instead of by four neighbours. Samples and missing
// neighbours have constant cells. Everything a half-step can do without its
// neighbours (Philox block, proposal and its cosine) is done between the
// barrier's arrival and its wait.
//
// Energies: an iteration only needs each block's sum of E_b(t) over the
// measured sweeps, E_b(t) = E_b(0) + the moves' changes up to sweep t, so a
// change of sweep s counts once for every measured sweep from s on. Each
// thread sums its changes with that weight in two-float arithmetic (products
// and sums error-free, 48 bits) and adds them to the block in FP64 once, where
// a half-step per launch sums every sweep's changes over warps in FP32.
#include <cuda_runtime.h>

#include <cstdint>

#include "mpr_launch.h"
#include "mpr_sweep.cuh"

namespace mpr {

namespace {

constexpr int kClusterCtas = 16;
constexpr int kClusterThreads = 1024;                       // half of them per colour
static_assert(kClusterCtas * kClusterThreads / 2 == kCalClusterSites, "sites per colour");

__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// A cell: (cos, sin) of q phi in the pair's even, then its odd realization.
// Cells of a CTA: one per owned site and colour, then four per thread for the
// neighbours that are not gap sites.
constexpr int kCells = kClusterThreads + 4 * kClusterThreads;
constexpr size_t kClusterSmem = (size_t)kCells * sizeof(float4);

__device__ __forceinline__ uint32_t cell_address(const float4* cell, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;"
        : "=r"(r)
        : "r"((uint32_t)__cvta_generic_to_shared(cell)), "r"(rank));
    return r;
}
__device__ __forceinline__ float4 cell_load(uint32_t at) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(at)
                 : "memory");
    return v;
}

// kOne: only the pair's even realization exists (a bisection's single chain).
template <bool kOne>
__global__ void __launch_bounds__(kClusterThreads, 1) k_cal_cluster(CalClusterArgs a) {
    extern __shared__ float4 cells[];
    const SweepArgs& sw = a.sw;
    const Model& m = sw.m;
    const int rank = (int)(blockIdx.x % kClusterCtas), p = (int)(blockIdx.x / kClusterCtas);
    constexpr int kHalf = kClusterThreads / 2;
    const int c = threadIdx.x / kHalf, slot = threadIdx.x % kHalf;
    const int n = a.n_list[c], per = (n + kClusterCtas - 1) / kClusterCtas;
    const int per_o = (a.n_list[c ^ 1] + kClusterCtas - 1) / kClusterCtas;
    const int e = rank * per + slot;
    const bool live = slot < per && e < n;
    const int rl = 2 * p;
    const bool run0 = rl < sw.R, run1 = rl + 1 < sw.R;
    const uint32_t tag = sw.ctl->tag, rpair = (sw.r_base + (uint32_t)rl) >> 1;
    uint32_t hs = 0, f = 0, site = 0, key1 = 0;
    int b = 0, left = 0;
    float2 beta = both(0.0f), ph = both(0.0f), co = ph, so = ph;
    float2* own = reinterpret_cast<float2*>(static_cast<float*>(sw.ang) + pair_plane(sw.g, p, c));
    const float2* oth = reinterpret_cast<const float2*>(static_cast<const float*>(sw.ang) +
                                                        pair_plane(sw.g, p, c ^ 1));
    float4* cell = cells + threadIdx.x;
    if (live) {
        const uint4 en = a.list[c][e];
        hs = en.x;
        f = en.y & ((1u << META_SHIFT) - 1u);
        site = en.z;
        left = (int)en.w;
        b = (int)(en.y >> META_SHIFT);
        key1 = slice_key1(sw.sl, slice_of(sw.sl, b));
        if (sw.beta_pts) {
            beta.x = sw.beta_pts[(size_t)(rl % sw.n_pts) * sw.g.nblk + b];
            beta.y = sw.beta_pts[(size_t)((rl + 1) % sw.n_pts) * sw.g.nblk + b];
        } else {
            beta.x = sw.beta[b];
            beta.y = sw.beta_odd ? sw.beta_odd[b] : beta.x;
        }
        ph = both(a.init_angle[b]);
        if (a.random_init) {
            uint32_t w[4];
            philox4x32_10_rk(site, 0xFFFFu << 16, rpair, 0u, sw.rng.rk0, key1, w);
            ph = make_float2(kTwoPi * u01(w[0]), kTwoPi * u01(w[2]));
        }
        sincos_2(__fmul2_rn(both(m.q), ph), so, co);
        *cell = make_float4(co.x, so.x, co.y, so.y);
        // The site's list index, where its neighbours look it up once.
        __stcg(own + hs, make_float2(__int_as_float(e), 0.0f));
    }
    cluster_arrive();
    cluster_wait();
    // The neighbours' cells: a gap site's in its owner's CTA, else a constant
    // one of this thread (a sample's cos / sin, or 0 where there is no site).
    uint32_t at[4] = {0u, 0u, 0u, 0u};
    if (live) {
        const float2* word[4] = {oth + (ptrdiff_t)left, oth + (ptrdiff_t)left + 1,
                                 oth + hs - (ptrdiff_t)sw.g.Wh, oth + hs + sw.g.Wh};
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            if (f & (GAP_L << d)) {
                const int i = __float_as_int(__ldcg(word[d]).x);
                at[d] = cell_address(cells + (c ^ 1) * kHalf + i % per_o, i / per_o);
            } else {
                float sj = 0.0f, cj = 0.0f;
                if (f & (NB_L << d)) __sincosf(m.q * __ldcg(word[d]).x, &sj, &cj);
                float4* k = cells + kClusterThreads + 4 * (int)threadIdx.x + d;
                *k = make_float4(cj, sj, cj, sj);
                at[d] = cell_address(k, rank);
            }
        }
    }
    Sum2 sum_o{both(0.0f), both(0.0f)}, sum_l = sum_o, sum_u = sum_o;
    // The next half-step's draws, proposal and its cosine and sine.
    float2 u1, php, cp, sp;
    auto propose = [&](int s) {
        uint32_t w[4];
        philox4x32_10_rk(site, (uint32_t)s | (tag << 16), rpair, 0u, sw.rng.rk0, key1, w);
        const float2 u0 = u01_2(w[0], w[2]);
        u1 = u01_2(w[1], w[3]);
        php = __fmul2_rn(both(kTwoPi), u0);
        sincos_2(__fmul2_rn(both(m.q), php), sp, cp);
    };
    propose(1);
    __syncthreads();
    for (int s = 1; s <= a.n_sweeps; ++s) {
        const float weight = (float)min(a.n_meas, a.n_sweeps - s + 1);
#pragma unroll 1
        for (int col = 0; col < 2; ++col) {
            if (col == c && live) {
                const float4 L = cell_load(at[0]), R = cell_load(at[1]), U = cell_load(at[2]),
                             D = cell_load(at[3]);
                float2 ao = both(0.0f), al = ao, au = ao;
                if constexpr (kOne) {
                    const float C = (L.x + R.x) + (U.x + D.x), Sn = (L.y + R.y) + (U.y + D.y);
                    const SiteNew nw = site_move<float>(ph.x, co.x, so.x, php.x, cp.x, sp.x, C, Sn,
                                                        u1.x, beta.x, m);
                    if (f & (EDGE_L | EDGE_U))
                        split_edge<float>(nw, ph.x, f, C, Sn, L.x, L.y, U.x, U.y, m, ao.x, al.x,
                                          au.x);
                    else
                        ao.x = nw.dE;
                    ph.x = nw.phi;
                    __sincosf(m.q * ph.x, &so.x, &co.x);
                } else {
                    const float2 v[8] = {{L.x, L.z}, {R.x, R.z}, {U.x, U.z}, {D.x, D.z},
                                         {L.y, L.w}, {R.y, R.w}, {U.y, U.w}, {D.y, D.w}};
                    const float2 C = sum4(v), Sn = sum4(v + 4);
                    const PairNew nw = pair_move<float>(ph, co, so, php, cp, sp, C, Sn, u1, beta, m);
                    if (f & (EDGE_L | EDGE_U))
                        split_edge_2<float>(nw, ph, f, C, Sn, v[0], v[4], v[2], v[6], m, ao, al, au);
                    else
                        ao = nw.dE;
                    ph = make_float2(run0 ? nw.phi.x : ph.x, run1 ? nw.phi.y : ph.y);
                    sincos_2(__fmul2_rn(both(m.q), ph), so, co);
                }
                *cell = make_float4(co.x, so.x, co.y, so.y);
                cluster_arrive();
                sum_o.add(ao, weight);
                if (f & (EDGE_L | EDGE_U)) {
                    sum_l.add(al, weight);
                    sum_u.add(au, weight);
                }
                propose(s + 1);
            } else {
                cluster_arrive();
            }
            cluster_wait();
        }
    }
    // (no CTA leaves while another may read its cells: the last wait is past
    // every read)
    if (live) own[hs] = ph;
    // The blocks' sums over the measured sweeps: the start's E_b once per
    // sweep, and the weighted changes.
    auto add = [&](int blk, int r, double v) {
        if (r >= sw.R) return;
        double* dst = a.points > 2 ? a.ebar_pts + (size_t)(r % a.points) * sw.g.nblk
                      : a.points == 2 && (r & 1) ? a.ebar_odd
                                                 : a.ebar;
        if (v != 0.0) atomicAdd(&dst[blk], v * a.inb[blk]);
    };
    for (int k = rank * kClusterThreads + (int)threadIdx.x; k < sw.g.nblk;
         k += kClusterCtas * kClusterThreads)
        for (int r = rl; r < rl + 2; ++r) add(k, r, (double)a.n_meas * a.E0[(size_t)k * sw.Rp + r]);
    if (!live) return;
    add(b, rl, (double)sum_o.hi.x + (double)sum_o.lo.x);
    add(b, rl + 1, (double)sum_o.hi.y + (double)sum_o.lo.y);
    if (f & EDGE_L) {
        add(b - 1, rl, (double)sum_l.hi.x + (double)sum_l.lo.x);
        add(b - 1, rl + 1, (double)sum_l.hi.y + (double)sum_l.lo.y);
    }
    if (f & EDGE_U) {
        add(b - sw.g.nbx, rl, (double)sum_u.hi.x + (double)sum_u.lo.x);
        add(b - sw.g.nbx, rl + 1, (double)sum_u.hi.y + (double)sum_u.lo.y);
    }
}

cudaLaunchConfig_t cluster_config(int n_pairs, cudaLaunchAttribute* attr, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = kClusterCtas;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(n_pairs * kClusterCtas));
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = kClusterSmem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

int cal_cluster_max_active() {
    int n = 1 << 30;
    const void* kernels[2] = {(const void*)k_cal_cluster<true>, (const void*)k_cal_cluster<false>};
    for (const void* k : kernels) {
        cudaLaunchAttribute attr[1];
        const cudaLaunchConfig_t cfg = cluster_config(1, attr, nullptr);
        int m = 0;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                cudaSuccess ||
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kClusterSmem) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&m, k, &cfg) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        n = m < n ? m : n;
    }
    return n;
}

cudaError_t launch_cal_cluster(const CalClusterArgs& a, cudaStream_t s) {
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = cluster_config(a.sw.Rp / 2, attr, s);
    return a.sw.R == 1 ? cudaLaunchKernelEx(&cfg, k_cal_cluster<true>, a)
                       : cudaLaunchKernelEx(&cfg, k_cal_cluster<false>, a);
}

}  // namespace mpr
