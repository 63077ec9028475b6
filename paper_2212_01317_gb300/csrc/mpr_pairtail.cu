// The stop tail of a realization batch with one cluster per realization pair.
//
// Realizations are independent chains (Sec. 3.4 reading: each (block,
// realization) pair sweeps until its first crossing of e_s,b, or n_max; the
// blocks without sample bonds of a realization stop once none of its
// targeted blocks runs), so the sweeps of one realization pair need no
// other pair's results. Late in a batch only a few of each pair's blocks
// still run; there, one cluster of CTAs per pair runs the pair's remaining
// sweeps with cluster barriers between the phases (colour 0, colour 1, the
// targeted stops, the closing stop part) instead of a launch per phase. Each
// CTA keeps its share of the running units in shared memory. Every phase runs
// the same device code as the per-launch loop (sweep_item, stop_targeted_range,
// stop_rest_range) on the same data, so the results are those of the per-launch
// loop up to the order of the FP64 energy atomics.
//
// A phase is a chain of dependent loads for each warp's units, one after the
// other: with one CTA per pair, a batch of few pairs (4096 running units over
// ten pairs) left 13 units to a warp, 56 us per sweep. As many CTAs per pair as
// fit the GPU with every cluster resident (1 to 16): 29 us; realizations of
// 128^2, 80 % missing, R = 10: 4.2 -> 2.4 ms, 256^2, half missing: 2.5 -> 1.7 ms.
// A cluster barrier with its writes to L2 costs about 1.5 us, so once a CTA has
// a warp for every unit left the first one goes on alone (at 32 units 2 % more
// time, at 64 and 128 more again).
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "mpr_launch.h"
#include "mpr_sweep.cuh"

namespace mpr {

namespace {

constexpr int kPairThreads = 512;    // (1024: 64 registers, the sweep spills)
constexpr int kPairWarps = kPairThreads / 32;
// Units of a pair above which a unit gets one warp. (The number of warps per
// unit decides how the block sums are grouped in FP32, so it depends on the
// pair's units only.)
constexpr int kPairUnits = 32;
constexpr uint32_t kAloneUnits = kPairWarps;   // the pair's first CTA goes on alone

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Barrier over the cluster's threads; their writes are visible after it.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// *p of CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t peer_load(const uint32_t* p, uint32_t rank) {
    uint32_t at, v;
    asm("mapa.shared::cluster.u32 %0, %1, %2;"
        : "=r"(at)
        : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
    return v;
}

template <typename S>
__global__ void __launch_bounds__(kPairThreads, 1) k_pair_tail(SimTailArgs a) {
    __shared__ uint32_t s_units[2][kPairTailCap];
    __shared__ uint32_t s_n[2], s_total;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int npairs = a.sw.Rp >> 1;
    const uint32_t rank = cluster_rank(), ctas = cluster_size();
    const int p = (int)(blockIdx.x / ctas);           // this cluster's realization pair
    Control* ctl = a.ctl;
    const uint32_t t0 = ctl->t, tag = ctl->tag;
    const uint32_t n0 = ctl->n_work[t0 & 1u];
    const uint32_t* work = a.work_all + (size_t)(t0 & 1u) * a.sw.work_stride;
    if (tid == 0) {
        s_n[0] = 0;
        s_n[1] = 0;
    }
    __syncthreads();
    // This CTA's share of the pair's units of the global worklist (the launch
    // is only made when the whole list fits one CTA's buffer): blocks dealt out
    // in turn, so that neighbours that stop together leave the shares even.
    for (uint32_t i = tid; i < n0; i += kPairThreads) {
        const uint32_t u = work[i];
        const uint32_t b = u / (uint32_t)npairs;
        if ((int)(u - b * (uint32_t)npairs) == p && b % ctas == rank) {
            const uint32_t j = atomicAdd(&s_n[0], 1u);
            if (j < (uint32_t)kPairTailCap) s_units[0][j] = u;
        }
    }
    __syncthreads();
    if (tid == 0 && s_n[0] > (uint32_t)kPairTailCap) s_n[0] = kPairTailCap;   // never (host check)
    cluster_sync();
    int cur = 0;
    uint32_t t = t0;
    bool alone = ctas == 1;      // the pair's units are all in this CTA
    auto phase_end = [&] {
        if (alone) __syncthreads();
        else cluster_sync();
    };
    for (;;) {
        uint32_t total = s_n[cur];
        if (!alone) {
            if (warp == 0) {
                const uint32_t v = (uint32_t)tid < ctas ? peer_load(&s_n[cur], (uint32_t)tid) : 0u;
                const uint32_t sum = __reduce_add_sync(0xffffffffu, v);
                if (tid == 0) s_total = sum;
            }
            __syncthreads();
            total = s_total;
            // Few units: the first CTA takes them all and goes on alone.
            if (total <= kAloneUnits) {
                if (rank == 0) {
                    uint32_t at = s_n[cur];
                    for (uint32_t o = 1; o < ctas; ++o) {
                        const uint32_t m = peer_load(&s_n[cur], o);
                        if ((uint32_t)tid < m)
                            s_units[cur][at + tid] = peer_load(&s_units[cur][tid], o);
                        at += m;
                    }
                }
                cluster_sync();
                if (rank != 0) return;
                if (tid == 0) s_n[cur] = total;
                alone = true;
                __syncthreads();
            }
        }
        const uint32_t n = s_n[cur];
        if (total == 0 || (int)t > a.st.n_max) break;   // (the same in every CTA)
        const uint32_t ctr1 = t | (tag << 16);
        // One warp per unit while the pair's units outnumber a CTA's warps; two
        // or four (splitting a block's entries) when they are few.
        int k = 1;
        while (k < 4 && (int)total * 2 * k <= kPairUnits) k *= 2;
        const int slot = warp / k, cw = warp - slot * k, nslot = kPairWarps / k;
        for (int c = 0; c < 2; ++c) {
            SweepArgs s = a.sw;
            s.colour = c;
            s.list = a.list[c];
            s.start = a.start[c];
            s.split = a.split[c];
            for (uint32_t it = slot; it < n; it += nslot) {
                const int b = (int)(s_units[cur][it] / (uint32_t)npairs);
                sweep_item<S>(s, b, p, cw, k, ctr1);
            }
            phase_end();
        }
        stop_targeted_range(a.st, t, s_units[cur], (int64_t)n * 2, (int64_t)n * 2, tid,
                            kPairThreads);
        if (tid == 0) s_n[cur ^ 1] = 0;
        phase_end();
        stop_rest_range(a.st, t, s_units[cur], n, n, s_units[cur ^ 1], &s_n[cur ^ 1], tid,
                        kPairThreads);
        phase_end();
        cur ^= 1;
        ++t;
    }
    if (!alone) cluster_sync();   // (no CTA leaves while another may read its count)
    if (rank != 0) return;
    // The last cluster to finish leaves the Control as the per-launch loop's
    // last closing stop kernel would: the sweep index after the last sweep
    // any pair ran, nothing running, empty worklists.
    if (tid == 0) {
        atomicMax(&ctl->t_tail, t);
        __threadfence();
        if (atomicAdd(&ctl->ticket, 1u) == gridDim.x / ctas - 1) {
            __threadfence();
            const uint32_t tm = atomicExch(&ctl->t_tail, 0u);
            ctl->t = tm > t0 ? tm : t0;
            ctl->n_running = 0;
            ctl->n_running_acc = 0;
            ctl->n_work[0] = 0;
            ctl->n_work[1] = 0;
            ctl->ticket = 0;
            __threadfence();
        }
    }
}

template <typename S> struct PairTag { using type = S; };
template <typename F> void with_storage_pair(int storage, F&& f) {
    if (storage == 1) f(PairTag<__nv_bfloat16>{});
    else if (storage == 2) f(PairTag<__half>{});
    else f(PairTag<float>{});
}

template <typename S>
cudaLaunchConfig_t tail_config(int n_pairs, int ctas, cudaLaunchAttribute* attr, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)ctas;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(n_pairs * ctas));
    cfg.blockDim = dim3(kPairThreads);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

int pair_tail_ctas(int storage, int n_pairs) {
    int best = 1;
    with_storage_pair(storage, [&](auto tag) {
        using S = typename decltype(tag)::type;
        if (cudaFuncSetAttribute(k_pair_tail<S>, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                 1) != cudaSuccess) {
            cudaGetLastError();
            return;
        }
        for (int ctas = 16; ctas > 1; ctas /= 2) {
            cudaLaunchAttribute attr[1];
            const cudaLaunchConfig_t cfg = tail_config<S>(1, ctas, attr, nullptr);
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, k_pair_tail<S>, &cfg) != cudaSuccess) {
                cudaGetLastError();
                continue;
            }
            if (n >= n_pairs) {
                best = ctas;
                return;
            }
        }
    });
    return best;
}

cudaError_t launch_pair_tail(const SimTailArgs& a, int storage, int n_pairs, int ctas,
                             cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    with_storage_pair(storage, [&](auto tag) {
        using S = typename decltype(tag)::type;
        cudaLaunchAttribute attr[1];
        const cudaLaunchConfig_t cfg = tail_config<S>(n_pairs, ctas, attr, s);
        e = cudaLaunchKernelEx(&cfg, k_pair_tail<S>, a);
    });
    return e;
}

}  // namespace mpr
