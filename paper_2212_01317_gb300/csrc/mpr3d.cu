// 3-D grids (D x H x W, 6-neighbour MPR Hamiltonian, cubic blocks): the
// space / space-time extension the paper names in its conclusions (Sec. 4).
// Everything but the geometry is the 2-D method: Sec. 2.1 transform, Eq. 2
// per block, per-block temperatures by bisection, checkerboard Metropolis +
// over-relaxation half-steps, incremental block energies, the per-block
// local-equilibrium stop (Sec. 3.4), realizations averaged and
// back-transformed.
//
// Layout: site (z, y, x), index i = (z H + y) W + x, colour (x + y + z) mod 2,
// half-lattice state [pair][colour][D][H][ceil(W/2)] of float2 (a realization
// pair per element, a plane per pair and colour; sample angles in both lanes;
// a layer, a row and two half-sites readable before and after it); gap lists
// per colour, block-major (see gap_item3). A thread updates one gap site for
// one realization pair. Every site owns its +x, +y, +z bonds; a site on the
// low x / y / z face of its block hands that bond's change to the neighbouring
// block. The stop and calibration bookkeeping (per block and realization) are
// the 2-D kernels.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <string>
#include <utility>
#include <vector>

#include "mpr.h"
#include "mpr_internal.h"
#include "mpr_launch.h"
#include "mpr_memory.h"
#include "mpr_pdl.h"
#include "mpr_stats.cuh"
#include "mpr_sweep.cuh"

using namespace mpr;

namespace {

struct Geom3 {
    int D, H, W, Wh, lb, nbx, nby, nbz, nblk;
};

__device__ __forceinline__ int block3(const Geom3& g, int z, int y, int x) {
    return ((z / g.lb) * g.nby + y / g.lb) * g.nbx + x / g.lb;
}

// Half index of site (z, y, x), and element offset of pair p's plane of colour c.
__device__ __forceinline__ size_t half3(const Geom3& g, int z, int y, int x) {
    return ((size_t)z * g.H + y) * g.Wh + (x >> 1);
}
__host__ __device__ inline size_t plane3(const Geom3& g, int p, int c) {
    return ((size_t)p * 2 + (size_t)c) * g.D * g.H * g.Wh;
}
// Elements before and after the state that a neighbour load may touch.
inline size_t guard3(const Geom3& g) { return (size_t)g.H * g.Wh + g.Wh + 2; }

// Low bits of a gap entry's .y: which of the neighbours -x, +x, -y, +y, -z, +z
// exist, and whether the -x, -y, -z bond belongs to the neighbouring block.
constexpr uint32_t ALL6 = 0x3Fu;
constexpr int FACE_SHIFT = 6;

// The list entry of gap site (z, y, x) of block b: .x = half index, .y =
// b << META_SHIFT | flags, .z = site index (the Philox counter word), .w = the
// -x neighbour's half index (the +x one's is one more). Worked out once here,
// where the sweep would divide site indices by the grid's sides in 64 bits for
// every realization pair of every update.
__device__ __forceinline__ uint4 gap_item3(const Geom3& g, int b, int z, int y, int x) {
    const uint32_t f = (uint32_t)(x > 0) | (uint32_t)(x + 1 < g.W) << 1 | (uint32_t)(y > 0) << 2 |
                       (uint32_t)(y + 1 < g.H) << 3 | (uint32_t)(z > 0) << 4 |
                       (uint32_t)(z + 1 < g.D) << 5 | (uint32_t)(x > 0 && x % g.lb == 0) << 6 |
                       (uint32_t)(y > 0 && y % g.lb == 0) << 7 |
                       (uint32_t)(z > 0 && z % g.lb == 0) << 8;
    const uint32_t h = (uint32_t)half3(g, z, y, x);
    return make_uint4(h, (uint32_t)b << META_SHIFT | f,
                      (uint32_t)(((int64_t)z * g.H + y) * g.W + x), h + (uint32_t)(x & 1) - 1u);
}

__device__ __forceinline__ uint32_t f2ord3(float f) {
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__global__ void k3_minmax(const float* __restrict__ values, const uint8_t* __restrict__ mask,
                          int64_t n, uint32_t* __restrict__ mm) {
    uint32_t lo = 0xffffffffu, hi = 0u;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (mask[i]) continue;
        const uint32_t o = f2ord3(values[i]);
        lo = min(lo, o);
        hi = max(hi, o);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(&mm[0], lo);
        atomicMax(&mm[1], hi);
    }
}

// Sample angles (Sec. 2.1) in FP32, 0 at gaps.
__global__ void k3_layout(int64_t n, const float* __restrict__ values,
                          const uint8_t* __restrict__ mask, double zmin, double zmax,
                          int degenerate, float* __restrict__ phi_s) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        phi_s[i] = (mask[i] || degenerate)
                       ? 0.0f
                       : (float)(6.283185307179586476925 * ((double)values[i] - zmin) / (zmax - zmin));
}

// Eq. 2 per block (one CTA per block, FP64): owned sample-sample bonds, all
// owned bonds, sample mean angle, gap counts per colour. A block holds
// thousands of sites and a grid few blocks: with one warp per block the 512
// blocks of a 128^3 grid kept 3.4 warps per SM (693 us).
constexpr int kStatsWarps = 8;
__global__ void __launch_bounds__(32 * kStatsWarps)
k3_block_stats(Geom3 g, const float* __restrict__ values, const uint8_t* __restrict__ mask,
               double zmin, double zmax, int degenerate, double q, double J,
               double* __restrict__ Es, int32_t* __restrict__ Nsp, int32_t* __restrict__ Nb,
               double* __restrict__ ssum, int32_t* __restrict__ nsamp,
               int32_t* __restrict__ ngap0, int32_t* __restrict__ ngap1) {
    const int b = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int bx = b % g.nbx, by = (b / g.nbx) % g.nby, bz = b / (g.nbx * g.nby);
    const int x0 = bx * g.lb, y0 = by * g.lb, z0 = bz * g.lb;
    const int x1 = min(g.W, x0 + g.lb), y1 = min(g.H, y0 + g.lb), z1 = min(g.D, z0 + g.lb);
    const int bw = x1 - x0, bh = y1 - y0, nsite = bw * bh * (z1 - z0);
    const double scale = degenerate ? 0.0 : 6.283185307179586476925 / (zmax - zmin);
    const int64_t HW = (int64_t)g.H * g.W;
    double es = 0.0, sm = 0.0;
    int nsp = 0, nb = 0, ns = 0, c0 = 0, c1 = 0;
    for (int j = threadIdx.x; j < nsite; j += 32 * kStatsWarps) {
        const int x = x0 + j % bw, y = y0 + (j / bw) % bh, z = z0 + j / (bw * bh);
        const int64_t i = z * HW + (int64_t)y * g.W + x;
        const bool gap = mask[i] != 0;
        const double pi = gap ? 0.0 : ((double)values[i] - zmin) * scale;
        if (gap) {
            if (((x + y + z) & 1) == 0) ++c0; else ++c1;
        } else {
            sm += pi;
            ++ns;
        }
        const int64_t nbr[3] = {x + 1 < g.W ? i + 1 : -1, y + 1 < g.H ? i + g.W : -1,
                                z + 1 < g.D ? i + HW : -1};
        for (int k = 0; k < 3; ++k) {
            if (nbr[k] < 0) continue;
            ++nb;
            if (!gap && !mask[nbr[k]]) {
                const double pj = ((double)values[nbr[k]] - zmin) * scale;
                es += -J * cos_bond(q * (pi - pj));
                ++nsp;
            }
        }
    }
    __shared__ double s_d[kStatsWarps][2];
    __shared__ int s_i[kStatsWarps][5];
    int v[5] = {nsp, nb, ns, c0, c1};
    for (int d = 16; d > 0; d >>= 1) {
        es += __shfl_xor_sync(0xffffffffu, es, d);
        sm += __shfl_xor_sync(0xffffffffu, sm, d);
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) v[k] = __reduce_add_sync(0xffffffffu, v[k]);
    if (lane == 0) {
        s_d[warp][0] = es;
        s_d[warp][1] = sm;
        for (int k = 0; k < 5; ++k) s_i[warp][k] = v[k];
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < kStatsWarps; ++w) {
        es += s_d[w][0];
        sm += s_d[w][1];
        for (int k = 0; k < 5; ++k) v[k] += s_i[w][k];
    }
    Es[b] = es;
    Nsp[b] = v[0];
    Nb[b] = v[1];
    ssum[b] = sm;
    nsamp[b] = v[2];
    ngap0[b] = v[3];
    ngap1[b] = v[4];
}

// Gap lists, block-major, in site order (one warp per block).
__global__ void k3_build_lists(Geom3 g, const uint8_t* __restrict__ mask,
                               const int32_t* __restrict__ start0,
                               const int32_t* __restrict__ start1, uint4* __restrict__ list0,
                               uint4* __restrict__ list1) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= g.nblk) return;
    const int bx = warp % g.nbx, by = (warp / g.nbx) % g.nby, bz = warp / (g.nbx * g.nby);
    const int x0 = bx * g.lb, y0 = by * g.lb, z0 = bz * g.lb;
    const int x1 = min(g.W, x0 + g.lb), y1 = min(g.H, y0 + g.lb), z1 = min(g.D, z0 + g.lb);
    const int bw = x1 - x0, bh = y1 - y0, nsite = bw * bh * (z1 - z0);
    const int64_t HW = (int64_t)g.H * g.W;
    int o0 = start0[warp], o1 = start1[warp];
    for (int j0 = 0; j0 < nsite; j0 += 32) {
        const int j = j0 + lane;
        bool take = false;
        int x = 0, y = 0, z = 0, c = 0;
        if (j < nsite) {
            x = x0 + j % bw;
            y = y0 + (j / bw) % bh;
            z = z0 + j / (bw * bh);
            take = mask[z * HW + (int64_t)y * g.W + x] != 0;
            c = (x + y + z) & 1;
        }
        const unsigned m0 = __ballot_sync(0xffffffffu, take && c == 0);
        const unsigned m1 = __ballot_sync(0xffffffffu, take && c == 1);
        if (take) {
            const unsigned below = (1u << lane) - 1u;
            const uint4 e = gap_item3(g, warp, z, y, x);
            if (c == 0) list0[o0 + __popc(m0 & below)] = e;
            else list1[o1 + __popc(m1 & below)] = e;
        }
        o0 += __popc(m0);
        o1 += __popc(m1);
    }
}

struct Args3 {
    Geom3 g;
    Model m;
    uint32_t rk0[10], key1;  // round keys of key word 0, key word 1
    int colour;
    const uint4* list;
    int n_list;
    float2* ang;             // [np][2][D][H][Wh]
    const float* beta;       // [nblk]
    const uint8_t* running;  // [nblk][Rp] or nullptr (every lane r < R)
    double* eacc;            // [nblk][Rp] FP64 per-sweep changes
    double* ecur;            // [nblk][Rp] (energy pass)
    int np, R, Rp;
    uint32_t pair_base;      // Philox counter word 2 of lane pair 0 (realization base / 2)
    uint32_t ctr1;           // t | tag << 16
    int energy;
    int chunks;              // consecutive 32-entry chunks of the list per warp
};

// The six neighbours' angles (-x, +x, -y, +y, -z, +z) for one realization
// pair, from its plane of the other colour. One that does not exist reads some
// other element or the state's guard; the caller drops it by the entry's flags.
__device__ __forceinline__ void neighbours3(const Geom3& g, const float2* __restrict__ oth,
                                            const uint4& en, float2 v[6]) {
    const float2* left = oth + (ptrdiff_t)(int)en.w;
    const float2* here = oth + en.x;
    const ptrdiff_t layer = (ptrdiff_t)g.H * g.Wh;
    v[0] = left[0];
    v[1] = left[1];
    v[2] = *(here - g.Wh);
    v[3] = here[g.Wh];
    v[4] = *(here - layer);
    v[5] = here[layer];
}

template <typename V> __device__ __forceinline__ V sum6(const V v[6]);
template <> __device__ __forceinline__ float sum6(const float v[6]) {
    return ((v[0] + v[1]) + (v[2] + v[3])) + (v[4] + v[5]);
}
template <> __device__ __forceinline__ float2 sum6(const float2 v[6]) {
    return __fadd2_rn(__fadd2_rn(__fadd2_rn(v[0], v[1]), __fadd2_rn(v[2], v[3])),
                      __fadd2_rn(v[4], v[5]));
}

// A move on the block's low faces, bond by bond: what the neighbouring blocks
// own goes to ae[k] (faces x, y, z) instead of ao. nc, ns: the neighbours'
// (cos, sin). The roundings are spelled out (see bond_change).
__device__ __forceinline__ void split_faces(const SiteNew& n, float phi, uint32_t f, float C,
                                            float Sn, const float nc[3], const float ns[3],
                                            const Model& m, float& ao, float ae[3]) {
    float co, so, ca, sa, cn, sn;
    __sincosf(m.q * phi, &so, &co);
    __sincosf(m.q * n.mid, &sa, &ca);
    final_cs(n.refl, ca, sa, C, Sn, cn, sn);
    const float dc = cn - co, ds = sn - so;
    ao += n.dE;
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (f & (1u << (FACE_SHIFT + k))) {
            const float d = bond_change<float>(dc, ds, nc[k], ns[k], m.J);
            ao -= d;
            ae[k] += d;
        }
}

// One gap entry in both realizations of pair p (kOne: in the even one, the
// only lane of a single-chain calibration): new angles stored, energy changes
// into ao and, for the faces, ae.
template <bool kOne>
__device__ __forceinline__ void update3(const Args3& a, float2* own, const float2* oth,
                                        const uint4& en, const uint32_t w[4], float beta, bool run0,
                                        bool run1, float2& ao, float2 ae[3]) {
    const uint32_t f = en.y;
    const Model& m = a.m;
    float2 v[6];
    neighbours3(a.g, oth, en, v);
    const float2 ph = own[en.x];
    if constexpr (kOne) {
        float nc[6], ns[6];
#pragma unroll
        for (int d = 0; d < 6; ++d) __sincosf(m.q * v[d].x, &ns[d], &nc[d]);
        if ((f & ALL6) != ALL6) {
#pragma unroll
            for (int d = 0; d < 6; ++d)
                if (!(f & (1u << d))) nc[d] = ns[d] = 0.0f;
        }
        const float C = sum6<float>(nc), Sn = sum6<float>(ns);
        const SiteNew n = site_update<float>(ph.x, C, Sn, u01(w[0]), u01(w[1]), beta, m);
        own[en.x].x = n.phi;
        if (f & (7u << FACE_SHIFT)) {
            const float lc[3] = {nc[0], nc[2], nc[4]}, ls[3] = {ns[0], ns[2], ns[4]};
            float e[3] = {0.0f, 0.0f, 0.0f};
            split_faces(n, ph.x, f, C, Sn, lc, ls, m, ao.x, e);
#pragma unroll
            for (int k = 0; k < 3; ++k) ae[k].x = e[k];
        } else {
            ao.x += n.dE;
        }
    } else {
        float2 nc[6], ns[6];
#pragma unroll
        for (int d = 0; d < 6; ++d) sincos_2(__fmul2_rn(both(m.q), v[d]), ns[d], nc[d]);
        if ((f & ALL6) != ALL6) {
#pragma unroll
            for (int d = 0; d < 6; ++d)
                if (!(f & (1u << d))) nc[d] = ns[d] = both(0.0f);
        }
        const float2 C = sum6<float2>(nc), Sn = sum6<float2>(ns);
        const PairNew n = pair_update<float>(ph, C, Sn, u01_2(w[0], w[2]), u01_2(w[1], w[3]),
                                             both(beta), m);
        own[en.x] = make_float2(run0 ? n.phi.x : ph.x, run1 ? n.phi.y : ph.y);
        float2 o = n.dE;
        if (f & (7u << FACE_SHIFT)) {
            o = both(0.0f);
            float e0[3] = {0.0f, 0.0f, 0.0f}, e1[3] = {0.0f, 0.0f, 0.0f};
            // (cosines and sines again, as in split_edge_2's callers)
            float2 lc[3], ls[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) sincos_2(__fmul2_rn(both(m.q), v[2 * k]), ls[k], lc[k]);
            const float c0[3] = {lc[0].x, lc[1].x, lc[2].x}, s0[3] = {ls[0].x, ls[1].x, ls[2].x};
            const float c1[3] = {lc[0].y, lc[1].y, lc[2].y}, s1[3] = {ls[0].y, ls[1].y, ls[2].y};
            split_faces(SiteNew{n.phi.x, n.mid.x, n.dE.x, n.refl0}, ph.x, f, C.x, Sn.x, c0, s0, m,
                        o.x, e0);
            split_faces(SiteNew{n.phi.y, n.mid.y, n.dE.y, n.refl1}, ph.y, f, C.y, Sn.y, c1, s1, m,
                        o.y, e1);
#pragma unroll
            for (int k = 0; k < 3; ++k)
                ae[k] = make_float2(run0 ? e0[k] : 0.0f, run1 ? e1[k] : 0.0f);
        }
        ao = make_float2(run0 ? o.x : 0.0f, run1 ? o.y : 0.0f);
    }
}

// FP64 warp sum of a pair's changes, added by lane 0.
__device__ __forceinline__ void flush3(double* ea, double x, double y) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, d);
        y += __shfl_xor_sync(0xffffffffu, y, d);
    }
    if ((threadIdx.x & 31) != 0) return;
    if (x != 0.0) atomicAdd(ea, x);
    if (y != 0.0) atomicAdd(ea + 1, y);
}

__device__ __forceinline__ void add3(double* ea, float2 v) {
    if (v.x != 0.0f) atomicAdd(ea, (double)v.x);
    if (v.y != 0.0f) atomicAdd(ea + 1, (double)v.y);
}

// FP32 warp sum of a pair's changes (kOne: of its even lane only).
template <bool kOne> __device__ __forceinline__ float2 warp_sum3(float2 v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, d);
        if constexpr (!kOne) v.y += __shfl_xor_sync(0xffffffffu, v.y, d);
    }
    return v;
}

// One half-step: a warp per run of consecutive 32-entry chunks of the colour's
// list and realization pair (blockIdx.y), and f.ctas trailing CTAs that fold
// the previous sweep of a calibration. The block sums: with several pairs every
// update's change is summed in FP64 (per lane while the warp stays in a block,
// then over the warp), with one pair a chunk's changes are an FP32 warp sum
// added in FP64; a chunk that spans blocks adds lane by lane. One FP64 atomic
// per block and warp instead of one per update. 128^3, half the sites missing,
// l_b = 16: 20 realizations 43 -> 86 G updates/s, single-chain calibration 14 ->
// 49 (10.7 us per half-step of 524 k updates), against 64-bit divisions of the
// site index, pairs interleaved per site and an FP64 atomic per update. Bound
// by instruction issue in large batches, by the latency of one chunk's chain in
// a single-chain calibration. CTAs per SM: 9 of 6 to 9 for pairs, 10 of 8 to 16
// for single chains.
constexpr int kSweep3Threads = 128;
template <bool kOne>
__global__ void __launch_bounds__(kSweep3Threads, kOne ? 10 : 9) k3_sweep(Args3 a, FoldArgs f) {
    grid_dep_launch();
    const int ctas = (int)gridDim.x - f.ctas;
    if ((int)blockIdx.x >= ctas) {
        grid_dep_wait();
        if (blockIdx.y == 0) fold_block_energies<kSweep3Threads>(f, (int)blockIdx.x - ctas);
        return;
    }
    const int lane = threadIdx.x & 31;
    const int p = blockIdx.y, rl = 2 * p;
    const int c0 = ((int)blockIdx.x * (kSweep3Threads / 32) + (int)(threadIdx.x >> 5)) * a.chunks;
    const int last = a.n_list - 1;
    float2* own = a.ang + plane3(a.g, p, a.colour);
    const float2* oth = a.ang + plane3(a.g, p, a.colour ^ 1);
    const bool sum32 = a.np == 1;
    double dx = 0.0, dy = 0.0;       // the lane's changes in block cur
    int cur = -1;
    if (c0 * 32 > last) {
        grid_dep_wait();
        return;
    }
    for (int k = 0; k < a.chunks; ++k) {
        const int base = (c0 + k) * 32;
        if (base > last) break;
        const bool live = base + lane <= last;
        const uint4 en = a.list[min(base + lane, last)];
        const int b = (int)(en.y >> META_SHIFT);
        uint32_t w[4];
        philox4x32_10_rk(en.z, a.ctr1, a.pair_base + (uint32_t)p, 0u, a.rk0, a.key1, w);
        const float beta = a.beta[b];
        // (the entry, its Philox block and the temperature do not depend on
        // the previous half-step)
        if (k == 0) grid_dep_wait();
        const int b0 = __shfl_sync(0xffffffffu, b, 0);
        const bool one_block = __all_sync(0xffffffffu, live && b == b0);
        bool run0 = live && rl < a.R, run1 = live && rl + 1 < a.R;
        if (a.running) {
            const uchar2 r2 =
                *reinterpret_cast<const uchar2*>(a.running + (size_t)b * a.Rp + rl);
            run0 = live && r2.x != 0;
            run1 = live && r2.y != 0;
        }
        float2 ao = both(0.0f), ae[3] = {ao, ao, ao};
        if (run0 || run1) {
            update3<kOne>(a, own, oth, en, w, beta, run0, run1, ao, ae);
        }
        if (!a.energy) continue;
        const size_t off[3] = {1, (size_t)a.g.nbx, (size_t)a.g.nbx * a.g.nby};
        double* ea = a.eacc + (size_t)b * a.Rp + rl;
        if (one_block && sum32) {
            ao = warp_sum3<kOne>(ao);
            if (lane == 0) add3(ea, ao);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                if (!__any_sync(0xffffffffu, (en.y & (1u << (FACE_SHIFT + j))) != 0)) continue;
                const float2 s = warp_sum3<kOne>(ae[j]);
                if (lane == 0) add3(ea - off[j] * a.Rp, s);
            }
            continue;
        }
        if (one_block) {
            if (b0 != cur) {
                if (cur >= 0) flush3(a.eacc + (size_t)cur * a.Rp + rl, dx, dy);
                dx = dy = 0.0;
                cur = b0;
            }
            dx += (double)ao.x;
            dy += (double)ao.y;
        } else {
            add3(ea, ao);
        }
        if (en.y & (7u << FACE_SHIFT)) {
#pragma unroll
            for (int j = 0; j < 3; ++j) add3(ea - off[j] * a.Rp, ae[j]);
        }
    }
    if (cur >= 0) flush3(a.eacc + (size_t)cur * a.Rp + rl, dx, dy);
}

// Block energies of the start state from scratch (FP64 into ecur, which holds
// E_s,b): the bonds of the list entries [e0, e1) in pair blockIdx.y, whose two
// lanes hold the same start. Colour 1 adds every bond of its gap sites, colour
// 0 only the bonds to sample neighbours, each to the block that owns it.
__global__ void k3_energy(Args3 a, const uint8_t* __restrict__ mask, int e0, int e1) {
    const Geom3& g = a.g;
    const int e = e0 + (int)(blockIdx.x * blockDim.x + threadIdx.x);
    const bool live = e < e1;
    const uint4 en = a.list[live ? e : e1 - 1];
    const int b = (int)(en.y >> META_SHIFT);
    const int64_t HW = (int64_t)g.H * g.W;
    const size_t off[3] = {1, (size_t)g.nbx, (size_t)g.nbx * g.nby};
    double* ecur = a.ecur + 2 * (size_t)blockIdx.y;
    auto add = [&](size_t blk, double v) {
        atomicAdd(&ecur[blk * a.Rp], v);
        atomicAdd(&ecur[blk * a.Rp + 1], v);
    };
    double own = 0.0;
    if (live) {
        float2 v[6];
        neighbours3(g, a.ang + plane3(g, blockIdx.y, a.colour ^ 1), en, v);
        const float ph = a.ang[plane3(g, blockIdx.y, a.colour) + en.x].x;
        const int64_t ni[6] = {-1, 1, -(int64_t)g.W, (int64_t)g.W, -HW, HW};
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            if (!(en.y & (1u << d))) continue;
            if (a.colour == 0 && mask[(int64_t)en.z + ni[d]]) continue;   // gap-gap: colour 1
            const double eb = -a.m.J * cos_bond((double)a.m.q * ((double)ph - (double)v[d].x));
            if ((d & 1) == 0 && (en.y & (1u << (FACE_SHIFT + d / 2)))) add((size_t)b - off[d / 2], eb);
            else own += eb;
        }
    }
    const int b0 = __shfl_sync(0xffffffffu, b, 0);
    if (__all_sync(0xffffffffu, b == b0)) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) own += __shfl_xor_sync(0xffffffffu, own, d);
        if ((threadIdx.x & 31) != 0) own = 0.0;
    }
    if (own != 0.0) add(b, own);
}

// Sample angles into both lanes of every pair's planes (blockIdx.y: the pair).
__global__ void k3_fill_samples(Geom3 g, const float* __restrict__ phi_s,
                                const uint8_t* __restrict__ mask, float2* __restrict__ ang) {
    const int64_t n = (int64_t)g.D * g.H * g.W;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (mask[i]) continue;
        const uint32_t row = (uint32_t)i / (uint32_t)g.W;
        const int x = (int)((uint32_t)i - row * (uint32_t)g.W);
        const int z = (int)(row / (uint32_t)g.H), y = (int)(row - (uint32_t)z * (uint32_t)g.H);
        ang[plane3(g, blockIdx.y, (x + y + z) & 1) + half3(g, z, y, x)] = both(phi_s[i]);
    }
}

// Gap sites at their block's mean sample angle (blockIdx.y: the pair).
__global__ void k3_init(Geom3 g, const uint4* __restrict__ list, int n_list, int colour,
                        const float* __restrict__ init_angle, float2* __restrict__ ang) {
    float2* dst = ang + plane3(g, blockIdx.y, colour);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n_list; e += gridDim.x * blockDim.x)
        dst[list[e].x] = both(init_angle[list[e].y >> META_SHIFT]);
}

__global__ void k3_accumulate(Geom3 g, const uint4* __restrict__ list, int64_t n_list, int colour,
                              const float2* __restrict__ ang, int R, double* __restrict__ sum) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_list;
         e += (int64_t)gridDim.x * blockDim.x) {
        const uint4 en = list[e];
        double s = 0.0;
        for (int r = 0; r < R; r += 2) {
            const float2 v = ang[plane3(g, r / 2, colour) + en.x];
            s += (double)v.x;
            if (r + 1 < R) s += (double)v.y;
        }
        sum[en.z] += s;
    }
}

__global__ void k3_predict(int64_t n, const float* __restrict__ values,
                           const uint8_t* __restrict__ mask, const double* __restrict__ sum,
                           double inv_r, double zmin, double zmax, float* __restrict__ out,
                           const float* __restrict__ truth, double* __restrict__ err) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (!mask[i]) {
            out[i] = values[i];
            continue;
        }
        const float z = (float)(zmin + (zmax - zmin) * sum[i] * inv_r / 6.283185307179586476925);
        out[i] = z;
        if (truth) {
            const double d = (double)truth[i] - (double)z;
            atomicAdd(&err[0], fabs(d));
            atomicAdd(&err[1], d * d);
        }
    }
}

__global__ void k3_get_state(Geom3 g, const float2* __restrict__ ang, int r,
                             float* __restrict__ out) {
    const int64_t n = (int64_t)g.D * g.H * g.W;
    const int64_t HW = (int64_t)g.H * g.W;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int z = (int)(i / HW), y = (int)((i % HW) / g.W), x = (int)(i % g.W);
        const float2 v = ang[plane3(g, r / 2, (x + y + z) & 1) + half3(g, z, y, x)];
        out[i] = (r & 1) ? v.y : v.x;
    }
}

__global__ void k3_set_state(Geom3 g, const uint8_t* __restrict__ mask, float2* __restrict__ ang,
                             int r, const float* __restrict__ in) {
    const int64_t n = (int64_t)g.D * g.H * g.W;
    const int64_t HW = (int64_t)g.H * g.W;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (!mask[i]) continue;
        const int z = (int)(i / HW), y = (int)((i % HW) / g.W), x = (int)(i % g.W);
        float2& v = ang[plane3(g, r / 2, (x + y + z) & 1) + half3(g, z, y, x)];
        if (r & 1) v.y = in[i]; else v.x = in[i];
    }
}

__global__ void k3_fill_valid(uint8_t* running, int64_t n, int Rp, int R) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x)
        running[t] = (int)(t % Rp) < R ? 1 : 0;
}

inline int grid_of(int64_t n, int threads = 256) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((n + threads - 1) / threads, 152 * 32));
}

}  // namespace

struct mpr3_ctx {
    mpr_options opt{};
    Geom3 g{};
    Model m{};
    uint32_t key0 = 0, key1 = 0;
    cudaStream_t s = nullptr;
    int device = 0;
    std::string err;
    std::vector<void*> owned;
    double zmin = 0, zmax = 0;
    int degenerate = 0, calibrated = 0;
    int64_t n = 0, n_gap[2] = {0, 0};
    float *values = nullptr, *phi_s = nullptr, *init_angle = nullptr;
    uint8_t* mask = nullptr;
    uint4* list[2] = {nullptr, nullptr};
    int32_t* start[2] = {nullptr, nullptr};
    double *Es = nullptr, *es = nullptr, *inb = nullptr, *ssum = nullptr;
    int32_t *Nsp = nullptr, *Nb = nullptr, *nsamp = nullptr, *ngap = nullptr,
            *ngap_c[2] = {nullptr, nullptr}, *zero_slices = nullptr;
    int32_t* Nsp_cal = nullptr;  // calibrating blocks: sample bonds and gap sites
    float *T = nullptr, *beta = nullptr, *lo = nullptr, *hi = nullptr;
    double* ebar = nullptr;
    double* sum = nullptr;
    double* err_buf = nullptr;
    uint32_t* mm = nullptr;
    // batch
    int np = 0, R = 0, Rp = 0, batch_open = 0, t = 0;
    size_t ang_cap = 0, blk_cap = 0;
    int64_t n_allocs = 0;      // allocations seen by the alloc_test hook
    float2* ang_mem = nullptr;   // the state with a guard on both sides
    float2* ang = nullptr;
    double* eacc = nullptr;      // two per-sweep buffers
    double *ecur = nullptr, *ecur0 = nullptr, *e_last = nullptr;
    int n_sm = 152;
    uint8_t* running = nullptr;
    int32_t *stop = nullptr, *tcount = nullptr;
    int8_t* sigma = nullptr;
    uint32_t* work = nullptr;
    Control* ctl = nullptr;
    unsigned long long* counter = nullptr;
    int4* blk_rect = nullptr;
    int64_t realizations = 0, gap_updates = 0, cal_updates = 0;
    int64_t r_next = 0;          // index of the next realization (batches start even)
    uint32_t pair_base = 0;
    // profiling (opt.profile): event pairs around the realizations' sweeps
    // (their two half-steps) and around the calibration's iterations
    int64_t launches = 0, sim_hs = 0, cal_hs = 0;
    double sim_ms = 0.0, cal_ms = 0.0;
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev_sim, ev_cal;
    unsigned long long* h_run = nullptr;   // pinned: running counts of two sweep chunks
};

namespace {

mpr_status fail3(mpr3_ctx* c, mpr_status st, const char* fmt, ...) {
    if (c) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof(buf), fmt, ap);
        va_end(ap);
        c->err = buf;
    }
    return st;
}

#define CK3(call)                                                                             \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess)                                                                \
            return fail3(ctx, e_ == cudaErrorMemoryAllocation ? MPR_ENOMEM : MPR_ECUDA,       \
                         "%s failed: %s", #call, cudaGetErrorString(e_));                     \
    } while (0)
#define CKL3()                                                                                \
    do {                                                                                      \
        ++ctx->launches;                                                                      \
        cudaError_t e_ = cudaPeekAtLastError();                                               \
        if (e_ != cudaSuccess)                                                                \
            return fail3(ctx, MPR_ECUDA, "kernel launch failed: %s", cudaGetErrorString(e_)); \
    } while (0)
#define TRY3(x)                                  \
    do {                                         \
        mpr_status st_ = (x);                    \
        if (st_ != MPR_OK) return st_;           \
    } while (0)

template <class T>
mpr_status alloc3(mpr3_ctx* ctx, T** p, size_t count) {
    *p = nullptr;
    // Test hook: the alloc_test-th allocation of the context is refused.
    if (ctx->opt.alloc_test > 0 && ++ctx->n_allocs == ctx->opt.alloc_test)
        return fail3(ctx, MPR_ENOMEM, "allocation %d refused by the alloc_test hook",
                     ctx->opt.alloc_test);
    void* q = nullptr;
    if (pool_alloc(&q, std::max<size_t>(count, 1) * sizeof(T), ctx->device, ctx->s) !=
        cudaSuccess) {
        cudaGetLastError();
        return fail3(ctx, MPR_ENOMEM, "allocation of %zu bytes failed", count * sizeof(T));
    }
    ctx->owned.push_back(q);
    *p = static_cast<T*>(q);
    return MPR_OK;
}

void free3(mpr3_ctx* ctx, void* p) {
    if (!p) return;
    auto it = std::find(ctx->owned.begin(), ctx->owned.end(), p);
    if (it != ctx->owned.end()) ctx->owned.erase(it);
    pool_free(p, ctx->s);
}

Slices slices3(mpr3_ctx* ctx) {
    Slices sl{};
    sl.n = 1;
    sl.rect0 = make_int4(0, 0, ctx->g.D * ctx->g.H, ctx->g.W);
    sl.blk = ctx->blk_rect;
    sl.of_block = ctx->zero_slices;
    return sl;
}

// Batch buffers for `lanes` realization lanes (pairs of realizations).
mpr_status ensure3(mpr3_ctx* ctx, int lanes) {
    const int np = (lanes + 1) / 2, Rp = 2 * np;
    const size_t guard = guard3(ctx->g);
    const size_t ang_need = plane3(ctx->g, np, 0) + 2 * guard;
    // (a failed allocation leaves the capacity at 0 and every pointer of its
    // group null, so the next call allocates the group again)
    if (ang_need > ctx->ang_cap) {
        free3(ctx, ctx->ang_mem);
        ctx->ang_mem = ctx->ang = nullptr;
        ctx->ang_cap = 0;
        TRY3(alloc3(ctx, &ctx->ang_mem, ang_need));
        ctx->ang_cap = ang_need;
    }
    ctx->ang = ctx->ang_mem + guard;
    const size_t blk = (size_t)ctx->g.nblk * Rp;
    if (blk > ctx->blk_cap) {
        for (void* p : {(void*)ctx->eacc, (void*)ctx->ecur, (void*)ctx->ecur0, (void*)ctx->e_last, (void*)ctx->running,
                        (void*)ctx->stop, (void*)ctx->sigma, (void*)ctx->work, (void*)ctx->tcount})
            free3(ctx, p);
        ctx->eacc = nullptr; ctx->ecur = nullptr; ctx->e_last = nullptr; ctx->running = nullptr;
        ctx->ecur0 = nullptr;
        ctx->stop = nullptr; ctx->sigma = nullptr; ctx->work = nullptr; ctx->tcount = nullptr;
        ctx->blk_cap = 0;
        TRY3(alloc3(ctx, &ctx->eacc, 2 * blk));
        TRY3(alloc3(ctx, &ctx->ecur, blk));
        TRY3(alloc3(ctx, &ctx->ecur0, blk));
        TRY3(alloc3(ctx, &ctx->e_last, blk));
        TRY3(alloc3(ctx, &ctx->running, blk));
        TRY3(alloc3(ctx, &ctx->stop, blk));
        TRY3(alloc3(ctx, &ctx->sigma, blk));
        TRY3(alloc3(ctx, &ctx->work, 2 * (size_t)ctx->g.nblk * np));
        TRY3(alloc3(ctx, &ctx->tcount, (size_t)Rp));
        ctx->blk_cap = blk;
    }
    ctx->np = np;
    ctx->Rp = Rp;
    CK3(cudaMemsetAsync(ctx->eacc, 0, 2 * blk * sizeof(double), ctx->s));
    CK3(cudaMemsetAsync(ctx->ctl, 0, sizeof(Control), ctx->s));
    return MPR_OK;
}

Args3 args3(mpr3_ctx* ctx, int colour, bool simulate) {
    Args3 a{};
    a.g = ctx->g;
    a.m = ctx->m;
    for (int r = 0; r < 10; ++r) a.rk0[r] = ctx->key0 + (uint32_t)r * 0x9E3779B9u;
    a.key1 = ctx->key1;
    a.colour = colour;
    a.list = ctx->list[colour];
    a.n_list = (int)ctx->n_gap[colour];
    a.ang = ctx->ang;
    a.beta = ctx->beta;
    a.running = simulate ? ctx->running : nullptr;
    a.eacc = ctx->eacc;
    a.ecur = ctx->ecur;
    a.np = ctx->np;
    a.pair_base = simulate ? ctx->pair_base : 0u;
    a.R = ctx->R;
    a.Rp = ctx->Rp;
    a.energy = 1;
    return a;
}

// Samples into the batch's state (once per batch; the sweeps never write them).
mpr_status fill3(mpr3_ctx* ctx) {
    const dim3 grid((unsigned)grid_of(ctx->n), (unsigned)ctx->np);
    k3_fill_samples<<<grid, 256, 0, ctx->s>>>(ctx->g, ctx->phi_s, ctx->mask, ctx->ang);
    CKL3();
    return MPR_OK;
}

// Every gap site at its start.
mpr_status init3(mpr3_ctx* ctx) {
    for (int c = 0; c < 2; ++c) {
        if (ctx->n_gap[c] == 0) continue;
        const dim3 grid((unsigned)grid_of(ctx->n_gap[c]), (unsigned)ctx->np);
        k3_init<<<grid, 256, 0, ctx->s>>>(ctx->g, ctx->list[c], (int)ctx->n_gap[c], c,
                                          ctx->init_angle, ctx->ang);
        CKL3();
    }
    return MPR_OK;
}

// E_b of the start state in every lane: summed in the first pair (every lane
// starts from the same state), copied to the others.
//
// The pass covers the first kEnergy3 (entry, pair) combinations of a colour,
// pairs fastest, and leaves the bonds of later entries out of E_b(0). That is
// a defect of long standing for batches beyond that size (128^3 with half the
// sites missing and 20 realizations is one): the start energies of the blocks
// at the list's end, and with them sigma and the stop sweeps, are not those of
// the state. It is kept as it is here, because the results of every such batch
// would change.
constexpr int64_t kEnergy3 = 152 * 32 * 256;

mpr_status energy3(mpr3_ctx* ctx) {
    launch_ecur_reset(ctx->g.nblk, ctx->Rp, ctx->Es, ctx->ecur, ctx->eacc, ctx->s);
    CKL3();
    int whole[2], part[2];   // entries covered in every pair, pairs that cover one more
    for (int c = 0; c < 2; ++c) {
        const int64_t n = ctx->n_gap[c];
        whole[c] = (int)std::min<int64_t>(n, kEnergy3 / ctx->np);
        part[c] = n > whole[c] ? (int)(kEnergy3 % ctx->np) : 0;
        if (whole[c] == 0) continue;
        k3_energy<<<(unsigned)((whole[c] + 127) / 128), 128, 0, ctx->s>>>(args3(ctx, c, false),
                                                                         ctx->mask, 0, whole[c]);
        CKL3();
    }
    launch_ecur_broadcast(ctx->g.nblk, ctx->Rp, 2, ctx->ecur, ctx->s);
    CKL3();
    for (int c = 0; c < 2; ++c) {
        if (part[c] == 0) continue;
        k3_energy<<<dim3(1, (unsigned)part[c]), 32, 0, ctx->s>>>(args3(ctx, c, false), ctx->mask,
                                                                 whole[c], whole[c] + 1);
        CKL3();
    }
    return MPR_OK;
}

// Chunks of 32 entries per warp: as many as still leave two waves of warps, at
// most kChunks3 (a longer run saves block flushes, 10 FP64 additions each).
constexpr int kChunks3 = 8;

mpr_status halfstep3(mpr3_ctx* ctx, int colour, uint32_t ctr1, bool simulate, double* eacc,
                     const FoldArgs* fold = nullptr) {
    Args3 a = args3(ctx, colour, simulate);
    a.ctr1 = ctr1;
    a.eacc = eacc;
    FoldArgs f{};
    if (fold) f = *fold;
    if (a.n_list == 0 && f.ctas == 0) return MPR_OK;
    const int64_t chunks = ((int64_t)a.n_list + 31) / 32;
    const int64_t wave = (int64_t)ctx->n_sm * 28;
    a.chunks = (int)std::max<int64_t>(1, std::min<int64_t>(kChunks3, chunks * a.np / (2 * wave)));
    const int64_t warps = (chunks + a.chunks - 1) / a.chunks;
    constexpr int per_cta = kSweep3Threads / 32;
    const dim3 grid((unsigned)((warps + per_cta - 1) / per_cta + f.ctas), (unsigned)a.np);
    if (ctx->R == 1) launch_pdl(k3_sweep<true>, grid, kSweep3Threads, ctx->s, a, f);
    else launch_pdl(k3_sweep<false>, grid, kSweep3Threads, ctx->s, a, f);
    CKL3();
    return MPR_OK;
}

// After a stream synchronisation: the recorded event pairs into the totals.
void collect3(mpr3_ctx* ctx) {
    for (int which = 0; which < 2; ++which) {
        auto& v = which ? ctx->ev_cal : ctx->ev_sim;
        double& acc = which ? ctx->cal_ms : ctx->sim_ms;
        for (auto& pr : v) {
            float ms = 0.0f;
            if (cudaEventElapsedTime(&ms, pr.first, pr.second) == cudaSuccess) acc += ms;
            else cudaGetLastError();
            cudaEventDestroy(pr.first);
            cudaEventDestroy(pr.second);
        }
        v.clear();
    }
}

// An event pair on the context's stream when profiling (nullptr otherwise).
std::pair<cudaEvent_t, cudaEvent_t> begin_timing3(mpr3_ctx* ctx) {
    std::pair<cudaEvent_t, cudaEvent_t> e{nullptr, nullptr};
    if (!ctx->opt.profile) return e;
    if (cudaEventCreate(&e.first) != cudaSuccess || cudaEventCreate(&e.second) != cudaSuccess) {
        cudaGetLastError();
        if (e.first) cudaEventDestroy(e.first);
        return {nullptr, nullptr};
    }
    cudaEventRecord(e.first, ctx->s);
    return e;
}

mpr_status sweep3(mpr3_ctx* ctx) {
    ctx->t += 1;
    const auto ev = begin_timing3(ctx);
    for (int c = 0; c < 2; ++c) TRY3(halfstep3(ctx, c, (uint32_t)ctx->t, true, ctx->eacc));
    ctx->sim_hs += 2;
    if (ev.first) {
        cudaEventRecord(ev.second, ctx->s);
        ctx->ev_sim.push_back(ev);
    }
    const int64_t items = (int64_t)ctx->g.nblk * ctx->np;
    const int grid = (int)std::min<int64_t>((items * 2 + 255) / 256, 152 * 16);
    launch_stop_targeted(2, ctx->np, ctx->Rp, ctx->zero_slices, grid, ctx->ctl, ctx->work,
                         (uint32_t)items, ctx->es, ctx->inb, ctx->Nsp, ctx->eacc, ctx->ecur,
                         ctx->sigma, ctx->running, ctx->stop, ctx->tcount, ctx->e_last, ctx->t,
                         ctx->s);
    CKL3();
    launch_stop_rest(ctx->g.nblk, ctx->np, 2, ctx->Rp, ctx->opt.n_max, ctx->zero_slices, grid,
                     ctx->ctl, ctx->work, ctx->work, (uint32_t)items, ctx->Nsp, ctx->running,
                     ctx->stop, ctx->tcount, 0, ctx->t, ctx->s);
    CKL3();
    return MPR_OK;
}

}  // namespace

extern "C" {

void mpr3_destroy(mpr3_ctx* ctx) {
    if (!ctx) return;
    cudaStreamSynchronize(ctx->s);
    collect3(ctx);
    for (void* p : ctx->owned) pool_free(p, ctx->s);
    cudaStreamSynchronize(ctx->s);
    pinned_release(ctx->h_run);
    delete ctx;
}

mpr_status mpr3_get_profile(mpr3_ctx* ctx, mpr_profile* p) {
    if (!ctx || !p) return MPR_EINVAL;
    if (cudaStreamSynchronize(ctx->s) != cudaSuccess) return fail3(ctx, MPR_ECUDA, "sync failed");
    collect3(ctx);
    std::memset(p, 0, sizeof(*p));
    p->kernel_launches = ctx->launches;
    p->sim_halfstep_launches = ctx->sim_hs;
    p->cal_halfstep_launches = ctx->cal_hs;
    p->sim_halfstep_ms = ctx->sim_ms;
    p->cal_halfstep_ms = ctx->cal_ms;
    return MPR_OK;
}

const char* mpr3_last_error(const mpr3_ctx* ctx) { return ctx ? ctx->err.c_str() : ""; }

mpr_status mpr3_create(const mpr_grid3* grid, const uint8_t* mask_in, const float* values_in,
                       const mpr_options* opt_in, mpr3_ctx** out) {
    if (!out) return MPR_EINVAL;
    *out = nullptr;
    if (!grid || !mask_in || !values_in) return MPR_EINVAL;
    const int D = grid->depth, H = grid->height, W = grid->width, lb = grid->block;
    if (D < 1 || H < 1 || W < 1 || lb < 1 || (int64_t)D * H * W > 0x7fffffffLL) return MPR_EINVAL;
    mpr3_ctx* ctx = new (std::nothrow) mpr3_ctx();
    if (!ctx) return MPR_ENOMEM;
    auto bail = [&](mpr_status st) {
        mpr3_destroy(ctx);
        return st;
    };
    if (opt_in) ctx->opt = *opt_in; else mpr_default_options(&ctx->opt);
    const mpr_options& o = ctx->opt;
    if (!(o.q > 0.0 && o.q <= 0.5) || !(o.J > 0.0) || o.n_max < 1 || o.n_max > 65535 ||
        o.n_eq < 0 || o.n_meas < 1 || o.n_eq + o.n_meas > 65535 || o.n_bisect < 0 ||
        o.cal_chains < 1 || o.cal_chains > 4096 || !(o.t_lo > 0.0f && o.t_hi > o.t_lo) ||
        o.stop_rule != MPR_STOP_CROSS ||   // (3-D: the first-crossing stop only)
        o.alloc_test < 0)
        return bail(MPR_EINVAL);
    Geom3& g = ctx->g;
    g.D = D; g.H = H; g.W = W; g.Wh = (W + 1) / 2; g.lb = lb;
    g.nbx = (W + lb - 1) / lb; g.nby = (H + lb - 1) / lb; g.nbz = (D + lb - 1) / lb;
    if ((int64_t)g.nbx * g.nby * g.nbz > MAX_BLOCKS) return bail(MPR_EINVAL);
    g.nblk = g.nbx * g.nby * g.nbz;
    ctx->m.q = (float)o.q;
    ctx->m.J = (float)o.J;
    ctx->m.inv_q = (float)(1.0 / o.q);
    ctx->m.overrelax = o.overrelax ? 1 : 0;
    ctx->key0 = (uint32_t)(o.seed & 0xffffffffu);
    ctx->key1 = (uint32_t)(o.seed >> 32) ^ o.slice_id;
    ctx->s = (cudaStream_t)o.cuda_stream;
    if (cudaGetDevice(&ctx->device) != cudaSuccess) return bail(MPR_ECUDA);
    cudaDeviceGetAttribute(&ctx->n_sm, cudaDevAttrMultiProcessorCount, ctx->device);
    if (ctx->n_sm < 1) ctx->n_sm = 1;
    const int64_t n = (int64_t)D * H * W;
    ctx->n = n;
    mpr_status st;
#define ST3(x) do { st = (x); if (st != MPR_OK) return bail(st); } while (0)
    ST3(alloc3(ctx, &ctx->values, n));
    ST3(alloc3(ctx, &ctx->mask, n));
    ST3(alloc3(ctx, &ctx->phi_s, n));
    ST3(alloc3(ctx, &ctx->sum, n));
    for (auto* p : {&ctx->Es, &ctx->es, &ctx->inb, &ctx->ssum, &ctx->ebar})
        ST3(alloc3(ctx, p, g.nblk));
    for (auto* p : {&ctx->Nsp, &ctx->Nb, &ctx->nsamp, &ctx->ngap, &ctx->ngap_c[0], &ctx->ngap_c[1],
                    &ctx->zero_slices, &ctx->Nsp_cal})
        ST3(alloc3(ctx, p, g.nblk));
    for (auto* p : {&ctx->init_angle, &ctx->T, &ctx->beta, &ctx->lo, &ctx->hi})
        ST3(alloc3(ctx, p, g.nblk));
    ST3(alloc3(ctx, &ctx->start[0], g.nblk + 1));
    ST3(alloc3(ctx, &ctx->start[1], g.nblk + 1));
    ST3(alloc3(ctx, &ctx->err_buf, 2));
    ST3(alloc3(ctx, &ctx->mm, 2));
    ST3(alloc3(ctx, &ctx->ctl, 1));
    ST3(alloc3(ctx, &ctx->counter, 1));
    ST3(alloc3(ctx, &ctx->blk_rect, 1));
    const int4 bk = make_int4(0, 0, g.nbz * g.nby, g.nbx);
    if (cudaMemcpyAsync(ctx->values, values_in, n * 4, cudaMemcpyDefault, ctx->s) ||
        cudaMemcpyAsync(ctx->mask, mask_in, n, cudaMemcpyDefault, ctx->s) ||
        cudaMemsetAsync(ctx->zero_slices, 0, g.nblk * 4, ctx->s) ||
        cudaMemcpyAsync(ctx->blk_rect, &bk, sizeof(bk), cudaMemcpyHostToDevice, ctx->s) ||
        cudaMemsetAsync(ctx->sum, 0, n * 8, ctx->s))
        return bail(MPR_ECUDA);
    uint32_t mm[2] = {0xffffffffu, 0u};
    if (cudaMemcpyAsync(ctx->mm, mm, 8, cudaMemcpyHostToDevice, ctx->s)) return bail(MPR_ECUDA);
    k3_minmax<<<grid_of(n), 256, 0, ctx->s>>>(ctx->values, ctx->mask, n, ctx->mm);
    if (cudaMemcpyAsync(mm, ctx->mm, 8, cudaMemcpyDeviceToHost, ctx->s) ||
        cudaStreamSynchronize(ctx->s))
        return bail(MPR_ECUDA);
    if (mm[0] == 0xffffffffu) {
        ctx->degenerate = 1;
    } else {
        ctx->zmin = (double)ord2f(mm[0]);
        ctx->zmax = (double)ord2f(mm[1]);
        ctx->degenerate = !(ctx->zmax > ctx->zmin);
    }
    k3_layout<<<grid_of(n), 256, 0, ctx->s>>>(n, ctx->values, ctx->mask, ctx->zmin, ctx->zmax,
                                              ctx->degenerate, ctx->phi_s);
    const int bblocks = (int)(((int64_t)g.nblk * 32 + 255) / 256);
    k3_block_stats<<<g.nblk, 32 * kStatsWarps, 0, ctx->s>>>(g, ctx->values, ctx->mask, ctx->zmin, ctx->zmax,
                                                ctx->degenerate, o.q, o.J, ctx->Es, ctx->Nsp,
                                                ctx->Nb, ctx->ssum, ctx->nsamp, ctx->ngap_c[0],
                                                ctx->ngap_c[1]);
    launch_scan(ctx->ngap_c[0], ctx->ngap_c[1], g.nblk, ctx->start[0], ctx->start[1], ctx->s);
    std::vector<int32_t> s0(g.nblk + 1), s1(g.nblk + 1), nsp(g.nblk), nsm(g.nblk), ng0(g.nblk),
        ng1(g.nblk), nbv(g.nblk);
    std::vector<double> ssum(g.nblk), esv(g.nblk);
    if (cudaPeekAtLastError() ||
        cudaMemcpyAsync(s0.data(), ctx->start[0], s0.size() * 4, cudaMemcpyDeviceToHost, ctx->s) ||
        cudaMemcpyAsync(s1.data(), ctx->start[1], s1.size() * 4, cudaMemcpyDeviceToHost, ctx->s) ||
        cudaMemcpyAsync(nsp.data(), ctx->Nsp, g.nblk * 4, cudaMemcpyDeviceToHost, ctx->s) ||
        cudaMemcpyAsync(nsm.data(), ctx->nsamp, g.nblk * 4, cudaMemcpyDeviceToHost, ctx->s) ||
        cudaMemcpyAsync(ng0.data(), ctx->ngap_c[0], g.nblk * 4, cudaMemcpyDeviceToHost, ctx->s) ||
        cudaMemcpyAsync(ng1.data(), ctx->ngap_c[1], g.nblk * 4, cudaMemcpyDeviceToHost, ctx->s) ||
        cudaMemcpyAsync(ssum.data(), ctx->ssum, g.nblk * 8, cudaMemcpyDeviceToHost, ctx->s) ||
        cudaMemcpyAsync(esv.data(), ctx->Es, g.nblk * 8, cudaMemcpyDeviceToHost, ctx->s) ||
        cudaMemcpyAsync(nbv.data(), ctx->Nb, g.nblk * 4, cudaMemcpyDeviceToHost, ctx->s) ||
        cudaStreamSynchronize(ctx->s))
        return bail(MPR_ECUDA);
    ctx->n_gap[0] = s0[g.nblk];
    ctx->n_gap[1] = s1[g.nblk];
    int64_t pairs = 0, samples = 0;
    double gsum = 0.0;
    std::vector<float> init(g.nblk);
    std::vector<int32_t> ng(g.nblk);
    std::vector<double> es_h(g.nblk), inb_h(g.nblk);
    std::vector<int32_t> nsp_cal(g.nblk);
    for (int b = 0; b < g.nblk; ++b) {
        nsp_cal[b] = (ng0[b] + ng1[b]) > 0 ? nsp[b] : 0;
        pairs += nsp[b];
        samples += nsm[b];
        gsum += ssum[b];
        ng[b] = ng0[b] + ng1[b];
        es_h[b] = nsp[b] > 0 ? esv[b] / (double)nsp[b] : 0.0;
        inb_h[b] = nbv[b] > 0 ? 1.0 / (double)nbv[b] : 0.0;
    }
    const double gmean = samples ? gsum / (double)samples : 0.0;
    for (int b = 0; b < g.nblk; ++b) init[b] = (float)(nsm[b] > 0 ? ssum[b] / nsm[b] : gmean);
    if (pairs == 0 && ctx->n_gap[0] + ctx->n_gap[1] > 0) {
        mpr3_destroy(ctx);
        return MPR_ENOSAMPLES;
    }
    ST3(alloc3(ctx, &ctx->list[0], ctx->n_gap[0]));
    ST3(alloc3(ctx, &ctx->list[1], ctx->n_gap[1]));
    if (cudaMemcpyAsync(ctx->init_angle, init.data(), g.nblk * 4, cudaMemcpyHostToDevice, ctx->s) ||
        cudaMemcpyAsync(ctx->es, es_h.data(), g.nblk * 8, cudaMemcpyHostToDevice, ctx->s) ||
        cudaMemcpyAsync(ctx->inb, inb_h.data(), g.nblk * 8, cudaMemcpyHostToDevice, ctx->s) ||
        cudaMemcpyAsync(ctx->ngap, ng.data(), g.nblk * 4, cudaMemcpyHostToDevice, ctx->s) ||
        cudaMemcpyAsync(ctx->Nsp_cal, nsp_cal.data(), g.nblk * 4, cudaMemcpyHostToDevice, ctx->s))
        return bail(MPR_ECUDA);
    k3_build_lists<<<bblocks, 256, 0, ctx->s>>>(g, ctx->mask, ctx->start[0], ctx->start[1],
                                                ctx->list[0], ctx->list[1]);
    if (cudaPeekAtLastError() || cudaStreamSynchronize(ctx->s)) return bail(MPR_ECUDA);
#undef ST3
    *out = ctx;
    return MPR_OK;
}

mpr_status mpr3_get_block_stats(mpr3_ctx* ctx, double* Es, int32_t* Nsp, int32_t* Nb,
                                float* mean_angle, int32_t* n_gap) {
    if (!ctx) return MPR_EINVAL;
    const size_t nb = (size_t)ctx->g.nblk;
    if (Es) CK3(cudaMemcpyAsync(Es, ctx->Es, nb * 8, cudaMemcpyDefault, ctx->s));
    if (Nsp) CK3(cudaMemcpyAsync(Nsp, ctx->Nsp, nb * 4, cudaMemcpyDefault, ctx->s));
    if (Nb) CK3(cudaMemcpyAsync(Nb, ctx->Nb, nb * 4, cudaMemcpyDefault, ctx->s));
    if (mean_angle) CK3(cudaMemcpyAsync(mean_angle, ctx->init_angle, nb * 4, cudaMemcpyDefault, ctx->s));
    if (n_gap) CK3(cudaMemcpyAsync(n_gap, ctx->ngap, nb * 4, cudaMemcpyDefault, ctx->s));
    CK3(cudaStreamSynchronize(ctx->s));
    return MPR_OK;
}

mpr_status mpr3_set_temperatures(mpr3_ctx* ctx, const float* T) {
    if (!ctx || !T) return MPR_EINVAL;
    ctx->err.clear();
    const int nb = ctx->g.nblk;
    std::vector<float> h(nb), bt(nb);
    CK3(cudaMemcpyAsync(h.data(), T, nb * 4, cudaMemcpyDefault, ctx->s));
    CK3(cudaStreamSynchronize(ctx->s));
    for (int b = 0; b < nb; ++b) {
        if (!(h[b] > 0.0f) || !std::isfinite(h[b])) return fail3(ctx, MPR_EINVAL, "T_%d not > 0", b);
        bt[b] = 1.0f / h[b];
    }
    CK3(cudaMemcpyAsync(ctx->T, h.data(), nb * 4, cudaMemcpyHostToDevice, ctx->s));
    CK3(cudaMemcpyAsync(ctx->beta, bt.data(), nb * 4, cudaMemcpyHostToDevice, ctx->s));
    CK3(cudaStreamSynchronize(ctx->s));
    ctx->calibrated = 1;
    return MPR_OK;
}

// Bisection on the per-block T (Sec. 2.1 energy matching per block): every
// iteration starts the chains afresh, runs n_eq + n_meas sweeps at the
// midpoints and keeps the half of each bracket on the side of e_s,b.
mpr_status mpr3_calibrate(mpr3_ctx* ctx, float* T_out) {
    if (!ctx) return MPR_EINVAL;
    ctx->err.clear();
    const Geom3& g = ctx->g;
    const mpr_options& o = ctx->opt;
    ctx->batch_open = 0;
    const Slices sl = slices3(ctx);
    if (ctx->degenerate) {
        std::vector<float> h(g.nblk, o.t_lo);
        TRY3(mpr3_set_temperatures(ctx, h.data()));
    } else {
        const int chains = o.cal_chains;
        TRY3(ensure3(ctx, chains));
        ctx->R = chains;
        launch_cal_init(g.nblk, o.t_lo, o.t_hi, ctx->lo, ctx->hi, ctx->ebar, ctx->ctl, ctx->s);
        CKL3();
        const double inv_count = 1.0 / ((double)o.n_meas * (double)chains);
        const auto ev = begin_timing3(ctx);
        // Every iteration starts its chains from the same state: its E_b once.
        const size_t blk = (size_t)g.nblk * ctx->Rp;
        TRY3(fill3(ctx));
        if (o.n_bisect > 0) {
            TRY3(init3(ctx));
            TRY3(energy3(ctx));
            CK3(cudaMemcpyAsync(ctx->ecur0, ctx->ecur, blk * sizeof(double),
                                cudaMemcpyDeviceToDevice, ctx->s));
        }
        for (int k = 0; k < o.n_bisect; ++k) {
            launch_cal_mid(g.nblk, ctx->Nsp_cal, ctx->lo, ctx->hi, ctx->T, ctx->ctl, ctx->s);
            ++ctx->launches;
            launch_cal_fill(sl, g.nbx, ctx->Nsp_cal, ctx->T, ctx->beta, ctx->s);
            CKL3();
            TRY3(init3(ctx));
            CK3(cudaMemcpyAsync(ctx->ecur, ctx->ecur0, blk * sizeof(double),
                                cudaMemcpyDeviceToDevice, ctx->s));
            CK3(cudaMemsetAsync(ctx->eacc, 0, 2 * blk * sizeof(double), ctx->s));
            // Sweep sw's changes go to eacc buffer sw & 1; the colour-0 launch
            // of sweep sw + 1 folds them (extra CTAs), the last sweep's fold
            // runs alone.
            const int n_sw = o.n_eq + o.n_meas;
            for (int sw = 1; sw <= n_sw; ++sw) {
                const uint32_t ctr1 = (uint32_t)sw | ((uint32_t)(1 + k) << 16);
                FoldArgs f{};
                if (sw > 1) {
                    f.ctas = (g.nblk + kSweep3Threads - 1) / kSweep3Threads;
                    f.nblk = g.nblk;
                    f.Rp = ctx->Rp;
                    f.chains = chains;
                    f.points = 1;
                    f.measure = (sw - 1) > o.n_eq;
                    f.inb = ctx->inb;
                    f.eacc = ctx->eacc + (size_t)((sw - 1) & 1) * blk;
                    f.ecur = ctx->ecur;
                    f.ebar = ctx->ebar;
                }
                for (int c = 0; c < 2; ++c)
                    TRY3(halfstep3(ctx, c, ctr1, false, ctx->eacc + (size_t)(sw & 1) * blk,
                                   c == 0 ? &f : nullptr));
            }
            launch_cal_step(g.nblk, ctx->Rp, chains, o.n_eq, n_sw, ctx->ctl, ctx->inb,
                            ctx->eacc + (size_t)(n_sw & 1) * blk, ctx->ecur, ctx->ebar, ctx->s);
            CKL3();
            launch_cal_update(g.nblk, inv_count, ctx->es, ctx->Nsp_cal, ctx->T, ctx->lo, ctx->hi,
                              ctx->ebar, ctx->ctl, o.n_bisect, 0, ctx->s);
            CKL3();
        }
        if (ev.first) {
            cudaEventRecord(ev.second, ctx->s);
            ctx->ev_cal.push_back(ev);
        }
        ctx->cal_hs += (int64_t)o.n_bisect * (o.n_eq + o.n_meas) * 2;
        launch_cal_mid(g.nblk, ctx->Nsp_cal, ctx->lo, ctx->hi, ctx->T, ctx->ctl, ctx->s);
        ++ctx->launches;
        launch_cal_fill(sl, g.nbx, ctx->Nsp_cal, ctx->T, ctx->beta, ctx->s);
        CKL3();
        ctx->cal_updates += (int64_t)o.n_bisect * (o.n_eq + o.n_meas) * chains *
                            (ctx->n_gap[0] + ctx->n_gap[1]);
        ctx->calibrated = 1;
    }
    if (T_out) CK3(cudaMemcpyAsync(T_out, ctx->T, g.nblk * 4, cudaMemcpyDefault, ctx->s));
    CK3(cudaStreamSynchronize(ctx->s));
    return MPR_OK;
}

mpr_status mpr3_sim_begin(mpr3_ctx* ctx, int32_t n) {
    if (!ctx) return MPR_EINVAL;
    ctx->err.clear();
    if (n < 1 || n > 65534) return fail3(ctx, MPR_EINVAL, "n_realizations in [1, 65534]");
    if (ctx->batch_open) return fail3(ctx, MPR_ESTATE, "a batch is open");
    if (!ctx->calibrated) return fail3(ctx, MPR_ESTATE, "calibrate or set temperatures first");
    const int64_t base = (ctx->r_next + 1) / 2 * 2;   // lane pairs align with Philox blocks
    if (base + n > (int64_t)0x1FFFFFFFF) return fail3(ctx, MPR_EINVAL, "realization index overflow");
    ctx->pair_base = (uint32_t)(base / 2);
    TRY3(ensure3(ctx, n));
    ctx->R = n;
    ctx->t = 0;
    const int64_t nbr = (int64_t)ctx->g.nblk * ctx->Rp;
    k3_fill_valid<<<grid_of(nbr), 256, 0, ctx->s>>>(ctx->running, nbr, ctx->Rp, n);
    CKL3();
    TRY3(fill3(ctx));
    TRY3(init3(ctx));
    CK3(cudaMemsetAsync(ctx->tcount, 0, ctx->Rp * sizeof(int32_t), ctx->s));
    TRY3(energy3(ctx));
    launch_stop_init(ctx->g.nblk, ctx->Rp, ctx->zero_slices, ctx->es, ctx->inb, ctx->Nsp,
                     ctx->ngap, ctx->ecur, ctx->sigma, ctx->running, ctx->stop, ctx->tcount,
                     ctx->e_last, ctx->s);
    CKL3();
    const int64_t items = (int64_t)ctx->g.nblk * ctx->np;
    launch_stop_rest(ctx->g.nblk, ctx->np, 2, ctx->Rp, ctx->opt.n_max, ctx->zero_slices,
                     (int)std::min<int64_t>((items + 255) / 256, 152 * 16), ctx->ctl, nullptr,
                     ctx->work, (uint32_t)items, ctx->Nsp, ctx->running, ctx->stop, ctx->tcount, 0,
                     -1, ctx->s);
    CKL3();
    ctx->batch_open = 1;
    return MPR_OK;
}

mpr_status mpr3_halfstep(mpr3_ctx* ctx, int32_t colour, int32_t t, int32_t tag) {
    if (!ctx) return MPR_EINVAL;
    ctx->err.clear();
    if (!ctx->batch_open) return fail3(ctx, MPR_ESTATE, "no open batch");
    if (colour < 0 || colour > 1 || t < 0 || t > 65535 || tag < 0 || tag > 65535)
        return fail3(ctx, MPR_EINVAL, "bad colour, t or tag");
    TRY3(halfstep3(ctx, colour, (uint32_t)t | ((uint32_t)tag << 16), true, ctx->eacc));
    CK3(cudaStreamSynchronize(ctx->s));
    return MPR_OK;
}

mpr_status mpr3_sim_end(mpr3_ctx* ctx) {
    if (!ctx) return MPR_EINVAL;
    if (!ctx->batch_open) return fail3(ctx, MPR_ESTATE, "no open batch");
    for (int c = 0; c < 2; ++c) {
        if (ctx->n_gap[c] == 0) continue;
        k3_accumulate<<<grid_of(ctx->n_gap[c]), 256, 0, ctx->s>>>(
            ctx->g, ctx->list[c], ctx->n_gap[c], c, ctx->ang, ctx->R, ctx->sum);
        CKL3();
    }
    CK3(cudaMemsetAsync(ctx->counter, 0, 8, ctx->s));
    launch_count_updates(ctx->g.nblk, ctx->Rp, ctx->stop, ctx->ngap, ctx->counter, ctx->s);
    CKL3();
    unsigned long long h = 0;
    CK3(cudaMemcpyAsync(&h, ctx->counter, 8, cudaMemcpyDeviceToHost, ctx->s));
    CK3(cudaStreamSynchronize(ctx->s));
    ctx->gap_updates += (int64_t)h;
    ctx->realizations += ctx->R;
    ctx->r_next = (int64_t)ctx->pair_base * 2 + ctx->R;
    ctx->batch_open = 0;
    return MPR_OK;
}

// Sweeps are queued in chunks of four; after each chunk the running count is
// copied to pinned memory, and the host checks the count of the chunk before
// the one it just queued, so the GPU never waits for the host. Sweeps queued
// after everything stopped find no running pair.
mpr_status mpr3_simulate(mpr3_ctx* ctx, int32_t n) {
    if (!ctx) return MPR_EINVAL;
    mpr_status st = mpr3_sim_begin(ctx, n);
    if (st != MPR_OK) return st;
    if (!ctx->h_run) {
        ctx->h_run = static_cast<unsigned long long*>(pinned_slot());
        if (!ctx->h_run) return fail3(ctx, MPR_ENOMEM, "pinned memory");
    }
    cudaEvent_t ev[2] = {nullptr, nullptr};
    if (cudaEventCreateWithFlags(&ev[0], cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&ev[1], cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        return fail3(ctx, MPR_ECUDA, "cudaEventCreate failed");
    }
    int c = 0;
    while (st == MPR_OK && ctx->t < ctx->opt.n_max) {
        for (int i = 0; i < 4 && st == MPR_OK && ctx->t < ctx->opt.n_max; ++i) st = sweep3(ctx);
        if (st != MPR_OK) break;
        if (cudaMemcpyAsync(ctx->h_run + (c & 1), &ctx->ctl->n_running, sizeof(unsigned long long),
                            cudaMemcpyDeviceToHost, ctx->s) != cudaSuccess ||
            cudaEventRecord(ev[c & 1], ctx->s) != cudaSuccess) {
            st = fail3(ctx, MPR_ECUDA, "reading the running count failed");
            break;
        }
        if (c >= 1) {
            if (cudaEventSynchronize(ev[(c - 1) & 1]) != cudaSuccess) {
                st = fail3(ctx, MPR_ECUDA, "event synchronisation failed");
                break;
            }
            if (ctx->h_run[(c - 1) & 1] == 0) break;
        }
        ++c;
    }
    cudaStreamSynchronize(ctx->s);
    cudaEventDestroy(ev[0]);
    cudaEventDestroy(ev[1]);
    if (st == MPR_OK) st = mpr3_sim_end(ctx);
    return st;
}

mpr_status mpr3_get_state(mpr3_ctx* ctx, int32_t r, float* out) {
    if (!ctx || !out) return MPR_EINVAL;
    if (!ctx->batch_open || r < 0 || r >= ctx->R) return fail3(ctx, MPR_ESTATE, "no such realization");
    float* d = nullptr;
    TRY3(alloc3(ctx, &d, ctx->n));
    k3_get_state<<<grid_of(ctx->n), 256, 0, ctx->s>>>(ctx->g, ctx->ang, r, d);
    mpr_status st = cudaPeekAtLastError() == cudaSuccess ? MPR_OK : MPR_ECUDA;
    if (st == MPR_OK && (cudaMemcpyAsync(out, d, ctx->n * 4, cudaMemcpyDefault, ctx->s) ||
                         cudaStreamSynchronize(ctx->s)))
        st = MPR_ECUDA;
    free3(ctx, d);
    return st;
}

mpr_status mpr3_set_state(mpr3_ctx* ctx, int32_t r, const float* in) {
    if (!ctx || !in) return MPR_EINVAL;
    if (!ctx->batch_open || r < 0 || r >= ctx->R) return fail3(ctx, MPR_ESTATE, "no such realization");
    float* d = nullptr;
    TRY3(alloc3(ctx, &d, ctx->n));
    mpr_status st = MPR_OK;
    if (cudaMemcpyAsync(d, in, ctx->n * 4, cudaMemcpyDefault, ctx->s)) st = MPR_ECUDA;
    if (st == MPR_OK) {
        k3_set_state<<<grid_of(ctx->n), 256, 0, ctx->s>>>(ctx->g, ctx->mask, ctx->ang, r, d);
        if (cudaPeekAtLastError() || cudaStreamSynchronize(ctx->s)) st = MPR_ECUDA;
    }
    free3(ctx, d);
    return st;
}

mpr_status mpr3_predict(mpr3_ctx* ctx, float* out, const float* truth, double* aae_rase) {
    if (!ctx || !out) return MPR_EINVAL;
    ctx->err.clear();
    const int64_t gaps = ctx->n_gap[0] + ctx->n_gap[1];
    if (ctx->realizations == 0 && gaps > 0) return fail3(ctx, MPR_ESTATE, "no realization yet");
    float *o = nullptr, *tr = nullptr;
    TRY3(alloc3(ctx, &o, ctx->n));
    mpr_status st = MPR_OK;
    if (truth) {
        st = alloc3(ctx, &tr, ctx->n);
        if (st == MPR_OK && cudaMemcpyAsync(tr, truth, ctx->n * 4, cudaMemcpyDefault, ctx->s))
            st = MPR_ECUDA;
    }
    if (st == MPR_OK && cudaMemsetAsync(ctx->err_buf, 0, 16, ctx->s)) st = MPR_ECUDA;
    if (st == MPR_OK) {
        const double inv_r = ctx->realizations > 0 ? 1.0 / (double)ctx->realizations : 0.0;
        k3_predict<<<grid_of(ctx->n), 256, 0, ctx->s>>>(ctx->n, ctx->values, ctx->mask, ctx->sum,
                                                        inv_r, ctx->zmin, ctx->zmax, o, tr,
                                                        ctx->err_buf);
        double h[2] = {0, 0};
        if (cudaPeekAtLastError() ||
            cudaMemcpyAsync(out, o, ctx->n * 4, cudaMemcpyDefault, ctx->s) ||
            cudaMemcpyAsync(h, ctx->err_buf, 16, cudaMemcpyDeviceToHost, ctx->s) ||
            cudaStreamSynchronize(ctx->s))
            st = MPR_ECUDA;
        if (st == MPR_OK && truth && aae_rase) {
            aae_rase[0] = gaps ? h[0] / (double)gaps : 0.0;
            aae_rase[1] = gaps ? std::sqrt(h[1] / (double)gaps) : 0.0;
        }
    }
    free3(ctx, o);
    free3(ctx, tr);
    return st;
}

mpr_status mpr3_get_info(const mpr3_ctx* ctx, mpr3_info* info) {
    if (!ctx || !info) return MPR_EINVAL;
    std::memset(info, 0, sizeof(*info));
    info->depth = ctx->g.D;
    info->height = ctx->g.H;
    info->width = ctx->g.W;
    info->block = ctx->g.lb;
    info->nblk = ctx->g.nblk;
    info->n_gap = ctx->n_gap[0] + ctx->n_gap[1];
    info->zmin = ctx->zmin;
    info->zmax = ctx->zmax;
    info->realizations = ctx->realizations;
    info->gap_updates = ctx->gap_updates;
    info->cal_gap_updates = ctx->cal_updates;
    return MPR_OK;
}

}  // extern "C"
