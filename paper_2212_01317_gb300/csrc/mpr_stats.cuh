// Eq. 2 per block: the sample-bond energy E_s,b, its bond count N_SP,b, the
// owned bonds N_b, and the block's sample-angle sum, sample count and gap
// counts per colour. One CTA per block; every site owns its right and down
// bonds (a bond belongs to the block of its left / upper site). Sums in FP64.
//
// FP64 runs at two operations per clock and SM on this GPU, so its operations
// are what the statistics cost: a cosine in a warp with one active lane costs as
// much as in a full one. Each warp therefore queues the sample-sample bonds it
// meets (the two values) in shared memory and takes cosines 32 at a time, with a
// polynomial for the bounded argument (cos_bond), short where the warp's bonds
// are all shallow. 4096^2, disc gaps of 60 %, l_b = 32 (sample angles written in
// the same pass), whole mpr_create: 2.63 -> 1.13 ms.
//
// Shared by the context path (k_block_stats: canvas masks, where 2 marks an
// absent site and no bond reaches one) and the allocation-free entry point
// (k_na_block_stats: the caller's mask, nonzero = gap), so both compute the
// statistics with the same arithmetic in the same order.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "mpr_internal.h"

namespace mpr {

// cos x for |x| <= pi (a bond's q times an angle difference: q <= 1/2, angles in
// [0, 2 pi]): 1 - 2 sin^2(x / 2) with the Taylor series of the sine up to the
// 21st power (remainder below 2e-18 on [-pi/2, pi/2]). FP64 runs at two
// operations per clock and SM here, so the fourteen this takes, without the
// range reduction of a general cosine, are what the statistics cost.
__device__ __forceinline__ double cos_bond(double x) {
    const double h = 0.5 * x, z = h * h;
    double p = 1.9572941063391261e-20;               // 1 / 21!
    p = fma(p, z, -8.2206352466243295e-18);          // -1 / 19!
    p = fma(p, z, 2.8114572543455206e-15);           // 1 / 17!
    p = fma(p, z, -7.6471637318198164e-13);          // -1 / 15!
    p = fma(p, z, 1.6059043836821613e-10);           // 1 / 13!
    p = fma(p, z, -2.5052108385441720e-08);          // -1 / 11!
    p = fma(p, z, 2.7557319223985893e-06);           // 1 / 9!
    p = fma(p, z, -1.9841269841269841e-04);          // -1 / 7!
    p = fma(p, z, 8.3333333333333333e-03);           // 1 / 5!
    p = fma(p, z, -1.6666666666666667e-01);          // -1 / 3!
    const double s = fma(p * z, h, h);
    return fma(-2.0 * s, s, 1.0);
}

// The same for |x| <= 1/2: the cosine's own series up to the 14th power
// (remainder below 8e-19).
__device__ __forceinline__ double cos_shallow(double x) {
    const double z = x * x;
    double p = -1.1470745597729725e-11;              // -1 / 14!
    p = fma(p, z, 2.0876756987868099e-09);           // 1 / 12!
    p = fma(p, z, -2.7557319223985888e-07);          // -1 / 10!
    p = fma(p, z, 2.4801587301587302e-05);           // 1 / 8!
    p = fma(p, z, -1.3888888888888889e-03);          // -1 / 6!
    p = fma(p, z, 4.1666666666666667e-02);           // 1 / 4!
    p = fma(p, z, -0.5);
    return fma(p, z, 1.0);
}

struct BlockSums {
    double es, sm;               // E_s,b; sum of the sample angles
    int nsp, nb, ns, g0, g1;     // N_SP,b, N_b, samples, gaps of colour 0 / 1
};

constexpr int kStatsMaxWarps = 8;
constexpr int kBondQueue = 96;   // less than 32 left over + 64 of one step

struct StatsShared {
    float2 bond[kStatsMaxWarps][kBondQueue];
    double d[kStatsMaxWarps][2];
    int i[kStatsMaxWarps][5];
};

// The FP32 sample angle: the FP64 value 2 pi (z - zmin) / (zmax - zmin) rounded.
// pi = (z - zmin) scale is within a few units in the last place of it and rounds
// to the same float unless it lies that close to the middle between two; only
// then (and for results too small to tell) the division is made.
__device__ __forceinline__ float sample_angle(double pi, float v, double zmin, double zmax) {
    const uint32_t low = (uint32_t)__double2loint(pi) & 0x1FFFFFFFu;   // bits a float drops
    if (low - (0x10000000u - 8u) > 16u && pi >= 1e-30) return (float)pi;
    if (!(zmax > zmin)) return 0.0f;
    return (float)(6.283185307179586476925 * ((double)v - zmin) / (zmax - zmin));
}

// Sites [x0, x1) x [y0, y1) of a W-wide grid by the threads of one CTA (at most
// 32 kStatsMaxWarps); right_ok / down_ok: the bonds across the block's right /
// lower edge exist. phi = (z - zmin) * scale. kCanvas: mask value 2 marks an
// absent site (else nonzero is a gap), and each site's FP32 angle (0 at gaps)
// goes to dang (half-lattice of row length Wh, planes `plane` apart). Thread 0
// gets the block's totals.
template <bool kCanvas>
__device__ __forceinline__ BlockSums block_sums(const float* __restrict__ values,
                                                const uint8_t* __restrict__ mask, int W, int y0,
                                                int x0, int y1, int x1, bool right_ok,
                                                bool down_ok, double zmin, double zmax,
                                                double scale, double q, double J, bool active,
                                                float* __restrict__ dang, int Wh, size_t plane,
                                                StatsShared& sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const int bw = x1 - x0, nsite = (y1 - y0) * bw;
    const int step_y = (int)blockDim.x / bw, step_x = (int)blockDim.x - step_y * bw;
    int y = y0 + (int)threadIdx.x / bw, x = x0 + (int)threadIdx.x % bw;
    float2* queue = sh.bond[warp];
    const double qs = q * scale;
    double es = 0.0, sm = 0.0;
    int v[5] = {0, 0, 0, 0, 0};   // nsp, nb, ns, g0, g1
    int cnt = 0;
    auto drain = [&](int n) {     // the last n (<= 32) bonds of the queue
        __syncwarp();
        double a = 0.0;
        if (lane < n) {
            const float2 b = queue[cnt - n + lane];
            a = ((double)b.x - (double)b.y) * qs;
        }
        const bool shallow = __all_sync(0xffffffffu, fabs(a) <= 0.5);
        const double c = shallow ? cos_shallow(a) : cos_bond(a);
        if (lane < n) es += c;
        cnt -= n;
        __syncwarp();
    };
    for (int j0 = 0; j0 < nsite; j0 += (int)blockDim.x) {
        const bool in = j0 + (int)threadIdx.x < nsite;
        bool right = false, down = false;
        float vi = 0.0f, vr = 0.0f, vd = 0.0f;
        if (in) {
            const int64_t i = (int64_t)y * W + x;
            const uint8_t mi = mask[i];
            const bool site = active && (!kCanvas || mi != MASK_ABSENT);
            const bool gap = kCanvas ? mi == MASK_GAP : mi != 0;
            float angle = 0.0f;
            if (site) {
                if (gap) {
                    if (((x + y) & 1) == 0) ++v[3]; else ++v[4];
                } else {
                    vi = values[i];
                    const double pi = ((double)vi - zmin) * scale;
                    sm += pi;
                    ++v[2];
                    if constexpr (kCanvas) angle = sample_angle(pi, vi, zmin, zmax);
                }
                if (x + 1 < x1 || right_ok) {
                    const uint8_t mj = mask[i + 1];
                    if (!kCanvas || mj != MASK_ABSENT) {
                        ++v[1];
                        right = !gap && mj == 0;
                        if (right) vr = values[i + 1];
                    }
                }
                if (y + 1 < y1 || down_ok) {
                    const uint8_t mj = mask[i + W];
                    if (!kCanvas || mj != MASK_ABSENT) {
                        ++v[1];
                        down = !gap && mj == 0;
                        if (down) vd = values[i + W];
                    }
                }
            }
            if constexpr (kCanvas)
                dang[((x + y) & 1) * plane + (size_t)y * Wh + (x >> 1)] = angle;
            x += step_x;
            y += step_y;
            if (x >= x1) {
                x -= bw;
                ++y;
            }
        }
        const unsigned br = __ballot_sync(0xffffffffu, right), bd = __ballot_sync(0xffffffffu, down);
        if (right) queue[cnt + __popc(br & below)] = make_float2(vi, vr);
        cnt += __popc(br);
        if (down) queue[cnt + __popc(bd & below)] = make_float2(vi, vd);
        cnt += __popc(bd);
        v[0] += (int)right + (int)down;
        while (cnt >= 32) drain(32);
    }
    if (cnt > 0) drain(cnt);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        es += __shfl_xor_sync(0xffffffffu, es, d);
        sm += __shfl_xor_sync(0xffffffffu, sm, d);
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) v[k] = __reduce_add_sync(0xffffffffu, v[k]);
    if (lane == 0) {
        sh.d[warp][0] = es;
        sh.d[warp][1] = sm;
        for (int k = 0; k < 5; ++k) sh.i[warp][k] = v[k];
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
            es += sh.d[w][0];
            sm += sh.d[w][1];
            for (int k = 0; k < 5; ++k) v[k] += sh.i[w][k];
        }
    return BlockSums{-J * es, sm, v[0], v[1], v[2], v[3], v[4]};
}

}  // namespace mpr
