// Device code of one checkerboard half-step (Sec. 2.2.2) and of the energy
// pass, shared by the per-launch kernels (mpr_kernels.cu) and the persistent
// calibration kernel (mpr_persist.cu).
//
// A unit is one block of the grid in one realization pair; the realizations'
// worklist hands out units, the calibration's flat kernel every entry. Each
// lane updates its site in both realizations of the pair, from one Philox
// block: words 0, 1 for the even realization, 2, 3 for the odd. Every pair has
// its own planes of the state: neighbouring half-sites are neighbouring words,
// so a warp's loads of one unit touch a quarter of the cache lines they would
// with eight realizations interleaved per site (FP32, 2048^2, l_b = 32, 32
// realizations: first sweeps 147 against 125 G updates/s).
//
// Block energies are kept incrementally. A move changes the energy of the
// site's four bonds by dE, and the reflection conserves it (up to the
// rounding of the stored angle, which the 16-bit forms account for), so the
// site's block gains dE. A site on the left or top edge of its block hands
// the change of its left / up bond to the neighbouring block that owns it (a
// bond is owned by the block of its left / upper site). Frozen sites never
// move, so stopped (block, realization) pairs cost nothing.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "mpr_device.cuh"
#include "mpr_internal.h"

namespace mpr {

// Element type of the batch state: a realization pair is two adjacent
// elements, one 8-byte (FP32) or 4-byte (FP16 / BF16) word; arithmetic is FP32
// throughout. The sample angles the method conditions on are never rounded:
// in the 16-bit forms a sample site's word holds its FP32 angle, so a
// neighbour is one load of the same size whether it is a gap or a sample, and
// decode() is told which.
template <typename S> struct Store;

template <> struct Store<float> {
    static constexpr bool kExact = true;
    using Word = float2;             // a realization pair as it lies in memory
    __device__ static float2 decode(Word w, bool) { return w; }
    __device__ static float2 load2(const float* p) { return *reinterpret_cast<const float2*>(p); }
    __device__ static void store2(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
    __device__ static float load1(const float* p) { return *p; }
    __device__ static void store1(float* p, float v) { *p = v; }
    __device__ static float round(float v) { return v; }
    __device__ static float2 round2(float2 v) { return v; }
};

template <> struct Store<__half> {
    static constexpr bool kExact = false;
    using Word = uint32_t;
    __device__ static float2 decode(Word w, bool gap) {
        const float s = __uint_as_float(w);
        const __half2 h = *reinterpret_cast<const __half2*>(&w);
        return gap ? __half22float2(h) : make_float2(s, s);
    }
    __device__ static float2 load2(const __half* p) {
        return __half22float2(*reinterpret_cast<const __half2*>(p));
    }
    __device__ static void store2(__half* p, float2 v) {
        *reinterpret_cast<__half2*>(p) = __floats2half2_rn(v.x, v.y);
    }
    __device__ static float load1(const __half* p) { return __half2float(*p); }
    __device__ static void store1(__half* p, float v) { *p = __float2half_rn(v); }
    __device__ static float round(float v) { return __half2float(__float2half_rn(v)); }
    __device__ static float2 round2(float2 v) {
        return __half22float2(__floats2half2_rn(v.x, v.y));
    }
};

template <> struct Store<__nv_bfloat16> {
    static constexpr bool kExact = false;
    using Word = uint32_t;
    __device__ static float2 decode(Word w, bool gap) {
        const float s = __uint_as_float(w);
        return make_float2(gap ? __uint_as_float(w << 16) : s,
                           gap ? __uint_as_float(w & 0xFFFF0000u) : s);
    }
    __device__ static float2 load2(const __nv_bfloat16* p) {
        return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
    }
    __device__ static void store2(__nv_bfloat16* p, float2 v) {
        *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(v.x, v.y);
    }
    __device__ static float load1(const __nv_bfloat16* p) { return __bfloat162float(*p); }
    __device__ static void store1(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
    __device__ static float round(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
    __device__ static float2 round2(float2 v) {
        return __bfloat1622float2(__floats2bfloat162_rn(v.x, v.y));
    }
};

// Site update with the state's rounding applied: the proposal is rounded
// before its energy is taken, so the Metropolis test judges the angle that
// is stored; the reflected angle is rounded too, and for the 16-bit forms
// dE is the exact change from the old to the stored final angle. (co, so):
// cos, sin of q phi; php, (cp, sp): the rounded proposal and its cos, sin;
// C, Sn: the local field. The roundings are spelled out (see bond_change).
template <typename S>
__device__ __forceinline__ SiteNew site_move(float phi, float co, float so, float php, float cp,
                                             float sp, float C, float Sn, float u1, float beta,
                                             const Model& m) {
    SiteNew n;
    const float e0 = __fmaf_rn(Sn, so, __fmul_rn(C, co));
    const float e1 = __fmaf_rn(Sn, sp, __fmul_rn(C, cp));
    const float dE = __fmul_rn(m.J, __fsub_rn(e0, e1));
    // exp(-dE beta) = 2^(-dE beta log2 e)
    const bool acc = (dE <= 0.0f) ||
                     (u1 < ex2_approx(__fmul_rn(__fmul_rn(dE, -beta), 1.44269504088896341f)));
    n.mid = acc ? php : phi;
    n.dE = acc ? dE : 0.0f;
    // Over-relaxation, without branches. The reflected angle (2 psi - q phi)/q
    // is >= 0 only if psi >= 0, i.e. S >= 0, so psi is taken from (|S|, C) and
    // the move is kept only when S >= 0 and the angle lies in [0, 2pi], as one
    // comparison of the bits: a negative number or the NaN of C = S = 0
    // compares above (-0 cannot arise from the fused difference).
    const float psi = atan2_upper(fabsf(Sn), C);
    const float por = __fmul_rn(__fmaf_rn(-m.q, n.mid, 2.0f * psi), m.inv_q);
    n.refl = m.overrelax && Sn >= 0.0f && __float_as_uint(por) <= __float_as_uint(kTwoPi);
    n.phi = n.refl ? Store<S>::round(por) : n.mid;
    if constexpr (!Store<S>::kExact) {
        float sf, cf;
        __sincosf(m.q * n.phi, &sf, &cf);
        n.dE = __fmul_rn(m.J, __fsub_rn(e0, __fmaf_rn(Sn, sf, __fmul_rn(C, cf))));
    }
    return n;
}

template <typename S>
__device__ __forceinline__ SiteNew site_update(float phi, float C, float Sn, float u0, float u1,
                                               float beta, const Model& m) {
    float co, so, cp, sp;
    __sincosf(m.q * phi, &so, &co);
    const float php = Store<S>::round(kTwoPi * u0);
    __sincosf(m.q * php, &sp, &cp);
    return site_move<S>(phi, co, so, php, cp, sp, C, Sn, u1, beta, m);
}

// site_update of a site in both realizations of a pair, with the same roundings
// (bit for bit): what is not a hardware function or a choice is packed two-wide
// FP32 arithmetic, one instruction for both realizations. The half-step is
// bound by instruction issue (60-66 %, no pipe above 55 %, DRAM below 30 %), so
// instructions are what it has to save: with the packed arithmetic, the list
// entries that hold what every pair would compute again (gap_item) and the
// pair planes, a warp pass of 32 entries x 2 realizations takes about 280
// instead of 400 instructions (FP32 state; 310 instead of 430 in BF16). First
// sweeps of a 2048^2 field, 32 realizations, half the sites missing: l_b = 32
// FP32 125 -> 147, BF16 104 -> 139, l_b = 16 (two units per warp) FP32
// 106 -> 120 G updates/s. Copying the next entry's words into shared memory
// ahead of time (cp.async) removed the long-scoreboard stalls but cost as many
// instructions and L1 wavefronts as it saved (2.21 against 2.03 ms per four
// BF16 sweeps); loads one entry ahead into registers, bulk prefetches of the
// next unit's rows into L2, and 7, 9 or 10 CTAs per SM were slower too.
template <typename S>
__device__ __forceinline__ PairNew pair_move(float2 phi, float2 co, float2 so, float2 php,
                                             float2 cp, float2 sp, float2 C, float2 Sn, float2 u1,
                                             float2 beta, const Model& m) {
    PairNew n;
    const float2 q2 = both(m.q), J2 = both(m.J);
    const float2 e0 = __ffma2_rn(Sn, so, __fmul2_rn(C, co));
    const float2 e1 = __ffma2_rn(Sn, sp, __fmul2_rn(C, cp));
    n.dE = __fmul2_rn(J2, __ffma2_rn(e1, both(-1.0f), e0));
    const float2 x = __fmul2_rn(__fmul2_rn(n.dE, make_float2(-beta.x, -beta.y)),
                                both(1.44269504088896341f));
    const bool acc0 = (n.dE.x <= 0.0f) || (u1.x < ex2_approx(x.x));
    const bool acc1 = (n.dE.y <= 0.0f) || (u1.y < ex2_approx(x.y));
    n.mid = make_float2(acc0 ? php.x : phi.x, acc1 ? php.y : phi.y);
    const float2 psi = atan2_upper_2(make_float2(fabsf(Sn.x), fabsf(Sn.y)), C);
    const float2 por = __fmul2_rn(
        __ffma2_rn(make_float2(-m.q, -m.q), n.mid, __fadd2_rn(psi, psi)), both(m.inv_q));
    n.refl0 = m.overrelax && Sn.x >= 0.0f && __float_as_uint(por.x) <= __float_as_uint(kTwoPi);
    n.refl1 = m.overrelax && Sn.y >= 0.0f && __float_as_uint(por.y) <= __float_as_uint(kTwoPi);
    const float2 pr = Store<S>::round2(por);
    n.phi = make_float2(n.refl0 ? pr.x : n.mid.x, n.refl1 ? pr.y : n.mid.y);
    if constexpr (Store<S>::kExact) {
        n.dE = make_float2(acc0 ? n.dE.x : 0.0f, acc1 ? n.dE.y : 0.0f);
    } else {
        float2 cf, sf;
        sincos_2(__fmul2_rn(q2, n.phi), sf, cf);
        const float2 e2 = __ffma2_rn(Sn, sf, __fmul2_rn(C, cf));
        n.dE = __fmul2_rn(J2, __ffma2_rn(e2, both(-1.0f), e0));
    }
    return n;
}

template <typename S>
__device__ __forceinline__ PairNew pair_update(float2 phi, float2 C, float2 Sn, float2 u0,
                                               float2 u1, float2 beta, const Model& m) {
    const float2 q2 = both(m.q);
    float2 co, so, cp, sp;
    sincos_2(__fmul2_rn(q2, phi), so, co);
    const float2 php = Store<S>::round2(__fmul2_rn(both(kTwoPi), u0));
    sincos_2(__fmul2_rn(q2, php), sp, cp);
    return pair_move<S>(phi, co, so, php, cp, sp, C, Sn, u1, beta, m);
}

// A block's change in one half-step: the FP32 warp sum of the unit's moves
// is added to eacc with an FP64 atomic, so every sum across units, half-steps
// and (in the stop test and the calibration fold) sweeps is FP64. (The warp
// sum stays FP32: GB300's FP64 pipe is narrow, and FP64 shuffle sums per unit
// doubled the half-step's time.)
__device__ __forceinline__ void flush_pair(double* ea, float v0, float v1) {
    if (!__any_sync(0xffffffffu, v0 != 0.0f || v1 != 0.0f)) return;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, s);
        v1 += __shfl_xor_sync(0xffffffffu, v1, s);
    }
    if ((threadIdx.x & 31) != 0) return;
    if (v0 != 0.0f) atomicAdd(ea, (double)v0);
    if (v1 != 0.0f) atomicAdd(ea + 1, (double)v1);
}

// Bond-by-bond split of a move at a block edge: (lc, ls) and (uc, us) are the
// left and upper neighbours' (cos, sin) of q phi_j. The roundings are spelled
// out, so that every form adds the same numbers whatever the compiler would
// contract in it.
template <typename S>
__device__ __forceinline__ float bond_change(float dc, float ds, float c, float s, float J) {
    return -J * (Store<S>::kExact ? __fmaf_rn(dc, c, __fmul_rn(ds, s))
                                  : __fmaf_rn(ds, s, __fmul_rn(dc, c)));
}

// phi: the angle before the update. The cosines and sines of the site's own
// angles are computed again here: only a block's edge sites come here, and
// kept values would cost every update registers.
template <typename S>
__device__ __forceinline__ void split_edge(const SiteNew& n, float phi, uint32_t f, float C,
                                           float Sn, float lc, float ls, float uc, float us,
                                           const Model& m, float& ao, float& al, float& au) {
    float co, so, cn, sn;
    __sincosf(m.q * phi, &so, &co);
    if constexpr (Store<S>::kExact) {
        float ca, sa;
        __sincosf(m.q * n.mid, &sa, &ca);
        final_cs(n.refl, ca, sa, C, Sn, cn, sn);
    } else {
        __sincosf(m.q * n.phi, &sn, &cn);
    }
    const float dc = cn - co, ds = sn - so;
    ao += n.dE;
    if (f & EDGE_L) {
        const float d = bond_change<S>(dc, ds, lc, ls, m.J);
        ao -= d;
        al += d;
    }
    if (f & EDGE_U) {
        const float d = bond_change<S>(dc, ds, uc, us, m.J);
        ao -= d;
        au += d;
    }
}

// The same for a pair (.x, .y).
template <typename S>
__device__ __forceinline__ void split_edge_2(const PairNew& n, float2 phi, uint32_t f, float2 C,
                                             float2 Sn, float2 lc, float2 ls, float2 uc, float2 us,
                                             const Model& m, float2& ao, float2& al, float2& au) {
    split_edge<S>(SiteNew{n.phi.x, n.mid.x, n.dE.x, n.refl0}, phi.x, f, C.x, Sn.x, lc.x, ls.x,
                  uc.x, us.x, m, ao.x, al.x, au.x);
    split_edge<S>(SiteNew{n.phi.y, n.mid.y, n.dE.y, n.refl1}, phi.y, f, C.y, Sn.y, lc.y, ls.y,
                  uc.y, us.y, m, ao.y, al.y, au.y);
}

// The neighbours' angles (left, right, up, down) in both realizations of the
// pair, from its plane of the other colour. A neighbour that does not exist
// reads some other site's word or the state's guard; neighbour_field drops it.
template <typename S>
__device__ __forceinline__ void load_neighbours(const Geom& g, const S* __restrict__ oth,
                                                const uint4& en, float2 v[4]) {
    using W = typename Store<S>::Word;
    const W* left = reinterpret_cast<const W*>(oth) + (ptrdiff_t)(int)en.w;
    const W* here = reinterpret_cast<const W*>(oth) + en.x;
    v[0] = Store<S>::decode(left[0], (en.y & GAP_L) != 0);
    v[1] = Store<S>::decode(left[1], (en.y & GAP_R) != 0);
    v[2] = Store<S>::decode(*(here - g.Wh), (en.y & GAP_U) != 0);
    v[3] = Store<S>::decode(here[g.Wh], (en.y & GAP_D) != 0);
}

// (cos, sin) of q phi_j of the four neighbours from their angles; 0 for a
// neighbour that does not exist.
__device__ __forceinline__ void neighbour_field(const Model& m, const float2 v[4], uint32_t f,
                                                float2 nc[4], float2 ns[4]) {
#pragma unroll
    for (int d = 0; d < 4; ++d) sincos_2(__fmul2_rn(both(m.q), v[d]), ns[d], nc[d]);
    if ((f & 0xFu) != 0xFu) {
#pragma unroll
        for (int d = 0; d < 4; ++d)
            if (!(f & (NB_L << d))) nc[d] = ns[d] = make_float2(0.0f, 0.0f);
    }
}

// Sum over the four neighbours, in the order every form uses.
__device__ __forceinline__ float2 sum4(const float2 v[4]) {
    return __fadd2_rn(__fadd2_rn(v[0], v[1]), __fadd2_rn(v[2], v[3]));
}

// One gap entry updated in both realizations of a pair: own angles ph, the
// four neighbours' angles v, Philox block w; returns the angles to store and
// adds the energy changes to ao / al / au (own block, left and upper
// neighbour's block).
template <typename S>
__device__ __forceinline__ float2 update_entry(const Model& m, float2 ph, const float2 v[4],
                                               uint32_t f, const uint32_t w[4], float2 beta,
                                               float2& ao, float2& al, float2& au) {
    float2 nc[4], ns[4];
    neighbour_field(m, v, f, nc, ns);
    const float2 C = sum4(nc), Sn = sum4(ns);
    const PairNew n = pair_update<S>(ph, C, Sn, u01_2(w[0], w[2]), u01_2(w[1], w[3]), beta, m);
    if (f & (EDGE_L | EDGE_U)) {
        // (the neighbours' cosines and sines again: see split_edge)
        float2 lc, ls, uc, us;
        sincos_2(__fmul2_rn(both(m.q), v[0]), ls, lc);
        sincos_2(__fmul2_rn(both(m.q), v[2]), us, uc);
        split_edge_2<S>(n, ph, f, C, Sn, lc, ls, uc, us, m, ao, al, au);
    } else {
        ao = __fadd2_rn(ao, n.dE);
    }
    return n.phi;
}

// The same in one realization of the pair (the other one does not run): its
// angle ph, its neighbours' angles v, its two Philox words.
template <typename S>
__device__ __forceinline__ float update_entry_one(const Model& m, float ph, const float v[4],
                                                  uint32_t f, uint32_t w0, uint32_t w1, float beta,
                                                  float& ao, float& al, float& au) {
    float nc[4], ns[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) __sincosf(m.q * v[d], &ns[d], &nc[d]);
    if ((f & 0xFu) != 0xFu) {
#pragma unroll
        for (int d = 0; d < 4; ++d)
            if (!(f & (NB_L << d))) nc[d] = ns[d] = 0.0f;
    }
    const float C = (nc[0] + nc[1]) + (nc[2] + nc[3]);
    const float Sn = (ns[0] + ns[1]) + (ns[2] + ns[3]);
    const SiteNew n = site_update<S>(ph, C, Sn, u01(w0), u01(w1), beta, m);
    if (f & (EDGE_L | EDGE_U))
        split_edge<S>(n, ph, f, C, Sn, nc[0], ns[0], nc[2], ns[2], m, ao, al, au);
    else
        ao += n.dE;
    return n.phi;
}

__device__ __forceinline__ void pair_running(const SweepArgs& a, int b, int rl, bool& run0,
                                             bool& run1) {
    if (a.running) {
        const uchar2 r2 = *reinterpret_cast<const uchar2*>(a.running + (size_t)b * a.Rp + rl);
        run0 = r2.x != 0;
        run1 = r2.y != 0;
    } else {
        run0 = rl < a.R;
        run1 = rl + 1 < a.R;
    }
}

// Clears the sums of the pair's realizations that do not run.
__device__ __forceinline__ void drop_idle(bool run0, bool run1, float2& ao, float2& al,
                                          float2& au) {
    if (!run0) ao.x = al.x = au.x = 0.0f;
    if (!run1) ao.y = al.y = au.y = 0.0f;
}

// The gap entries e, e + step, ... < e1 of one unit, by one lane; the next
// list entry is loaded while the current one is updated. kAll: both
// realizations run; else one that does not keeps its angles, and its sums are
// cleared at the end.
template <typename S, bool kAll>
__device__ __forceinline__ void sweep_entries(const SweepArgs& a, int e, int e1, int step, S* own,
                                              const S* oth, uint32_t ctr1, uint32_t rpair,
                                              uint32_t key1, float2 beta, bool run0, bool run1,
                                              float2& ao, float2& al, float2& au) {
    const float* bs =
        a.beta_site ? a.beta_site + (size_t)a.colour * a.g.H * a.g.Wh : nullptr;
    uint4 nx = e < e1 ? a.list[e] : make_uint4(0u, 0u, 0u, 0u);
    for (; e < e1; e += step) {
        const uint4 en = nx;
        if (e + step < e1) nx = a.list[e + step];
        uint32_t w[4];
        philox4x32_10_rk(en.z, ctr1, rpair, 0u, a.rng.rk0, key1, w);
        S* po = own + 2 * (size_t)en.x;
        const float2 ph = Store<S>::load2(po);
        float2 v[4];
        load_neighbours<S>(a.g, oth, en, v);
        const float2 bt = bs ? both(bs[en.x]) : beta;
        float2 out = update_entry<S>(a.m, ph, v, en.y, w, bt, ao, al, au);
        if constexpr (!kAll) out = make_float2(run0 ? out.x : ph.x, run1 ? out.y : ph.y);
        Store<S>::store2(po, out);
    }
    if constexpr (!kAll) drop_idle(run0, run1, ao, al, au);
}

// All gap sites of colour c of one unit: block b in realization pair p, by CW
// warps that split its entries 32 at a time (cw: this warp's index among
// them). The block's list puts its edge entries first, so the branch that
// splits an edge move bond by bond diverges in the first 32 entries only.
// kCal: the calibration's chains, whose two lanes of a pair may sit at
// different temperatures (the trisection's two points, or the k-point
// section's lane r at point r mod n_pts), as in sweep_flat.
template <typename S, bool kCal = false, bool kAll = false>
__device__ __forceinline__ void sweep_item(const SweepArgs& a, int b, int p, int cw, int CW,
                                           uint32_t ctr1) {
    const int lane = threadIdx.x & 31;
    const int e0 = a.start[b], e1 = a.start[b + 1];
    if (e0 >= e1) return;
    const int rl = 2 * p;
    bool run0, run1;
    pair_running(a, b, rl, run0, run1);
    if (!(run0 || run1)) return;
    S* own = static_cast<S*>(a.ang) + pair_plane(a.g, p, a.colour);
    const S* oth = static_cast<const S*>(a.ang) + pair_plane(a.g, p, a.colour ^ 1);
    float beta = a.beta[b], beta_odd = beta;
    if constexpr (kCal) {
        if (a.beta_pts) {
            beta = a.beta_pts[(size_t)(rl % a.n_pts) * a.g.nblk + b];
            beta_odd = a.beta_pts[(size_t)((rl + 1) % a.n_pts) * a.g.nblk + b];
        } else if (a.beta_odd) {
            beta_odd = a.beta_odd[b];
        }
    }
    const uint32_t rpair = (a.r_base + (uint32_t)rl) >> 1;
    const uint32_t key1 = slice_key1(a.sl, slice_of(a.sl, b));
    float2 ao = both(0.0f), al = ao, au = ao;
    const int e = e0 + cw * 32 + lane, step = CW * 32;
    const float2 bt = make_float2(beta, beta_odd);
    if constexpr (kCal) {
        // A calibration's lists and state of many waves stream from memory (a
        // realization batch reads its lists again and again), and an entry's
        // words are known only once the entry is: the block's rows are asked
        // for at once, a row per lane. 4096^2, l_b = 32, half of the sites
        // missing, two points: 73.9 -> 69.3 us per half-step. Ahead of the list
        // (from the block's place) 71.0, a wave of units ahead 77.8, an entry
        // ahead per lane 74.6 us; in the realizations' kernels 2 % slower.
        const uint32_t h0 = a.list[e0].x, h1 = a.list[e1 - 1].x, Wh = (uint32_t)a.g.Wh;
        const uint32_t y0 = h0 / Wh, x = h0 - y0 * Wh;
        for (uint32_t y = y0 + lane; y <= h1 / Wh; y += 32) {
            const size_t at = 2 * ((size_t)y * Wh + x);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(own + at));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(oth + at));
        }
    }
    sweep_entries<S, kAll>(a, e, e1, step, own, oth, ctr1, rpair, key1, bt, run0, run1, ao, al,
                           au);
    if (!a.energy) return;
    double* ea = a.eacc + (size_t)b * a.Rp + rl;
    flush_pair(ea, ao.x, ao.y);
    flush_pair(ea - a.Rp, al.x, al.y);
    flush_pair(ea - (size_t)a.g.nbx * a.Rp, au.x, au.y);
}

// Energy flush of one half-warp's unit: the FP32 sum over its 16 lanes, added
// by its lane 0 with an FP64 atomic (act: the half has a running unit).
// Every lane of the warp calls it.
__device__ __forceinline__ void flush_pair_half(double* ea, float v0, float v1, bool act) {
    if (!__any_sync(0xffffffffu, v0 != 0.0f || v1 != 0.0f)) return;
#pragma unroll
    for (int s = 8; s > 0; s >>= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, s);
        v1 += __shfl_xor_sync(0xffffffffu, v1, s);
    }
    if ((threadIdx.x & 15) != 0 || !act) return;
    if (v0 != 0.0f) atomicAdd(ea, (double)v0);
    if (v1 != 0.0f) atomicAdd(ea + 1, (double)v1);
}

// Two units per warp: lanes 0-15 take one (block, realization pair) unit,
// lanes 16-31 another, each half 16 gap entries at a time. For blocks whose
// colour holds few entries (about 64 at l_b = 16 and half the sites missing)
// the last, partial pass wastes fewer lanes, and the warp's per-unit work
// (bounds, flags, energy sums) serves two units. have: this half has a unit
// (block b, pair p); every lane of the warp calls this.
template <typename S>
__device__ __forceinline__ void sweep_item_half(const SweepArgs& a, int b, int p, bool have,
                                                uint32_t ctr1) {
    const int hl = threadIdx.x & 15;
    int e0 = 0, e1 = 0;
    bool run0 = false, run1 = false;
    const int rl = 2 * p;
    if (have) {
        e0 = a.start[b];
        e1 = a.start[b + 1];
        pair_running(a, b, rl, run0, run1);
    }
    const bool act = have && e0 < e1 && (run0 || run1);
    float2 ao = both(0.0f), al = ao, au = ao;
    if (act) {
        S* own = static_cast<S*>(a.ang) + pair_plane(a.g, p, a.colour);
        const S* oth = static_cast<const S*>(a.ang) + pair_plane(a.g, p, a.colour ^ 1);
        const float beta = a.beta[b];
        const uint32_t rpair = (a.r_base + (uint32_t)rl) >> 1;
        const uint32_t key1 = slice_key1(a.sl, slice_of(a.sl, b));
        // (one loop for both: the two halves of a warp would take turns in two)
        sweep_entries<S, false>(a, e0 + hl, e1, 16, own, oth, ctr1, rpair, key1, both(beta), run0,
                                run1, ao, al, au);
    }
    if (!a.energy) return;
    double* ea = a.eacc + (size_t)b * a.Rp + rl;
    flush_pair_half(ea, ao.x, ao.y, act);
    flush_pair_half(ea - a.Rp, al.x, al.y, act);
    flush_pair_half(ea - (size_t)a.g.nbx * a.Rp, au.x, au.y, act);
}

// One half-step over the whole list of one colour, flat: one thread per
// (gap entry, realization pair). For calibration, where every block runs
// and only one or a few chains exist, this puts every site's
// latency chain into one wave. The block-energy change is summed per CTA in
// shared memory (the list is block-major, so a CTA spans few blocks) and
// flushed with one atomic per (block, realization); changes that belong to
// another block (left / up bonds of edge sites) go straight to global memory.
// The per-CTA sums are FP32; the global accumulation is FP64.
constexpr int kFlatThreads = 256;
constexpr int kFlatBlocks = 64;     // local blocks summed in shared memory per CTA

// Programmatic dependent launch: a launch may start while the previous
// kernel on the stream finishes. griddepcontrol.wait blocks until every
// prerequisite grid has completed and its writes are visible; every thread of
// such a kernel executes it (so its completion implies its predecessors').
// launch_dependents lets the next launch begin once every CTA of this one
// has issued it or exited.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The list entry, its Philox block and the temperatures do not depend on the
// previous half-step, so they are taken before the dependency wait and
// overlap the previous launch's tail.
//
// A CTA takes kFlatThreads entries of one pair (blockIdx.y), so no thread is
// left to the padding lanes of a group of G; the sums keep the group's shares:
// G / 2 sections of a CTA, each with shared-memory sums of its own, and warp
// sums of 64 / G entries. With an entry's G / 2 pairs on neighbouring threads,
// four chains (G = 8) left half of the threads idle: forward and backward of a
// 1024^2 field 2.85 ms, now 2.17; three chains 3.15 -> 2.05, eight (no padding)
// 3.07 -> 3.10.
template <int G>
__device__ __forceinline__ void sweep_flat(const SweepArgs& a, int64_t n_list, uint32_t ctr1) {
    constexpr int kSections = G / 2;
    constexpr int kSection = kFlatThreads / kSections;
    constexpr int kSum = 32 / kSections;
    __shared__ float acc[kSections][kFlatBlocks * 2];
    const int sec = (int)threadIdx.x / kSection;
    const int64_t e0 = (int64_t)blockIdx.x * kFlatThreads;
    const int64_t e = e0 + threadIdx.x;
    for (int i = threadIdx.x; i < kSections * kFlatBlocks * 2; i += kFlatThreads) (&acc[0][0])[i] = 0.0f;
    const int64_t s0 = e0 + sec * kSection;
    const int b0 = kSections == 1 || s0 < n_list ? (int)(a.list[s0].y >> META_SHIFT) : 0;
    const bool live = e < n_list;
    const int rl = 2 * (int)blockIdx.y;
    uint4 en = make_uint4(0u, 0u, 0u, 0u);
    int b = b0;
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    float beta = 0.0f, beta1 = 0.0f;
    if (live) {
        en = a.list[e];
        b = (int)(en.y >> META_SHIFT);
        philox4x32_10_rk(en.z, ctr1, (a.r_base + (uint32_t)rl) >> 1, 0u, a.rng.rk0,
                         slice_key1(a.sl, slice_of(a.sl, b)), w);
        if (a.beta_pts) {
            beta = a.beta_pts[(size_t)(rl % a.n_pts) * a.g.nblk + b];
            beta1 = a.beta_pts[(size_t)((rl + 1) % a.n_pts) * a.g.nblk + b];
        } else {
            beta = a.beta[b];
            beta1 = a.beta_odd ? a.beta_odd[b] : beta;
        }
    }
    grid_dep_wait();
    __syncthreads();
    float2 ao = both(0.0f), al = ao, au = ao;
    uint32_t f = 0;
    if (live) {
        bool run0, run1;
        pair_running(a, b, rl, run0, run1);
        if (run0 || run1) {
            f = en.y;
            float* po = static_cast<float*>(a.ang) + pair_plane(a.g, rl >> 1, a.colour) +
                        2 * (size_t)en.x;
            const float* oth =
                static_cast<const float*>(a.ang) + pair_plane(a.g, rl >> 1, a.colour ^ 1);
            float2 v[4];
            load_neighbours<float>(a.g, oth, en, v);
            if (run0 && run1) {
                Store<float>::store2(po, update_entry<float>(a.m, Store<float>::load2(po), v, f, w,
                                                             make_float2(beta, beta1), ao, al, au));
            } else {
                // one lane runs (a bisection's single chain): the other's arithmetic left out
                const int o = run0 ? 0 : 1;
                const float v1[4] = {run0 ? v[0].x : v[0].y, run0 ? v[1].x : v[1].y,
                                     run0 ? v[2].x : v[2].y, run0 ? v[3].x : v[3].y};
                po[o] = update_entry_one<float>(a.m, po[o], v1, f, w[2 * o], w[2 * o + 1],
                                                run0 ? beta : beta1, run0 ? ao.x : ao.y,
                                                run0 ? al.x : al.y, run0 ? au.x : au.y);
            }
        }
    }
    if (!a.energy) return;
    // The block's share: one sum per realization when all kSum entries lie in
    // one block (the usual case: the list is block-major), else an atomic per
    // lane; shared-memory sums for the section's first blocks.
    const int lane = threadIdx.x & 31;
    const int first = lane & ~(kSum - 1);
    bool whole;
    float2 sum = ao;
    if constexpr (kSections == 1) {
        whole = __all_sync(0xffffffffu, b == __shfl_sync(0xffffffffu, b, 0));
    } else {
        const uint32_t same = __ballot_sync(0xffffffffu, b == __shfl_sync(0xffffffffu, b, first));
        whole = ((same >> first) & ((1u << (kSum & 31)) - 1u)) == (1u << (kSum & 31)) - 1u;
    }
    if (kSections > 1 || whole) {
#pragma unroll
        for (int d = kSum / 2; d >= 1; d >>= 1) {
            sum.x += __shfl_xor_sync(0xffffffffu, sum.x, d);
            sum.y += __shfl_xor_sync(0xffffffffu, sum.y, d);
        }
    }
    if (whole ? lane == first : live) {
        if (!whole) sum = ao;
        const int loc = b - b0;
        if (loc < kFlatBlocks) {
            if (sum.x != 0.0f) atomicAdd(&acc[sec][loc * 2], sum.x);
            if (sum.y != 0.0f) atomicAdd(&acc[sec][loc * 2 + 1], sum.y);
        } else {
            double* ea = a.eacc + (size_t)b * a.Rp + rl;
            if (sum.x != 0.0f) atomicAdd(ea, (double)sum.x);
            if (sum.y != 0.0f) atomicAdd(ea + 1, (double)sum.y);
        }
    }
    // Left / up bonds of edge sites belong to the neighbouring blocks.
    if (f & (EDGE_L | EDGE_U)) {
        double* ea = a.eacc + (size_t)b * a.Rp + rl;
        if (al.x != 0.0f) atomicAdd(ea - a.Rp, (double)al.x);
        if (al.y != 0.0f) atomicAdd(ea - a.Rp + 1, (double)al.y);
        const size_t up = (size_t)a.g.nbx * a.Rp;
        if (au.x != 0.0f) atomicAdd(ea - up, (double)au.x);
        if (au.y != 0.0f) atomicAdd(ea - up + 1, (double)au.y);
    }
    __syncthreads();
    for (int i = (int)threadIdx.x % kSection; i < kFlatBlocks * 2; i += kSection) {
        const float v = acc[sec][i];
        if (v != 0.0f) atomicAdd(&a.eacc[(size_t)(b0 + i / 2) * a.Rp + rl + (i & 1)], (double)v);
    }
}

// Fold of the previous sweep's block energies by CTA `cta` of f.ctas: E_b of
// every (block, chain lane) gains the sweep's change, and during the measured
// sweeps each point's mean e_b gains E_b / N_b. It touches eacc of the other
// parity and ecur, which the half-step does not. kThreads: the CTA size.
template <int kThreads>
__device__ __forceinline__ void fold_block_energies(const FoldArgs& f, int cta) {
    for (int b = cta * kThreads + (int)threadIdx.x; b < f.nblk; b += f.ctas * kThreads) {
        double s[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (int r = 0; r < f.chains * f.points; ++r) {
            const size_t k = (size_t)b * f.Rp + r;
            const double E = f.ecur[k] + f.eacc[k];
            f.ecur[k] = E;
            f.eacc[k] = 0.0;
            s[r % f.points] += E * f.inb[b];
        }
        if (f.measure) {
            if (f.points > 2) {
                for (int p = 0; p < f.points; ++p) f.ebar_pts[(size_t)p * f.nblk + b] += s[p];
            } else {
                f.ebar[b] += s[0];
                if (f.points == 2) f.ebar_odd[b] += s[1];
            }
        }
    }
}

// Energies from scratch (no move) of one item: the bonds that touch a gap
// site of this colour and belong to no gap site of the other colour (colour
// 1 counts all bonds of its gap sites, colour 0 only those to sample
// neighbours). Each lane sums its few bonds in FP32; the warp sums and the
// block totals are FP64.
// The FP32 partial sums of the lanes depend on how the warps
// split the entries: warp wi of a block's four takes pair wi mod NP of lane
// group grp, and the 4 / NP warps of a pair split them 32 at a time.
template <typename S>
__device__ __forceinline__ void energy_item(const SweepArgs& a, int b, int grp, int NP, int wi,
                                            int wpi) {
    const int lane = threadIdx.x & 31;
    const int q = wi % NP, cw = wi / NP, CW = wpi / NP;
    const int c = a.colour;
    const int rl = 2 * (grp * NP + q);
    const int e0 = a.start[b], e1 = a.start[b + 1];
    const S* own = static_cast<const S*>(a.ang) + pair_plane(a.g, rl >> 1, c);
    const S* oth = static_cast<const S*>(a.ang) + pair_plane(a.g, rl >> 1, c ^ 1);
    float o0 = 0.f, o1 = 0.f, l0 = 0.f, l1 = 0.f, u0 = 0.f, u1 = 0.f;
    for (int e = e0 + cw * 32 + lane; e < e1; e += CW * 32) {
        const uint4 en = a.list[e];
        const uint32_t f = en.y;
        const float2 ph = Store<S>::load2(own + 2 * (size_t)en.x);
        float2 v[4], nc[4], ns[4];
        load_neighbours<S>(a.g, oth, en, v);
        neighbour_field(a.m, v, f, nc, ns);
        float s0, c0, s1, c1;
        __sincosf(a.m.q * ph.x, &s0, &c0);
        __sincosf(a.m.q * ph.y, &s1, &c1);
        const uint32_t take = (c == 1) ? 0xFu : (~(f >> 4) & 0xFu);
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            if (!((f & (NB_L << d)) && (take & (1u << d)))) continue;
            const float b0 = -a.m.J * (c0 * nc[d].x + s0 * ns[d].x);
            const float b1 = -a.m.J * (c1 * nc[d].y + s1 * ns[d].y);
            if (d == 0 && (f & EDGE_L)) { l0 += b0; l1 += b1; }
            else if (d == 2 && (f & EDGE_U)) { u0 += b0; u1 += b1; }
            else { o0 += b0; o1 += b1; }
        }
    }
    double v[6] = {o0, o1, l0, l1, u0, u1};
#pragma unroll
    for (int s = 16; s > 0; s >>= 1)
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], s);
    if (lane != 0) return;
    double* ea = a.ecur + (size_t)b * a.Rp + rl;
    const size_t up = (size_t)a.g.nbx * a.Rp;
    if (v[0] != 0.0) atomicAdd(ea, v[0]);
    if (v[1] != 0.0) atomicAdd(ea + 1, v[1]);
    if (v[2] != 0.0) atomicAdd(ea - a.Rp, v[2]);
    if (v[3] != 0.0) atomicAdd(ea - a.Rp + 1, v[3]);
    if (v[4] != 0.0) atomicAdd(ea - up, v[4]);
    if (v[5] != 0.0) atomicAdd(ea - up + 1, v[5]);
}

// The stop test after sweep t_sweep, on the items of the sweep's worklist
// (every running (block, realization) pair belongs to one of them), in two
// parts: the second needs the final per-realization count of running
// targeted blocks, which the first completes.
//
// Targeted part: E_b += the sweep's change (eacc, then cleared); e_b = E_b / N_b;
// a targeted block stops once sigma (e_b(t) - e_s,b) >= 0 (CROSS), or, under the
// WINDOW rule, at a test sweep t = n_fit + n_f + k n_f once the least-squares
// slope of e_b over sweeps t - n_fit + 1 .. t no longer has the sign sigma
// (its numerator sum_j (2 j - (n_fit - 1)) e_b(t - n_fit + 1 + j)). Entries
// i = i0, i0 + step, ... < n of (item, lane) pairs (n = items * G). Entries
// below `cap` are readable whatever n is (the worklist buffer's length times
// G; past n they hold stale items), so the first item is read without waiting
// for n; every value of an entry is then read at once, and only then tested.
// U entries per pass: a pass reads all of its entries' values before it tests
// any of them, so U loads of each kind are in flight per thread (the test is
// latency-bound: an entry's loads wait for the worklist word naming its
// block). Entries are independent (each (block, realization) appears once).
template <int U = 1>
__device__ __forceinline__ void stop_targeted_range(const StopArgs& s, uint32_t t_sweep,
                                                    const uint32_t* __restrict__ w, int64_t n,
                                                    int64_t cap, int64_t i0, int64_t step) {
    for (int64_t ib = i0; ib < n; ib += (int64_t)U * step) {
        uint32_t item[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = ib + (int64_t)u * step;
            item[u] = i < cap ? w[i / s.G] : 0u;
        }
        size_t k[U];
        int b[U], r[U], sg[U];
        int32_t nsp[U], ob[U];
        uint8_t run[U];
        double E[U], inb[U], es[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = ib + (int64_t)u * step;
            b[u] = (int)(item[u] / (uint32_t)s.groups);
            r[u] = (int)(item[u] % (uint32_t)s.groups) * s.G + (int)(i % s.G);
            k[u] = (size_t)b[u] * s.Rp + r[u];
            const bool v = i < n;
            run[u] = v ? s.running[k[u]] : (uint8_t)0;
            E[u] = v ? s.ecur[k[u]] + s.eacc[k[u]] : 0.0;
            inb[u] = v ? s.inb[b[u]] : 0.0;
            es[u] = v ? s.es[b[u]] : 0.0;
            nsp[u] = v ? s.Nsp[b[u]] : 0;
            ob[u] = v ? s.of_block[b[u]] : 0;
            sg[u] = v ? s.sigma[k[u]] : 0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (!run[u]) continue;
            s.eacc[k[u]] = 0.0;
            s.ecur[k[u]] = E[u];
            const double e = E[u] * inb[u];
            s.e_last[k[u]] = e;
            bool reached;
            if (s.win.rule == 1) {
                const int nf = s.win.n_fit;
                s.win.hist[(size_t)(t_sweep % (uint32_t)nf) * s.win.stride + k[u]] = e;
                if (nsp[u] == 0) continue;
                const uint32_t first = (uint32_t)(nf + s.win.n_f);
                if (t_sweep < first || (t_sweep - first) % (uint32_t)s.win.n_f != 0) continue;
                double num = 0.0;
                for (int j = 0; j < nf; ++j) {
                    const uint32_t sw = t_sweep - (uint32_t)nf + 1u + (uint32_t)j;
                    num += (double)(2 * j - (nf - 1)) *
                           s.win.hist[(size_t)(sw % (uint32_t)nf) * s.win.stride + k[u]];
                }
                reached = (double)sg[u] * num <= 0.0;
            } else {
                if (nsp[u] == 0) continue;
                reached = sg[u] > 0 ? (e >= es[u]) : (sg[u] < 0 ? (e <= es[u]) : true);
            }
            if (reached) {
                s.running[k[u]] = 0;
                s.stop[k[u]] = (int32_t)t_sweep;
                atomicSub(&s.tcount[ob[u] * s.Rp + r[u]], 1);
            }
        }
    }
}

// Closing part: blocks without sample bonds stop when no targeted block of
// their realization runs; everything stops at n_max. Items with a lane still
// running are appended to `out` (counter *n_out, one atomic per warp, items in
// lane order). Items i = i0, i0 + step, ... < n of the worklist w (nullptr:
// every item); `cap` as for the targeted part. Returns this thread's count of
// lanes still running.
__device__ __forceinline__ unsigned stop_rest_range(const StopArgs& s, uint32_t t_sweep,
                                                    const uint32_t* __restrict__ w, int64_t n,
                                                    int64_t cap, uint32_t* __restrict__ out,
                                                    uint32_t* n_out, int64_t i0, int64_t step) {
    unsigned cnt = 0;
    uint32_t item = w ? (i0 < cap ? w[i0] : 0u) : (uint32_t)i0;
    for (int64_t i = i0; i < n; i += step) {
        if (i != i0) item = w ? w[i] : (uint32_t)i;
        const int b = (int)(item / (uint32_t)s.groups), grp = (int)(item % (uint32_t)s.groups);
        const int32_t ob = s.of_block[b], nsp = s.Nsp[b];
        const int32_t* tc = s.tcount + (size_t)(ob < 0 ? 0 : ob) * s.Rp;
        bool any = false;
        for (int g = 0; g < s.G; ++g) {
            const int r = grp * s.G + g;
            const size_t k = (size_t)b * s.Rp + r;
            if (!s.running[k]) continue;
            if ((nsp == 0 && tc[r] == 0) || (int)t_sweep >= s.n_max) {
                s.running[k] = 0;
                s.stop[k] = (int32_t)t_sweep;
            } else {
                ++cnt;
                any = true;
            }
        }
        const unsigned act = __activemask();
        const unsigned vote = __ballot_sync(act, any);
        if (vote) {
            const int lane = threadIdx.x & 31;
            const int leader = __ffs(vote) - 1;
            uint32_t base = 0;
            if (lane == leader) base = atomicAdd(n_out, (uint32_t)__popc(vote));
            base = __shfl_sync(act, base, leader);
            if (any) out[base + __popc(vote & ((1u << lane) - 1u))] = item;
        }
    }
    return cnt;
}

// ------------------------------------------------- grid-wide barrier --
// For cooperative launches (the persistent calibration and the simulation's
// stop tail). The barrier never waits forever: a CTA that has waited `limit`
// polls sets the error flag and returns false, and every CTA that sees the
// flag returns false too; the host then reports MPR_ETIMEOUT. A test hook
// (`extra`) makes the barrier wait for arrivals that never come, to exercise
// that path.
__device__ __forceinline__ unsigned int ld_acquire(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Barrier over all CTAs of the launch. `gen` is the generation this CTA last
// passed (kept by thread 0). The last CTA to arrive runs last() (thread 0)
// before it releases the others, so its writes are visible to every CTA
// after the barrier. Returns false if the wait gave up here or elsewhere.
template <typename F>
__device__ bool grid_sync_then(GridBarrier* bar, unsigned int& gen, unsigned long long limit,
                               F&& last) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = ld_acquire(&bar->err) == 0;
        if (ok) {
            const unsigned int target = gen + 1;
            const unsigned int expect = gridDim.x + bar->extra;
            __threadfence();
            const unsigned int arrived = atomicAdd(&bar->arrive, 1u) + 1u;
            if (arrived == expect) {
                __threadfence();
                last();
                atomicExch(&bar->arrive, 0u);
                __threadfence();
                atomicExch(&bar->gen, target);
            } else {
                unsigned long long spins = 0;
                while (ld_acquire(&bar->gen) != target) {
                    if (ld_acquire(&bar->err) != 0) {
                        ok = 0;
                        break;
                    }
                    if (++spins > limit) {
                        atomicExch(&bar->err, 1u);
                        ok = 0;
                        break;
                    }
                    __nanosleep(100);
                }
            }
            __threadfence();
            gen = target;
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

__device__ __forceinline__ bool grid_sync(GridBarrier* bar, unsigned int& gen,
                                          unsigned long long limit) {
    return grid_sync_then(bar, gen, limit, [] {});
}

// Median of the targeted blocks' T by a radix select over the (positive)
// float bit patterns, run by one CTA over the blocks of one slice (the block
// rectangle bk = (by0, bx0, nby_s, nbx_s) of a canvas nbx blocks wide); k is
// the 0-based rank.
__device__ inline uint32_t select_kth(const float* __restrict__ T, const int32_t* __restrict__ Nsp,
                                      int4 bk, int nbx, uint32_t k, uint32_t* hist,
                                      uint32_t* s_digit, uint32_t* s_k) {
    const int nb = bk.z * bk.w;
    uint32_t prefix = 0, pmask = 0;
    for (int pass = 0; pass < 4; ++pass) {
        const int shift = 24 - 8 * pass;
        for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
        __syncthreads();
        for (int j = threadIdx.x; j < nb; j += blockDim.x) {
            const int b = (bk.x + j / bk.w) * nbx + bk.y + j % bk.w;
            if (Nsp[b] <= 0) continue;
            const uint32_t v = __float_as_uint(T[b]);
            if ((v & pmask) == prefix) atomicAdd(&hist[(v >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t kk = k, d = 0;
            while (d < 255 && kk >= hist[d]) { kk -= hist[d]; ++d; }
            *s_digit = d;
            *s_k = kk;
        }
        __syncthreads();
        prefix |= (*s_digit) << shift;
        pmask |= 255u << shift;
        k = *s_k;
        __syncthreads();
    }
    return prefix;
}

// Median (mean of the two middle values for an even count) of the targeted
// blocks' T within one slice, by one CTA; 0 when no block is targeted.
__device__ inline float median_targeted(const float* __restrict__ T, const int32_t* __restrict__ Nsp,
                                        int4 bk, int nbx) {
    __shared__ uint32_t hist[256];
    __shared__ uint32_t s_digit, s_k, s_n;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int nb = bk.z * bk.w;
    uint32_t cnt = 0;
    for (int j = threadIdx.x; j < nb; j += blockDim.x)
        cnt += Nsp[(bk.x + j / bk.w) * nbx + bk.y + j % bk.w] > 0;
    atomicAdd(&s_n, cnt);
    __syncthreads();
    const uint32_t n = s_n;
    float med = 0.0f;
    if (n > 0) {
        const float lo =
            __uint_as_float(select_kth(T, Nsp, bk, nbx, (n - 1) / 2, hist, &s_digit, &s_k));
        const float hi = (n & 1) ? lo
                                 : __uint_as_float(select_kth(T, Nsp, bk, nbx, n / 2, hist,
                                                              &s_digit, &s_k));
        med = 0.5f * (lo + hi);
    }
    return med;
}

}  // namespace mpr
