// One calibration iteration of a field that the GPU holds in one wave, as one
// cooperative launch: for each realization pair a group of CTAs, each with its
// stretch of both colours' lists in shared memory, runs the pair's start, all
// n_eq + n_meas sweeps and the energy averages of the measured ones.
//
// A half-step as a launch of its own takes 8.1 us for the 262 k gap sites per
// colour of a 1024^2 field and two realizations, two thirds of it launch, list
// and state loads (1.9 us of instruction issue at full rate). Here it takes 5.5,
// and 1.85 instead of 3.3 us for the 33 k sites of a 256^2 field, which is the
// way of a message and a site's update: a site's angle, (cos, sin) of q times the
// angle and everything its updates need stay in shared memory, a cosine is taken
// once instead of by four neighbours, and the next half-step's random numbers
// and proposals are worked out while messages are under way.
//
// A lattice update needs only adjacent sites, so there is no grid-wide order
// either: a CTA starts a half-step when it has the angles of its sites'
// neighbours that other CTAs own (a few per hundred: the lists are block-major),
// each of which carries the half-step it belongs to. (With a flag per CTA behind
// a fence, and the cells read after it: 3.2 us per half-step of the 256^2 field.
// With a copy of the update's code per colour: 2.4 us, for its instruction
// fetches.) A site's next angle is sent only after the adjacent sites' previous
// ones have come, whose owner had read this one before, so a message is not
// overwritten before it is read. Every wait is bounded; a CTA that gives up marks
// the launch, the others follow, and the host runs the calibration with a launch
// per half-step.
//
// Energies as in mpr_calcluster.cu (changes weighted by the measured sweeps they
// count for), but with the FP32 warp sums of the launch-per-half-step form, so
// that both round alike; everything above a warp is summed in FP64, a change
// that belongs to another block error-free in two floats.
#include <cuda_runtime.h>

#include <cstdint>

#include "mpr_launch.h"
#include "mpr_sweep.cuh"

namespace mpr {

namespace {

constexpr int kThreads = kCalResidentThreads;
constexpr int kRounds = kCalResidentSites / kThreads;   // sites per thread and colour

// meta word of a site: bit 0: other CTAs read it; EDGE_L, EDGE_U as in the
// list; then its block (counted from the CTA's first) and its edge record.
constexpr uint32_t kExported = 1u;
constexpr int kBlockShift = 10, kEdgeShift = 21;
constexpr uint32_t kBlockMask = (1u << (kEdgeShift - kBlockShift)) - 1u;
static_assert((EDGE_L | EDGE_U) < (1u << kBlockShift), "flags below the block");

// Shared memory, in this order: cells of the even realization, then of the odd
// one (own sites of both colours, then the neighbours owned elsewhere), cells of
// samples (the same in both), angles, edge records, site records, blocks, warp
// sums, sources of the neighbours' cells.
struct Layout {
    int cells;     // cells per realization
    size_t angles, edges, sites, blocks, sums, sources, bytes;
    __host__ __device__ explicit Layout(const CalResidentArgs& a) {
        cells = a.sites + 2 * a.halo;
        angles = (size_t)(2 * cells + a.consts) * sizeof(float2);
        edges = angles + (size_t)a.sites * sizeof(float2);
        sites = edges + (size_t)a.edges * sizeof(float4);
        blocks = sites + (size_t)a.sites * sizeof(uint4);
        sums = blocks + (size_t)a.blocks * sizeof(float4);
        sources = sums + (size_t)(a.sites / 32) * sizeof(float4);
        bytes = sources + (size_t)2 * a.halo * sizeof(uint32_t);
    }
};

__device__ __forceinline__ uint32_t load_acquire(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// An exported angle pair with the half-step it is of: 16 bytes, written and read
// as one (PTX: 128-bit accesses of a scope are single-copy atomic), so that the
// reader polls the message itself, with no flag and no fence.
__device__ __forceinline__ void send(float4* to, float2 ph, uint32_t h) {
    asm volatile("{\n\t.reg .b64 x, y;\n\t.reg .b128 v;\n\tmov.b64 x, {%1, %2};\n\t"
                 "mov.b64 y, {%3, %4};\n\tmov.b128 v, {x, y};\n\t"
                 "st.relaxed.gpu.global.b128 [%0], v;\n\t}" ::"l"(to),
                 "f"(ph.x), "f"(ph.y), "r"(h), "r"(0u)
                 : "memory");
}
__device__ __forceinline__ uint32_t look(const float4* from, float2& ph) {
    uint32_t h, unused;
    asm volatile("{\n\t.reg .b64 x, y;\n\t.reg .b128 v;\n\t"
                 "ld.relaxed.gpu.global.b128 v, [%4];\n\tmov.b128 {x, y}, v;\n\t"
                 "mov.b64 {%0, %1}, x;\n\tmov.b64 {%2, %3}, y;\n\t}"
                 : "=f"(ph.x), "=f"(ph.y), "=r"(h), "=r"(unused)
                 : "l"(from)
                 : "memory");
    return h;
}

// Polls until done() holds. False (and the launch marked) after `limit` polls,
// or when another wait gave up.
template <typename F>
__device__ __forceinline__ bool poll(uint32_t* error, uint32_t limit, F&& done) {
    for (uint32_t polls = 0; !done();) {
        if (++polls >= limit) {
            atomicExch(error, 1u);
            return false;
        }
        if ((polls & 63u) == 0 && load_acquire(error) != 0) return false;
    }
    return true;
}

// kOne: only the pair's even realization exists (a bisection's single chain).
template <bool kOne>
__global__ void __launch_bounds__(kThreads, 1) k_cal_resident(CalResidentArgs a) {
    extern __shared__ float4 smem[];
    __shared__ int s_part[2][kCalResidentCtas + 1];
    __shared__ int s_consts, s_edges, s_halo[2], s_bad;
    const CalClusterArgs& k = a.cal;
    const SweepArgs& sw = k.sw;
    const Model& m = sw.m;
    const Layout at(a);
    unsigned char* base = reinterpret_cast<unsigned char*>(smem);
    float2* cells = reinterpret_cast<float2*>(smem);
    float2* angles = reinterpret_cast<float2*>(base + at.angles);
    float4* edges = reinterpret_cast<float4*>(base + at.edges);
    uint4* sites = reinterpret_cast<uint4*>(base + at.sites);
    float4* blocks = reinterpret_cast<float4*>(base + at.blocks);
    float* sums = reinterpret_cast<float*>(base + at.sums);
    uint32_t* sources = reinterpret_cast<uint32_t*>(base + at.sources);
    const int odd = at.cells;               // an odd realization's cell lies this far on
    const int tid = threadIdx.x, lane = tid & 31;
    const int p = (int)(blockIdx.x / a.ctas), rank = (int)(blockIdx.x % a.ctas);
    const int rl = 2 * p;
    const bool run0 = rl < sw.R, run1 = rl + 1 < sw.R;
    const uint32_t tag = sw.ctl->tag, rpair = (sw.r_base + (uint32_t)rl) >> 1;
    uint32_t* error = a.sync;
    float4* exports = a.exports + (size_t)p * a.ctas * 2 * a.cap;

    if (tid == 0) {
        s_bad = load_acquire(error) != 0;
        s_consts = 1;                       // the first: no neighbour
        s_edges = 0;
        s_halo[0] = s_halo[1] = 0;
        cells[2 * at.cells] = both(0.0f);
    }
    for (int i = tid; i < 2 * (a.ctas + 1); i += kThreads)
        s_part[i / (a.ctas + 1)][i % (a.ctas + 1)] = a.part[i];
    __syncthreads();
    if (s_bad) return;
    const int e0[2] = {s_part[0][rank], s_part[1][rank]};
    const int n[2] = {s_part[0][rank + 1] - e0[0], s_part[1][rank + 1] - e0[1]};
    const int off1 = (n[0] + 31) / 32 * 32;   // where colour 1's sites start
    int b0 = 0x7fffffff, b1 = -1;           // the blocks of the CTA's sites
    for (int c = 0; c < 2; ++c) {
        if (n[c] == 0) continue;
        b0 = min(b0, (int)(k.list[c][e0[c]].y >> META_SHIFT));
        b1 = max(b1, (int)(k.list[c][e0[c] + n[c] - 1].y >> META_SHIFT));
    }
    for (int b = b0 + tid; b <= b1; b += kThreads) {
        float2 beta;
        if (sw.beta_pts) {
            beta.x = sw.beta_pts[(size_t)(rl % sw.n_pts) * sw.g.nblk + b];
            beta.y = sw.beta_pts[(size_t)((rl + 1) % sw.n_pts) * sw.g.nblk + b];
        } else {
            beta.x = sw.beta[b];
            beta.y = sw.beta_odd ? sw.beta_odd[b] : beta.x;
        }
        blocks[b - b0] = make_float4(beta.x, beta.y,
                                     __uint_as_float(slice_key1(sw.sl, slice_of(sw.sl, b))), 0.0f);
    }
    // The start. Each site's list index goes where its neighbours look it up.
    for (int c = 0; c < 2; ++c) {
        float2* own = reinterpret_cast<float2*>(static_cast<float*>(sw.ang) + pair_plane(sw.g, p, c));
        for (int i = tid; i < n[c]; i += kThreads) {
            const uint4 en = k.list[c][e0[c] + i];
            const int b = (int)(en.y >> META_SHIFT);
            float2 ph = both(k.init_angle[b]);
            if (k.random_init) {
                uint32_t w[4];
                philox4x32_10_rk(en.z, 0xFFFFu << 16, rpair, 0u, sw.rng.rk0,
                                 slice_key1(sw.sl, slice_of(sw.sl, b)), w);
                ph = make_float2(kTwoPi * u01(w[0]), kTwoPi * u01(w[2]));
            }
            float2 co, so;
            sincos_2(__fmul2_rn(both(m.q), ph), so, co);
            angles[c * off1 + i] = ph;
            cells[c * off1 + i] = make_float2(co.x, so.x);
            cells[odd + c * off1 + i] = make_float2(co.y, so.y);
            __stcg(own + en.x, make_float2(__int_as_float(e0[c] + i), 0.0f));
        }
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        atomicAdd(a.sync + 1, 1u);
        if (!poll(error, a.spin_limit, [&] { return load_acquire(a.sync + 1) >= a.arrivals; }))
            s_bad = 1;
    }
    __syncthreads();
    if (s_bad) return;
    // Site records: the four neighbours' cells, the Philox word, the meta word.
    for (int c = 0; c < 2; ++c) {
        const float2* oth = reinterpret_cast<const float2*>(static_cast<const float*>(sw.ang) +
                                                            pair_plane(sw.g, p, c ^ 1));
        for (int i = tid; i < n[c]; i += kThreads) {
            const uint4 en = k.list[c][e0[c] + i];
            const float2* word[4] = {oth + (ptrdiff_t)(int)en.w, oth + (ptrdiff_t)(int)en.w + 1,
                                     oth + en.x - (ptrdiff_t)sw.g.Wh, oth + en.x + sw.g.Wh};
            uint32_t ref[4], meta = en.y & (EDGE_L | EDGE_U);
            meta |= ((en.y >> META_SHIFT) - (uint32_t)b0) << kBlockShift;
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                if (en.y & (GAP_L << d)) {
                    const int e = __float_as_int(__ldcg(word[d]).x), i1 = e - e0[c ^ 1];
                    if (i1 >= 0 && i1 < n[c ^ 1]) {
                        ref[d] = (uint32_t)((c ^ 1) * off1 + i1);
                        continue;
                    }
                    int lo = 0, hi = a.ctas;      // the owner: part[lo] <= e < part[lo + 1]
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (s_part[c ^ 1][mid] <= e) lo = mid;
                        else hi = mid;
                    }
                    const int j = atomicAdd(&s_halo[c ^ 1], 1);
                    meta |= kExported;
                    ref[d] = (uint32_t)(a.sites + (c ^ 1) * a.halo + j);
                    if (j < a.halo)
                        sources[(c ^ 1) * a.halo + j] =
                            (uint32_t)((lo * 2 + (c ^ 1)) * a.cap + e - s_part[c ^ 1][lo]);
                    else
                        s_bad = 1;
                } else if (en.y & (NB_L << d)) {
                    float sj, cj;
                    __sincosf(m.q * __ldcg(word[d]).x, &sj, &cj);
                    const int j = atomicAdd(&s_consts, 1);
                    ref[d] = (uint32_t)(2 * at.cells + j);
                    if (j < a.consts) cells[2 * at.cells + j] = make_float2(cj, sj);
                    else s_bad = 1;
                } else {
                    ref[d] = (uint32_t)(2 * at.cells);
                }
            }
            if (meta & (EDGE_L | EDGE_U)) {
                const int two = (meta & EDGE_L) && (meta & EDGE_U);
                const int j = atomicAdd(&s_edges, 1 + two);
                if (j + two < a.edges) {
                    edges[j] = edges[j + two] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    meta |= (uint32_t)j << kEdgeShift;
                } else {
                    s_bad = 1;
                }
            }
            sites[c * off1 + i] = make_uint4(ref[0] | ref[1] << 16, ref[2] | ref[3] << 16, en.z, meta);
            if (c == 1 && (meta & kExported))       // what the first half-step reads
                send(exports + (size_t)(rank * 2 + c) * a.cap + i, angles[c * off1 + i], 1u);
        }
    }
    __syncthreads();
    if (s_bad) {                            // (never with the plan's capacities but for the halo)
        if (tid == 0) atomicExch(error, 2u);
        return;
    }

    // The cells of colour c owned elsewhere, as half-step h reads them.
    auto receive = [&](int c, uint32_t h) {
        bool ok = true;
        for (int j = tid; j < s_halo[c]; j += kThreads) {
            const float4* from = exports + sources[c * a.halo + j];
            float2 ph, co, so;
            ok = ok && poll(error, a.spin_limit, [&] { return look(from, ph) == h; });
            sincos_2(__fmul2_rn(both(m.q), ph), so, co);
            float2* to = cells + a.sites + c * a.halo + j;
            to[0] = make_float2(co.x, so.x);
            to[odd] = make_float2(co.y, so.y);
        }
        return ok;
    };

    // The next half-step's draws, proposals and their cosines and sines.
    float2 u1[kRounds], php[kRounds], cp[kRounds], sp[kRounds];
    auto propose = [&](int c, int s) {
#pragma unroll
        for (int r = 0; r < kRounds; ++r) {
            const int i = r * kThreads + tid;
            if (i < n[c]) {
                const uint2 zw = *reinterpret_cast<const uint2*>(&sites[c * off1 + i].z);
                const uint32_t key1 = __float_as_uint(blocks[(zw.y >> kBlockShift) & kBlockMask].z);
                uint32_t w[4];
                philox4x32_10_rk(zw.x, (uint32_t)s | (tag << 16), rpair, 0u, sw.rng.rk0, key1, w);
                u1[r] = u01_2(w[1], w[3]);
                php[r] = __fmul2_rn(both(kTwoPi), u01_2(w[0], w[2]));
                sincos_2(__fmul2_rn(both(m.q), php[r]), sp[r], cp[r]);
            }
        }
    };
    auto add = [&](int b, int r, double v) {
        if (r >= sw.R || v == 0.0) return;
        double* dst = k.points > 2 ? k.ebar_pts + (size_t)(r % k.points) * sw.g.nblk
                      : k.points == 2 && (r & 1) ? k.ebar_odd
                                                 : k.ebar;
        atomicAdd(&dst[b], v * k.inb[b]);
    };
    // Thread t sums the changes of warp group t / 4 (32 entries in a row): of
    // its first entry's block (even realization, odd one), then of its last's.
    double total0 = 0.0, total1 = 0.0;
    propose(0, 1);
    if (!__syncthreads_and(receive(1, 1u))) return;
#pragma unroll 1
    for (int h = 1; h <= 2 * k.n_sweeps; ++h) {
        const int c = (h - 1) & 1, s = (h + 1) >> 1;
        const float weight = (float)min(k.n_meas, k.n_sweeps - s + 1);
#pragma unroll
        for (int r = 0; r < kRounds; ++r) {
            const int i = r * kThreads + tid;
            if (i - lane >= n[c]) break;    // (a warp's entries)
            float2 ao = both(0.0f);
            uint32_t blk = 0;
            if (i < n[c]) {
                const uint4 st = sites[c * off1 + i];
                const uint32_t f = st.w & (EDGE_L | EDGE_U);
                blk = (st.w >> kBlockShift) & kBlockMask;
                const uint32_t ref[4] = {st.x & 0xffffu, st.x >> 16, st.y & 0xffffu, st.y >> 16};
                const float4 bl = blocks[blk];
                float2* cell = cells + c * off1 + i;
                float2* angle = angles + c * off1 + i;
                float2 ph = *angle;
                float2 al = both(0.0f), au = al;
                if constexpr (kOne) {
                    const float2 L = cells[ref[0]], Rt = cells[ref[1]], U = cells[ref[2]],
                                 D = cells[ref[3]], o = *cell;
                    const float C = (L.x + Rt.x) + (U.x + D.x), Sn = (L.y + Rt.y) + (U.y + D.y);
                    const SiteNew nw = site_move<float>(ph.x, o.x, o.y, php[r].x, cp[r].x, sp[r].x,
                                                        C, Sn, u1[r].x, bl.x, m);
                    if (f)
                        split_edge<float>(nw, ph.x, f, C, Sn, L.x, L.y, U.x, U.y, m, ao.x, al.x,
                                          au.x);
                    else
                        ao.x = nw.dE;
                    ph.x = nw.phi;
                    float sn, cs;
                    __sincosf(m.q * ph.x, &sn, &cs);
                    angle->x = ph.x;
                    *cell = make_float2(cs, sn);
                    if (st.w & kExported)
                        send(exports + (size_t)(rank * 2 + c) * a.cap + i, ph, (uint32_t)h + 1u);
                } else {
                    float2 v[8];
#pragma unroll
                    for (int d = 0; d < 4; ++d) {
                        const float2 x = cells[ref[d]];
                        const float2 y = cells[ref[d] + (ref[d] < (uint32_t)odd ? odd : 0)];
                        v[d] = make_float2(x.x, y.x);
                        v[4 + d] = make_float2(x.y, y.y);
                    }
                    const float2 o0 = cell[0], o1 = cell[odd];
                    const float2 C = sum4(v), Sn = sum4(v + 4);
                    float2 co = make_float2(o0.x, o1.x), so = make_float2(o0.y, o1.y);
                    const PairNew nw = pair_move<float>(ph, co, so, php[r], cp[r], sp[r], C, Sn,
                                                        u1[r], make_float2(bl.x, bl.y), m);
                    if (f)
                        split_edge_2<float>(nw, ph, f, C, Sn, v[0], v[4], v[2], v[6], m, ao, al, au);
                    else
                        ao = nw.dE;
                    ph = make_float2(run0 ? nw.phi.x : ph.x, run1 ? nw.phi.y : ph.y);
                    sincos_2(__fmul2_rn(both(m.q), ph), so, co);
                    *angle = ph;
                    cell[0] = make_float2(co.x, so.x);
                    cell[odd] = make_float2(co.y, so.y);
                    if (st.w & kExported)
                        send(exports + (size_t)(rank * 2 + c) * a.cap + i, ph, (uint32_t)h + 1u);
                }
                if (f) {
                    float4* rec = edges + (st.w >> kEdgeShift);
                    auto record = [&](float4* to, float2 x) {
                        const float4 v = *to;
                        Sum2 t{make_float2(v.x, v.y), make_float2(v.z, v.w)};
                        t.add(x, weight);
                        *to = make_float4(t.hi.x, t.hi.y, t.lo.x, t.lo.y);
                    };
                    if (f & EDGE_L) record(rec++, al);
                    if (f & EDGE_U) record(rec, au);
                }
            }
            // The warp's sums: usually one block's, else the first and the last
            // entry's blocks; blocks between them are added one by one.
            const int last_lane = min(31, n[c] - 1 - (i - lane));
            const uint32_t first = __shfl_sync(0xffffffffu, blk, 0);
            const uint32_t last = __shfl_sync(0xffffffffu, blk, last_lane);
            const bool in_first = blk == first || lane > last_lane;
            float4 out = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            float2 x = in_first ? ao : both(0.0f);
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) {
                x.x += __shfl_xor_sync(0xffffffffu, x.x, d);
                if constexpr (!kOne) x.y += __shfl_xor_sync(0xffffffffu, x.y, d);
            }
            out.x = x.x;
            out.y = x.y;
            if (first != last) {
                x = !in_first && blk == last ? ao : both(0.0f);
#pragma unroll
                for (int d = 16; d >= 1; d >>= 1) {
                    x.x += __shfl_xor_sync(0xffffffffu, x.x, d);
                    if constexpr (!kOne) x.y += __shfl_xor_sync(0xffffffffu, x.y, d);
                }
                out.z = x.x;
                out.w = x.y;
                if (!in_first && blk != last) {
                    add(b0 + (int)blk, rl, (double)weight * (double)ao.x);
                    add(b0 + (int)blk, rl + 1, (double)weight * (double)ao.y);
                }
            }
            if (lane == 0)
                reinterpret_cast<float4*>(sums)[c * (off1 / 32) + (i >> 5)] = out;
        }
        propose(c ^ 1, (h + 2) >> 1);
        if (!__syncthreads_and(h == 2 * k.n_sweeps || receive(c, (uint32_t)h + 1u))) return;
        if (tid < 4 * ((n[c] + 31) >> 5)) {
            const double v = (double)weight * (double)sums[c * (off1 / 8) + tid];
            if (c == 0) total0 += v;
            else total1 += v;
        }
    }
    for (int c = 0; c < 2; ++c) {
        if (tid < 4 * ((n[c] + 31) >> 5)) {
            const int at_e = (tid & 2) ? min((tid >> 2) * 32 + 31, n[c] - 1) : (tid >> 2) * 32;
            add((int)(k.list[c][e0[c] + at_e].y >> META_SHIFT), rl + (tid & 1), c ? total1 : total0);
        }
        float2* own = reinterpret_cast<float2*>(static_cast<float*>(sw.ang) + pair_plane(sw.g, p, c));
        for (int i = tid; i < n[c]; i += kThreads) {
            const uint4 en = k.list[c][e0[c] + i];
            own[en.x] = angles[c * off1 + i];
            if (!(en.y & (EDGE_L | EDGE_U))) continue;
            const float4* rec = edges + (sites[c * off1 + i].w >> kEdgeShift);
            const int b = (int)(en.y >> META_SHIFT);
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                if (!(en.y & (EDGE_L << d))) continue;
                const int to = d == 0 ? b - 1 : b - sw.g.nbx;
                add(to, rl, (double)rec->x + (double)rec->z);
                add(to, rl + 1, (double)rec->y + (double)rec->w);
                ++rec;
            }
        }
    }
    for (int b = rank * kThreads + tid; b < sw.g.nblk; b += a.ctas * kThreads)
        for (int r = rl; r < rl + 2; ++r) add(b, r, (double)k.n_meas * k.E0[(size_t)b * sw.Rp + r]);
}

// Each CTA's stretch of the two lists: colour 0 in equal shares, in whole warps
// of entries (the groups whose changes are summed in FP32), colour 1 up to the
// same place of the same block.
__device__ int2 part_start(const uint4* l0, const int32_t* start0, const int32_t* start1,
                           int64_t n0, int64_t n1, int i, int ctas) {
    if (i == 0) return make_int2(0, 0);
    if (i >= ctas) return make_int2((int)n0, (int)n1);
    const int64_t x0 = (n0 * i / ctas + 16) / 32 * 32;
    if (x0 >= n0) return make_int2((int)n0, (int)n1);
    const int b = (int)(l0[x0].y >> META_SHIFT);
    const int64_t num = x0 - start0[b], den = start0[b + 1] - start0[b];
    const int64_t x1 = (start1[b] + num * (start1[b + 1] - start1[b]) / den + 16) / 32 * 32;
    return make_int2((int)x0, (int)(x1 < n1 ? x1 : n1));
}

__global__ void __launch_bounds__(256) k_cal_resident_plan(
    const uint4* l0, const uint4* l1, const int32_t* start0, const int32_t* start1, int64_t n0,
    int64_t n1, int ctas, int* part, int* res) {
    __shared__ int s_n[2];
    const int i = blockIdx.x;
    const int2 from = part_start(l0, start0, start1, n0, n1, i, ctas);
    const int2 to = part_start(l0, start0, start1, n0, n1, i + 1, ctas);
    if (threadIdx.x < 2) s_n[threadIdx.x] = 0;
    __syncthreads();
    int consts = 0, edges = 0;
    for (int c = 0; c < 2; ++c) {
        const uint4* l = c ? l1 : l0;
        for (int e = (c ? from.y : from.x) + (int)threadIdx.x; e < (c ? to.y : to.x); e += 256) {
            const uint32_t f = l[e].y;
            consts += __popc(f & (NB_L * 15u)) - __popc(f & (GAP_L * 15u));
            edges += __popc(f & (EDGE_L | EDGE_U));
        }
    }
    atomicAdd(&s_n[0], consts);
    atomicAdd(&s_n[1], edges);
    __syncthreads();
    if (threadIdx.x != 0) return;
    int b0 = 0x7fffffff, b1 = -1;
    for (int c = 0; c < 2; ++c) {
        const int e = c ? from.y : from.x, e1 = c ? to.y : to.x;
        part[c * (ctas + 1) + i] = e;
        if (i + 1 == ctas) part[c * (ctas + 1) + ctas] = e1;
        if (e1 <= e) continue;
        const uint4* l = c ? l1 : l0;
        b0 = min(b0, (int)(l[e].y >> META_SHIFT));
        b1 = max(b1, (int)(l[e1 - 1].y >> META_SHIFT));
    }
    atomicMax(&res[0], max(to.x - from.x, to.y - from.y));
    atomicMax(&res[1], s_n[0]);
    atomicMax(&res[2], s_n[1]);
    atomicMax(&res[3], b1 - b0 + 1);
    atomicMax(&res[4], (to.x - from.x + 31) / 32 * 32 + (to.y - from.y + 31) / 32 * 32);
}

const void* kernel_of(bool one) {
    return one ? (const void*)k_cal_resident<true> : (const void*)k_cal_resident<false>;
}

}  // namespace

void launch_cal_resident_plan(const uint4* const list[2], const int32_t* const start[2],
                              const int64_t n[2], int ctas, int* part, int* res, cudaStream_t s) {
    cudaMemsetAsync(res, 0, sizeof(CalResidentPlan), s);
    k_cal_resident_plan<<<ctas, 256, 0, s>>>(list[0], list[1], start[0], start[1], n[0], n[1], ctas,
                                             part, res);
}

size_t cal_resident_smem_max(int device) {
    int optin = 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) !=
        cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    size_t most = (size_t)optin;
    for (int one = 0; one < 2; ++one) {
        cudaFuncAttributes fa{};
        if (cudaFuncGetAttributes(&fa, kernel_of(one)) != cudaSuccess ||
            fa.sharedSizeBytes >= (size_t)optin ||
            cudaFuncSetAttribute(kernel_of(one), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 optin - (int)fa.sharedSizeBytes) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        if ((size_t)optin - fa.sharedSizeBytes < most) most = (size_t)optin - fa.sharedSizeBytes;
    }
    return most;
}

size_t cal_resident_smem(const CalResidentArgs& a) { return Layout(a).bytes; }

cudaError_t launch_cal_resident(const CalResidentArgs& a, cudaStream_t s) {
    cudaLaunchAttribute attr[1] = {};
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((a.cal.sw.R + 1) / 2 * a.ctas));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Layout(a).bytes;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return a.cal.sw.R == 1 ? cudaLaunchKernelEx(&cfg, k_cal_resident<true>, a)
                           : cudaLaunchKernelEx(&cfg, k_cal_resident<false>, a);
}

}  // namespace mpr
