// mergepath.cuh -- cooperative merge walk for few pairs: one pair is split
// across a group of threads (a warp, a CTA, or a cluster of CTAs).
//
// When a call has too few 32 x 32 tiles to occupy every SM (small N), a pair
// is cut along its merge instead.  The walk of a pair is the merge of the two
// sorted lists of finite interval ends X = te_f[0..n_f-2] and
// Y = te_g[0..n_g-2] (f first on equal ends, the same order as the tile
// walk).  A thread finds where its share of the advances starts by a binary
// search along the cross diagonal (merge path, Green, McColl and Bader 2012),
// and walks it exactly like the tile walk.  A CTA takes the merge in slabs of S
// = 256 * kMpItems advances: it copies the next S + 2 elements of each PCF into
// shared memory (coalesced), and its threads share the slab, adding to the same
// accumulators slab after slab.  The threads' partial integrals are combined
// in float64 in a fixed order, so results do not depend on scheduling; they
// differ from one left-to-right sum only in rounding.
//
// What bounds it.  Few long pairs: latency.  A lane that walks its share
// straight from global memory waits for an L2 sector nearly every step (32
// lanes, each with two streams of 4 or 2 elements per sector): 880 cycles per
// step on 25 PCFs of 54,000 breakpoints, with one warp per pair.  Staging makes
// the waits shared and coalesced, and a CTA or a cluster per pair uses the whole
// GPU.  Many pairs: throughput.  The waits of 32 warps per SM overlap, and
// staging, one binary search per eight advances and barriers cost more than
// they save.  So there are two kernels (rule and measurements at
// launch_mergepath_t):
//   mergepath_kernel       a warp per pair, its 32 shares walked from global
//                          memory (float64 pairs of up to kMpShort advances
//                          from a copy in shared memory)
//   mergepath_cta_kernel   a 256-thread CTA per pair, or a cluster of 2, 4 or 8
//                          of them with a part of the pair each (the parts are
//                          summed through distributed shared memory, in part
//                          order), in staged slabs
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "walk.cuh"

namespace pcfgb {

// Pair index -> (row, column) of the pair queue, longest first.
__device__ __forceinline__ void decode_pair(const WalkArgs& a, int64_t t, int64_t& i, int64_t& j)
{
    if (a.symmetric) {
        const int64_t N = a.n_r;
        const int64_t m = upper_line(N, t);
        j = N - 1 - m;
        i = j - (t - (m * N - m * (m - 1) / 2));
    } else {
        const int64_t q = (((uint64_t)t | (uint64_t)a.n_c) >> 32) == 0
                              ? (int64_t)((uint32_t)t / (uint32_t)a.n_c) : t / a.n_c;
        i = a.n_r - 1 - q;
        j = a.n_c - 1 - (t - q * a.n_c);
    }
}

// End-time order of the two walk forms: values (float64 through the integer
// pipe) or order keys.
template <typename K> __device__ __forceinline__ bool key_after(K x, K y) { return ends_after(x, y); }
template <> __device__ __forceinline__ bool key_after<uint32_t>(uint32_t x, uint32_t y) { return x > y; }

constexpr int kMpThreads = 256;     // threads per CTA
constexpr int kMpItems = 8;         // advances per thread and slab, at most
constexpr int kMpShort = 256;       // advances of a pair that a warp copies first (float64)
// elements staged per PCF and slab: the one before the slab .. the one after it
constexpr int kMpSlabElems = kMpThreads * kMpItems + 2;
constexpr size_t mp_cta_smem(size_t elem) { return 2 * kMpSlabElems * elem; }
constexpr int kMpShortElems = kMpShort + 2;            // of both PCFs of a short pair
constexpr size_t mp_short_smem(size_t elem) { return (size_t)(kMpThreads / 32) * kMpShortElems * elem; }

// An element read from global memory (written before the launch, which is an
// ordinary one: the read-only path is open to it).
template <typename E> __device__ __forceinline__ E mp_load(const E* p) { return __ldg(p); }
template <> __device__ __forceinline__ KElem mp_load<KElem>(const KElem* p)
{
    const uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
    KElem e;
    e.k = u.x;
    e.hi = __uint_as_float(u.y);
    e.lo = __uint_as_float(u.z);
    e.v = __uint_as_float(u.w);
    return e;
}

// Tail rule, root and output of one pair, by one thread.
template <typename T, int COMBO, typename WF, typename E>
__device__ __forceinline__ void mp_store(const WalkArgs& a, int64_t gi, int64_t gj, const E* F, int nf,
                                         const E* G, int ng, const double* I)
{
    constexpr int NM = combo_n(COMBO);
    const T lfv = WF::val(F[nf - 1]), lgv = WF::val(G[ng - 1]);
    const int64_t i = a.perm_r[gi], j = a.perm_c[gj];
    auto store = [&](auto m_c) {
        constexpr int m = decltype(m_c)::value;
        constexpr int MI = combo_metric(COMBO, m);
        const int sgn = tail_sign<MI>(lfv, lgv);
        double Iv = I[m];
        if (sgn) Iv = sgn > 0 ? (double)INFINITY : -(double)INFINITY;
        const double Fv = finalize_root<MI>(a.root[m], a.p[m], Iv);
        void* out = a.out[m];
        auto put = [&](int64_t idx) {
            if (a.out_f64) reinterpret_cast<double*>(out)[idx] = Fv;
            else reinterpret_cast<float*>(out)[idx] = (float)Fv;
        };
        if (!a.symmetric) {
            put(i * a.ld_out + j);
        } else if (a.layout == PCF_OUT_FULL) {
            put(i * a.ld_out + j);
            if (gi != gj) put(j * a.ld_out + i);
        } else if (a.layout == kOutRowsInputColsSorted) {
            put(i * a.ld_out + gj);
            if (gi != gj) put(j * a.ld_out + gi);
        } else if (a.layout == PCF_OUT_FULL_SORTED) {
            put(gi * a.ld_out + gj);
            if (gi != gj) put(gj * a.ld_out + gi);
        } else {
            const int64_t N = a.ld_out;
            const int64_t lo2 = i < j ? i : j, hi2 = i < j ? j : i;
            put(lo2 * N - lo2 * (lo2 - 1) / 2 + (hi2 - lo2));
        }
    };
    store(std::integral_constant<int, 0>{});
    if constexpr (NM > 1) store(std::integral_constant<int, 1>{});
    if constexpr (NM > 2) store(std::integral_constant<int, 2>{});
}

// Advances [s0, s1) of the merge of F (lx finite ends) and G (ly), added to acc.
// load: an element of F or G; flushed every 16 terms (block-compensated sums).
template <typename T, int PREC, int COMBO, bool KEYED, typename E, typename Load>
__device__ __forceinline__ void mp_walk_share(Acc<PREC>* acc, const E* F, int64_t lx, const E* G,
                                              int64_t ly, int64_t s0, int64_t s1, T p0, Load load)
{
    using WF = WalkForm<T, KEYED>;
    constexpr int NM = combo_n(COMBO);
    auto flush = [&] {
#pragma unroll
        for (int m = 0; m < NM; ++m) acc[m].flush();
    };
    if (s1 <= s0) return;
    // x = advances of F among the first s0
    int64_t lo = s0 - ly > 0 ? s0 - ly : 0, hi = s0 < lx ? s0 : lx;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (!key_after(WF::key(load(F + mid)), WF::key(load(G + (s0 - 1 - mid))))) lo = mid + 1;
        else hi = mid;
    }
    const E* f = F + lo;
    const E* g = G + (s0 - lo);
    E ef = load(f), eg = load(g);
    const int cnt = (int)(s1 - s0);
    if constexpr (KEYED) {
        // start time: the later of the two interval ends passed so far
        float tc = 0.f, tcl = 0.f;
        uint32_t kc = 0;
        if (f > F) { const E e = load(f - 1); tc = e.hi; tcl = e.lo; kc = e.k; }
        if (g > G) {
            const E e = load(g - 1);
            if (e.k > kc) { tc = e.hi; tcl = e.lo; }
        }
        for (int q = 0; q < cnt; ++q) {
            if ((q & 15) == 0) flush();
            const bool adv_f = ef.k <= eg.k;
            const float hn = adv_f ? ef.hi : eg.hi, ln = adv_f ? ef.lo : eg.lo;
            const float dt = __fadd_rn(__fsub_rn(hn, tc), __fsub_rn(ln, tcl));
            tc = hn;
            tcl = ln;
            accumulate<COMBO, PREC, T>(acc, ef.v, eg.v, dt, p0);
            if (adv_f) ef = load(++f);
            else eg = load(++g);
        }
    } else {
        T tc = T(0);
        if (f > F) tc = load(f - 1).x;
        if (g > G) { const T e = load(g - 1).x; tc = ends_after(e, tc) ? e : tc; }
        for (int q = 0; q < cnt; ++q) {
            if ((q & 15) == 0) flush();
            const bool adv_f = !ends_after(ef.x, eg.x);
            const T tn = adv_f ? ef.x : eg.x;
            const T dt = tn - tc;
            tc = tn;
            accumulate<COMBO, PREC, T>(acc, ef.y, eg.y, dt, p0);
            if (adv_f) ef = load(++f);
            else eg = load(++g);
        }
    }
    flush();
}

// A warp per pair.  COPY: pairs of up to kMpShort advances are copied into the
// warp's shared memory first.
template <typename T, int PREC, int COMBO, bool KEYED, bool COPY>
__global__ void __launch_bounds__(kMpThreads, COPY ? 3 : 4) mergepath_kernel(const WalkArgs a,
                                                                             int64_t npairs)
{
    using WF = WalkForm<T, KEYED>;
    using E = typename WF::E;
    constexpr int NM = combo_n(COMBO);
    if (gated_off(a.gate, a.gate_want64)) return;   // the other walk of an AUTO64 call
    if (steps_gated_off(a)) return;                 // another kernel of the call walks
    if (a.hdr->err != kNoError) return;             // recorded before this launch: every CTA agrees
    extern __shared__ __align__(16) unsigned char mp_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const T p0 = (T)a.p[0];
    const E* R = reinterpret_cast<const E*>(a.pack_r);
    const E* C = reinterpret_cast<const E*>(a.pack_c);
    const int64_t ustep = (int64_t)gridDim.x * (kMpThreads / 32);

    for (int64_t u = (int64_t)blockIdx.x * (kMpThreads / 32) + warp;; u += ustep) {
        const int64_t t = a.shard_index + u * a.shard_count;
        if (t >= npairs) break;
        int64_t gi, gj;
        decode_pair(a, t, gi, gj);
        const E* F = R + a.poff_r[gi];
        const E* G = C + a.poff_c[gj];
        const int nf = a.slen_r[gi], ng = a.slen_c[gj];
        const int64_t lx = nf - 1, ly = ng - 1, total = lx + ly;
        Acc<PREC> acc[NM];
        bool walked = false;
        if constexpr (COPY) {
            if (total <= kMpShort) {
                E* const sF = reinterpret_cast<E*>(mp_smem) + warp * kMpShortElems;
                E* const sG = sF + nf;
                for (int q = lane; q < nf; q += 32) sF[q] = F[q];
                for (int q = lane; q < ng; q += 32) sG[q] = G[q];
                __syncwarp();
                const int cnt = (int)total, items = (cnt + 31) / 32;
                const int s0 = lane * items < cnt ? lane * items : cnt;
                const int s1 = s0 + items < cnt ? s0 + items : cnt;
                mp_walk_share<T, PREC, COMBO, KEYED>(acc, (const E*)sF, lx, (const E*)sG, ly, s0, s1, p0,
                                                     [](const E* p) { return *p; });
                __syncwarp();
                walked = true;
            }
        }
        if (!walked)
            mp_walk_share<T, PREC, COMBO, KEYED>(acc, F, lx, G, ly, total * lane / 32,
                                                 total * (lane + 1) / 32, p0,
                                                 [](const E* p) { return mp_load(p); });
        // fixed-order float64 combine of the lanes
        double I[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            double v = acc[m].value();
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            I[m] = v;
        }
        if (lane == 0) mp_store<T, COMBO, WF>(a, gi, gj, F, nf, G, ng, I);
    }
}

// A CTA per pair, or a cluster of `parts` of them.
template <typename T, int PREC, int COMBO, bool KEYED>
__global__ void __launch_bounds__(kMpThreads) mergepath_cta_kernel(const WalkArgs a, int64_t npairs,
                                                                   int parts)
{
    using WF = WalkForm<T, KEYED>;
    using E = typename WF::E;
    constexpr int NM = combo_n(COMBO);
    constexpr int S = kMpThreads * kMpItems;
    if (gated_off(a.gate, a.gate_want64)) return;   // the other walk of an AUTO64 call
    if (steps_gated_off(a)) return;                 // another kernel of the call walks
    if (a.hdr->err != kNoError) return;             // recorded before this launch: every CTA agrees
    extern __shared__ __align__(16) unsigned char mp_smem[];
    __shared__ int s_split[2];
    __shared__ double s_part[NM][kMpThreads / 32];
    __shared__ double s_sum[NM];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    E* const sF = reinterpret_cast<E*>(mp_smem);
    E* const sG = sF + kMpSlabElems;
    const E* const f = sF + 1;                              // f[x]: element kf + x
    const E* const g = sG + 1;
    const T p0 = (T)a.p[0];
    const E* R = reinterpret_cast<const E*>(a.pack_r);
    const E* C = reinterpret_cast<const E*>(a.pack_c);
    const int part = (int)(blockIdx.x % (unsigned)parts);
    const int64_t ustep = gridDim.x / (unsigned)parts;

    for (int64_t u = blockIdx.x / (unsigned)parts;; u += ustep) {
        const int64_t t = a.shard_index + u * a.shard_count;
        if (t >= npairs) break;
        int64_t gi, gj;
        decode_pair(a, t, gi, gj);
        const E* F = R + a.poff_r[gi];
        const E* G = C + a.poff_c[gj];
        const int nf = a.slen_r[gi], ng = a.slen_c[gj];
        const int lx = nf - 1, ly = ng - 1;
        const int64_t total = (int64_t)lx + ly;
        // this part's advances [s, s_end), after kf advances of f and kg of g
        int64_t s = total * part / parts;
        const int64_t s_end = total * (part + 1) / parts;
        int kf = 0, kg = 0;
        if (s > 0) {
            int64_t lo = s - ly > 0 ? s - ly : 0, hi = s < lx ? s : lx;
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (!key_after(WF::key(F[mid]), WF::key(G[s - 1 - mid]))) lo = mid + 1; else hi = mid;
            }
            kf = (int)lo;
            kg = (int)(s - lo);
        }

        Acc<PREC> acc[NM];
        while (s < s_end) {
            const int cnt = s_end - s < S ? (int)(s_end - s) : S;
            // elements kf - 1 .. kf + cnt of f and kg - 1 .. kg + cnt of g, where they exist
            for (int q = tid; q < cnt + 2; q += kMpThreads) {
                const int64_t fi = (int64_t)kf - 1 + q, gq = (int64_t)kg - 1 + q;
                if (fi >= 0 && fi < nf) sF[q] = F[fi];
                if (gq >= 0 && gq < ng) sG[q] = G[gq];
            }
            __syncthreads();
            const int items = (cnt + kMpThreads - 1) / kMpThreads;    // advances per thread, <= kMpItems
            const int i0 = tid * items < cnt ? tid * items : cnt;
            const int i1 = i0 + items < cnt ? i0 + items : cnt;
            const int last = (cnt - 1) / items;             // thread of the slab's last advance
            int x = 0, y = 0;
            if (i1 > i0) {
                // x = advances of f among the slab's first i0
                const int rf = lx - kf, rg = ly - kg;
                int lo = i0 - rg > 0 ? i0 - rg : 0, hi = i0 < rf ? i0 : rf;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (!key_after(WF::key(f[mid]), WF::key(g[i0 - 1 - mid]))) lo = mid + 1; else hi = mid;
                }
                x = lo;
                y = i0 - lo;
                E ef = f[x], eg = g[y];
                if constexpr (KEYED) {
                    // start time: the later of the two interval ends passed so far
                    float tc = 0.f, tcl = 0.f;
                    uint32_t kc = 0;
                    if (kf + x > 0) { const E e = f[x - 1]; tc = e.hi; tcl = e.lo; kc = e.k; }
                    if (kg + y > 0) {
                        const E e = g[y - 1];
                        if (e.k > kc) { tc = e.hi; tcl = e.lo; }
                    }
                    for (int q = i0; q < i1; ++q) {
                        const bool adv_f = ef.k <= eg.k;
                        const float hn = adv_f ? ef.hi : eg.hi, ln = adv_f ? ef.lo : eg.lo;
                        const float dt = __fadd_rn(__fsub_rn(hn, tc), __fsub_rn(ln, tcl));
                        tc = hn;
                        tcl = ln;
                        accumulate<COMBO, PREC, T>(acc, ef.v, eg.v, dt, p0);
                        if (adv_f) ef = f[++x];
                        else eg = g[++y];
                    }
                } else {
                    T tc = T(0);
                    if (kf + x > 0) tc = f[x - 1].x;
                    if (kg + y > 0) { const T e = g[y - 1].x; tc = ends_after(e, tc) ? e : tc; }
                    for (int q = i0; q < i1; ++q) {
                        const bool adv_f = !ends_after(ef.x, eg.x);
                        const T tn = adv_f ? ef.x : eg.x;
                        const T dt = tn - tc;
                        tc = tn;
                        accumulate<COMBO, PREC, T>(acc, ef.y, eg.y, dt, p0);
                        if (adv_f) ef = f[++x];
                        else eg = g[++y];
                    }
                }
                // compensated blocks: at most kMpItems (<= 16) terms
#pragma unroll
                for (int m = 0; m < NM; ++m) acc[m].flush();
            }
            // the thread with the slab's last advance has the next slab's start
            if (tid == last) { s_split[0] = x; s_split[1] = y; }
            __syncthreads();
            x = s_split[0];
            y = s_split[1];
            kf += x;
            kg += y;
            s += cnt;
        }
        // fixed-order float64 combine: lanes, then warps, then the cluster's parts
        double I[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            double v = acc[m].value();
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            I[m] = v;
        }
        if (lane == 0) {
#pragma unroll
            for (int m = 0; m < NM; ++m) s_part[m][warp] = I[m];
        }
        __syncthreads();
        if (tid == 0) {
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                I[m] = s_part[m][0];
                for (int w = 1; w < kMpThreads / 32; ++w) I[m] += s_part[m][w];
                s_sum[m] = I[m];
            }
        }
        if (parts > 1) {
            auto cluster = cooperative_groups::this_cluster();
            cluster.sync();
            if (part == 0 && tid == 0) {
#pragma unroll
                for (int m = 0; m < NM; ++m)
                    for (int r = 1; r < parts; ++r) I[m] += *cluster.map_shared_rank(&s_sum[m], r);
            }
            cluster.sync();     // s_sum and s_part may be written again
        } else {
            __syncthreads();
        }
        if (tid == 0 && part == 0) mp_store<T, COMBO, WF>(a, gi, gj, F, nf, G, ng, I);
    }
}

// Which of the two kernels walks the pairs: whole CTAs when the call's longest
// pair would take a warp longer than all pairs take the CTAs, that is when its
// advances exceed pairs * (kMpCtaPair + mean / kMpCtaSteps).  A warp takes 6 to 12
// ns per advance of the longest pair (less when the elements are in L2 already)
// and 2.1 ps per advance in all; CTAs 6 ns per pair (15 with three metrics) and 4
// ps per advance.  Measured (us, warp / CTA, walk alone): 25 even float32 curves
// of 1,350 points 23 / 13, 60 of 5,400 70 / 80, 160 of 1,350 83 / 134 (three
// metrics 99 / 234), 350 of 1,350 318 / 658; two of 50,000 points among 100 of 50
// 541 / 136; ten of 20,000 among 160 of 10 226 / 156; float64 25 of 1,350 31 / 19,
// 160 of 1,350 218 / 332.  The longest pair is known on the device only: when its
// bounds (the mean, and all breakpoints but one per PCF) do not decide, both
// kernels are launched and the header's lengths say which of them walks.  Below
// kMpLongSteps on average it is not worth a second launch.  (npairs: of all
// shards, so that every rank of a split takes the same kernel.)
constexpr int64_t kMpLongSteps = 1024;
constexpr int64_t kMpCtaSteps = 1500;
constexpr double kMpCtaPair = 0.9, kMpCtaPair3 = 2.2;   // (2.2: float32, three metrics)

// A float64 warp copies its pairs to shared memory up to this many advances on
// average (100 / 299 curves of 55 points with one metric 19 / 76 us, from global
// memory 19 / 85; with three 31 / 183, 38 / 226; of 275 points with one 40 / 208,
// 33 / 181).  In float32 it does not pay at any length.
constexpr int64_t kMpCopySteps = 256;

// The walk of `npairs` pairs (args.mean_steps, max_steps: their lengths as far as
// the host knows them), if the longest is in (args.steps_lo, args.steps_hi].
template <typename T, int PREC, bool KEYED = false>
cudaError_t launch_mergepath_t(int combo, const WalkArgs& args, int64_t npairs, cudaStream_t s)
{
    using E = typename WalkForm<T, KEYED>::E;
    const int64_t sms = device_sm_count();
    const int64_t mine = (npairs - args.shard_index + args.shard_count - 1) / args.shard_count;
    if (mine < 1) return cudaSuccess;
    WalkArgs a = args;
    const int64_t mean = a.mean_steps;
    const double cta_from = (double)npairs * ((sizeof(T) == 4 && a.nout > 1 ? kMpCtaPair3 : kMpCtaPair) +
                                              (double)mean / (double)kMpCtaSteps);
    bool warps = true, ctas = false;
    if (mean > kMpLongSteps) {
        warps = (double)mean <= cta_from;
        ctas = (double)a.max_steps > cta_from;
        if (!warps && !ctas) ctas = true;
    }
    const int64_t limit = cta_from < 9e18 ? (int64_t)cta_from : INT64_MAX;
    // (not launched by launch_next: clusters placed before the pack has left
    // its SMs end up unevenly spread, 25 long curves 216 -> 231 us per call)
    auto go = [&](auto kern, int64_t grid, int parts, size_t smem, auto... tail) -> cudaError_t {
        if (smem > 48 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(
                kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3(kMpThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)parts;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = parts > 1 ? 1 : 0;
        return cudaLaunchKernelEx(&cfg, kern, a, npairs, tail...);
    };
    auto pick = [&](auto combo_c) -> cudaError_t {
        constexpr int CB = decltype(combo_c)::value;
        const int64_t lo = args.steps_lo, hi = args.steps_hi;
        if (warps) {
            // with both kernels in play the warps take (lo, limit]
            a.steps_lo = lo;
            a.steps_hi = ctas && limit < hi ? limit : hi;
            if (a.steps_lo < a.steps_hi) {
                // (a launch that may have to return at once: no more CTAs than run together)
                int64_t grid = (mine + kMpThreads / 32 - 1) / (kMpThreads / 32);
                const int64_t most = sms * (a.steps_lo > 0 || a.steps_hi < kAnySteps ? 4 : 16);
                if (grid > most) grid = most;
                cudaError_t e = cudaSuccess;
                if constexpr (sizeof(T) == 8) {
                    e = mean <= kMpCopySteps
                            ? go(mergepath_kernel<T, PREC, CB, KEYED, true>, grid, 1, mp_short_smem(sizeof(E)))
                            : go(mergepath_kernel<T, PREC, CB, KEYED, false>, grid, 1, 0);
                } else {
                    e = go(mergepath_kernel<T, PREC, CB, KEYED, false>, grid, 1, 0);
                }
                if (e != cudaSuccess) return e;
            }
        }
        if (!ctas) return cudaSuccess;
        a.steps_lo = warps && limit > lo ? limit : lo;
        a.steps_hi = hi;
        if (a.steps_lo >= a.steps_hi) return cudaSuccess;
        // parts: enough CTAs for six per SM, each with two slabs or more (by the
        // pairs of all shards, so that a shard's results have the whole call's bits)
        int parts = 1;
        while (parts < 8 && npairs * parts < 6 * sms &&
               mean >= 2 * parts * 2 * (int64_t)kMpThreads * kMpItems)
            parts *= 2;
        const int64_t grid = mine < sms * 64 ? mine : sms * 64;
        return go(mergepath_cta_kernel<T, PREC, CB, KEYED>, grid * parts, parts, mp_cta_smem(sizeof(E)),
                  parts);
    };
    switch (combo) {
    case kComboL1: return pick(std::integral_constant<int, kComboL1>{});
    case kComboL2: return pick(std::integral_constant<int, kComboL2>{});
    case kComboGram: return pick(std::integral_constant<int, kComboGram>{});
    case kComboLP: return pick(std::integral_constant<int, kComboLP>{});
    case kComboL3: return pick(std::integral_constant<int, kComboL3>{});
    case kComboL1L2Gram: return pick(std::integral_constant<int, kComboL1L2Gram>{});
    case kComboL1L2L3: return pick(std::integral_constant<int, kComboL1L2L3>{});
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace pcfgb
