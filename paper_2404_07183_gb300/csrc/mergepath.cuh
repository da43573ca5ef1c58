// mergepath.cuh -- cooperative merge walk for few pairs: one pair is split
// across a group of threads (a warp, a CTA, or a cluster of CTAs).
//
// When a call has too few 32 x 32 tiles to occupy every SM (small N), a pair
// is cut along its merge instead.  The walk of a pair is the merge of the two
// sorted lists of finite interval ends X = te_f[0..n_f-2] and
// Y = te_g[0..n_g-2] (f first on equal ends, the same order as the tile
// walk).  The group takes it in slabs of S = GROUP * kMpItems advances: it
// copies the next S + 2 elements of each PCF into shared memory (coalesced),
// every thread finds where its share of the advances starts by a binary search
// along the cross diagonal in shared memory (merge path, Green, McColl and
// Bader 2012), and walks them exactly like the tile walk, adding to the same
// accumulators slab after slab.  The threads' partial integrals are combined
// in float64 in a fixed order, so results do not depend on scheduling; they
// differ from one left-to-right sum only in rounding.
//
// What bounds it: latency.  A lane that walks its share straight from global
// memory waits for an L2 sector nearly every step (32 lanes, each with two
// streams of 4 or 2 elements per sector): 880 cycles per step on 25 PCFs of
// 54,000 breakpoints, with one warp per pair.  Staging makes the waits shared
// and coalesced, and the group is as large as the pair's length allows:
//   GROUP 32   pairs of up to kMpLongSteps advances, eight pairs per CTA
//   GROUP 256  longer ones, one pair per CTA or per cluster of 2, 4 or 8
//              CTAs, each with its part of the pair, when the pairs alone
//              would leave the GPU idle (the parts are summed through
//              distributed shared memory, in part order)
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
// elements staged per PCF and slab: the one before the slab .. the one after it
template <int GROUP> __host__ __device__ constexpr int mp_slab_elems() { return GROUP * kMpItems + 2; }
template <int GROUP> __host__ __device__ constexpr size_t mp_smem_bytes(size_t elem)
{
    return (size_t)(kMpThreads / GROUP) * 2 * mp_slab_elems<GROUP>() * elem;
}

// parts: CTAs per pair (the cluster size; 1 for GROUP 32).
template <typename T, int PREC, int COMBO, bool KEYED, int GROUP>
__global__ void __launch_bounds__(kMpThreads) mergepath_kernel(const WalkArgs a, int64_t npairs,
                                                               int parts)
{
    using WF = WalkForm<T, KEYED>;
    using E = typename WF::E;
    constexpr int NM = combo_n(COMBO);
    constexpr int S = GROUP * kMpItems, SE = mp_slab_elems<GROUP>();
    constexpr bool kWarp = GROUP == 32;
    constexpr int kGroups = kMpThreads / GROUP;             // pairs a CTA walks at a time
    if (gated_off(a.gate, a.gate_want64)) return;   // the other walk of an AUTO64 call
    if (a.hdr->err != kNoError) return;             // recorded before this launch: every CTA agrees
    extern __shared__ __align__(16) unsigned char mp_smem[];
    __shared__ int s_split[2];
    __shared__ double s_part[NM][kMpThreads / 32];
    __shared__ double s_sum[NM];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tid = threadIdx.x & (GROUP - 1);              // thread of the group
    E* const sF = reinterpret_cast<E*>(mp_smem) + (size_t)(threadIdx.x / GROUP) * 2 * SE;
    E* const sG = sF + SE;
    const E* const f = sF + 1;                              // f[x]: element kf + x
    const E* const g = sG + 1;
    auto group_sync = [] { if constexpr (kWarp) __syncwarp(); else __syncthreads(); };
    const T p0 = (T)a.p[0];
    const E* R = reinterpret_cast<const E*>(a.pack_r);
    const E* C = reinterpret_cast<const E*>(a.pack_c);
    const int part = (int)(blockIdx.x % (unsigned)parts);
    const int64_t u0 = (int64_t)(blockIdx.x / (unsigned)parts) * kGroups + threadIdx.x / GROUP;
    const int64_t ustep = (int64_t)(gridDim.x / (unsigned)parts) * kGroups;

    for (int64_t u = u0;; u += ustep) {
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
            for (int q = tid; q < cnt + 2; q += GROUP) {
                const int64_t fi = (int64_t)kf - 1 + q, gq = (int64_t)kg - 1 + q;
                if (fi >= 0 && fi < nf) sF[q] = F[fi];
                if (gq >= 0 && gq < ng) sG[q] = G[gq];
            }
            group_sync();
            const int items = (cnt + GROUP - 1) / GROUP;    // advances per thread, <= kMpItems
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
            if constexpr (kWarp) {
                x = __shfl_sync(0xffffffffu, x, last);
                y = __shfl_sync(0xffffffffu, y, last);
                __syncwarp();
            } else {
                if (tid == last) { s_split[0] = x; s_split[1] = y; }
                __syncthreads();
                x = s_split[0];
                y = s_split[1];
            }
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
        if constexpr (!kWarp) {
            if (lane == 0) {
#pragma unroll
                for (int m = 0; m < NM; ++m) s_part[m][warp] = I[m];
            }
            __syncthreads();
            if (threadIdx.x == 0) {
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
                if (part == 0 && threadIdx.x == 0) {
#pragma unroll
                    for (int m = 0; m < NM; ++m)
                        for (int r = 1; r < parts; ++r) I[m] += *cluster.map_shared_rank(&s_sum[m], r);
                }
                cluster.sync();     // s_sum and s_part may be written again
            } else {
                __syncthreads();
            }
        }
        if (tid == 0 && part == 0) {
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
    }
}

// Pairs whose two PCFs hold more than this many breakpoints on average are
// walked by whole CTAs.  (Host rule: the call knows the mean lengths only.)
constexpr int64_t kMpLongSteps = 1024;

template <typename T, int PREC, bool KEYED = false>
cudaError_t launch_mergepath_t(int combo, const WalkArgs& a, int64_t npairs, int64_t mean_steps,
                               cudaStream_t s)
{
    using E = typename WalkForm<T, KEYED>::E;
    const int64_t sms = device_sm_count();
    const int64_t mine = (npairs - a.shard_index + a.shard_count - 1) / a.shard_count;
    if (mine < 1) return cudaSuccess;
    // (not launched by launch_next: clusters placed before the pack has left
    // its SMs end up unevenly spread, 25 long curves 216 -> 231 us per call)
    auto go = [&](auto kern, int64_t grid, int parts, size_t smem) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
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
        return cudaLaunchKernelEx(&cfg, kern, a, npairs, parts);
    };
    auto pick = [&](auto combo_c) -> cudaError_t {
        constexpr int CB = decltype(combo_c)::value;
        if (mean_steps <= kMpLongSteps) {
            int64_t grid = (mine + kMpThreads / 32 - 1) / (kMpThreads / 32);
            if (grid > sms * 16) grid = sms * 16;
            return go(mergepath_kernel<T, PREC, CB, KEYED, 32>, grid, 1, mp_smem_bytes<32>(sizeof(E)));
        }
        // parts: enough CTAs for six per SM, each with two slabs or more
        int parts = 1;
        while (parts < 8 && mine * parts < 6 * sms &&
               mean_steps >= 2 * parts * 2 * (int64_t)kMpThreads * kMpItems)
            parts *= 2;
        int64_t grid = mine < sms * 64 ? mine : sms * 64;
        return go(mergepath_kernel<T, PREC, CB, KEYED, kMpThreads>, grid * parts, parts,
                  mp_smem_bytes<kMpThreads>(sizeof(E)));
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
