// keys.cu -- exact order keys of float64 interval ends for the float32 walks.
//
// A float32 walk over float64 input must still decide every comparison of
// Alg. 1 (which interval ends first, and ties) on the float64 times.  Rounding
// the times to float32 would merge distinct breakpoints closer than one
// float32 ulp and reorder others.  Instead every finite interval end te of
// the call's collections gets a 32-bit rank: twice the number of distinct
// end times below it, plus 2, so that equal times get equal ranks and the
// order of the ranks is the order of the times; the last interval of a PCF
// (te = +inf) has rank 0xFFFFFFFF.  A query time q that is not an interval
// end (an integration bound) gets 2 * (distinct ends below q) + 1, which
// orders it exactly against every end.  The walk then compares ranks with
// one unsigned compare, and forms interval widths from a float32 hi/lo split
// of each time (packed next to the rank).
//
// The ranks come from a device-wide stable LSD radix sort of the (time bits,
// packed position) pairs: non-negative float64 values order like their bit
// patterns read as unsigned 64-bit integers.  One kernel counts all eight
// 8-bit digits (they do not depend on the order) and plans the passes: a digit
// that all keys share needs none.  Each pass is one kernel: a CTA takes a tile
// of 8,192 keys by ticket, ranks them stably (warp ballots, per-warp digit
// counts), learns how many of each digit the tiles before it hold by decoupled
// look-back (thread d waits for digit d; tickets make every predecessor a
// running or finished CTA, and every wait is bounded), orders the tile in
// shared memory and writes it in runs of one digit.  A last kernel counts
// distinct keys the same way and writes every key's rank into the packed
// element its payload names.
//
// A wait that gives up records kErrWait and leaves its tile unwritten.  From
// then on no kernel may trust the buffers (a pass would scatter stale keys by
// digit counts that are not theirs, the rank kernel would store through stale
// payloads): every CTA of the passes, of the rank kernel and of the bounds
// reads the recorded error first and returns.
//
// What bounds it: few keys, the latency of ten launches in a row; many, the
// 24 bytes per key and pass.  A histogram, two scans and an unordered scatter
// per pass (35 launches) came before: three matrices of 701 stable-rank curves
// (193,000 keys) took 0.78 ms per call and 0.47 with this sort, of 20,000 (5.5
// million) 117.0 and 116.2.
//
// The number of keys is known on the device only (it depends on the lengths
// of the rows a call packs); the kernels read it from the header and are
// launched for the workspace's capacity.
#include "internal.cuh"

namespace pcfgb {

constexpr int kSortThreads2 = 512;
constexpr int kSortWarps = kSortThreads2 / 32;
constexpr int kSortItems = 16;
constexpr int kSortTile = kSortThreads2 * kSortItems;   // keys per tile (8,192)

// KeySort::misc (32-bit words): the digit counts (then their exclusive scans)
// of the eight passes, the pass plan, the sorted buffer, the tickets of the
// passes and of the rank kernel, the finished counter of the histogram.
constexpr int kMiscPlan = 8 * 256;         // [8]: buffer the pass reads, or 2 = no pass
constexpr int kMiscFinal = kMiscPlan + 8;  // buffer that holds the sorted keys
constexpr int kMiscTicket = kMiscFinal + 1;    // [9]
constexpr int kMiscDone = kMiscTicket + 9;
constexpr int kMiscWords = 8 * 256 + 64;
static_assert(kMiscDone < kMiscWords, "misc layout");

int64_t key_tiles(int64_t cap) { return cap > 0 ? (cap + kSortTile - 1) / kSortTile : 1; }

size_t keysort_bytes(int64_t cap)
{
    const int64_t tiles = key_tiles(cap);
    size_t b = 0;
    b += 2 * align_up(sizeof(uint64_t) * (size_t)(cap > 0 ? cap : 1));
    b += 2 * align_up(sizeof(uint32_t) * (size_t)(cap > 0 ? cap : 1));
    b += align_up(sizeof(uint32_t) * 256 * (size_t)tiles);
    b += align_up(sizeof(uint32_t) * (size_t)(tiles + 1));
    b += align_up(sizeof(uint32_t) * kMiscWords);
    return b;
}

KeySort carve_keysort(char*& cur, int64_t cap)
{
    KeySort k;
    const int64_t c = cap > 0 ? cap : 1;
    k.cap = cap;
    k.tiles = key_tiles(cap);
    auto take = [&](size_t bytes) { char* p = cur; cur += align_up(bytes); return p; };
    k.key[0] = reinterpret_cast<uint64_t*>(take(sizeof(uint64_t) * (size_t)c));
    k.key[1] = reinterpret_cast<uint64_t*>(take(sizeof(uint64_t) * (size_t)c));
    k.pay[0] = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * (size_t)c));
    k.pay[1] = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * (size_t)c));
    k.status = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * 256 * (size_t)k.tiles));
    k.tsum = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * (size_t)(k.tiles + 1)));
    k.misc = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * kMiscWords));
    return k;
}

// Number of keys of a call: sum over its collections of (breakpoints - PCFs),
// from the packed offsets poff[n] of each set.  Clears the sort's counters.
__global__ void __launch_bounds__(256) count_keys_kernel(Header* hdr, const int64_t* poff0, int64_t n0,
                                                         const int64_t* poff1, int64_t n1,
                                                         uint32_t* misc)
{
    chain_start();
    for (int i = threadIdx.x; i < kMiscWords; i += 256) misc[i] = 0;
    if (threadIdx.x != 0) return;
    // no keys after an input error, or when an AUTO64 call walks in float64
    if (hdr->err != kNoError || hdr->need64 != 0u) { hdr->nkeys = 0; return; }
    unsigned long long m = 0;
    if (poff0) m += (unsigned long long)(poff0[n0] - n0);
    if (poff1) m += (unsigned long long)(poff1[n1] - n1);
    hdr->nkeys = m;
}

// Chunk states of a decoupled look-back, 32 bits: a tile's own count, then its
// inclusive prefix.  Narrow form (fewer than 2^27 keys): the pass number marks
// the state, so that one array serves all passes without being cleared; wide
// form: 0 = nothing yet, the array is cleared before each pass.
struct TileState {
    uint32_t epoch;
    int wide;
    __device__ __forceinline__ uint32_t own(uint32_t c) const
    {
        return wide ? c + 1u : (epoch << 28) | c;
    }
    __device__ __forceinline__ uint32_t incl(uint32_t c) const
    {
        return wide ? 0x80000000u | c : (epoch << 28) | 0x08000000u | c;
    }
    __device__ __forceinline__ bool empty(uint32_t w) const { return wide ? w == 0u : (w >> 28) != epoch; }
    __device__ __forceinline__ bool is_incl(uint32_t w) const
    {
        return wide ? (w >> 31) != 0u : (w & 0x08000000u) != 0u;
    }
    __device__ __forceinline__ uint32_t value(uint32_t w) const
    {
        return wide ? ((w >> 31) ? w & 0x7fffffffu : w - 1u) : w & 0x07ffffffu;
    }
};
constexpr int64_t kNarrowKeys = 1ll << 27;

// Polls before a look-back wait gives up (64 ns sleeps: 0.27 s and more).
constexpr int kSortPolls = 1 << 22;

// A CTA's tile of a pass (one thread): the next ticket, or -1 (stop) when an
// error is recorded.
__device__ __forceinline__ int64_t take_tile(uint32_t* ticket, const Header* hdr)
{
    const unsigned long long err = __ldcg(&hdr->err);
    const int64_t t = (int64_t)atomicAdd(ticket, 1u);
    return err == kNoError ? t : -1;
}

// Sum of the counts of the tiles before `tile` (stride words apart), by one
// thread.  False when a wait gave up (after max_polls polls, or because
// another one has).
__device__ __forceinline__ bool tile_prefix(const uint32_t* st, int64_t tile, int stride,
                                            const TileState& ts, const Header* hdr, int max_polls,
                                            uint32_t& prefix)
{
    constexpr int kAhead = 8;               // states read at a time: one L2 latency for eight
    uint32_t sum = 0;
    for (int64_t t0 = tile - 1; t0 >= 0; t0 -= kAhead) {
        uint32_t w[kAhead];
#pragma unroll
        for (int q = 0; q < kAhead; ++q) w[q] = t0 - q >= 0 ? __ldcg(st + (t0 - q) * stride) : 0u;
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            const int64_t t = t0 - q;
            if (t < 0) break;                // (tile 0 publishes an inclusive prefix at once)
            for (int polls = 0; ts.empty(w[q]); ++polls) {
                if (polls > max_polls || ((polls & 1023) == 1023 && __ldcg(&hdr->err) != kNoError))
                    return false;
                if (polls > 8) __nanosleep(64);
                w[q] = __ldcg(st + t * stride);
            }
            sum += ts.value(w[q]);
            if (ts.is_incl(w[q])) { prefix = sum; return true; }
        }
    }
    prefix = sum;
    return true;
}

// Counts of all eight digits; the CTA that finishes last turns them into
// exclusive scans and plans the passes.  Clears the states of the first pass
// that needs it and of the rank kernel.
__global__ void __launch_bounds__(256)
radix_hist_kernel(const uint64_t* key, uint32_t* misc, uint32_t* status, int64_t nstatus,
                  uint32_t* tsum, int64_t ntsum, const Header* hdr)
{
    __shared__ uint32_t cnt[8][256];
    __shared__ uint32_t wsum[8];
    __shared__ int last, trivial[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t gid = (int64_t)blockIdx.x * 256 + tid, gsz = (int64_t)gridDim.x * 256;
    chain_start();
    for (int64_t i = gid; i < nstatus; i += gsz) status[i] = 0;
    for (int64_t i = gid; i < ntsum; i += gsz) tsum[i] = 0;
    for (int d = 0; d < 8; ++d) cnt[d][tid] = 0;
    __syncthreads();
    const int64_t m = (int64_t)hdr->nkeys;
    for (int64_t i0 = gid - lane; i0 < m; i0 += gsz) {      // warp-uniform
        const bool valid = i0 + lane < m;
        const uint64_t k = key[valid ? i0 + lane : i0];
        const unsigned live = __ballot_sync(0xffffffffu, valid);
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            const unsigned g = (unsigned)(k >> (8 * d)) & 255u;
            if (d >= 6) {
                // sign, exponent and the first mantissa bits: mostly one value per warp
                const unsigned g0 = __shfl_sync(0xffffffffu, g, 0);
                if (__all_sync(0xffffffffu, g == g0)) {
                    if (lane == 0) atomicAdd(&cnt[d][g0], (unsigned)__popc(live));
                    continue;
                }
            }
            if (valid) atomicAdd(&cnt[d][g], 1u);
        }
    }
    __syncthreads();
    for (int d = 0; d < 8; ++d)
        if (cnt[d][tid]) atomicAdd(&misc[d * 256 + tid], cnt[d][tid]);
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(&misc[kMiscDone], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int d = 0; d < 8; ++d) {
        const uint32_t x = __ldcg(&misc[d * 256 + tid]);
        const int all = __syncthreads_or((int64_t)x == m);   // one digit holds every key
        if (tid == 0) trivial[d] = all;
        uint32_t incl = x;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        uint32_t before = 0;
        for (int w = 0; w < warp; ++w) before += wsum[w];
        misc[d * 256 + tid] = before + incl - x;
        __syncthreads();
    }
    if (tid == 0) {
        uint32_t src = 0;
        for (int d = 0; d < 8; ++d) {
            misc[kMiscPlan + d] = trivial[d] ? 2u : src;
            if (!trivial[d]) src ^= 1u;
        }
        misc[kMiscFinal] = src;
    }
}

constexpr size_t radix_pass_smem()
{
    return (size_t)kSortTile * 12 + (size_t)kSortWarps * 256 * 2;
}

// Lanes of the warp whose 8-bit digit equals this lane's, from eight ballots
// (match.any costs several times that with thirty-odd distinct digits in a warp).
__device__ __forceinline__ unsigned digit_peers(unsigned d)
{
    unsigned peers = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool set = (d >> b) & 1u;
        const unsigned m = __ballot_sync(0xffffffffu, set);
        peers &= set ? m : ~m;
    }
    return peers;
}

// One stable pass by the digit at 8 * pass (see the file's head).
__global__ void __launch_bounds__(kSortThreads2, 2)
radix_pass_kernel(uint64_t* key0, uint64_t* key1, uint32_t* pay0, uint32_t* pay1,
                  uint32_t* status, uint32_t* misc, int pass, int wide, int max_polls,
                  Header* hdr)
{
    extern __shared__ __align__(16) unsigned char rsm[];
    uint64_t* skey = reinterpret_cast<uint64_t*>(rsm);
    uint32_t* spay = reinterpret_cast<uint32_t*>(rsm + (size_t)kSortTile * 8);
    uint16_t* wcnt = reinterpret_cast<uint16_t*>(rsm + (size_t)kSortTile * 12);   // [warp][digit]
    __shared__ uint32_t dstart[256];      // first place of a digit in the ordered tile
    __shared__ uint32_t gstart[256];      // its place in the output, minus dstart
    __shared__ uint32_t wsum[8];
    __shared__ int64_t s_tile;
    __shared__ int s_fail;
    chain_start();
    const uint32_t plan = misc[kMiscPlan + pass];
    if (plan > 1u) return;                                  // all keys share this digit
    const uint64_t* kin = plan ? key1 : key0;
    const uint32_t* pin = plan ? pay1 : pay0;
    uint64_t* kout = plan ? key0 : key1;
    uint32_t* pout = plan ? pay0 : pay1;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const TileState ts{(uint32_t)pass + 1u, wide};
    if (tid == 0) {
        s_tile = take_tile(&misc[kMiscTicket + pass], hdr);
        s_fail = 0;
    }
    for (int i = tid; i < kSortWarps * 256 / 2; i += kSortThreads2) reinterpret_cast<uint32_t*>(wcnt)[i] = 0;
    __syncthreads();
    const int64_t tile = s_tile, m = (int64_t)hdr->nkeys;
    const int64_t base = tile * kSortTile;
    if (tile < 0 || base >= m) return;                      // block-uniform (nor any tile after it)
    const int cnt = m - base < kSortTile ? (int)(m - base) : kSortTile;
    const int shift = 8 * pass;
    // warp w holds the tile's keys w * 512 .., item j of lane l is key 32 j + l
    // of them; past the end: all ones, which order after every key of the tile
    const int wbase = warp * 32 * kSortItems + lane;
    uint64_t k[kSortItems];
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const int i = wbase + 32 * j;
        k[j] = i < cnt ? kin[base + i] : ~0ull;
    }
    uint16_t* my = wcnt + warp * 256;
    uint32_t rank2[kSortItems / 2];                         // 16-bit ranks in the warp's digit
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const unsigned d = (unsigned)(k[j] >> shift) & 255u;
        const unsigned peers = digit_peers(d);
        const unsigned before = my[d];
        const unsigned r = before + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
        if ((__ffs(peers) - 1) == lane) my[d] = (uint16_t)(before + __popc(peers));
        __syncwarp();
        if (j & 1) rank2[j / 2] |= r << 16; else rank2[j / 2] = r;
    }
    __syncthreads();
    // per digit: places of the warps, the tile's count, its prefix
    uint32_t total = 0;
    if (tid < 256) {
        for (int w = 0; w < kSortWarps; ++w) {
            const uint32_t c = wcnt[w * 256 + tid];
            wcnt[w * 256 + tid] = (uint16_t)total;
            total += c;
        }
        const uint32_t real = total - (tid == 255 ? (uint32_t)(kSortTile - cnt) : 0u);
        uint32_t* st = status + tid;
        atomicExch(st + tile * 256, tile == 0 ? ts.incl(real) : ts.own(real));
        uint32_t incl = total;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
        dstart[tid] = incl - total;                         // within the warp, for now
        uint32_t prefix = 0;
        if (tile > 0) {
            if (tile_prefix(st, tile, 256, ts, hdr, max_polls, prefix))
                atomicExch(st + tile * 256, ts.incl(prefix + real));
            else
                s_fail = 1;
        }
        gstart[tid] = misc[pass * 256 + tid] + prefix;
    }
    __syncthreads();
    if (tid < 256) {
        uint32_t before = 0;
        for (int w = 0; w < warp; ++w) before += wsum[w];
        dstart[tid] += before;
        gstart[tid] -= dstart[tid];
    }
    if (s_fail) {                                           // block-uniform
        if (tid == 0) record_error(hdr, kErrWait, tile);
        return;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const unsigned d = (unsigned)(k[j] >> shift) & 255u;
        const uint32_t r = (j & 1) ? rank2[j / 2] >> 16 : rank2[j / 2] & 0xffffu;
        const uint32_t pos = dstart[d] + my[d] + r;         // < kSortTile
        skey[pos] = k[j];
        const int i = wbase + 32 * j;
        if (i < cnt) spay[pos] = pin[base + i];
    }
    __syncthreads();
    for (int i = tid; i < cnt; i += kSortThreads2) {
        const uint64_t kk = skey[i];
        const uint32_t at = gstart[(unsigned)(kk >> shift) & 255u] + (uint32_t)i;
        kout[at] = kk;
        pout[at] = spay[i];
    }
}

// Rank of every sorted key: 2 * (distinct keys up to and including it),
// written into the rank field of the packed element its payload names
// (bit 31 selects the set: 0 = set0, 1 = set1).
__global__ void __launch_bounds__(kSortThreads2)
rank_write_kernel(const uint64_t* key0, const uint64_t* key1, const uint32_t* pay0,
                  const uint32_t* pay1, uint32_t* tsum, uint32_t* misc, KElem* pack0, KElem* pack1,
                  int max_polls, Header* hdr)
{
    __shared__ uint32_t wcount[kSortWarps];
    __shared__ uint32_t s_prefix;
    __shared__ int64_t s_tile;
    __shared__ int s_fail;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    chain_start();
    const bool one = misc[kMiscFinal] != 0u;
    const uint64_t* key = one ? key1 : key0;
    const uint32_t* pay = one ? pay1 : pay0;
    if (tid == 0) {
        s_tile = take_tile(&misc[kMiscTicket + 8], hdr);
        s_fail = 0;
    }
    __syncthreads();
    const int64_t tile = s_tile, m = (int64_t)hdr->nkeys;
    const int64_t base = tile * kSortTile;
    if (tile < 0 || base >= m) return;
    const int64_t w0 = base + warp * 32 * kSortItems;       // the warp's keys, in order
    uint32_t heads[kSortItems];                             // ballots: key differs from the one before
    uint32_t count = 0;
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const int64_t i = w0 + 32 * j + lane;
        const uint64_t k = i < m ? key[i] : 0;
        uint64_t kp = __shfl_up_sync(0xffffffffu, k, 1);
        if (lane == 0 && i > 0 && i < m) kp = key[i - 1];
        heads[j] = __ballot_sync(0xffffffffu, i < m && (i == 0 || k != kp));
        count += __popc(heads[j]);
    }
    if (lane == 0) wcount[warp] = count;
    __syncthreads();
    if (tid == 0) {
        const TileState ts{0u, 1};
        uint32_t total = 0, prefix = 0;
        for (int w = 0; w < kSortWarps; ++w) { const uint32_t c = wcount[w]; wcount[w] = total; total += c; }
        atomicExch(tsum + tile, tile == 0 ? ts.incl(total) : ts.own(total));
        if (tile > 0) {
            if (tile_prefix(tsum, tile, 1, ts, hdr, max_polls, prefix)) atomicExch(tsum + tile, ts.incl(prefix + total));
            else s_fail = 1;
        }
        s_prefix = prefix;
    }
    __syncthreads();
    if (s_fail) {                                           // block-uniform
        if (tid == 0) record_error(hdr, kErrWait, tile);
        return;
    }
    uint32_t before = s_prefix + wcount[warp];
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const int64_t i = w0 + 32 * j + lane;
        if (i < m) {
            const uint32_t d = before + __popc(heads[j] & (0xffffffffu >> (31 - lane)));
            const uint32_t p = pay[i];
            KElem* dst = (p >> 31) ? pack1 : pack0;
            dst[p & 0x7fffffffu].k = 2u * d;
        }
        before += __popc(heads[j]);
    }
}

// Keys of the integration bounds a and b (one thread): 2 * (distinct ends
// below q) + 1, or + 2 when q is itself an interval end; b = inf maps to the
// rank of the last intervals.  Written to hdr->bound_key[0..1].
__global__ void bound_keys_kernel(const uint64_t* key0, const uint64_t* key1, const uint32_t* pay0,
                                  const uint32_t* pay1, const uint32_t* misc, const KElem* pack0,
                                  const KElem* pack1, double a, double b, Header* hdr)
{
    chain_start();
    if (hdr->err != kNoError) return;       // the payloads may not be the sort's
    const int64_t m = (int64_t)hdr->nkeys;
    const uint64_t* key = misc[kMiscFinal] ? key1 : key0;
    const uint32_t* pay = misc[kMiscFinal] ? pay1 : pay0;
    const double q2[2] = {a, b};
    for (int w = 0; w < 2; ++w) {
        const double q = q2[w];
        if (isinf(q)) { hdr->bound_key[w] = 0xFFFFFFFFu; continue; }
        const uint64_t qb = (uint64_t)__double_as_longlong(q);
        int64_t lo = 0, hi = m;                 // first sorted key >= q
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (key[mid] < qb) lo = mid + 1; else hi = mid;
        }
        uint32_t below = 0;                      // distinct keys < q
        if (lo > 0) {
            const uint32_t p = pay[lo - 1];
            below = ((p >> 31) ? pack1 : pack0)[p & 0x7fffffffu].k / 2u;
        }
        hdr->bound_key[w] = 2u * below + ((lo < m && key[lo] == qb) ? 2u : 1u);
    }
}

// The sort and the ranks, from the keys of ks.key[0], ks.pay[0] (hdr->nkeys of
// them) and cleared counters.
static cudaError_t sort_and_rank(const KeySort& ks, KElem* pack0, KElem* pack1, int max_polls,
                                 Header* hdr, cudaStream_t s)
{
    const unsigned tiles = (unsigned)ks.tiles;
    const int wide = ks.cap >= kNarrowKeys ? 1 : 0;
    cudaError_t e = cudaFuncSetAttribute(radix_pass_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)radix_pass_smem());
    if (e != cudaSuccess) return e;
    // a CTA per 2,048 keys up to four per SM
    int64_t hgrid = (ks.cap + 2047) / 2048;
    const int64_t hcap = (int64_t)device_sm_count() * 4;
    if (hgrid > hcap) hgrid = hcap;
    if (hgrid < 1) hgrid = 1;
    launch_next(radix_hist_kernel, hgrid, 256, 0, s, ks.key[0], ks.misc, ks.status, ks.tiles * 256,
                                                      ks.tsum, ks.tiles + 1, hdr);
    for (int pass = 0; pass < 8; ++pass) {
        if (wide && pass > 0) {
            e = cudaMemsetAsync(ks.status, 0, sizeof(uint32_t) * 256 * (size_t)ks.tiles, s);
            if (e != cudaSuccess) return e;
        }
        launch_next(radix_pass_kernel, tiles, kSortThreads2, radix_pass_smem(), s,
            ks.key[0], ks.key[1], ks.pay[0], ks.pay[1], ks.status, ks.misc, pass, wide, max_polls, hdr);
    }
    launch_next(rank_write_kernel, tiles, kSortThreads2, 0, s, ks.key[0], ks.key[1], ks.pay[0], ks.pay[1], ks.tsum,
                                                      ks.misc, pack0, pack1, max_polls, hdr);
    return cudaGetLastError();
}

cudaError_t rank_keys(const KeySort& ks, KElem* pack0, const int64_t* poff0, int64_t n0,
                      KElem* pack1, const int64_t* poff1, int64_t n1, Header* hdr, cudaStream_t s)
{
    launch_next(count_keys_kernel, 1, 256, 0, s, hdr, poff0, n0, poff1, n1, ks.misc);
    return sort_and_rank(ks, pack0, pack1, kSortPolls, hdr, s);
}

cudaError_t bound_keys(const KeySort& ks, const KElem* pack0, const KElem* pack1, double a, double b,
                       Header* hdr, cudaStream_t s)
{
    launch_next(bound_keys_kernel, 1, 1, 0, s, ks.key[0], ks.key[1], ks.pay[0], ks.pay[1], ks.misc, pack0, pack1, a, b, hdr);
    return cudaGetLastError();
}

// Self-test input: well mixed 63-bit keys, their own positions as payloads,
// ranks zero; with missing >= 0, tile 0 of that pass is never handed out.
__global__ void __launch_bounds__(256) sort_selftest_kernel(Header* hdr, uint64_t* key, uint32_t* pay,
                                                            KElem* pack, int64_t keys, uint32_t* misc,
                                                            int missing)
{
    const int64_t gid = (int64_t)blockIdx.x * 256 + threadIdx.x, gsz = (int64_t)gridDim.x * 256;
    for (int64_t i = gid; i < keys; i += gsz) {
        key[i] = ((uint64_t)(i + 1) * 0x9e3779b97f4a7c15ull) >> 1;
        pay[i] = (uint32_t)i;
        pack[i] = KElem{0u, 0.f, 0.f, 0.f};
    }
    for (int64_t i = gid; i < kMiscWords; i += gsz)
        misc[i] = missing >= 0 && i == kMiscTicket + missing ? 1u : 0u;
    if (gid == 0) {
        hdr->err = kNoError;
        hdr->nkeys = (unsigned long long)keys;
    }
}

}  // namespace pcfgb

extern "C" int pcf_selftest_sort_wait(int64_t keys, int missing_pass, int64_t polls, void* workspace,
                                      size_t workspace_bytes, size_t* used, cudaStream_t stream)
{
    using namespace pcfgb;
    if (keys < 1 || keys > (1ll << 28) || missing_pass < -1 || missing_pass > 8 || polls < 1 ||
        polls > (1ll << 20) || !used)
        return PCF_EINVAL;
    // (with one tile there is no successor to wait for the missing one)
    if (missing_pass >= 0 && keys <= kSortTile) return PCF_EINVAL;
    *used = align_up(sizeof(Header)) + keysort_bytes(keys) + align_up(sizeof(KElem) * (size_t)keys);
    if (!workspace || ((uintptr_t)workspace % kAlign) || workspace_bytes < *used) return PCF_ENOWS;
    Header* hdr = (Header*)workspace;
    char* cur = (char*)workspace + align_up(sizeof(Header));
    const KeySort ks = carve_keysort(cur, keys);
    KElem* pack = (KElem*)cur;
    int64_t grid = (keys + 255) / 256;
    if (grid > device_sm_count() * 8) grid = device_sm_count() * 8;
    sort_selftest_kernel<<<(unsigned)grid, 256, 0, stream>>>(hdr, ks.key[0], ks.pay[0], pack, keys,
                                                             ks.misc, missing_pass);
    if (cudaGetLastError() != cudaSuccess) return PCF_ECUDA;
    return sort_and_rank(ks, pack, nullptr, (int)polls, hdr, stream) == cudaSuccess ? PCF_OK
                                                                                     : PCF_ECUDA;
}
