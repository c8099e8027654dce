// Cell binning: stable counting sort of particles by key = cell * S + species (particles collide per cell of
// volume dV, Sec. 2), and a gather through the resulting permutation.
//
// histogram (atomic counts) -> exclusive scan -> scatter to the counted places (order within a segment arbitrary)
// -> per-segment sort: by particle index, which restores the stable order, or straight by weight. The result does not
// depend on the order in which the atomics were served. Lanes of a warp with equal keys add once (key_group); the count's
// atomic also gives each particle its place in the segment, so the scatter needs none.
// Segments of up to 512 entries are sorted by one warp in its slice of shared memory (warp barriers only), larger ones
// by a whole CTA. What bounds it: atomics and random sectors on shuffled input (3.3e7 particles, 2e5 segments: 1.64 ms with a
// match in every warp, cursors and bitonic sorts, 1.09 so); the segment sorts after a push (17% moved: 0.92 -> 0.81 ms, 0.47 of
// it the sorts; in weight order 1.63 -> 0.94). 1.34e8 particles: shuffled 7.6 -> 5.9 ms, after a push 3.49 -> 3.05, in weight
// order 6.3 -> 3.5. 60% moved, which no push does, is the one input found where the network in every segment was
// faster (0.97 against 1.07 ms). A two-pass radix sort of (key, index) pairs took 1.43 ms shuffled and lost on nearly binned
// input, where a warp here has few atomics.
#include <mutex>

#include "mcc_kernels.h"

// Counters of mcc_bin_static: every device that loads the library holds this array until the process exits.
// counts | cursors | large-segment list, the layout bin_core expects for kStaticBinKeys segments.
constexpr int64_t kStaticBinKeys = 1 << 21;
constexpr size_t kStaticBinHalf = ((size_t)kStaticBinKeys * sizeof(int32_t) + 255) & ~(size_t)255;
constexpr size_t kStaticBinList = ((size_t)(kStaticBinKeys + 1) * sizeof(int32_t) + 255) & ~(size_t)255;
static __device__ __align__(256) int32_t g_bin_static_scratch[(2 * kStaticBinHalf + kStaticBinList) / sizeof(int32_t)];

namespace mcc {
namespace {

constexpr int kBinThreads = 256;
constexpr int kScanThreads = 1024;
constexpr int kSegCap = 12288;  // indices sorted in shared memory per segment; larger segments sort in place
constexpr int kSegCapW = 4096;  // weight-order keys sorted in shared memory per segment; larger ones in the workspace

constexpr int kWarpSeg = 512;  // segments up to this size are sorted by one warp

// Key of particle i (cell * S + species), or -1 past the end or out of range (latched).
__device__ __forceinline__ long long bin_key(const int32_t* __restrict__ cell, const int32_t* __restrict__ species,
                                             int64_t i, int64_t n, int32_t n_cells, int32_t S, int32_t* status)
{
    if (i >= n) return -1;
    const int32_t c = cell[i], s = species[i];
    if (c < 0 || c >= n_cells || s < 0 || s >= S) {
        if (status) latch(status, kErrBounds);
        return -1;
    }
    return (long long)c * S + s;
}

// Lanes of a warp that count as one: this lane's group has `len` lanes, this one is number `rank`, the first is lane `lead`.
// Either all lanes with equal keys (a warp match) or runs of equal keys in neighbouring lanes (two ballots). The match takes
// time with the number of different keys, about 64 cycles of an SM for 32 of them, the atomics it saves take more: it is
// taken when a warp's keys repeat, that is when at most kRunHeads runs begin (nearly binned input, such as a re-bin after
// a push), when kSameKey lanes hold lane 0's key (species in turns within binned cells) or when there are few segments,
// whose counters the atomics queue for. Shuffled input (32 runs of one lane) takes the runs. Count, and scatter with cursors, us:
// 3.3e7 particles in 2e5 segments, 17% moved by a push, 100 and 176 (runs alone 162 and 294), shuffled 330 and 350 (a match in
// every warp 460 and 520); 1e7 particles in 192 segments 2360 and 1170 (runs alone 2650 and 1300).
constexpr int kRunHeads = 28, kSameKey = 4;
constexpr int64_t kFewSegments = 512;

__device__ __forceinline__ void key_group(long long key, bool few, int& lead, int& rank, int& len)
{
    const int lane = threadIdx.x & 31;
    const long long prev = __shfl_up_sync(0xffffffffu, key, 1);
    const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || key != prev);
    const unsigned same0 = __ballot_sync(0xffffffffu, key == __shfl_sync(0xffffffffu, key, 0));
    if (few || __popc(heads) <= kRunHeads || __popc(same0) >= kSameKey) {
        const unsigned m = __match_any_sync(0xffffffffu, key);
        lead = __ffs(m) - 1;
        rank = __popc(m & ((1u << lane) - 1u));
        len = __popc(m);
        return;
    }
    const unsigned upto = (2u << lane) - 1u;  // this lane and those below
    lead = 31 - __clz(heads & upto);
    rank = lane - lead;
    const unsigned after = heads & ~upto;
    len = (after ? __ffs(after) - 1 : 32) - lead;
}

// All lanes of a warp run the same trips (the loop index is the warp's base), so the shuffles see the full warp. One element
// per thread and iteration: four, a grid's stride apart, with their atomics in flight together took 202 / 208 us (count / scatter)
// where one takes 144 / 156 after a push (the counters of four places at once); on shuffled input they gain little (1.34e8
// particles 5.79 against 5.92 ms, 3.3e7 1.09 against 1.10). Both kernels have to take the rows in the same order, or a segment's
// places are written at different times (four in one of them only: 6.8 and 7.4 ms).
// PLACE: place[i] = the particle's place in its segment, in the order the atomics were served.
template <bool PLACE>
__global__ void __launch_bounds__(kBinThreads) k_hist(const int32_t* __restrict__ cell, const int32_t* __restrict__ species,
                                                      int64_t n, int32_t n_cells, int32_t S, int32_t* __restrict__ counts,
                                                      int32_t* __restrict__ place, int32_t* status)
{
    const int lane = threadIdx.x & 31;
    const bool few = (int64_t)n_cells * S <= kFewSegments;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        const long long key = bin_key(cell, species, base + lane, n, n_cells, S, status);
        int lead, rank, len, at = 0;
        key_group(key, few, lead, rank, len);
        if (key >= 0 && lane == lead) at = atomicAdd(&counts[key], len);
        if (PLACE) {
            at = __shfl_sync(0xffffffffu, at, lead) + rank;
            if (key >= 0) place[base + lane] = at;
        }
    }
}

// Exclusive scan of nk counts into nk + 1 offsets, in three passes over tiles of kScanTile keys: each CTA scans its
// tile (tile-local offsets) and leaves the tile's total in counts[first key of the tile]; one CTA scans the tile
// totals in place (their exclusive prefixes) and writes offsets[nk]; each CTA adds its tile's prefix. The counts are
// not read again after the scan, so their tile-start slots can carry the totals.
constexpr int kScanTile = 4 * kScanThreads;

// Exclusive scan of v over the CTA (kScanThreads threads); returns this thread's exclusive prefix, *total the sum.
__device__ __forceinline__ int64_t block_exclusive_scan(int64_t v, int64_t* wsum, int64_t* total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int64_t t = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        wsum[lane] = t;
    }
    __syncthreads();
    *total = wsum[31];
    return x - v + (wid > 0 ? wsum[wid - 1] : 0);
}

__global__ void __launch_bounds__(kScanThreads) k_scan_tile(int32_t* __restrict__ counts, int64_t nk,
                                                            int64_t* __restrict__ offsets, int32_t* status)
{
    __shared__ int64_t wsum[kScanThreads / 32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + 4 * threadIdx.x;
    int32_t c[4];
    int64_t s = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        c[j] = base + j < nk ? counts[base + j] : 0;
        if (c[j] > (1 << kPermBits)) latch(status, kErrTooLarge);
        s += c[j];
    }
    int64_t total;
    int64_t run = block_exclusive_scan(s, wsum, &total);  // every thread has read its counts before this returns
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (base + j < nk) offsets[base + j] = run;
        run += c[j];
    }
    if (threadIdx.x == 0) {
        counts[(int64_t)blockIdx.x * kScanTile] = (int32_t)total;  // total <= n <= INT32_MAX
        if (gridDim.x == 1) offsets[nk] = total;                   // one tile: done
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_top(int32_t* __restrict__ counts, int64_t nk, int64_t tiles,
                                                           int64_t* __restrict__ offsets)
{
    __shared__ int64_t wsum[kScanThreads / 32];
    const int64_t chunk = (tiles + kScanThreads - 1) / kScanThreads;
    const int64_t b = (int64_t)threadIdx.x * chunk;
    const int64_t e = b + chunk < tiles ? b + chunk : tiles;
    int64_t s = 0;
    for (int64_t t = b; t < e; ++t) s += counts[t * kScanTile];
    int64_t total;
    int64_t run = block_exclusive_scan(s, wsum, &total);
    for (int64_t t = b; t < e; ++t) {
        const int32_t x = counts[t * kScanTile];
        counts[t * kScanTile] = (int32_t)run;
        run += x;
    }
    if (threadIdx.x == 0) offsets[nk] = total;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_add(const int32_t* __restrict__ counts, int64_t nk,
                                                           int64_t* __restrict__ offsets)
{
    if (blockIdx.x == 0) return;
    const int64_t pre = counts[(int64_t)blockIdx.x * kScanTile];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    for (int j = threadIdx.x; j < kScanTile; j += kScanThreads)
        if (base + j < nk) offsets[base + j] += pre;
}

// PLACE: each particle's place was counted (place); else it is taken from the segment's cursor.
template <bool PLACE>
__global__ void __launch_bounds__(kBinThreads) k_scatter(const int32_t* __restrict__ cell, const int32_t* __restrict__ species,
                                                         int64_t n, int32_t n_cells, int32_t S,
                                                         const int64_t* __restrict__ offsets, int32_t* __restrict__ cursor,
                                                         const int32_t* __restrict__ place, int32_t* __restrict__ perm)
{
    const int lane = threadIdx.x & 31;
    const bool few = (int64_t)n_cells * S <= kFewSegments;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        const long long key = bin_key(cell, species, base + lane, n, n_cells, S, nullptr);
        int at = 0;
        if (PLACE) {
            if (key >= 0) at = place[base + lane];
        } else {
            int lead, rank, len;
            key_group(key, few, lead, rank, len);
            if (key >= 0 && lane == lead) at = atomicAdd(&cursor[key], len);
            at = __shfl_sync(0xffffffffu, at, lead) + rank;
        }
        if (key >= 0) perm[offsets[key] + at] = (int32_t)(base + lane);
    }
}

// Ascending sort of n <= kWarpSeg entries in the calling warp's shared-memory slice: the bitonic network in its
// "flip" form (every comparator puts the smaller entry at the lower index, so positions >= n act as +infinity and
// are skipped), one warp barrier per stage. Loops stay rolled: the code is small enough to stay in the instruction
// cache. cmpx(lo, hi) orders the entries at two positions.
template <class Cmpx>
__device__ __forceinline__ void warp_sort_smem(int n, Cmpx cmpx)
{
    const int lane = threadIdx.x & 31;
    int logP = 0;
    while ((1 << logP) < n) ++logP;
    const int half_work = 1 << (logP - 1);
#pragma unroll 1
    for (int lg = 1; lg <= logP; ++lg) {
        const int size = 1 << lg, hmask = (size >> 1) - 1;
#pragma unroll 1
        for (int i = lane; i < half_work; i += 32) {
            const int base = (i >> (lg - 1)) << lg;
            const int lo = base + (i & hmask), hi = base + size - 1 - (i & hmask);
            if (hi < n) cmpx(lo, hi);
        }
        __syncwarp();
#pragma unroll 1
        for (int ls = lg - 2; ls >= 0; --ls) {
            const int stride = 1 << ls;
#pragma unroll 1
            for (int i = lane; i < half_work; i += 32) {
                const int lo = ((i >> ls) << (ls + 1)) + (i & (stride - 1)), hi = lo + stride;
                if (hi < n) cmpx(lo, hi);
            }
            __syncwarp();
        }
    }
}

// Small segments (2 .. kWarpSeg entries), one warp each, sorted in the warp's shared-memory slice (the loop index is
// warp-uniform, so whole warps take the same branches). Not WEIGHTED: by particle index. WEIGHTED: straight into the weight
// order of mcc_bin_weighted, pairs (weight key with a zero rank field, particle index) in lexicographic order, which is
// descending truncated weight with ties in increasing index. The ids of the larger segments are appended to `large` (large[0]
// the count, zeroed before) for the CTA-wide sorts.
// A segment in order already is left. Otherwise a counting sort on a linear map of the keys' top words (the indices) to n or
// more buckets, then an insertion sort within a bucket. Indices of shuffled particles spread evenly, and so do weights over
// decades, as the IEEE bits of a weight are nearly linear in its logarithm. After a particle push most indices of a segment
// are neighbours, those that stayed, and the rest come from anywhere: one bucket of the linear map would hold nearly all.
// The map of such a segment (of 32 entries looked at, kCrowd in the bucket of a middling one) has three pieces: half the buckets
// for the 2.5 n indices around that entry, a quarter each for those below and above, by the logarithm of their distance (what
// moved in comes from the next cells, rows and planes of the grid, orders of magnitude apart). A segment of which a third
// comes from elsewhere, or one that still fills a bucket beyond kBucketMost, takes the bitonic network; up to 32 indices
// take it in registers. 3.3e7 particles, 17% moved: 616 us by the network in every segment, 734 by a futile count and then
// the network, 470 by three pieces.
constexpr int kOrderWarps = 4;   // warps per CTA
constexpr int kBucketMost = 12;  // longest bucket for the insertion sort
constexpr int kCrowd = 8;        // of 32 entries looked at, in one bucket: a crowd

template <bool WEIGHTED>
__global__ void __launch_bounds__(32 * kOrderWarps) k_segsort_warp(const int64_t* __restrict__ offsets, int64_t nk,
                                                                  const double* __restrict__ w,
                                                                  int32_t* __restrict__ perm, int32_t* __restrict__ large)
{
    __shared__ uint64_t kslab[WEIGHTED ? kOrderWarps : 1][WEIGHTED ? kWarpSeg : 1];
    __shared__ int32_t islab[kOrderWarps][kWarpSeg];
    __shared__ uint32_t cslab[kOrderWarps][kWarpSeg];
    __shared__ uint16_t oslab[kOrderWarps][kWarpSeg];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t* kb = kslab[WEIGHTED ? wid : 0];
    int32_t* ib = islab[wid];
    uint32_t* cnt = cslab[wid];
    uint16_t* ord = oslab[wid];
    auto top = [&](int i) -> uint32_t { return WEIGHTED ? (uint32_t)(kb[i] >> 32) : (uint32_t)ib[i]; };
    auto after = [&](int i, int j) -> bool {  // entry i comes after entry j
        return WEIGHTED ? (kb[i] > kb[j] || (kb[i] == kb[j] && ib[i] > ib[j])) : ib[i] > ib[j];
    };
    const int64_t nwarps = (int64_t)gridDim.x * kOrderWarps;
    for (int64_t seg = (int64_t)blockIdx.x * kOrderWarps + wid; seg < nk; seg += nwarps) {
        const int64_t b = offsets[seg];
        const int n = (int)(offsets[seg + 1] - b);
        if (n > kWarpSeg && lane == 0) large[1 + atomicAdd(&large[0], 1)] = (int32_t)seg;
        if (n < 2 || n > kWarpSeg) continue;
        int32_t* p = perm + b;
        if (!WEIGHTED && n <= 32) {  // one index per lane: the network in registers, no shared memory
            int32_t v = lane < n ? p[lane] : INT32_MAX;
#pragma unroll
            for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
                for (int j = k / 2; j > 0; j >>= 1) {
                    const int32_t y = __shfl_xor_sync(0xffffffffu, v, j);
                    v = ((lane & j) == 0) == ((lane & k) == 0) ? min(v, y) : max(v, y);
                }
            if (lane < n) p[lane] = v;
            continue;
        }
        uint32_t lo = 0xFFFFFFFFu, hi = 0u;
        for (int i = lane; i < n; i += 32) {
            const int32_t q = p[i];
            ib[i] = q;
            if (WEIGHTED) kb[i] = weight_key(w[q], 0u);
            lo = min(lo, top(i));
            hi = max(hi, top(i));
        }
        __syncwarp();
        bool out = false;
        for (int i = lane; i + 1 < n; i += 32) out |= after(i, i + 1);
        if (!__any_sync(0xffffffffu, out)) continue;
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        auto network = [&] {
            warp_sort_smem(n, [&](int x, int y) {
                if (after(x, y)) {
                    const int32_t a = ib[x];
                    ib[x] = ib[y];
                    ib[y] = a;
                    if (WEIGHTED) {
                        const uint64_t k = kb[x];
                        kb[x] = kb[y];
                        kb[y] = k;
                    }
                }
            });
            for (int i = lane; i < n; i += 32) p[i] = ib[i];
            __syncwarp();
        };
        int lg = 5;
        while ((1 << lg) < n) ++lg;
        const int nb = 1 << lg, per = nb / 32;  // nb <= kWarpSeg
        // bucket = (key - lo) nb / (hi - lo + 1), rounded down: below nb, and never decreasing in the key
        const uint32_t span = hi - lo;
        // (a piece of width d with k buckets: (key - its start) k / d, the factor 0 where every key has a bucket of its own)
        auto factor = [](uint32_t k, uint64_t d) { return d <= k ? 0u : (uint32_t)(((uint64_t)k << 32) / d); };
        auto place = [](uint32_t x, uint32_t f) { return f ? __umulhi(x, f) : x; };
        const uint32_t mult = factor((uint32_t)nb, (uint64_t)span + 1u);
        uint32_t w0 = 0u, w1 = 0u, mw = 0u, side = 0u;  // side > 0: three pieces, side | 2 side | side buckets
        if (!WEIGHTED) {
            const uint32_t x = top(n / 4), y = top(n / 2), z = top(n - 1 - n / 4);
            const uint32_t mid = max(min(x, y), min(max(x, y), z));
            const uint32_t at = place(mid - lo, mult), mine = top(lane * n >> 5);  // every lane an entry in turn
            if (__popc(__ballot_sync(0xffffffffu, place(mine - lo, mult) == at)) >= kCrowd) {
                const uint32_t half = (uint32_t)(n + n / 4);
                w0 = mid - lo > half ? mid - half : lo;  // the window [w0, w1)
                w1 = hi - mid >= half ? mid + half : hi + 1u;
                if (__popc(__ballot_sync(0xffffffffu, mine >= w0 && mine < w1)) < 21) {  // many from elsewhere, in clumps
                    network();
                    continue;
                }
                side = (uint32_t)nb / 4;
                mw = factor(2 * side, (uint64_t)(w1 - w0));
            }
        }
        // distance d = 1 .. 2^31 to a bucket below nb / 4: its exponent and leading bits, 31 octaves over nb / 4 buckets
        auto octave = [&](uint32_t d) -> uint32_t { return (__float_as_uint((float)d) - 0x3F800000u) >> (30 - lg); };
        auto bucket = [&](int i) -> int {
            const uint32_t t = top(i);
            if (WEIGHTED || side == 0u) return (int)place(t - lo, mult);
            return (int)(t < w0 ? side - 1u - octave(w0 - t)
                                : (t < w1 ? side + place(t - w0, mw) : 3 * side + octave(t - w1 + 1u)));
        };
        for (int i = lane; i < nb; i += 32) cnt[i] = 0;
        __syncwarp();
        for (int i = lane; i < n; i += 32) atomicAdd(&cnt[bucket(i)], 1u);
        __syncwarp();
        uint32_t sum = 0, most = 0;
        for (int i = 0; i < per; ++i) {
            const uint32_t x = cnt[lane * per + i];
            sum += x;
            most = max(most, x);
        }
        if (__reduce_max_sync(0xffffffffu, most) > kBucketMost) {
            network();
            continue;
        }
        uint32_t inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        uint32_t run = inc - sum;
        for (int i = 0; i < per; ++i) {
            const uint32_t x = cnt[lane * per + i];
            cnt[lane * per + i] = run;
            run += x;
        }
        __syncwarp();
        for (int i = lane; i < n; i += 32) ord[atomicAdd(&cnt[bucket(i)], 1u)] = (uint16_t)i;
        __syncwarp();
        for (int i = lane; i < nb; i += 32) {  // cnt[i] is now the end of bucket i
            const int end = (int)cnt[i], start = i ? (int)cnt[i - 1] : 0;
            for (int x = start + 1; x < end; ++x) {
                const uint16_t v = ord[x];
                int y = x - 1;
                while (y >= start && after(ord[y], v)) {
                    ord[y + 1] = ord[y];
                    --y;
                }
                ord[y + 1] = v;
            }
        }
        __syncwarp();
        for (int i = lane; i < n; i += 32) p[i] = ib[ord[i]];
        __syncwarp();
    }
}

__global__ void __launch_bounds__(kBinThreads) k_segsort(const int64_t* __restrict__ offsets,
                                                         const int32_t* __restrict__ large, int32_t* __restrict__ perm)
{
    __shared__ int32_t buf[kSegCap];
    const int32_t n_large = large[0];
    for (int32_t q = blockIdx.x; q < n_large; q += gridDim.x) {
        const int64_t seg = large[1 + q];
        const int64_t b = offsets[seg];
        const int n = (int)(offsets[seg + 1] - b);
        if (n <= kSegCap) {
            for (int i = threadIdx.x; i < n; i += kBinThreads) buf[i] = perm[b + i];
            __syncthreads();
            block_sort_i32(buf, n);
            for (int i = threadIdx.x; i < n; i += kBinThreads) perm[b + i] = buf[i];
        } else {
            block_sort_i32(perm + b, n);
        }
        __syncthreads();
    }
}

// Weight order of every large segment (run after k_segsort, so a segment's entries are in increasing particle index):
// keys = weight_key(w, rank) (descending weight truncated to 32 fraction bits, ties by rank = by index), sorted, then
// each slot takes the index its key's rank points to. keys: [n] workspace, holds the keys of large segments and
// the reordered indices before they are copied back.
__global__ void __launch_bounds__(kBinThreads) k_segsort_w(const int64_t* __restrict__ offsets,
                                                           const int32_t* __restrict__ large,
                                                           const double* __restrict__ w, int32_t* __restrict__ perm,
                                                           uint64_t* __restrict__ keys)
{
    __shared__ uint64_t buf[kSegCapW];
    const int32_t n_large = large[0];
    for (int32_t q = blockIdx.x; q < n_large; q += gridDim.x) {
        const int64_t seg = large[1 + q];
        const int64_t b = offsets[seg];
        const int n = (int)(offsets[seg + 1] - b);
        uint64_t* k = n <= kSegCapW ? buf : keys + b;
        for (int i = threadIdx.x; i < n; i += kBinThreads) k[i] = weight_key(w[perm[b + i]], (uint32_t)i);
        __syncthreads();
        block_sort_u64(k, n);
        // each thread reads only its own slot of k before writing that slot of keys
        for (int i = threadIdx.x; i < n; i += kBinThreads)
            keys[b + i] = (uint64_t)(uint32_t)perm[b + (int)(k[i] & kPermMask)];
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += kBinThreads) perm[b + i] = (int32_t)(uint32_t)keys[b + i];
        __syncthreads();
    }
}

// Four elements per thread and iteration, their permuted reads issued together (more reads in flight). A shuffled
// permutation reads a whole sector per element, so what bounds it is how much of `in` stays in L2. STREAM: the permutation and
// the output, touched once, are marked to leave first. Without / with, us, on one GPU: floats in nearly the output's order 90 /
// 84 (33 million), 302 / 280 (134 million), shuffled 336 / 322 and 2663 / 2662; doubles in nearly the output's order 120 / 119
// (33 million), 224 / 223 (67 million), but 425 / 501 (134 million), shuffled 560 / 555 and 3026 / 3040. Doubles go without
// from 64 million on, where it gains nothing yet loses nothing.
constexpr int64_t kStreamDoubles = 64'000'000;

template <class T, bool STREAM>
__global__ void k_gather(const T* __restrict__ in, const int32_t* __restrict__ perm, int64_t n, T* __restrict__ out)
{
    constexpr int U = 4;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; base < n; base += U * stride) {
        int32_t p[U];
        T v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) p[u] = base + u * stride < n ? (STREAM ? __ldcs(perm + base + u * stride) : perm[base + u * stride]) : 0;
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = base + u * stride < n ? __ldg(in + p[u]) : T(0);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (base + u * stride < n) {
                if (STREAM) __stcs(out + base + u * stride, v[u]);
                else out[base + u * stride] = v[u];
            }
    }
}

int grid_for(int64_t n, int threads)
{
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t want = (n + threads - 1) / threads;
    const int64_t cap = (int64_t)sms * 16;
    return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

}  // namespace

static size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// Counters: counts | cursors (one int32 per segment each) | large-segment list (count, then segment ids). The workspace of
// mcc_bin adds each particle's place in its segment (int32), that of mcc_bin_weighted the keys of large segments (64 bits,
// over the places, which are done with by then).
static size_t counter_bytes(int64_t n_keys)
{
    return 2 * up256((size_t)n_keys * sizeof(int32_t)) + up256((size_t)(n_keys + 1) * sizeof(int32_t));
}

size_t bin_workspace_bytes(int64_t n, int64_t n_keys)
{
    return counter_bytes(n_keys) + up256((size_t)n * sizeof(int32_t));
}

static int32_t* large_list(void* ws, int64_t nk)
{
    return reinterpret_cast<int32_t*>(reinterpret_cast<char*>(ws) + 2 * up256((size_t)nk * sizeof(int32_t)));
}

// hist -> scan -> scatter -> small segments by one warp each (index order, or with w the weight order directly)
// -> large segments by index, one CTA each. place: [n] or null (the scatter then takes its places from the cursors).
static cudaError_t bin_core(const int32_t* cell, const int32_t* species, int64_t n, int32_t n_cells,
                            int32_t n_species, const double* w, int32_t* perm, int64_t* offsets, void* ws, int32_t* place,
                            int32_t* status, cudaStream_t st, int64_t* launches)
{
    const int64_t nk = (int64_t)n_cells * n_species;
    int32_t* counts = reinterpret_cast<int32_t*>(ws);
    int32_t* cursor = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(ws) + up256((size_t)nk * sizeof(int32_t)));
    int32_t* large = large_list(ws, nk);
    cudaError_t e = cudaMemsetAsync(ws, 0, counter_bytes(nk), st);
    if (e != cudaSuccess) return e;
    const int g = grid_for(n, kBinThreads);
    if (n > 0) {
        if (place) k_hist<true><<<g, kBinThreads, 0, st>>>(cell, species, n, n_cells, n_species, counts, place, status);
        else k_hist<false><<<g, kBinThreads, 0, st>>>(cell, species, n, n_cells, n_species, counts, place, status);
    }
    const int64_t tiles = (nk + kScanTile - 1) / kScanTile;
    k_scan_tile<<<(unsigned)tiles, kScanThreads, 0, st>>>(counts, nk, offsets, status);
    *launches += 1;
    // small sorts are bound by their launches (100 cells x 300 in weight order with a gather: 71 -> 61 us): one tile of segments
    // needs no second pass, and no segment exceeds the particles there are
    if (tiles > 1) {
        k_scan_top<<<1, kScanThreads, 0, st>>>(counts, nk, tiles, offsets);
        k_scan_add<<<(unsigned)tiles, kScanThreads, 0, st>>>(counts, nk, offsets);
        *launches += 2;
    }
    if (n > 0) {
        if (place)
            k_scatter<true><<<g, kBinThreads, 0, st>>>(cell, species, n, n_cells, n_species, offsets, cursor, place, perm);
        else
            k_scatter<false><<<g, kBinThreads, 0, st>>>(cell, species, n, n_cells, n_species, offsets, cursor, place, perm);
        const int gw = grid_for(nk * 32, 32 * kOrderWarps);
        if (w) k_segsort_warp<true><<<gw, 32 * kOrderWarps, 0, st>>>(offsets, nk, w, perm, large);
        else k_segsort_warp<false><<<gw, 32 * kOrderWarps, 0, st>>>(offsets, nk, w, perm, large);
        *launches += 3;
        if (n > kWarpSeg) {
            k_segsort<<<grid_for(n / (kWarpSeg + 1) * kBinThreads, kBinThreads), kBinThreads, 0, st>>>(offsets, large,
                                                                                                     perm);
            *launches += 1;
        }
    }
    return cudaGetLastError();
}

cudaError_t launch_bin(const int32_t* cell, const int32_t* species, int64_t n, int32_t n_cells, int32_t n_species,
                       int32_t* perm, int64_t* offsets, void* ws, int32_t* status, cudaStream_t st, int64_t* launches)
{
    int32_t* place = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(ws) + counter_bytes((int64_t)n_cells * n_species));
    return bin_core(cell, species, n, n_cells, n_species, nullptr, perm, offsets, ws, place, status, st, launches);
}

size_t bin_weighted_workspace_bytes(int64_t n, int64_t n_keys)
{
    return counter_bytes(n_keys) + up256((size_t)n * sizeof(uint64_t));
}

cudaError_t launch_bin_weighted(const int32_t* cell, const int32_t* species, const double* w, int64_t n,
                                int32_t n_cells, int32_t n_species, int32_t* perm, int64_t* offsets, void* ws,
                                int32_t* status, cudaStream_t st, int64_t* launches)
{
    const int64_t nk = (int64_t)n_cells * n_species;
    uint64_t* keys = reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(ws) + counter_bytes(nk));
    cudaError_t e = bin_core(cell, species, n, n_cells, n_species, w, perm, offsets, ws, reinterpret_cast<int32_t*>(keys),
                             status, st, launches);
    if (e != cudaSuccess || n <= kWarpSeg) return e;
    const int32_t* large = large_list(ws, nk);  // the segments above kWarpSeg, already in index order
    k_segsort_w<<<grid_for(n / (kWarpSeg + 1) * kBinThreads, kBinThreads), kBinThreads, 0, st>>>(offsets, large, w,
                                                                                               perm, keys);
    *launches += 1;
    return cudaGetLastError();
}

// Device address of g_bin_static_scratch on the current device. The host-side name is only a stand-in, so the
// address is looked up once per device (with that device current) and cached.
static void* static_bin_scratch(int* err)
{
    static std::mutex mu;
    static void* addr[256] = {nullptr};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) {
        *err = 1;
        return nullptr;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_bin_static_scratch) != cudaSuccess || !p) {
            *err = 1;
            return nullptr;
        }
        addr[dev] = p;
    }
    *err = 0;
    return addr[dev];
}

int64_t static_bin_max_keys() { return kStaticBinKeys; }

cudaError_t launch_bin_static(const int32_t* cell, const int32_t* species, int64_t n, int32_t n_cells,
                              int32_t n_species, int32_t* perm, int64_t* offsets, cudaStream_t st)
{
    int err = 0;
    void* ws = static_bin_scratch(&err);
    if (err) return cudaErrorInvalidSymbol;
    int64_t launches = 0;
    // bin_core clears both counter arrays on the stream before its kernels; no place array and no status word
    // (out-of-range particles are dropped, visible as offsets[last] < n)
    return bin_core(cell, species, n, n_cells, n_species, nullptr, perm, offsets, ws, nullptr, nullptr, st, &launches);
}

cudaError_t launch_gather(const void* in, const int32_t* perm, int64_t n, int elem_bytes, void* out, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    const int g = grid_for(n, kBinThreads);
    if (elem_bytes == 8) {
        const auto kernel = n < kStreamDoubles ? k_gather<uint64_t, true> : k_gather<uint64_t, false>;
        kernel<<<g, kBinThreads, 0, st>>>(reinterpret_cast<const uint64_t*>(in), perm, n, reinterpret_cast<uint64_t*>(out));
    } else {
        k_gather<uint32_t, true><<<g, kBinThreads, 0, st>>>(reinterpret_cast<const uint32_t*>(in), perm, n,
                                                            reinterpret_cast<uint32_t*>(out));
    }
    return cudaGetLastError();
}

}  // namespace mcc
