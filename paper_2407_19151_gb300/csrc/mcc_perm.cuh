// Random permutations of a cell's species segments by one CTA (kThreads threads), shared by the one-CTA step kernel and the
// adjoint.
#pragma once

#include "mcc_device.cuh"

namespace mcc {

// Random permutations of the interaction's one or two species segments: local indices ordered by their 64-bit
// Philox keys (44 random bits above the index). The random bits are uniform, so a counting sort on their top
// log2(B) bits (B = next power of two >= n buckets) already places almost every key; each bucket holding several
// keys is finished by an insertion sort on the full key. The result is the sort by full key (keys are distinct).
// One Philox block gives the keys of two consecutive indices, so each thread draws for a pair. The permutation is
// stored as cell-local particle indices (segment start included).
// keys, perm: [cell]; cnt: bucket counters, next_pow2(na) + next_pow2(nb) entries; iscan: shared, kWarps + 1 values.
__device__ inline void cta_permutations(const RngKey& rng, uint32_t step, uint64_t* keys, uint32_t* cnt, int32_t* perm,
                                        int* iscan, int c, uint32_t ictr, int nside, int a0, int na, int b0, int nb)
{
    const int s0v[2] = {a0, b0}, nv[2] = {na, nb};
    int lgB[2] = {0, 0}, Bv[2] = {0, 0};
    for (int side = 0; side < nside; ++side) {
        while ((1 << lgB[side]) < nv[side]) ++lgB[side];
        Bv[side] = 1 << lgB[side];
    }
    const int base1 = Bv[0];
    const int L = Bv[0] + (nside > 1 ? Bv[1] : 0);
    for (int side = 0; side < nside; ++side) {
        const int s0 = s0v[side], n = nv[side];
        const uint32_t tag = side ? kTagPermB : kTagPermA;
        for (int h = threadIdx.x; 2 * h < n; h += kThreads) {
            const uint4 r = draw_at(rng, step, (uint32_t)h, (uint32_t)c, ictr, tag);
            keys[s0 + 2 * h] = ((((uint64_t)r.x << 32) | r.y) & ~kPermMask) | (uint64_t)(2 * h);
            if (2 * h + 1 < n) keys[s0 + 2 * h + 1] = ((((uint64_t)r.z << 32) | r.w) & ~kPermMask) | (uint64_t)(2 * h + 1);
        }
    }
    for (int b = threadIdx.x; b < L; b += kThreads) cnt[b] = 0;
    __syncthreads();
    for (int side = 0; side < nside; ++side) {
        const int base = side ? base1 : 0;
        for (int q = threadIdx.x; q < nv[side]; q += kThreads) {
            const uint64_t k = keys[s0v[side] + q];
            const int b = lgB[side] ? (int)(k >> (64 - lgB[side])) : 0;
            atomicAdd(&cnt[base + b], 1u);
        }
    }
    __syncthreads();
    // exclusive scan over both sides' buckets (side 1's positions are offset by na)
    {
        const int chunk = (L + kThreads - 1) / kThreads;
        const int lo = threadIdx.x * chunk, hi = min(L, lo + chunk);
        int local = 0;
        for (int b = lo; b < hi; ++b) local += (int)cnt[b];
        int total;
        int run = block_exclusive_scan<int>(local, iscan, total);
        for (int b = lo; b < hi; ++b) {
            const int x = (int)cnt[b];
            cnt[b] = (uint32_t)run;
            run += x;
        }
    }
    __syncthreads();
    for (int side = 0; side < nside; ++side) {
        const int base = side ? base1 : 0, off = side ? na : 0, s0 = s0v[side];
        for (int q = threadIdx.x; q < nv[side]; q += kThreads) {
            const uint64_t k = keys[s0 + q];
            const int b = lgB[side] ? (int)(k >> (64 - lgB[side])) : 0;
            const int pos = (int)atomicAdd(&cnt[base + b], 1u) - off;
            perm[s0 + pos] = s0 + q;
        }
    }
    __syncthreads();
    // cnt[b] now holds the end of bucket b: finish buckets with several keys
    for (int side = 0; side < nside; ++side) {
        const int base = side ? base1 : 0, off = side ? na : 0, s0 = s0v[side];
        for (int b = threadIdx.x; b < Bv[side]; b += kThreads) {
            const int end = (int)cnt[base + b] - off;
            const int start = b ? (int)cnt[base + b - 1] - off : 0;
            for (int x = start + 1; x < end; ++x) {
                const int v = perm[s0 + x];
                const uint64_t kv = keys[v];
                int y = x - 1;
                while (y >= start && keys[perm[s0 + y]] > kv) {
                    perm[s0 + y + 1] = perm[s0 + y];
                    --y;
                }
                perm[s0 + y + 1] = v;
            }
        }
    }
    __syncthreads();
}

}  // namespace mcc
