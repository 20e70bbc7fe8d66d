// Stable radix sort of (32-bit key, 32-bit value) pairs, used while a graph is
// loaded: one least-significant-digit pass per 8 key bits.
//
// A pass is bound by memory (it reads each key twice and each value once and
// writes both), so the tile is sized for long coalesced runs: a block ranks
// 8,192 pairs in shared memory and writes them out sorted by digit, about 32
// consecutive pairs per digit.  Ranks are stable because every warp owns 512
// consecutive pairs and goes through them 32 at a time: lanes with the same digit
// find one another with a match, and a per-warp counter per digit carries over.
// The reverse adjacency of 20 M edges (three passes) takes 0.75 ms; a bitonic
// sort of 2^25 64-bit keys in 120 launches took 10.9 ms.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mhr_util.cuh"

namespace mhr {

constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 16;  // pairs per thread
constexpr int kSortTile = kSortThreads * kSortItems;

struct SortSmem {
    uint32_t key[kSortTile], val[kSortTile];
    uint32_t cnt[kSortWarps][256];  // per warp: running count, then first rank, of a digit
    uint32_t gbase[256];            // output position of the tile's digit run, minus its tile position
    uint32_t lbase[256];            // tile position of the digit run
    uint32_t red[33];
};

// counts[digit * tiles + tile] of digit (key >> shift) & 255
static __global__ void __launch_bounds__(kSortThreads)
    k_sort_count(const uint32_t* __restrict__ keys, uint32_t n, int shift, uint32_t tiles, uint32_t* __restrict__ counts) {
    __shared__ uint32_t hist[256];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0u;
    __syncthreads();
    const uint64_t base = static_cast<uint64_t>(blockIdx.x) * kSortTile;
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const uint64_t i = base + j * kSortThreads + threadIdx.x;
        if (i < n) atomicAdd(&hist[(keys[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < 256; d += blockDim.x)
        counts[static_cast<uint64_t>(d) * tiles + blockIdx.x] = hist[d];
}

// vals_in == NULL: value i is i; keys_out == NULL: only the values are written;
// offsets == NULL: few tiles, whose counts every block adds up itself (none needed
// for a single tile)
static __global__ void __launch_bounds__(kSortThreads)
    k_sort_scatter(const uint32_t* __restrict__ keys_in, const uint32_t* __restrict__ vals_in, uint32_t n, int shift,
                   uint32_t tiles, const int64_t* __restrict__ offsets, const uint32_t* __restrict__ counts,
                   uint32_t* __restrict__ keys_out,
                   uint32_t* __restrict__ vals_out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SortSmem& sm = *reinterpret_cast<SortSmem*>(smem_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t base = static_cast<uint64_t>(blockIdx.x) * kSortTile;
    const uint32_t m = static_cast<uint32_t>(n - base < kSortTile ? n - base : kSortTile);
    for (int i = threadIdx.x; i < kSortWarps * 256; i += blockDim.x) (&sm.cnt[0][0])[i] = 0u;
    __syncthreads();
    uint32_t key[kSortItems], val[kSortItems], rank[kSortItems];
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const uint32_t i = warp * (32 * kSortItems) + j * 32 + lane;
        key[j] = i < m ? keys_in[base + i] : 0u;
        val[j] = i < m ? (vals_in ? vals_in[base + i] : static_cast<uint32_t>(base + i)) : 0u;
    }
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const bool live = warp * (32 * kSortItems) + j * 32 + lane < m;
        const uint32_t d = live ? (key[j] >> shift) & 255u : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        uint32_t c = 0u;
        if (live) c = sm.cnt[warp][d];
        rank[j] = c + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
        if (live && lane == __ffs(peers) - 1) sm.cnt[warp][d] = c + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    uint32_t tot = 0u;
    if (threadIdx.x < 256) {
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) {
            const uint32_t c = sm.cnt[w][threadIdx.x];
            sm.cnt[w][threadIdx.x] = tot;
            tot += c;
        }
    }
    const uint32_t lb = block_excl_scan<uint32_t>(tot, sm.red, nullptr);
    if (offsets) {
        if (threadIdx.x < 256)
            sm.gbase[threadIdx.x] =
                static_cast<uint32_t>(offsets[static_cast<uint64_t>(threadIdx.x) * tiles + blockIdx.x]) - lb;
    } else if (tiles == 1) {
        if (threadIdx.x < 256) sm.gbase[threadIdx.x] = 0u;
    } else {  // block-uniform
        uint32_t all = 0u, before = 0u;
        if (threadIdx.x < 256)
            for (uint32_t t = 0; t < tiles; ++t) {
                const uint32_t c = counts[threadIdx.x * tiles + t];
                all += c;
                if (t < blockIdx.x) before += c;
            }
        const uint32_t first = block_excl_scan<uint32_t>(all, sm.red, nullptr);
        if (threadIdx.x < 256) sm.gbase[threadIdx.x] = first + before - lb;
    }
    if (threadIdx.x < 256) sm.lbase[threadIdx.x] = lb;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        if (warp * (32 * kSortItems) + j * 32 + lane < m) {
            const uint32_t d = (key[j] >> shift) & 255u;
            const uint32_t p = sm.lbase[d] + sm.cnt[warp][d] + rank[j];
            sm.key[p] = key[j];
            sm.val[p] = val[j];
        }
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < m; i += blockDim.x) {
        const uint32_t k = sm.key[i];
        const uint32_t p = sm.gbase[(k >> shift) & 255u] + i;  // modulo 2^32
        if (keys_out) keys_out[p] = k;
        vals_out[p] = sm.val[i];
    }
}

// Scratch of a sort of up to n pairs (device memory of the caller)
struct SortScratch {
    uint32_t* key[2];   // [n] each
    uint32_t* val[2];   // [n] each
    uint32_t* counts;   // [256 * tiles]
    int64_t* offsets;   // [256 * tiles + 1]
    int64_t* n_counts;  // device copy of 256 * tiles
    int64_t* partials;  // kScanPartials, zero
};

// Up to this many tiles (131,072 pairs) a pass needs no scan of the counts, and one
// tile no counts: one or two launches instead of four, of about 3 us each when there is
// next to nothing to sort.
constexpr uint32_t kSortFewTiles = 16;

inline uint32_t sort_tiles(uint64_t n) { return static_cast<uint32_t>((n + kSortTile - 1) / kSortTile); }

// Sorts the pairs (keys[i], vals[i]) (vals == NULL: (keys[i], i)) by the low
// `bits` bits of the key, stable; *out is the sorted value list (one of s.val;
// vals may be the other one).  The input keys may be s.key[0] or s.key[1].
inline cudaError_t radix_sort_pairs(const uint32_t* keys, const uint32_t* vals, uint32_t n, int bits,
                                    const SortScratch& s, uint32_t** out, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_sort_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(sizeof(SortSmem)));
    if (e != cudaSuccess) return e;
    const uint32_t tiles = sort_tiles(n);
    int side = vals == s.val[0] || keys == s.key[0] ? 1 : 0;  // never in place
    for (int shift = 0; shift < bits || shift == 0; shift += 8) {
        const bool last = shift + 8 >= bits;
        const bool few = tiles <= kSortFewTiles;
        if (tiles > 1) k_sort_count<<<tiles, kSortThreads, 0, st>>>(keys, n, shift, tiles, s.counts);
        if (!few) {
            e = device_excl_scan<uint32_t>(s.counts, s.n_counts, s.partials, s.offsets, st);
            if (e != cudaSuccess) return e;
        }
        k_sort_scatter<<<tiles, kSortThreads, sizeof(SortSmem), st>>>(keys, vals, n, shift, tiles,
                                                                      few ? nullptr : s.offsets, s.counts,
                                                                      last ? nullptr : s.key[side], s.val[side]);
        keys = s.key[side];
        vals = s.val[side];
        side ^= 1;
    }
    *out = const_cast<uint32_t*>(vals);
    return cudaGetLastError();
}

}  // namespace mhr
