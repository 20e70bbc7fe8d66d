// Threshold search of one query by one thread block, over the weight index.
//
// A path s -> u -> v -> t is a near slot (an edge of one endpoint's row), a
// middle edge of that slot's vertex and a far slot (an edge of the other
// endpoint's row).  The index keeps the fp32 weight of every edge and every row
// sorted by it, so a path's screening score fl(fl(w_near + w_mid) + w_far) needs
// no embedding, and the middle edges that can still matter are a prefix of each
// row: with `thr` a lower bound of the K-th best score, only edges with
// fl(w_near + w_mid) >= tau, tau just below thr - 2E - max w_far, are read.  The
// index also holds, per slot, p = w + (largest weight of a middle edge there) and,
// per vertex, the largest w and p of its row and the row's middle edges S, so
// nothing is computed per slot before the rows are filtered by p.
//
//   seed    the first middle edges of the rows with the largest p, joined with the
//           far slots of largest p: the K-th best score found is a first threshold
//           (any set of paths gives a valid one).  Its candidates are dropped.
//   side    with a threshold a side costs the edges in its prefixes, which S says
//           little about: both are estimated from a few ranks kept per row, the
//           smaller is scanned.  While that is many more than were read so far,
//           probes read about a sixteenth of them (the best ones) for a better
//           threshold first
//   far     a shared-memory table of 65,536 bytes, indexed by a hash of the vertex:
//           the largest weight of the far slots there, rounded up to 254 levels.  An
//           edge passes when fl(w_near + w_mid) + that weight can reach thr: one
//           byte load and a compare, and about one edge in a hundred passes
//   main    near slots with p >= tau in natural order, gathered into batches; each
//           thread finds its slot's prefix, the prefixes are cut into pieces of up
//           to 32 edges, one lane per piece reads whole 32-byte sectors (four
//           edges).  A lane per piece needs the owner of an edge once per piece; a
//           warp over consecutive edges, which needs it per 32 edges, took 180
//           instructions per 32 edges, most of them for that.  An edge that passes the far
//           table is looked up in the endpoint's row (sorted by vertex), every path
//           at or above thr - 2E is kept, and the threshold rises between slices
//
// What bounds it: latency (a few dependent loads and barriers per phase) and the
// issue of the scan.  Two 512-thread blocks per SM fill one another's barriers
// when there are queries enough for all SMs, one 1,024-thread block shortens a
// query's phases otherwise.  Measured, whole call, against the join that reads
// and weighs every edge of every row whose bound reaches the band: 4,096 queries
// over 10 M vertices and 200 M edges (128 bf16 values, K = 50) 112.7 -> 3.8 ms
// (4 % of the middle edges read); 256 over 1 M vertices and 20 M edges (256 fp32
// values, DistMult, K = 100) 3.2 -> 0.72 ms, 64 of them (128 values, TransE)
// 1.6 -> 0.28 ms.
//
// A query whose candidates overflow the buffers (ties) or whose prefixes are very
// long (fewer than K paths, a hub on both sides) is handed back (redo): one without a
// threshold after `alone` middle edges, which the join's blocks read together sooner.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mhr_internal.cuh"
#include "mhr_query.cuh"
#include "mhr_util.cuh"

namespace mhr {

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ float neg_inf() { return __int_as_float(0xff800000); }

// thr - 2E rounded toward -inf, as float (conservative keep threshold)
__device__ __forceinline__ float keep_threshold(uint32_t key, double two_err) {
    if (key == 0u) return neg_inf();
    return __double2float_rd(__dsub_rd(static_cast<double>(key2f(key)), two_err));
}

// K-th largest order key among n keys (1 <= K <= n) by 4-pass radix select.
// key_at(i) gives key i; all threads call; hist has 256 slots.
template <typename KeyAt>
__device__ uint32_t block_select_kth(KeyAt key_at, int64_t n, int K, uint32_t* hist, uint32_t* bcast) {
    uint32_t prefix = 0, mask = 0;
    uint32_t remaining = static_cast<uint32_t>(K);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int pass = 0; pass < 4; ++pass) {
        const int shift = 24 - 8 * pass;
        for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
        __syncthreads();
        for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
            uint32_t k = key_at(i);
            if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (wid == 0) {
            // lane l owns bins 255-8l .. 248-8l (descending)
            uint32_t c = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) c += hist[255 - 8 * lane - j];
            uint32_t cum = warp_incl_scan(c);
            unsigned b = __ballot_sync(0xffffffffu, cum >= remaining);
            int L = __ffs(b) - 1;
            if (lane == L) {
                uint32_t before = cum - c;
                for (int j = 0; j < 8; ++j) {
                    uint32_t bin = 255 - 8 * lane - j;
                    uint32_t h = hist[bin];
                    if (before + h >= remaining) {
                        bcast[0] = prefix | (bin << shift);
                        bcast[1] = remaining - before;
                        break;
                    }
                    before += h;
                }
            }
        }
        __syncthreads();
        prefix = bcast[0];
        remaining = bcast[1];
        mask |= 255u << shift;
        __syncthreads();
    }
    return prefix;
}

constexpr int kSrCand = 1024;        // candidates in shared memory (further ones in `spill`)
constexpr int kSrHash = 8192;        // slots of the seed's far table (vertex -> weight)
constexpr int kSrHashMax = 6144;     // far slots it takes
constexpr uint32_t kSrSegment = 2048;  // near slots gathered at a time
constexpr uint32_t kSrSmall = 4096;  // middle edges below which no seed is worth its phases
// Middle edges worth a better threshold first: a probe costs about 60,000.  Over four sets of
// inputs of each of three batches (64, 256 and 4,096 queries) 98,304 is 1.5 % slower in
// the mean and faster on one of the twelve; 60,000 and 250,000 were slower as well.
constexpr uint32_t kSrProbe = 160000;
constexpr uint32_t kSrSlice = 16384; // middle edges between threshold updates
constexpr uint32_t kSrSample = 4096; // slots looked at for a cut
constexpr uint32_t kSrRuns = 48;     // runs of 32 slots looked at for an estimate
constexpr uint32_t kSrOther = 32768; // middle edges below which the other side is not estimated
constexpr int kSrRank = 512;         // candidates up to which the K-th best is found by comparing pairs
constexpr uint32_t kSrNone = 0xffffffffu;
constexpr int kSrQueue = 256;        // edges that passed the far table, in shared memory
constexpr int kSrSpillQueue = 8192;  // and past it, per block

// one endpoint's row and the middle adjacency seen from its slots
struct SearchSide {
    const uint32_t* col;   // slots' vertices (the row of s, or the in-row of t)
    const uint16_t* rel;
    const float* w;
    const float* p;        // w + largest middle weight at the slot's vertex (-inf: it has no middle edge)
    const VertexRec* rec;  // per vertex: its middle row
    const uint2* se;
    const uint16_t* sr;
    uint32_t n;
    float maxw, maxp;      // largest w and p of the row (excluded slots included)
    unsigned long long S;  // middle edges of its slots
};

template <int NT>
struct SearchSmem {
    Cand cand[kSrCand];
    uint32_t tab[2 * kSrHash];  // seed: keys, then weight keys; else 65,536 bytes
    uint32_t list[NT + kSrSegment];
    uint32_t ea[NT], eb[NT], pre[NT], ei[NT];  // a batch: first and end edge, pieces before, slot
    float ew[NT];                              // its near weight
    SrPass queue[kSrQueue];
    uint32_t hist[256];
    uint32_t bc[4];
    unsigned long long red[33];
    SearchSide side[2];  // 0: row of s, 1: in-row of t
    uint32_t s, t;
    int K, part_count, part_index;
    const uint8_t* cons;
    const uint8_t* vtypes;
    int R;
    double two_err;
    Cand* spill;
    SrPass* spill_queue;
    int cap;             // candidates in all
    int fwd, rowmode;    // rowmode: no far table, every edge is looked up in the row
    int cand_cnt, list_cnt, ins, queue_cnt;
    int redo;
    uint32_t thr_key;
    float thr_keep, tau, maxf, cutp, err;
    float est;
    float far_p, far_w;  // far slots below either cannot reach thr_keep
    float top, step;     // byte table: code k > 0 is a weight of at most top - (255 - k) * step
    unsigned long long scanned, hits, paths, near_edges;
};

// The block's search state, at the start of its dynamic shared memory.  Every
// function names it itself: a reference passed to one that is not inlined would
// lose the shared address space.
extern __shared__ __align__(128) unsigned char sr_smem_raw[];
template <int NT>
__device__ __forceinline__ SearchSmem<NT>& sr_smem() {
    return *reinterpret_cast<SearchSmem<NT>*>(sr_smem_raw);
}

template <int NT>
__device__ __forceinline__ Cand& sr_cand(SearchSmem<NT>& sm, int i) {
    return i < kSrCand ? sm.cand[i] : sm.spill[i - kSrCand];
}

// whether slot i (vertex v) of a side may lie on a path
template <int NT>
__device__ __forceinline__ bool sr_slot_ok(const SearchSmem<NT>& sm, int sd, uint32_t i, uint32_t v) {
    bool ok = v != sm.s && v != sm.t;
    if (sd == 0 && sm.part_count > 1)
        ok = ok && v % static_cast<uint32_t>(sm.part_count) == static_cast<uint32_t>(sm.part_index);
    if (sm.cons && ok) {
        const int R = sm.R;
        ok = sm.cons[(sd ? 2 * R : 0) + sm.side[sd].rel[i]] != 0 && sm.cons[3 * R + (sd ? 256 : 0) + sm.vtypes[v]] != 0;
    }
    return ok;
}

// A p such that about `want` slots of the side lie at or above it, from up to
// kSrSample slots: whole runs of NT, evenly spaced (rows are sorted by vertex id,
// which says nothing of the weight).
template <int NT>
__device__ __noinline__ float sr_cut(int sd, uint32_t want) {
    SearchSmem<NT>& sm = sr_smem<NT>();
    const SearchSide& S = sm.side[sd];
    const uint32_t n = S.n;
    if (n <= want) return neg_inf();
    const uint32_t stride = (n + kSrSample - 1) / kSrSample;
    for (int i = threadIdx.x; i < 256; i += NT) sm.hist[i] = 0u;
    if (threadIdx.x == 0) sm.bc[0] = 0xffffffffu;
    __syncthreads();
    // the least p of the first run bounds the levels from below
    {
        const float p = threadIdx.x < n ? S.p[threadIdx.x] : neg_inf();
        const uint32_t k = __reduce_min_sync(0xffffffffu, p == neg_inf() ? 0xffffffffu : f2key(p));
        if ((threadIdx.x & 31) == 0) atomicMin(&sm.bc[0], k);
    }
    __syncthreads();
    const float hi = S.maxp, lo = sm.bc[0] == 0xffffffffu ? hi : key2f(sm.bc[0]);
    const float scale = hi > lo ? 256.f / (hi - lo) : 0.f;
    uint32_t seen = 0u;
    constexpr int U = 4;  // runs in flight
    for (uint64_t base = 0; base < n; base += static_cast<uint64_t>(U) * NT * stride) {
        float p[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t b = base + static_cast<uint64_t>(u) * NT * stride, i = b + threadIdx.x;
            p[u] = i < n ? S.p[i] : neg_inf();
            if (b < n) seen += static_cast<uint32_t>(min(static_cast<uint64_t>(NT), n - b));
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (p[u] != neg_inf()) atomicAdd(&sm.hist[max(0, min(255, static_cast<int>((hi - p[u]) * scale)))], 1u);
    }
    const float share = static_cast<float>(want) * static_cast<float>(seen) / static_cast<float>(n);
    __syncthreads();
    if (threadIdx.x < 32) {
        const int l = threadIdx.x;
        uint32_t c[8], tot = 0u;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            c[j] = sm.hist[8 * l + j];
            tot += c[j];
        }
        uint32_t cum = warp_incl_scan(tot) - tot;
        int at = 256;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            cum += c[j];
            if (static_cast<float>(cum) >= share && at == 256) at = 8 * l + j;
        }
        at = __reduce_min_sync(0xffffffffu, at);
        if (l == 0) sm.cutp = scale > 0.f && at < 255 ? hi - static_cast<float>(at + 1) / scale : neg_inf();
    }
    __syncthreads();
    return sm.cutp;
}

__device__ __forceinline__ uint32_t sr_mix(uint32_t v) { return v * 2654435769u; }

// The seed's far table: up to kSrHashMax far slots with p >= far_p, vertex -> key
// of its largest such weight.
template <int NT>
__device__ __noinline__ void sr_build_hash() {
    SearchSmem<NT>& sm = sr_smem<NT>();
    for (int i = threadIdx.x; i < kSrHash; i += NT) {
        sm.tab[i] = kSrNone;
        sm.tab[kSrHash + i] = 0u;
    }
    if (threadIdx.x == 0) sm.ins = 0;
    __syncthreads();
    const SearchSide& F = sm.side[sm.fwd];
    const float fp = sm.far_p;
    const uint32_t n = F.n;
    constexpr int U = 4;  // slots in flight per thread
    for (uint32_t i0 = threadIdx.x; i0 < n; i0 += U * NT) {
        float p[U], w[U];
        uint32_t v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t i = i0 + u * NT;
            const bool in = i < n && i >= i0;
            p[u] = in ? F.p[i] : neg_inf();
            w[u] = in ? F.w[i] : 0.f;
            v[u] = in ? F.col[i] : 0u;
        }
#pragma unroll 1
        for (int u = 0; u < U; ++u) {
            const float pu = u == 0 ? p[0] : u == 1 ? p[1] : u == 2 ? p[2] : p[3];
            if (pu == neg_inf() || pu < fp) continue;
            const uint32_t vu = u == 0 ? v[0] : u == 1 ? v[1] : u == 2 ? v[2] : v[3];
            const uint32_t k = f2key(u == 0 ? w[0] : u == 1 ? w[1] : u == 2 ? w[2] : w[3]);
            if (!sr_slot_ok(sm, sm.fwd, i0 + u * NT, vu)) continue;
            if (atomicAdd(&sm.ins, 1) >= kSrHashMax) break;
            uint32_t h = sr_mix(vu) >> 19;
            for (;;) {
                const uint32_t old = atomicCAS(&sm.tab[h], kSrNone, vu);
                if (old == kSrNone || old == vu) {
                    atomicMax(&sm.tab[kSrHash + h], k);
                    break;
                }
                h = (h + 1) & (kSrHash - 1);
            }
        }
        if (n - i0 <= U * NT) break;  // before i0 can wrap
    }
    __syncthreads();
}
static_assert(kSrHash == 1 << 13 && kSrHashMax < kSrHash, "hash bits and load");

// thr_keep - best - E, rounded down: a slot or edge whose own part of a path's
// score is below it cannot reach thr_keep with the other part at most `best`.  E,
// the proven bound of a path's screening error, covers the fp32 additions.
template <int NT>
__device__ __forceinline__ float sr_part(const SearchSmem<NT>& sm, float best) {
    return __fsub_rd(__fsub_rd(sm.thr_keep, best), sm.err);
}

template <int NT>
__device__ __forceinline__ void sr_set_threshold(SearchSmem<NT>& sm) {  // thread 0
    sm.thr_keep = keep_threshold(sm.thr_key, sm.two_err);
    sm.tau = sr_part(sm, sm.maxf);
}

// scan from the row of s (fwd 1, the far side is the in-row of t) or the other way
template <int NT>
__device__ __forceinline__ void sr_face(int fwd) {
    SearchSmem<NT>& sm = sr_smem<NT>();
    __syncthreads();
    if (threadIdx.x == 0) {
        sm.fwd = fwd;
        sm.maxf = sm.side[fwd].maxw;
        sr_set_threshold(sm);
    }
    __syncthreads();
}

// The byte table of the far slots that can still reach the threshold; rowmode
// when there are so few middle edges that reading the far row costs more.  A probe
// takes only the slots with p >= least_p.
template <int NT>
__device__ __noinline__ void sr_build_far(float least_p) {
    SearchSmem<NT>& sm = sr_smem<NT>();
    __syncthreads();
    const SearchSide& N = sm.side[1 - sm.fwd];
    const SearchSide& F = sm.side[sm.fwd];
    const bool row = N.S * 8 < F.n;
    if (threadIdx.x == 0) {
        sm.far_p = sr_part(sm, N.maxw);
        sm.far_w = sr_part(sm, N.maxp);
        sm.rowmode = row ? 1 : 0;
        const float span = F.maxw - sm.far_w;
        sm.top = F.maxw;
        // a level is never finer than the rounding of the scores it is compared with
        sm.step = span < 1e30f ? fmaxf(span * (1.f / 254.f), fmaxf(sm.err, 1e-30f)) : 1e30f;
    }
    if (!row)
        for (int i = threadIdx.x; i < 2 * kSrHash; i += NT) sm.tab[i] = 0u;
    __syncthreads();
    if (row) return;
    const float fp = fmaxf(sm.far_p, least_p), fw = sm.far_w, top = sm.top, inv = 1.f / sm.step;
    const uint32_t n = F.n;
    constexpr int U = 4;
    for (uint32_t base = 0; base < n; base += min(n - base, static_cast<uint32_t>(U * NT))) {  // uniform
        const uint32_t i0 = base + threadIdx.x;
        float p[U], w[U];
        uint32_t v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t i = i0 + u * NT;
            p[u] = i < n ? F.p[i] : neg_inf();
            w[u] = i < n ? F.w[i] : neg_inf();
            v[u] = i < n ? F.col[i] : 0u;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool in = p[u] != neg_inf() && p[u] >= fp && w[u] >= fw && sr_slot_ok(sm, sm.fwd, i0 + u * NT, v[u]);
            const uint32_t k = in ? 255u - min(254u, static_cast<uint32_t>((top - w[u]) * inv)) : 0u;
            const uint32_t h = sr_mix(v[u]) >> 16, sh = (h & 3u) * 8u;
            uint32_t* word = sm.tab + (h >> 2);
            uint32_t old = in ? *reinterpret_cast<volatile uint32_t*>(word) : 0u;
            while (((old >> sh) & 255u) < k) {
                const uint32_t seen = atomicCAS(word, old, (old & ~(255u << sh)) | (k << sh));
                if (seen == old) break;
                old = seen;
            }
            __syncwarp();
        }
    }
    __syncthreads();
}
static_assert(2 * kSrHash * 4 == 65536, "one byte per 16-bit hash");

// first slot of vertex v in the far row, or the row's length
__device__ __forceinline__ uint32_t sr_row_find(const SearchSide& F, uint32_t v) {
    uint32_t lo = 0, hi = F.n;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__ldg(F.col + mid) < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// K-th best candidate -> threshold.  All threads call.
template <int NT>
__device__ __noinline__ void sr_select(int n) {
    SearchSmem<NT>& sm = sr_smem<NT>();
    if (n <= kSrRank) {  // fewer barriers than the radix passes
        for (int i = threadIdx.x; i < n; i += NT) {
            const float mine = sm.cand[i].s32;
            int above = 0, same = 0;
#pragma unroll 8
            for (int j = 0; j < n; ++j) {
                const float x = sm.cand[j].s32;
                above += x > mine ? 1 : 0;
                same += x == mine ? 1 : 0;
            }
            if (above < sm.K && above + same >= sm.K) sm.bc[0] = f2key(mine);  // equal values, if several
        }
        __syncthreads();
        if (threadIdx.x == 0 && sm.bc[0] > sm.thr_key) {
            sm.thr_key = sm.bc[0];
            sr_set_threshold(sm);
        }
        __syncthreads();
        return;
    }
    const uint32_t key = block_select_kth([&](int64_t i) { return f2key(sr_cand(sm, static_cast<int>(i)).s32); }, n,
                                          sm.K, sm.hist, sm.bc);
    if (threadIdx.x == 0 && key > sm.thr_key) {
        sm.thr_key = key;
        sr_set_threshold(sm);
    }
    __syncthreads();
}

// candidates below thr_keep are dropped
template <int NT>
__device__ __noinline__ void sr_compact(int n) {
    SearchSmem<NT>& sm = sr_smem<NT>();
    const float thr = sm.thr_keep;
    int w = 0;
    for (int base = 0; base < n; base += NT) {
        const int i = base + threadIdx.x;
        Cand c;
        bool keep = false;
        if (i < n) {
            c = sr_cand(sm, i);
            keep = c.s32 >= thr;
        }
        int tot;
        const int pos = block_excl_scan(keep ? 1 : 0, reinterpret_cast<int*>(sm.red), &tot);
        if (keep) sr_cand(sm, w + pos) = c;
        w += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) sm.cand_cnt = w;
    __syncthreads();
}

template <int NT>
__device__ __forceinline__ void sr_keep(SearchSmem<NT>& sm, float s32, uint32_t near_i, uint32_t far_i, uint32_t r2) {
    const int slot = atomicAdd(&sm.cand_cnt, 1);
    if (slot < sm.cap) {
        Cand cd;
        cd.s32 = s32;
        cd.a_idx = sm.fwd ? near_i : far_i;
        cd.c_idx = sm.fwd ? far_i : near_i;
        cd.r2 = static_cast<uint16_t>(r2);
        cd.pad = 0;
        sr_cand(sm, slot) = cd;
    }
}

// Middle edge e to vertex v over near slot i, which passed the far table: keeps
// every path over it at or above thr_keep.  Returns their number.
template <int NT>
__device__ __noinline__ uint32_t sr_edge(uint32_t i, uint32_t e, uint32_t v, float phi, float thr_keep) {
    SearchSmem<NT>& sm = sr_smem<NT>();
    const SearchSide& N = sm.side[1 - sm.fwd];
    const SearchSide& F = sm.side[sm.fwd];
    uint32_t c = sr_row_find(F, v), paths = 0u;
    if (c >= F.n || F.col[c] != v) return 0u;
    const uint32_t r2 = N.sr[e];
    if (sm.cons && !sm.cons[sm.R + r2]) return 0u;
    const int fsd = sm.fwd;
    for (; c < F.n && F.col[c] == v; ++c) {
        const float s32 = __fadd_rn(phi, F.w[c]);
        if (!(s32 >= thr_keep) || !sr_slot_ok(sm, fsd, c, v)) continue;
        ++paths;
        sr_keep(sm, s32, i, c, r2);
    }
    return paths;
}

// Gathers near slots with p >= cut from `next` on into sm.list, at least NT of
// them unless the row ends.  Returns their number.
template <int NT>
__device__ __noinline__ int sr_gather(float cut, uint32_t& next) {
    SearchSmem<NT>& sm = sr_smem<NT>();
    const SearchSide& N = sm.side[1 - sm.fwd];
    const int lane = threadIdx.x & 31;
    const uint32_t nN = N.n;
    __syncthreads();  // the list and its count are no longer read
    if (threadIdx.x == 0) sm.list_cnt = 0;
    __syncthreads();
    for (;;) {
        float p[kSrSegment / NT];
#pragma unroll
        for (uint32_t j = 0; j < kSrSegment / NT; ++j) {
            const uint32_t i = next + j * NT + threadIdx.x;
            p[j] = i < nN ? N.p[i] : neg_inf();
        }
#pragma unroll
        for (uint32_t j = 0; j < kSrSegment / NT; ++j) {
            const uint32_t i = next + j * NT + threadIdx.x;
            const bool act = p[j] != neg_inf() && p[j] >= cut;
            const unsigned b = __ballot_sync(0xffffffffu, act);
            if (!b) continue;
            int base = 0;
            if (lane == 0) base = atomicAdd(&sm.list_cnt, __popc(b));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (act) sm.list[base + __popc(b & lanemask_lt())] = i;
        }
        next = nN - next > kSrSegment ? next + kSrSegment : nN;
        __syncthreads();
        const int cnt = sm.list_cnt;
        if (cnt >= NT || next >= nN) return cnt;
        __syncthreads();  // the count is read before the next segment adds to it
    }
}

// Estimate of the near side's middle edges at or above tau, from the kept ranks of
// up to kSrRuns * 32 slots' rows (a row's edges between two known ranks are taken as
// spread evenly between their weights; past the last one the fall of the weight
// per factor of eight is extrapolated).  *level: about a sixteenth of them lie
// above it.
template <int NT>
__device__ __noinline__ float sr_estimate(float* level) {
    SearchSmem<NT>& sm = sr_smem<NT>();
    constexpr int kLevels = 64;
    const SearchSide& N = sm.side[1 - sm.fwd];
    const float tau = sm.tau, top = N.maxp;
    const float scale = top > tau ? kLevels / (top - tau) : 0.f;
    // evenly spaced runs, a run per warp: what it costs is the chain of loads and the
    // counters' conflicts of every slot (35,000 cycles for 4,096 slots)
    const uint32_t runs = (N.n + 31) >> 5, stride = (runs + kSrRuns - 1) / kSrRuns, visits = (runs + stride - 1) / stride;
    // counts in units that keep every sum below 2^32
    const float unit = static_cast<float>(N.S) > 1e9f ? 1e9f / static_cast<float>(N.S) : 1.f;
    __syncthreads();
    for (int i = threadIdx.x; i < kLevels; i += NT) sm.hist[i] = 0u;
    __syncthreads();
    for (uint32_t v = threadIdx.x >> 5; v < visits; v += NT / 32) {
        const uint32_t i = v * stride * 32u + (threadIdx.x & 31);
        const bool in = i < N.n;
        const float pi = in ? N.p[i] : neg_inf(), wn = in ? N.w[i] : 0.f;
        const uint32_t u = in ? N.col[i] : 0u;
        if (pi >= tau && pi != neg_inf()) {
            const VertexRec rec = N.rec[u];
            const float deg = static_cast<float>(rec.deg);
            float r0 = 0.f, f0 = __fadd_rn(wn, rec.maxw), r1 = 4.f, fall = 0.f;
#pragma unroll 1
            for (int k = 0; k < 15 && r0 < deg; ++k) {
                const float wk = k == 0 ? rec.rank[0] : k == 1 ? rec.rank[1] : k == 2 ? rec.rank[2] : rec.rank[3];
                float f1;
                if (k < 4 && wk != neg_inf()) f1 = __fadd_rn(wn, wk);
                else f1 = fall > 0.f ? f0 - fall : f0 - 0.25f * (top - tau);
                float m = fminf(r1, deg) - r0, fe = f1;
                if (f1 < tau) {
                    const float part = f0 > f1 ? (f0 - tau) / (f0 - f1) : 1.f;
                    m *= part * part;
                    fe = tau;
                }
                atomicAdd(&sm.hist[max(0, min(kLevels - 1, static_cast<int>((top - 0.5f * (f0 + fe)) * scale)))],
                          static_cast<uint32_t>(m * unit) + 1u);
                if (f1 < tau) break;
                fall = f0 - f1;
                r0 = r1;
                f0 = f1;
                r1 *= 8.f;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {  // two levels per lane
        const int l = threadIdx.x;
        const float c0 = static_cast<float>(sm.hist[2 * l]), c1 = static_cast<float>(sm.hist[2 * l + 1]);
        const float incl = warp_incl_scan(c0 + c1), tot = __shfl_sync(0xffffffffu, incl, 31);
        const float want = tot * (1.f / 16.f);
        const int at = incl - c1 >= want ? 2 * l : incl >= want ? 2 * l + 1 : kLevels - 1;
        const int b = __reduce_min_sync(0xffffffffu, at);
        if (l == 0) {
            sm.cutp = scale > 0.f ? top - static_cast<float>(b + 1) / scale : tau;
            sm.est = tot / unit * (static_cast<float>(runs) / static_cast<float>(visits));
        }
    }
    static_assert(kLevels == 64, "two levels per lane");
    __syncthreads();
    *level = sm.cutp;
    const float est = sm.est;
    __syncthreads();
    return est;
}

// four consecutive edges of a sorted row (one aligned 32-byte sector)
__device__ __forceinline__ void sr_load4(const uint2* se, uint32_t sector, uint2 (&x)[4]) {
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(x[0].x), "=r"(x[0].y), "=r"(x[1].x), "=r"(x[1].y), "=r"(x[2].x), "=r"(x[2].y), "=r"(x[3].x), "=r"(x[3].y)
        : "l"(se + static_cast<uint64_t>(sector) * 4));
}

// Joins the near slots' middle edges with the far table.
//   SEED      the first `limit` edges of the slots with p >= sm.cutp, until `budget`
//             edges are read, against the seed's table; the score of the best path
//             over each edge that joins is all that is kept
//   else      every edge at or above tau and `level`; past `budget` the scan ends
//             and, unless it is a probe, hands the query back
// Returns the edges read.
template <int NT, bool SEED>
__device__ __noinline__ unsigned long long sr_scan(bool probe, uint32_t limit, float level, unsigned long long budget) {
    SearchSmem<NT>& sm = sr_smem<NT>();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const SearchSide& N = sm.side[1 - sm.fwd];
    const bool row = !SEED && sm.rowmode;
    const uint2* __restrict__ se = N.se;
    const uint8_t* bytes = reinterpret_cast<const uint8_t*>(sm.tab);
    uint32_t hits = 0u, paths = 0u;
    uint32_t next = 0;
    unsigned long long read = 0ull;
    while (next < N.n) {
        const int cnt = sr_gather<NT>(SEED ? sm.cutp : fmaxf(sm.tau, level), next);
        for (int b0 = 0; b0 < cnt; b0 += NT) {
            const int nent = min(NT, cnt - b0);
            uint32_t ne = 0u, rs = 0u, i = 0u;
            float wn = 0.f;
            if (static_cast<int>(threadIdx.x) < nent) {
                i = sm.list[b0 + threadIdx.x];
                const uint32_t u = N.col[i];
                wn = N.w[i];
                const VertexRec rec = N.rec[u];
                const uint32_t deg = rec.deg;
                rs = rec.row;
                const float tau = fmaxf(sm.tau, level);
                if (SEED) {
                    ne = min(deg, limit);
                } else if (tau == neg_inf()) {
                    ne = deg;
                } else {
                    // between the kept ranks, then bisect: [0, lo) is at or above tau, hi is not (or the end)
                    uint32_t lo = 0u, hi = deg;
                    if (__fadd_rn(wn, rec.rank[0]) < tau) hi = min(deg, 4u);
                    else if (__fadd_rn(wn, rec.rank[1]) < tau) lo = 5u, hi = min(deg, 32u);
                    else if (__fadd_rn(wn, rec.rank[2]) < tau) lo = 33u, hi = min(deg, 256u);
                    else if (__fadd_rn(wn, rec.rank[3]) < tau) lo = 257u, hi = min(deg, 2048u);
                    else lo = 2049u;
                    while (lo < hi) {
                        const uint32_t mid = (lo + hi) >> 1;
                        if (__fadd_rn(wn, __uint_as_float(__ldg(&se[rs + mid].y))) >= tau) lo = mid + 1u;
                        else hi = mid;
                    }
                    ne = lo;
                }
                if (!sr_slot_ok(sm, 1 - sm.fwd, i, u)) ne = 0u;
            }
            unsigned long long total;
            block_excl_scan<unsigned long long>(ne, sm.red, &total);
            read += total;
            if (read > budget) {  // block-uniform
                read -= total;
                if (!SEED && !probe && threadIdx.x == 0) sm.redo = 1;
                next = N.n;
                break;
            }
            // pieces of 4 to 32 edges (whole sectors), at least two per thread when there are enough
            int psh = 2;
            while (psh < 5 && (total >> psh) > 4u * NT) ++psh;
            const uint32_t np = ne ? ((rs + ne - 1u) >> psh) - (rs >> psh) + 1u : 0u;
            uint32_t P;
            const uint32_t ex = block_excl_scan<uint32_t>(np, reinterpret_cast<uint32_t*>(sm.red), &P);
            sm.ea[threadIdx.x] = rs;
            sm.eb[threadIdx.x] = rs + ne;
            sm.pre[threadIdx.x] = static_cast<int>(threadIdx.x) < nent ? ex : 0xffffffffu;
            sm.ei[threadIdx.x] = i;
            sm.ew[threadIdx.x] = wn;
            __syncthreads();
            uint32_t sl = 0;
            while (sl < P) {
                const uint32_t slice = max(static_cast<uint32_t>(NT), (SEED ? ~0u : kSrSlice) >> psh);
                const uint32_t hi = P - sl > slice ? sl + slice : P;
                const float thr_keep = sm.thr_keep;
                // An edge passes when its far weight lies at most (phi - least) / step
                // levels below the largest, `least` being the phi that the largest
                // lifts to thr_keep; one level of slack for the rounding.
                const float inv = SEED || row ? 0.f : 1.f / sm.step, least = SEED ? 0.f : thr_keep - sm.top;
                const bool all = row || thr_keep == neg_inf();
                for (uint32_t c0 = sl + warp * 32; c0 < hi; c0 += NT) {  // one piece per lane
                    // row of the first piece among the batch's prefixes, then of each lane's
                    uint32_t lo = 0, span = nent;
                    while (span > 32) {
                        const uint32_t step = (span + 31) >> 5;
                        const uint32_t j = lane * step;
                        const bool le = j < span && sm.pre[lo + j] <= c0;
                        const uint32_t c = __popc(__ballot_sync(0xffffffffu, le));
                        const uint32_t nlo = (c - 1) * step;
                        span = min(step, span - nlo);
                        lo += nlo;
                    }
                    const bool le = lane < static_cast<int>(span) && sm.pre[lo + lane] <= c0;
                    lo += __popc(__ballot_sync(0xffffffffu, le)) - 1;
                    const uint32_t pc = c0 + lane;
                    const uint32_t jn = lo + 1 + lane;
                    const uint32_t nxt = jn < static_cast<uint32_t>(nent) ? sm.pre[jn] : 0xffffffffu;
                    uint32_t own = 0;
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1) {
                        const uint32_t pv = __shfl_sync(0xffffffffu, nxt, own + step - 1);
                        if (pv <= pc) own += step;
                    }
                    own += lo;
                    if (__shfl_sync(0xffffffffu, nxt, 31) <= pc) {
                        // more than 31 rows start here (rows without edges)
                        uint32_t a = lo + 32, b2 = nent;
                        while (a < b2) {
                            const uint32_t mid = (a + b2) >> 1;
                            if (sm.pre[mid] <= pc) a = mid + 1;
                            else b2 = mid;
                        }
                        own = a - 1;
                    }
                    if (pc >= hi) continue;
                    const uint32_t a = sm.ea[own], b = sm.eb[own];
                    const float w1 = sm.ew[own];
                    const uint32_t blk = (a >> psh) + (pc - sm.pre[own]);
                    const uint32_t e0 = max(a, blk << psh), e1 = ((b - 1u) >> psh) == blk ? b : (blk + 1u) << psh;
                    const uint32_t last = (e1 - 1u) >> 2;
#pragma unroll 2
                    for (uint32_t sec = e0 >> 2; sec <= last; ++sec) {
                        uint2 x[4];
                        sr_load4(se, sec, x);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t e = 4u * sec + j;
                            const bool in = e >= e0 && e < e1;
                            const float phi = __fadd_rn(w1, __uint_as_float(x[j].y));
                            const uint32_t m = sr_mix(x[j].x);
                            if (SEED) {
                                if (!in) continue;
                                uint32_t h = m >> 19, k = sm.tab[h];
                                while (k != x[j].x && k != kSrNone) {
                                    h = (h + 1) & (kSrHash - 1);
                                    k = sm.tab[h];
                                }
                                if (k == kSrNone) continue;
                                if (sm.cons && !sm.cons[sm.R + N.sr[e]]) continue;
                                sr_keep(sm, __fadd_rn(phi, key2f(sm.tab[kSrHash + h])), 0u, 0u, 0u);
                            } else {
                                const int code = bytes[m >> 16];
                                bool pass;
                                if (!all) pass = code >= max(1, 254 - __float2int_rd(__fsub_rn(phi, least) * inv));
                                else pass = row || code;
                                if (pass && in) {
                                    ++hits;
                                    const int at = atomicAdd(&sm.queue_cnt, 1);
                                    const SrPass y{sm.ei[own], e, x[j].x, phi};
                                    if (at < kSrQueue) sm.queue[at] = y;
                                    else if (at < kSrQueue + kSrSpillQueue) sm.spill_queue[at - kSrQueue] = y;
                                    else paths += sr_edge<NT>(sm.ei[own], e, x[j].x, phi, thr_keep);
                                }
                            }
                        }
                    }
                }
                sl = hi;
                __syncthreads();
                if (SEED) continue;
                // The passing edges, one per thread, once there are enough or the batch
                // ends: a look-up is a chain of some fifteen loads, which the few warps
                // that hold the best rows would run one by one.
                int nq = sm.queue_cnt;
                __syncthreads();
                if (nq == 0 || (sl < P && nq < kSrQueue)) continue;
                nq = min(nq, kSrQueue + kSrSpillQueue);
                for (int k = threadIdx.x; k < nq; k += NT) {
                    const SrPass x = k < kSrQueue ? sm.queue[k] : sm.spill_queue[k - kSrQueue];
                    paths += sr_edge<NT>(x.i, x.e, x.v, x.phi, sm.thr_keep);
                }
                __syncthreads();
                if (threadIdx.x == 0) sm.queue_cnt = 0;
                int nc = sm.cand_cnt;
                __syncthreads();
                if (nc > sm.cap && !probe) {  // ties: the buffers cannot hold the band
                    if (threadIdx.x == 0) sm.redo = 1;
                    __syncthreads();
                    return read;
                }
                nc = min(nc, sm.cap);
                if (nc >= sm.K && (sm.thr_key == 0u || nc >= sm.K + max(sm.K / 2, 64))) {
                    sr_select<NT>(nc);
                    sr_compact<NT>(nc);
                }
            }
        }
    }
    // work counters (a seed's and a probe's edges count as read; their paths are found again)
    hits = __reduce_add_sync(0xffffffffu, hits);
    paths = __reduce_add_sync(0xffffffffu, paths);
    if (lane == 0 && !SEED && !probe) {
        atomicAdd(&sm.hits, static_cast<unsigned long long>(hits));
        atomicAdd(&sm.paths, static_cast<unsigned long long>(paths));
    }
    if (threadIdx.x == 0) sm.scanned += read;
    __syncthreads();
    return read;
}

// middle edges of the near slots that may lie on a path
template <int NT>
__device__ __noinline__ unsigned long long sr_open_edges() {
    SearchSmem<NT>& sm = sr_smem<NT>();
    const SearchSide& N = sm.side[1 - sm.fwd];
    unsigned long long mine = 0ull;
#pragma unroll 4
    for (uint32_t base = 0; base < N.n; base += NT) {
        const uint32_t i = base + threadIdx.x;
        if (i >= N.n) break;
        const uint32_t u = N.col[i];
        if (sr_slot_ok(sm, 1 - sm.fwd, i, u)) mine += N.rec[u].deg;
        if (N.n - base <= NT) break;  // before base can wrap
    }
    return block_sum<unsigned long long>(mine, sm.red);
}

// The whole search of the query described by sm.s, t, K, two_err, cons, part_*,
// spill and cap.  Afterwards sm.redo tells whether the query is handed back;
// otherwise sr_cand(0 .. sm.cand_cnt) are all paths that can be among the K
// best.  heavy: middle edges after which the query is handed back; alone: the same
// while no threshold is known.
template <int NT>
__device__ void search_query(const DevGraph& g, unsigned long long heavy, unsigned long long alone) {
    SearchSmem<NT>& sm = sr_smem<NT>();
    if (threadIdx.x < 2) {
        SearchSide& S = sm.side[threadIdx.x];
        const bool a = threadIdx.x == 0;
        const int64_t* off = a ? g.off : g.roff;
        const uint32_t x = a ? sm.s : sm.t;
        const int64_t lo = off[x];
        const VertexRec rec = (a ? g.vout : g.vin)[x];
        S.n = static_cast<uint32_t>(off[x + 1] - lo);
        S.col = (a ? g.col : g.rcol) + lo;
        S.rel = (a ? g.rel : g.rrel) + lo;
        S.w = (a ? g.w : g.rw) + lo;
        S.p = (a ? g.p : g.rp) + lo;
        S.rec = a ? g.vout : g.vin;
        S.se = a ? g.se : g.rse;
        S.sr = a ? g.sr : g.rsr;
        S.maxw = rec.maxw;
        S.maxp = key2f(rec.maxp_key);
        S.S = (a ? g.sout : g.sin)[x];
        if (a) {
            sm.cand_cnt = 0;
            sm.queue_cnt = 0;
            sm.redo = 0;
            sm.thr_key = 0u;
            sm.thr_keep = neg_inf();
            sm.tau = neg_inf();
            sm.vtypes = g.vtypes;
            sm.err = __double2float_ru(0.5 * sm.two_err);
            sm.scanned = sm.hits = sm.paths = sm.near_edges = 0ull;
        }
    }
    __syncthreads();
    if (sm.side[0].S == 0ull || sm.side[1].S == 0ull) return;  // no slot with a middle edge on one side
    sr_face<NT>(sm.side[0].S <= sm.side[1].S ? 1 : 0);
    const unsigned long long S_near = sm.side[1 - sm.fwd].S;
    if (threadIdx.x == 0) sm.near_edges = S_near;
    unsigned long long S_open = S_near;  // of slots that may lie on a path
    if (S_near > kSrSmall && (sm.cons || sm.part_count > 1)) {
        S_open = sr_open_edges<NT>();
        // Constraints past the near slots are tested hit by hit: seeds and thresholds
        // fail on most, and with many edges the join's blocks are faster together
        // (middle relation and one type allowed, two hubs, 5 M edges, K = 1,000: 1.87 ms
        // here, 0.42 ms there; 256 such queries 7.7 and 6.3 ms)
        if (sm.cons && S_open > alone) {
            if (threadIdx.x == 0) sm.redo = 1;
            __syncthreads();
            return;
        }
    }
    if (S_near > kSrSmall) {
        // seed: rows and edges per row grow until K paths are found
        const int nsd = 1 - sm.fwd, fsd = sm.fwd;
        uint32_t rows = 256u + static_cast<uint32_t>(sm.K), limit = 32u;
        const float cutf = sm.side[fsd].n > kSrHashMax ? sr_cut<NT>(fsd, kSrHashMax * 3 / 4) : neg_inf();
        if (threadIdx.x == 0) sm.far_p = cutf;
        __syncthreads();
        sr_build_hash<NT>();
        unsigned long long spent = 0, left = alone;
        for (int trial = 0; trial < 4; ++trial) {
            const float cut = sr_cut<NT>(nsd, rows);
            __syncthreads();
            if (threadIdx.x == 0) {
                sm.cutp = cut;
                sm.cand_cnt = 0;
            }
            __syncthreads();
            spent = sr_scan<NT, true>(false, limit, neg_inf(),
                                      min(left, static_cast<unsigned long long>(rows) * limit * 2));
            left -= spent;
            const int nc = min(sm.cand_cnt, sm.cap);
            __syncthreads();
            if (nc >= sm.K) {
                sr_select<NT>(nc);
                break;
            }
            // half of it read, or too few paths for a threshold at this rate
            if (spent * 2 > S_open) break;
            if (spent >= kSrSmall && 2ull * nc * S_open < spent * static_cast<unsigned long long>(sm.K)) break;
            rows *= 4;
            limit *= 8;
        }
        if (!sm.thr_key && S_open > alone) {
            if (threadIdx.x == 0) {
                sm.cand_cnt = 0;
                sm.redo = 1;
            }
            __syncthreads();
            return;
        }
        // side and probes
        float last = INFINITY, cut = cutf;
        int cut_side = fsd;
        for (int trial = 0; trial < 4 && sm.thr_key; ++trial) {
            float level, level1;
            float n = sr_estimate<NT>(&level);
            if (n > static_cast<float>(kSrOther) && trial == 0) {
                const int f0 = sm.fwd;
                sr_face<NT>(1 - f0);
                const float n1 = sr_estimate<NT>(&level1);
                if (n1 < n) n = n1, level = level1;
                else sr_face<NT>(f0);
            }
            // the last probe has to have been worth its phases
            if (n <= static_cast<float>(kSrProbe) || n <= 4.f * static_cast<float>(spent) || n > 0.6f * last) break;
            last = n;
            const float before = sm.thr_keep;
            if (sm.fwd != cut_side) {  // the other row is the far one now
                cut_side = sm.fwd;
                cut = sm.side[cut_side].n > kSrHashMax ? sr_cut<NT>(cut_side, kSrHashMax * 3 / 4) : neg_inf();
            }
            sr_build_far<NT>(cut);
            if (threadIdx.x == 0) sm.cand_cnt = 0;
            __syncthreads();
            spent = sr_scan<NT, false>(true, 0u, level, static_cast<unsigned long long>(n * 0.25f));
            const int nc = min(sm.cand_cnt, sm.cap);
            __syncthreads();
            if (nc >= sm.K) sr_select<NT>(nc);
            if (!(sm.thr_keep > before)) break;
        }
        if (threadIdx.x == 0) sm.cand_cnt = 0;
        __syncthreads();
    }
    sr_build_far<NT>(neg_inf());
    sr_scan<NT, false>(false, 0u, neg_inf(), heavy);
    if (sm.redo) return;
    const int nc = sm.cand_cnt;
    __syncthreads();
    if (nc >= sm.K) {
        sr_select<NT>(nc);
        sr_compact<NT>(nc);
    }
}

}  // namespace mhr
