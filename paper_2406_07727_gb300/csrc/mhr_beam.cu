// Generic H-hop search with a per-path beam (Alg. 6, Alg. 7), batched over
// queries, exact.
//
// Level l holds, per query, up to K^l paths in fixed slots (slot j of level
// l+1 is child j mod K of slot j / K of level l).  On a graph with a weight
// index one warp per held path reads only what can be kept (k_beam_step): its
// edges into t, found by a search in the row, and the front of its row sorted
// by weight, down to the band below its K-th extension.  Paths whose band or
// parallel edges into t overflow a warp's lists, and every path on a graph
// without an index, take a CTA per path (k_beam_level):
//   - every out-edge (x, r, y) of the path's last vertex x is scored in fp32;
//     the K-th largest fp32 weight among the path's extensions sets a band (the
//     graph's proven fp32 error, twice, plus the spacing of the rounded path
//     scores), and only the extensions inside it and the edges into t are
//     scored in fp64 in the canonical operation order (the path score is the
//     parent's score plus the edge weight, left to right, as the reference
//     definition);
//   - y already on the path: skipped (Alg. 7); y == t: a result (reaching the
//     target ends the path); otherwise an extension;
//   - the path keeps its K best extensions (score desc, then relation, then
//     vertex ascending) and its K best results, merged chunk by chunk (256
//     edges) into shared-memory lists with a bitonic sort;
//   - the K best extensions become the children's slots of level l+1 (unused
//     child slots are marked empty), the K best results are appended to the
//     query's result list.
// A final CTA per query keeps the K best results (score desc, hop count asc,
// then (y_1, r_1, ..., y_{h-1}, r_{h-1}, r_h) asc) and writes them in order.
// Every kept score is fp64 with the reference's operation order, so selection
// decisions and output equal the fp64 brute force exactly.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <type_traits>
#include <vector>

#include "mhr_exact.cuh"
#include "mhr_internal.cuh"

namespace mhr {

// Work buffers kept between calls (one call at a time per handle), up to
// kBeamKeep bytes; a call that needs more allocates its own and frees them.
struct BeamCache {
    void* buf = nullptr;
    size_t bytes = 0;
    ~BeamCache() {
        if (buf) cudaFree(buf);
    }
};
constexpr size_t kBeamKeep = size_t(64) << 20;

void destroy_beam(mhr_graph* g) {
    delete g->beam;
    g->beam = nullptr;
}

namespace {

constexpr int kBeamThreads = 256;
constexpr int kBeamChunk = 256;      // edges per merge step
constexpr int kBeamMaxK = 64;        // MHR_BEAM_K_MAX
constexpr int kBeamMaxH = 8;         // MHR_BEAM_MAX_H
constexpr int kBeamBuf = 512;        // >= kBeamMaxK + kBeamChunk, power of two

struct BeamPath {                    // same layout as mhr_beam_path (64 B)
    double score;
    int32_t hops;                    // -1: empty slot
    uint32_t v[kBeamMaxH + 1];
    uint16_t r[kBeamMaxH];
};
static_assert(sizeof(BeamPath) == 64, "beam path record is 64 bytes");
static_assert(kBeamBuf >= kBeamMaxK + kBeamChunk, "merge buffer holds the kept list and one chunk");

struct Ext {                         // one scored out-edge of a held path
    double score;
    uint32_t y;
    uint32_t r;                      // relation; 0xffffffff pads the sort
};

// extensions of one path: score desc, then relation asc, then vertex asc
__device__ __forceinline__ bool ext_before(const Ext& a, const Ext& b) {
    if (a.score != b.score) return a.score > b.score;
    if (a.r != b.r) return a.r < b.r;
    return a.y < b.y;
}

// results: score desc, hop count asc, then (y_1, r_1, ..., y_{h-1}, r_{h-1}, r_h) asc
__device__ __forceinline__ bool result_before(const BeamPath& a, const BeamPath& b) {
    if (a.score != b.score) return a.score > b.score;
    if (a.hops != b.hops) return a.hops < b.hops;
    for (int i = 1; i < a.hops; ++i) {
        if (a.v[i] != b.v[i]) return a.v[i] < b.v[i];
        if (a.r[i - 1] != b.r[i - 1]) return a.r[i - 1] < b.r[i - 1];
    }
    return a.r[a.hops - 1] < b.r[b.hops - 1];
}

__device__ __forceinline__ Ext ext_pad() { return Ext{-INFINITY, 0xffffffffu, 0xffffffffu}; }

// bitonic sort of P (power of two) records in shared memory, best first
template <typename T, typename Before>
__device__ void block_bitonic(T* a, unsigned P, Before before) {
    for (unsigned size = 2; size <= P; size <<= 1) {
        for (unsigned stride = size >> 1; stride > 0; stride >>= 1) {
            for (unsigned i = threadIdx.x; i < P; i += blockDim.x) {
                const unsigned j = i ^ stride;
                if (j > i) {
                    const T x = a[i], y = a[j];
                    const bool best_first = (i & size) == 0;
                    if (best_first ? before(y, x) : before(x, y)) {
                        a[i] = y;
                        a[j] = x;
                    }
                }
            }
            __syncthreads();
        }
    }
}

__device__ __forceinline__ unsigned pow2_at_least(unsigned m) {
    unsigned P = 1;
    while (P < m) P <<= 1;
    return P;
}

// level 0: the one-vertex path (s) of every query
__global__ void k_beam_init(const uint32_t* __restrict__ s, int nq, BeamPath* __restrict__ level0,
                            unsigned* __restrict__ n_res) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nq) return;
    BeamPath p;
    p.score = 0.0;
    p.hops = 0;
    for (int i = 0; i <= kBeamMaxH; ++i) p.v[i] = 0u;
    for (int i = 0; i < kBeamMaxH; ++i) p.r[i] = 0;
    p.v[0] = s[q];
    level0[q] = p;
    n_res[q] = 0u;
}

struct LevelArgs {
    DevGraph g;
    const uint32_t* t;             // [nq] targets
    int level, H, K;
    int64_t slots;                 // K^level slots per query at this level
    const BeamPath* cur;           // [nq * slots]
    BeamPath* next;                // [nq * slots * K] when level + 1 < H
    BeamPath* res;                 // [nq * res_cap]
    int64_t res_cap;
    unsigned* n_res;               // [nq]
    unsigned long long* n_scored;  // edges scored (one counter), NULL: not counted
    unsigned long long* n_exact;   // extensions scored in fp64 (one counter)
    double e1;                     // bound on |w32 - w64| of one edge
    int64_t n_slots;               // slots of all queries
    uint32_t* left;                // [n_slots] slots a warp left to a CTA (graphs with an index)
    unsigned* n_left;
};

// Screening of a path's extensions.  With T the K-th largest fp32 weight
// w32 among them and E1 the bound on |w32 - w64|, every extension of the true
// K best (by fl64(score(p) + w64), then relation, then vertex) has
//   w32 >= T - 2 E1 - 2^-51 (|score(p)| + |w32| + E1)   (rounded down below):
// at least one of the K extensions with w32 >= T ranks after it, so its w64 is
// at least that one's w64 minus the spacing of the doubles around the
// (equal) rounded path scores.  Only those extensions are scored in fp64.
__device__ __forceinline__ bool in_band(float w32, float T, double P, double e1) {
    if (T == -INFINITY) return true;
    const double a = fabs(P) + fabs(static_cast<double>(w32)) + e1 + 1.0;
    return static_cast<double>(w32) >= static_cast<double>(T) - 2.0 * e1 - ldexp(a, -50);
}

// one held path of this level, by the whole CTA
__device__ void beam_slot(const LevelArgs& a, const int64_t slot) {
    __shared__ Ext ext[kBeamBuf];
    __shared__ Ext res[kBeamBuf];
    __shared__ unsigned n_ext, n_rl, c_ext, c_res, res_base;
    const int64_t q = slot / a.slots;
    const BeamPath p = a.cur[slot];
    const bool more = a.level + 1 < a.H;
    const int K = a.K;
    if (p.hops != a.level) {  // an empty slot has empty children
        if (more)
            for (int c = threadIdx.x; c < K; c += blockDim.x) a.next[slot * K + c].hops = -1;
        return;
    }
    const uint32_t x = p.v[a.level];
    const uint32_t tq = a.t[q];
    const int64_t e0 = a.g.off[x], e1 = a.g.off[x + 1];
    __shared__ float topw[kBeamBuf];  // screening: the K largest fp32 extension weights, then staging
    __shared__ unsigned n_top, c_top;
    __shared__ float thr_adm;         // admission threshold of the staging (K-th largest so far)
    __shared__ unsigned long long n_fp64;
    if (threadIdx.x == 0) {
        n_ext = 0u;
        n_rl = 0u;
        n_top = 0u;
        n_fp64 = 0ull;
        thr_adm = -INFINITY;
        if (a.n_scored && e1 > e0) atomicAdd(a.n_scored, static_cast<unsigned long long>(e1 - e0));
    }
    __syncthreads();
    // 0. fp32 pass over the extensions: T = the K-th largest w32 (-inf when
    //    there are at most K extensions: every one is kept)
    float T = -INFINITY;
    if (more && e1 - e0 > K) {
        for (int64_t base = e0; base < e1; base += kBeamChunk) {
            if (threadIdx.x == 0) c_top = 0u;
            __syncthreads();
            const int64_t e = base + threadIdx.x;
            if (threadIdx.x < kBeamChunk && e < e1) {
                const uint32_t y = a.g.col[e];
                bool on_path = y == tq;
                for (int i = 0; i <= a.level; ++i) on_path |= (p.v[i] == y);
                if (!on_path) {
                    const float w = a.g.w ? a.g.w[e] : edge_w32_group(a.g, x, a.g.rel[e], y, 0, 1);
                    if (w >= thr_adm) topw[n_top + atomicAdd(&c_top, 1u)] = w;
                }
            }
            __syncthreads();
            const unsigned m = n_top + c_top;
            const bool last = base + kBeamChunk >= e1;
            // keep the K largest once the staging could not take another chunk, and
            // at the end (sorted, so that entry K - 1 is the K-th largest)
            if (m + kBeamChunk > static_cast<unsigned>(kBeamBuf) || last) {
                if (m > static_cast<unsigned>(K) || (last && m == static_cast<unsigned>(K))) {
                    const unsigned P2 = pow2_at_least(m);
                    for (unsigned i = m + threadIdx.x; i < P2; i += blockDim.x) topw[i] = -INFINITY;
                    __syncthreads();
                    block_bitonic(topw, P2, [](float u, float v) { return u > v; });
                    if (threadIdx.x == 0) {
                        n_top = static_cast<unsigned>(K);
                        thr_adm = topw[K - 1];
                    }
                } else if (threadIdx.x == 0) {
                    n_top = m;
                }
            } else if (threadIdx.x == 0) {
                n_top = m;
            }
            __syncthreads();
        }
        if (n_top >= static_cast<unsigned>(K)) T = topw[K - 1];
        __syncthreads();
    }
    for (int64_t base = e0; base < e1; base += kBeamChunk) {
        if (threadIdx.x == 0) {
            c_ext = 0u;
            c_res = 0u;
        }
        __syncthreads();
        // 1. score this chunk's edges; append behind the kept lists
        const int64_t e = base + threadIdx.x;
        if (threadIdx.x < kBeamChunk && e < e1) {
            const uint32_t y = a.g.col[e];
            const uint32_t r = a.g.rel[e];
            bool on_path = false;
            for (int i = 0; i <= a.level; ++i) on_path |= (p.v[i] == y);
            if (!on_path && (y == tq || more)) {
                // an extension outside the screening band cannot be among the K best
                const bool keep = y == tq || T == -INFINITY ||
                                  in_band(a.g.w ? a.g.w[e] : edge_w32_group(a.g, x, r, y, 0, 1), T, p.score, a.e1);
                if (keep) {
                    const double sc = __dadd_rn(p.score, edge_w64(a.g, x, r, y));
                    if (y == tq) res[n_rl + atomicAdd(&c_res, 1u)] = Ext{sc, y, r};
                    else ext[n_ext + atomicAdd(&c_ext, 1u)] = Ext{sc, y, r};
                    atomicAdd(&n_fp64, 1ull);
                }
            }
        }
        __syncthreads();
        // 2. keep the K best of each list
        const unsigned me = n_ext + c_ext, mr = n_rl + c_res;
        if (me > static_cast<unsigned>(K)) {
            const unsigned P = pow2_at_least(me);
            for (unsigned i = me + threadIdx.x; i < P; i += blockDim.x) ext[i] = ext_pad();
            __syncthreads();
            block_bitonic(ext, P, ext_before);
        }
        if (mr > static_cast<unsigned>(K)) {
            const unsigned P = pow2_at_least(mr);
            for (unsigned i = mr + threadIdx.x; i < P; i += blockDim.x) res[i] = ext_pad();
            __syncthreads();
            block_bitonic(res, P, ext_before);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            n_ext = min(me, static_cast<unsigned>(K));
            n_rl = min(mr, static_cast<unsigned>(K));
        }
        __syncthreads();
    }
    if (threadIdx.x == 0 && a.n_scored && n_fp64) atomicAdd(a.n_exact, n_fp64);
    // 3. children: the kept extensions (any order); the other child slots empty
    if (more) {
        for (int c = threadIdx.x; c < K; c += blockDim.x) {
            BeamPath* ch = a.next + slot * K + c;
            if (static_cast<unsigned>(c) < n_ext) {
                BeamPath cp = p;
                cp.score = ext[c].score;
                cp.r[a.level] = static_cast<uint16_t>(ext[c].r);
                cp.hops = a.level + 1;
                cp.v[a.level + 1] = ext[c].y;
                *ch = cp;
            } else {
                ch->hops = -1;
            }
        }
    }
    // 4. results: appended to the query's list
    if (n_rl) {
        if (threadIdx.x == 0) res_base = atomicAdd(a.n_res + q, n_rl);
        __syncthreads();
        for (unsigned c = threadIdx.x; c < n_rl; c += blockDim.x) {
            const int64_t pos = static_cast<int64_t>(res_base) + c;
            if (pos >= a.res_cap) continue;
            BeamPath rp = p;
            rp.score = res[c].score;
            rp.r[a.level] = static_cast<uint16_t>(res[c].r);
            rp.hops = a.level + 1;
            rp.v[a.level + 1] = tq;
            a.res[q * a.res_cap + pos] = rp;
        }
    }
}

__global__ void __launch_bounds__(kBeamThreads) k_beam_level(LevelArgs a) {
    const int64_t n = a.left ? static_cast<int64_t>(*a.n_left) : a.n_slots;
    for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
        beam_slot(a, a.left ? static_cast<int64_t>(a.left[i]) : i);
        __syncthreads();
    }
}

// One warp per held path, on the weight index.  A path keeps K of its x's
// extensions, and the row sorted by weight starts with them: the warp walks it in
// steps of 32 edges until K that may extend the path are counted (T) and the band
// below T (in_band) has ended, then scores those few in fp64, in integers where
// the coordinates allow it.  Edges into t are one run of the CSR row, found by a
// 32-way search.  What bounds it: the chain of dependent loads of a path (record,
// row, edges, embedding rows), about 20 us per level.  64 queries of H = 3, K = 10
// on 1M vertices / 20M edges: 57 us for the three levels, where a CTA per path read
// and scored all 17M edges of the held rows twice in 6.5 ms (the whole call 7.8 ->
// 0.27 ms, 1.4 ms of it from buffers that are kept).
constexpr int kStepWarps = 4;
constexpr int kStepCand = 128;  // candidates of a path: K <= 64 and its band
__global__ void __launch_bounds__(kStepWarps * 32) k_beam_step(LevelArgs a) {
    __shared__ double s_stage[kStepWarps][32 * 33];
    __shared__ double s_sc[kStepWarps][kStepCand];
    __shared__ uint32_t s_y[kStepWarps][kStepCand];
    __shared__ uint16_t s_r[kStepWarps][kStepCand];
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int64_t slot = blockIdx.x * static_cast<int64_t>(kStepWarps) + wi;
    if (slot >= a.n_slots) return;  // no block-wide step below
    const int K = a.K, level = a.level;
    const bool more = level + 1 < a.H;
    BeamPath* kids = a.next + slot * K;
    // the record by words: 0-1 score, 2 hops, 3 .. 11 vertices, 12 .. 15 relations (lanes 16 .. 31 repeat it)
    const uint32_t pw = reinterpret_cast<const uint32_t*>(a.cur + slot)[lane & 15];
    if (static_cast<int>(__shfl_sync(FULL, pw, 2)) != level) {  // an empty slot has empty children
        if (more)
            for (int c = lane; c < K; c += 32) kids[c].hops = -1;
        return;
    }
    const uint32_t x = __shfl_sync(FULL, pw, 3 + level);
    const double P = __hiloint2double(static_cast<int>(__shfl_sync(FULL, pw, 1)), static_cast<int>(__shfl_sync(FULL, pw, 0)));
    const int64_t q = slot / a.slots;
    const uint32_t tq = a.t[q];
    const int64_t e0 = a.g.off[x], e1 = a.g.off[x + 1];
    const int64_t deg = e1 - e0;
    // edges into t: [lo, lo + nt)
    int64_t lo = e0, hi = e1;
    while (hi - lo > 32) {
        const int64_t step = (hi - lo + 31) >> 5, at = lo + (lane + 1) * step - 1;
        const int c = __popc(__ballot_sync(FULL, at < hi && a.g.col[at] < tq));  // whole pieces before t
        lo += c * step;
        hi = min(hi, lo + step);
    }
    {
        const int64_t at = lo + lane;
        lo += __popc(__ballot_sync(FULL, at < hi && a.g.col[at] < tq));
    }
    const int64_t at = lo + lane;
    const bool to_t = at < e1 && a.g.col[at] == tq;
    const int nt = __popc(__ballot_sync(FULL, to_t));
    const uint32_t rt = to_t ? a.g.rel[at] : 0u;
    bool fits = nt < 32 && nt <= K;

    // the extensions that may be among the K best
    int nc = 0;
    if (more && fits) {
        const int64_t row = a.g.vout[x].row;
        float T = -INFINITY;
        int nv = 0;
        for (int64_t i = 0; i < deg; i += 32) {
            const bool in = i + lane < deg;
            const uint2 ed = in ? a.g.se[row + i + lane] : make_uint2(tq, 0u);
            const uint32_t r = in ? a.g.sr[row + i + lane] : 0u;
            bool ok = ed.x != tq;
            for (int k = 0; k <= level; ++k) ok &= __shfl_sync(FULL, pw, 3 + k) != ed.x;
            const float w = __uint_as_float(ed.y);
            const unsigned m = __ballot_sync(FULL, ok);
            if (nv < K && nv + __popc(m) >= K) {
                const bool kth = ok && nv + __popc(m & ((1u << lane) - 1u)) == K - 1;
                T = __shfl_sync(FULL, w, __ffs(__ballot_sync(FULL, kth)) - 1);
            }
            nv += __popc(m);
            const bool band = in_band(w, T, P, a.e1);
            const unsigned keep = __ballot_sync(FULL, ok && band);
            if (nc + __popc(keep) > kStepCand) {
                fits = false;
                break;
            }
            if (ok && band) {
                const int c = nc + __popc(keep & ((1u << lane) - 1u));
                s_y[wi][c] = ed.x;
                s_r[wi][c] = static_cast<uint16_t>(r);
            }
            nc += __popc(keep);
            if (__any_sync(FULL, in && !band)) break;  // the row descends: the band has ended
        }
        __syncwarp();
    }
    if (!fits) {
        if (lane == 0) a.left[atomicAdd(a.n_left, 1u)] = static_cast<uint32_t>(slot);
        return;
    }
    if (a.n_scored && lane == 0) {
        if (deg) atomicAdd(a.n_scored, static_cast<unsigned long long>(deg));
        if (nc + nt) atomicAdd(a.n_exact, static_cast<unsigned long long>(nc + nt));
    }
    // fp64 scores: the candidates, 32 at a time, and then the edges into t
    double sc_t = 0.0;
    const int rounds = (nc + 31) >> 5;
    for (int b = 0; b < rounds + (nt > 0 ? 1 : 0); ++b) {
        const bool ext = b < rounds;
        const int n = ext ? min(32, nc - 32 * b) : nt;
        const bool live = lane < n;
        uint32_t y = tq, r = rt;
        if (ext && live) {
            y = s_y[wi][32 * b + lane];
            r = s_r[wi][32 * b + lane];
        }
        double w64 = 0.0;
        bool open = live;  // for the fp64 route
        if (a.g.fn == MHR_SCORE_TRANSE_L1) {
#pragma unroll 2
            for (int k = 0; k < n; ++k) {
                bool ok;
                const double v = warp_w64_fixed(a.g, x, __shfl_sync(FULL, r, k), __shfl_sync(FULL, y, k), lane, &ok);
                if (lane == k && ok) {
                    w64 = v;
                    open = false;
                }
            }
        }
        if (__any_sync(FULL, open)) {
            const double v = warp_w64_staged(a.g, x, r, y, open, s_stage[wi], lane);
            if (open) w64 = v;
        }
        const double sc = __dadd_rn(P, w64);
        if (!ext) sc_t = sc;
        else if (live) s_sc[wi][32 * b + lane] = sc;
    }
    __syncwarp();
    // children: the K best extensions, each in the slot of its rank; the other slots empty
    if (more) {
        for (int b = 0; b < nc; b += 32) {
            const int c = b + lane;
            const Ext mine = c < nc ? Ext{s_sc[wi][c], s_y[wi][c], s_r[wi][c]} : ext_pad();
            int rank = 0;
            if (nc <= K) rank = c;  // children have no order of their own
            else
                for (int k = 0; k < nc; ++k) rank += ext_before(Ext{s_sc[wi][k], s_y[wi][k], s_r[wi][k]}, mine) ? 1 : 0;
            if (c < nc && rank < K) {
                const uint32_t keep = static_cast<uint32_t>(rank);
                s_stage[wi][keep] = __hiloint2double(0, c);  // whose record goes to that slot
            }
        }
        __syncwarp();
        const int held = min(nc, K);
        for (int c0 = 0; c0 < K; c0 += 2) {  // half a warp writes one child
            const int c = c0 + (lane >> 4), word = lane & 15;
            uint32_t v = pw;
            if (c < held) {
                const int e = __double2loint(s_stage[wi][c]);
                const double sc = s_sc[wi][e];
                if (word == 0) v = static_cast<uint32_t>(__double2loint(sc));
                if (word == 1) v = static_cast<uint32_t>(__double2hiint(sc));
                if (word == 2) v = static_cast<uint32_t>(level + 1);
                if (word == 3 + level + 1) v = s_y[wi][e];
                if (word == 12 + (level >> 1))
                    v = (level & 1) ? (v & 0xffffu) | (static_cast<uint32_t>(s_r[wi][e]) << 16)
                                    : (v & 0xffff0000u) | s_r[wi][e];
            } else {
                v = 0xffffffffu;
            }
            if (c < held || (c < K && word == 2)) reinterpret_cast<uint32_t*>(kids + c)[word] = v;
        }
    }
    // results: appended to the query's list
    if (nt) {
        unsigned base = 0u;
        if (lane == 0) base = atomicAdd(a.n_res + q, static_cast<unsigned>(nt));
        base = __shfl_sync(FULL, base, 0);
        for (int c = 0; c < nt; ++c) {
            const double sc = __shfl_sync(FULL, sc_t, c);
            const uint32_t r = __shfl_sync(FULL, rt, c);
            uint32_t v = pw;
            if (lane == 0) v = static_cast<uint32_t>(__double2loint(sc));
            if (lane == 1) v = static_cast<uint32_t>(__double2hiint(sc));
            if (lane == 2) v = static_cast<uint32_t>(level + 1);
            if (lane == 3 + level + 1) v = tq;
            if (lane == 12 + (level >> 1)) v = (level & 1) ? (v & 0xffffu) | (r << 16) : (v & 0xffff0000u) | r;
            const int64_t pos = static_cast<int64_t>(base) + c;
            if (lane < 16 && pos < a.res_cap) reinterpret_cast<uint32_t*>(a.res + q * a.res_cap + pos)[lane] = v;
        }
    }
}

__device__ __forceinline__ BeamPath result_pad() {
    BeamPath p;
    p.score = -INFINITY;
    p.hops = 0x7fffffff;
    for (int i = 0; i <= kBeamMaxH; ++i) p.v[i] = 0xffffffffu;
    for (int i = 0; i < kBeamMaxH; ++i) p.r[i] = 0xffff;
    return p;
}

// One CTA per query: the K best results in order.  Up to kBeamBuf results are
// compared pair by pair (no two rank alike, so a result's place is the number of
// results before it: one barrier, where sorting the 64-byte records took up to 45
// and 54 us for 64 queries, now 13 us); more are first cut to the K best, chunk by chunk.
__global__ void __launch_bounds__(kBeamThreads) k_beam_final(const BeamPath* __restrict__ res, int64_t res_cap,
                                                             const unsigned* __restrict__ n_res, int K,
                                                             BeamPath* __restrict__ out, int32_t* __restrict__ n_out) {
    __shared__ __align__(16) BeamPath buf[kBeamBuf];
    const int64_t q = blockIdx.x;
    const int64_t n = min(static_cast<int64_t>(n_res[q]), res_cap);
    const BeamPath* a = res + q * res_cap;
    unsigned kept = 0;
    if (n <= kBeamBuf) {
        kept = static_cast<unsigned>(n);
        const uint4* from = reinterpret_cast<const uint4*>(a);
        for (unsigned i = threadIdx.x; i < 4 * kept; i += blockDim.x) reinterpret_cast<uint4*>(buf)[i] = from[i];
    } else {
        for (int64_t base = 0; base < n; base += kBeamChunk) {
            const unsigned c = static_cast<unsigned>(min(static_cast<int64_t>(kBeamChunk), n - base));
            for (unsigned i = threadIdx.x; i < c; i += blockDim.x) buf[kept + i] = a[base + i];
            __syncthreads();
            const unsigned m = kept + c;
            if (m > static_cast<unsigned>(K)) {
                const unsigned P = pow2_at_least(m);
                for (unsigned i = m + threadIdx.x; i < P; i += blockDim.x) buf[i] = result_pad();
                __syncthreads();
                block_bitonic(buf, P, result_before);
            }
            kept = min(m, static_cast<unsigned>(K));
            __syncthreads();
        }
    }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < kept; i += blockDim.x) {
        int rank = 0;
        for (unsigned j = 0; j < kept && rank < K; ++j) {
            const double s = buf[j].score, mine = buf[i].score;  // most pairs differ in score
            rank += s != mine ? s > mine : result_before(buf[j], buf[i]);
        }
        if (rank < K) out[q * K + rank] = buf[i];
    }
    if (threadIdx.x == 0) n_out[q] = static_cast<int32_t>(min(kept, static_cast<unsigned>(K)));
}

}  // namespace
}  // namespace mhr

using namespace mhr;

extern "C" mhr_status mhr_beam_paths(const mhr_graph* g, int32_t nq, const uint32_t* s, const uint32_t* t,
                                     int32_t H, int32_t K, mhr_beam_path* out, int32_t* n_out, mhr_mem mem,
                                     mhr_stats* stats, void* cuda_stream) {
    const auto t_start = std::chrono::steady_clock::now();
    MHR_TRY(check_graph(g));
    if (nq < 0) return fail(MHR_EINVAL, "nq must be >= 0");
    if (H < 1 || H > MHR_BEAM_MAX_H) return fail(MHR_EINVAL, "H must be in [1, MHR_BEAM_MAX_H]");
    if (K < 1) return fail(MHR_EINVAL, "K must be >= 1");
    if (K > MHR_BEAM_K_MAX) return fail(MHR_ERANGE, "K exceeds MHR_BEAM_K_MAX");
    if (mem != MHR_MEM_HOST && mem != MHR_MEM_DEVICE) return fail(MHR_EINVAL, "unknown mem kind");
    // level l holds K^l slots per query; the widest level is H - 1
    int64_t widest = 1, held_total = 0;
    for (int l = 0; l < H; ++l) {
        held_total += widest;
        if (l + 1 < H) {
            widest *= K;
            if (widest > (int64_t(1) << 16)) return fail(MHR_ERANGE, "K^(H-1) exceeds 65536");
        }
    }
    const int64_t res_cap = held_total * K;
    if (stats) *stats = mhr_stats{};
    if (nq == 0) return MHR_OK;
    if (!s || !t || !out || !n_out) return fail(MHR_EINVAL, "NULL array");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);

    std::vector<uint32_t> hs(nq), ht(nq);
    if (mem == MHR_MEM_HOST) {
        std::copy(s, s + nq, hs.begin());
        std::copy(t, t + nq, ht.begin());
    } else {
        MHR_CUDA_TRY(cudaMemcpyAsync(hs.data(), s, 4ull * nq, cudaMemcpyDeviceToHost, st));
        MHR_CUDA_TRY(cudaMemcpyAsync(ht.data(), t, 4ull * nq, cudaMemcpyDeviceToHost, st));
        MHR_CUDA_TRY(cudaStreamSynchronize(st));
    }
    for (int i = 0; i < nq; ++i) {
        if (static_cast<int64_t>(hs[i]) >= g->dg.n || static_cast<int64_t>(ht[i]) >= g->dg.n)
            return fail(MHR_EINVAL, "vertex out of range");
        if (hs[i] == ht[i]) return fail(MHR_EINVAL, "s == t");
    }

    // queries per round so that the level buffers and results stay within 1 GiB
    const size_t per_query = sizeof(BeamPath) * static_cast<size_t>(2 * widest + res_cap) + 64;
    const int QB = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(nq, (int64_t(1) << 30) / per_query)));
    const double e1 = (g->eps32_edge + g->eps64_edge) * (1.0 + 1e-6);
    const bool index = g->dg.w != nullptr;
    BeamPath *A = nullptr, *B = nullptr, *R = nullptr, *d_out = reinterpret_cast<BeamPath*>(out);
    uint32_t *d_s = const_cast<uint32_t*>(s), *d_t = const_cast<uint32_t*>(t), *d_left = nullptr;
    unsigned *d_nres = nullptr, *d_nleft = nullptr;
    int32_t* d_nout = n_out;
    unsigned long long* d_scored = nullptr;  // [0] edges scored in fp32, [1] scored in fp64
    // one buffer: laid out once to size it, once more to hand out the pieces
    char* base = nullptr;
    size_t used = 0;
    auto take = [&](auto** p, size_t count) {
        *p = reinterpret_cast<std::remove_reference_t<decltype(*p)>>(base + used);
        used = (used + sizeof(**p) * count + 255) / 256 * 256;
    };
    auto lay_out = [&]() {
        used = 0;
        take(&A, static_cast<size_t>(QB) * widest);
        take(&B, static_cast<size_t>(QB) * widest);
        take(&R, static_cast<size_t>(QB) * res_cap);
        take(&d_nres, QB);
        take(&d_scored, 2);
        take(&d_nleft, H);
        if (index) take(&d_left, static_cast<size_t>(QB) * widest);
        if (mem == MHR_MEM_HOST) {
            take(&d_out, static_cast<size_t>(nq) * K);
            take(&d_nout, nq);
            take(&d_s, nq);
            take(&d_t, nq);
        }
    };
    lay_out();
    mhr_graph* gm = const_cast<mhr_graph*>(g);
    if (!gm->beam) gm->beam = new BeamCache();
    BeamCache* bc = gm->beam;
    void* own = nullptr;  // a buffer of this call alone
    cudaError_t e = cudaSuccess;
    if (used > kBeamKeep) {
        e = cudaMalloc(&own, used);
        base = static_cast<char*>(own);
    } else {
        if (used > bc->bytes) {
            if (bc->buf) cudaFree(bc->buf);
            bc->buf = nullptr;
            bc->bytes = 0;
            e = cudaMalloc(&bc->buf, used);
            if (e == cudaSuccess) bc->bytes = used;
            else bc->buf = nullptr;
        }
        base = static_cast<char*>(bc->buf);
    }
    if (e != cudaSuccess) return cuda_fail(e, "beam buffers");
    lay_out();
    auto cleanup = [&]() {
        if (own) cudaFree(own);
    };
    if (mem == MHR_MEM_HOST) {
        e = cudaMemcpyAsync(d_s, hs.data(), 4ull * nq, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(d_t, ht.data(), 4ull * nq, cudaMemcpyHostToDevice, st);
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(d_scored, 0, 16, st);
    if (e != cudaSuccess) {
        cudaStreamSynchronize(st);
        cleanup();
        return cuda_fail(e, "beam buffers");
    }
    for (int c0 = 0; c0 < nq && e == cudaSuccess; c0 += QB) {
        const int qb = std::min(QB, nq - c0);
        k_beam_init<<<(qb + 255) / 256, 256, 0, st>>>(d_s + c0, qb, A, d_nres);
        if (index) e = cudaMemsetAsync(d_nleft, 0, sizeof(unsigned) * H, st);
        if (e != cudaSuccess) break;
        BeamPath *cur = A, *nxt = B;
        int64_t slots = 1;
        for (int l = 0; l < H; ++l) {
            LevelArgs a;
            a.g = g->dg;
            a.t = d_t + c0;
            a.level = l;
            a.H = H;
            a.K = K;
            a.slots = slots;
            a.cur = cur;
            a.next = nxt;
            a.res = R;
            a.res_cap = res_cap;
            a.n_res = d_nres;
            a.n_scored = stats ? d_scored : nullptr;  // one address for all paths
            a.n_exact = d_scored + 1;
            a.e1 = e1;
            a.n_slots = qb * slots;
            a.left = d_left;
            a.n_left = d_nleft + l;
            if (index)
                k_beam_step<<<static_cast<unsigned>((a.n_slots + kStepWarps - 1) / kStepWarps), kStepWarps * 32, 0, st>>>(a);
            // the paths left to a CTA: as many CTAs as are resident at once
            const int64_t ctas = index ? std::min<int64_t>(a.n_slots, int64_t(8) * std::max(1, g->num_sms)) : a.n_slots;
            k_beam_level<<<static_cast<unsigned>(ctas), kBeamThreads, 0, st>>>(a);
            std::swap(cur, nxt);
            slots *= K;
        }
        k_beam_final<<<qb, kBeamThreads, 0, st>>>(R, res_cap, d_nres, K, d_out + static_cast<int64_t>(c0) * K,
                                                  d_nout + c0);
        e = cudaGetLastError();
    }
    unsigned long long scored[2] = {0ull, 0ull};
    if (e == cudaSuccess && mem == MHR_MEM_HOST) {
        e = cudaMemcpyAsync(out, d_out, sizeof(BeamPath) * static_cast<size_t>(nq) * K, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(n_out, d_nout, 4ull * nq, cudaMemcpyDeviceToHost, st);
    }
    if (e == cudaSuccess && stats) e = cudaMemcpyAsync(scored, d_scored, 16, cudaMemcpyDeviceToHost, st);
    const cudaError_t done = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = done;
    cleanup();
    if (e != cudaSuccess) return cuda_fail(e, "beam search");
    if (stats) {
        stats->edges_scanned = static_cast<int64_t>(scored[0]);
        stats->rescored = static_cast<int64_t>(scored[1]);
        stats->ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t_start).count();
    }
    return MHR_OK;
}
