// Tail prediction (Alg. 3, Alg. 4): for a head h and a relation r, score every
// candidate vertex c of one type with the edge weight w(h, r, c) and keep the
// K best (score descending, then c ascending).
//
// Alg. 3 and Alg. 4 loop over every person / university with one thread-private
// heap per OpenMP thread and merge the heaps with a tree (Alg. 2).  The GB300
// form streams the candidates' embedding rows once per batch of queries:
//
//   1. candidate list of the type (built once per type, ordered compaction);
//   2. sampling pass: the fp32 scores of an evenly strided sample of M
//      candidates; per query, the K-th best sampled score minus twice the
//      per-edge error bound is a threshold that can drop no candidate of the
//      exact top K (the K-th best of a subset is at most the K-th best of all);
//   3. full pass (k_tail_scan*): every candidate row is read with 16-byte loads
//      where its length allows it, held in registers by a group of lanes and scored
//      against the queries of a chunk (query vectors e_h + w_r or e_h * w_r in shared
//      memory); scores at or above the threshold are appended to the query's
//      survivor list;
//   4. per query (k_tail_final): the exact K-th best fp32 survivor score by a
//      radix select, the band of survivors within twice the error bound of it
//      rescored in fp64 in the canonical operation order (TransE in integers by
//      eight lanes per member; otherwise one member per thread, e_h + w_r formed once
//      in fp64 in shared memory), and the K best of the band put in order, a short band by
//      comparing every pair (64 queries, K = 50: 33 -> 16 us).
//
// Exactness: |S32 - w64| <= E = eps32 + eps64 for every candidate (the bound of
// mhr_graph.cu holds for any (u, r, v) triple and any summation order).  If c
// is in the exact top K then S32(c) >= w64_K - E >= S32_K - 2E, so the band
// holds every result, and sorting the band by (w64, c) gives them in order.
// A survivor list that overflows its sized buffer is detected on the host and
// that query is rescanned alone with room for every candidate.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <vector>

#include "mhr_exact.cuh"
#include "mhr_internal.cuh"
#include "mhr_util.cuh"

namespace mhr {

struct TailCache {
    uint32_t* cands[256] = {};  // candidate ids per vertex type (device; nullptr = not built)
    int64_t ncand[256] = {};
    void* scratch = nullptr;
    size_t scratch_bytes = 0;
    void* big = nullptr;  // survivors + band of one query rescanned alone
    size_t big_bytes = 0;
    char* pinned = nullptr;  // kPinned bytes: the queries' ids and the counts of a batch, read back
    cudaEvent_t ev[4] = {};

    ~TailCache() {
        for (uint32_t* p : cands)
            if (p) cudaFree(p);
        if (scratch) cudaFree(scratch);
        if (big) cudaFree(big);
        if (pinned) cudaFreeHost(pinned);
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
    }
};

void destroy_tail(mhr_graph* g) {
    delete g->tail;
    g->tail = nullptr;
}

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanWarps = kScanThreads / 32;
constexpr int kFinalThreads = 1024;
constexpr int kSortMax = MHR_TAIL_K_MAX;       // power of two
constexpr size_t kQueryBytes = 64 * 1024;      // query vectors + thresholds per scan launch
constexpr int kMaxBatch = 256;                 // queries per scan launch
constexpr size_t kScratchBudget = size_t(1) << 30;
constexpr int kCompactBlocks = 512;
constexpr size_t kPinned = 32 * 1024;
constexpr int kRankMax = 512;                  // records ordered by comparing every pair

static_assert((kSortMax & (kSortMax - 1)) == 0, "sort size must be a power of two");

struct SurvRec {
    float s;     // fp32 screening score
    uint32_t v;  // candidate
};

struct BandRec {
    double w;  // fp64 score, canonical order
    uint32_t v;
    uint32_t pad;
};

struct ScanArgs {
    DevGraph g;
    const uint32_t* h;     // [nq] heads
    const uint16_t* r;     // [nq] relations
    int nq;
    int chunk;             // queries of one block (blockIdx.y)
    int G;                 // lanes per candidate row (power of two, vector kernels)
    const uint32_t* cand;  // candidate ids; nullptr: candidate i is vertex i
    int64_t n_visit;       // candidates visited: positions i * stride for i < n_visit
    int64_t stride;
    const float* thr;      // [nq] keep scores >= thr[q]; nullptr keeps every score
    SurvRec* surv;         // query q's survivors at surv[q * cap]
    int64_t cap;
    unsigned int* cnt;     // [nq] survivors found (may exceed cap)
};

// ---------------------------------------------------------------------------
// candidate lists: ids of the vertices of one type, increasing
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_type_count(const uint8_t* __restrict__ vt, int64_t n, int type,
                                                     int64_t per_block, int64_t* __restrict__ counts) {
    const int64_t lo = blockIdx.x * per_block, hi = min(n, lo + per_block);
    int64_t c = 0;
    for (int64_t base = lo; base < hi; base += blockDim.x) {
        const int64_t i = base + threadIdx.x;
        c += __syncthreads_count(i < hi && vt[i] == type);
    }
    if (threadIdx.x == 0) counts[blockIdx.x] = c;
}

__global__ void __launch_bounds__(1024) k_type_offsets(int64_t* __restrict__ counts, int nb) {
    // exclusive scan of nb <= 1024 block counts in place; counts[nb] = total
    __shared__ int64_t sm[33];
    const int64_t x = threadIdx.x < nb ? counts[threadIdx.x] : 0;
    int64_t total;
    const int64_t ex = block_excl_scan<int64_t>(x, sm, &total);
    if (threadIdx.x < nb) counts[threadIdx.x] = ex;
    if (threadIdx.x == 0) counts[nb] = total;
}

__global__ void __launch_bounds__(1024) k_type_write(const uint8_t* __restrict__ vt, int64_t n, int type,
                                                     int64_t per_block, const int64_t* __restrict__ offsets,
                                                     uint32_t* __restrict__ out) {
    __shared__ int64_t sm[33];
    const int64_t lo = blockIdx.x * per_block, hi = min(n, lo + per_block);
    int64_t pos = offsets[blockIdx.x];
    for (int64_t base = lo; base < hi; base += blockDim.x) {
        const int64_t i = base + threadIdx.x;
        const int64_t f = (i < hi && vt[i] == type) ? 1 : 0;
        int64_t tile;
        const int64_t ex = block_excl_scan<int64_t>(f, sm, &tile);
        if (f) out[pos + ex] = static_cast<uint32_t>(i);
        pos += tile;
    }
}

// ---------------------------------------------------------------------------
// query vectors: q = fl32(e_h + w_r) (TransE) or fl32(e_h * w_r) (DistMult),
// the first rounding of the screening arithmetic of every edge weight.  A block
// takes the queries q0 .. q0 + n - 1 of its chunk, each padded with zeros to dp, and
// zero vectors up to a multiple of QP.
// ---------------------------------------------------------------------------
template <int QP>
__device__ __forceinline__ int load_queries(const ScanArgs& a, int dp, float* sq, float* sthr, int* first) {
    const int d = a.g.d;
    const bool transe = a.g.fn == MHR_SCORE_TRANSE_L1;
    const int q0 = blockIdx.y * a.chunk, n = min(a.chunk, a.nq - q0);
    for (int qi = threadIdx.x >> 5; qi < (n + QP - 1) / QP * QP; qi += kScanWarps) {
        const bool real = qi < n;
        const uint32_t h = real ? a.h[q0 + qi] : 0u, r = real ? a.r[q0 + qi] : 0u;
#pragma unroll 4
        for (int j = threadIdx.x & 31; j < dp; j += 32) {
            float x = 0.f;
            if (real && j < d) {
                const float e = emb_f32(a.g.vemb, a.g.dtype, h, d, j), w = emb_f32(a.g.remb, a.g.dtype, r, d, j);
                x = transe ? __fadd_rn(e, w) : __fmul_rn(e, w);
            }
            sq[static_cast<int64_t>(qi) * dp + j] = x;
        }
    }
    for (int qi = threadIdx.x; qi < n + QP; qi += blockDim.x)
        sthr[qi] = qi >= n ? INFINITY : (a.thr ? a.thr[q0 + qi] : -INFINITY);
    if (a.thr == nullptr && blockIdx.x == 0)  // every score is kept
        for (int qi = threadIdx.x; qi < n; qi += blockDim.x) a.cnt[q0 + qi] = static_cast<unsigned>(a.n_visit);
    __syncthreads();
    *first = q0;
    return n;
}

// ---------------------------------------------------------------------------
// The scans.  A lane group holds ROWS candidate rows in registers (up to 16 elements
// of each per lane), and each query vector load from shared memory feeds all of
// them; QP queries are scored at a time.  Their ROWS * QP partial sums are reduced
// together: each exchange step halves the sums a lane carries, so with eight of
// them and eight lanes every lane ends with one score and tests it.
//
// What bounds them: many queries, the issue of the fp32 pipe (TransE: half a paired
// subtraction and an addition per element); a few, the rows' bandwidth.  64 queries
// x 167,000 candidates of 128 fp32 values, TransE: 247 us (two rows, each sum reduced
// and tested by itself) -> 131 us, the sample's 8,192 candidates 55 -> 15 us by
// cutting the queries into chunks as well; one query over 1M candidates 75 us, 6.8
// TB/s, before and after.
// ---------------------------------------------------------------------------

template <bool BF16>
__device__ __forceinline__ void unpack_row(const uint4& w, float* x) {
    if constexpr (BF16) {
        x[0] = bf_lo(w.x);
        x[1] = bf_hi(w.x);
        x[2] = bf_lo(w.y);
        x[3] = bf_hi(w.y);
        x[4] = bf_lo(w.z);
        x[5] = bf_hi(w.z);
        x[6] = bf_lo(w.w);
        x[7] = bf_hi(w.w);
    } else {
        x[0] = __uint_as_float(w.x);
        x[1] = __uint_as_float(w.y);
        x[2] = __uint_as_float(w.z);
        x[3] = __uint_as_float(w.w);
    }
}

// The score of query qi for candidate i of the visit order, on the lanes with
// `mine`.  Keep-every-score mode (no threshold): candidate i owns slot i, no counter
// needed; otherwise the few lanes that pass append, one counter update per query.
__device__ __forceinline__ void emit(const ScanArgs& a, int qi, bool mine, float s32, int64_t i, int lane, float thr) {
    const bool keep = mine && s32 >= thr;
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    if (!keep) return;
    const int64_t at = i * a.stride;
    const uint32_t v = a.cand ? __ldg(a.cand + at) : static_cast<uint32_t>(at);
    int64_t pos = i;
    if (a.thr) {
        const unsigned peers = __match_any_sync(m, qi);
        const int leader = __ffs(peers) - 1;
        unsigned base = 0;
        if (lane == leader) base = atomicAdd(a.cnt + qi, static_cast<unsigned>(__popc(peers)));
        pos = __shfl_sync(peers, base, leader) + static_cast<unsigned>(__popc(peers & ((1u << lane) - 1u)));
        if (pos >= a.cap) return;
    }
    a.surv[static_cast<int64_t>(qi) * a.cap + pos] = SurvRec{s32, v};
}

// two fp32 operations at once (a 64-bit register pair), each rounded as by itself
__device__ __forceinline__ float2 sub2(float2 x, float2 y) {
    float2 r;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(reinterpret_cast<unsigned long long&>(r))
        : "l"(reinterpret_cast<unsigned long long&>(x)), "l"(reinterpret_cast<unsigned long long&>(y)));
    return r;
}
__device__ __forceinline__ float2 fma2(float2 x, float2 y, float2 z) {
    float2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(reinterpret_cast<unsigned long long&>(r))
        : "l"(reinterpret_cast<unsigned long long&>(x)), "l"(reinterpret_cast<unsigned long long&>(y)),
          "l"(reinterpret_cast<unsigned long long&>(z)));
    return r;
}

// acc[r] += the row's terms of two elements: TransE into acc[r].x, DistMult into both halves
template <bool TRANSE>
__device__ __forceinline__ void add_terms(float2& acc, float2 q, float2 x) {
    if constexpr (TRANSE) {
        const float2 t = sub2(q, x);
        acc.x += fabsf(t.x);
        acc.y += fabsf(t.y);
    } else {
        acc = fma2(q, x, acc);
    }
}

// Sums over a group of G lanes of N values per lane.  L exchange steps (2^L <= G, N)
// leave N >> L sums per lane: value (returned index + j) in v[j], each on the lanes
// s < 2^L and their repetitions.
template <int N, int L>
__device__ __forceinline__ int reduce_group(float (&v)[N], int s, int G) {
    int first = 0;
#pragma unroll
    for (int k = 0; k < L; ++k) {
        const int half = N >> (k + 1);
        const bool hi = ((s >> k) & 1) != 0;
#pragma unroll
        for (int j = 0; j < half; ++j) {
            const float send = hi ? v[j] : v[j + half], keep = hi ? v[j + half] : v[j];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, send, 1 << k);
        }
        first += hi ? half : 0;
    }
    for (int o = 1 << L; o < G; o <<= 1) {
#pragma unroll
        for (int j = 0; j < (N >> L); ++j) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
    }
    return first;
}

// the scores of ROWS rows from i0 for QP queries from qi (values q * ROWS + row)
template <int ROWS, int QP, int L, bool TRANSE>
__device__ __forceinline__ void finish_rows(const ScanArgs& a, float (&v)[ROWS * QP], int s, int G, int64_t i0, int q0,
                                            int qi, const float* sthr, int lane) {
    const int first = reduce_group<ROWS * QP, L>(v, s, G);
#pragma unroll
    for (int j = 0; j < ((ROWS * QP) >> L); ++j) {
        const int id = first + j, q = qi + id / ROWS;
        const int64_t i = i0 + id % ROWS;
        emit(a, q0 + q, s < (1 << L) && i < a.n_visit, TRANSE ? __fsub_rn(a.g.gamma32, v[j]) : v[j], i, lane, sthr[q]);
    }
}

// rows of whole 16-byte vectors: lane s of a group holds vectors s, s + G, ... (NV of
// them per row), so the group's loads of one step are consecutive.  Rows and query
// vectors are padded with zeros to G * NV vectors, whose terms are zero.  G >= 2^L.
template <int NV, int ROWS, int QP, int L, bool BF16, bool TRANSE>
__global__ void __launch_bounds__(kScanThreads, ROWS == 2 ? 4 : 2) k_tail_scan(const __grid_constant__ ScanArgs a) {
    extern __shared__ float4 smem4[];
    float* sq = reinterpret_cast<float*>(smem4);
    constexpr int EV = BF16 ? 8 : 4;
    const int d = a.g.d, G = a.G, dp = G * NV * EV;
    float* sthr = sq + static_cast<int64_t>((a.chunk + QP - 1) / QP * QP) * dp;
    int q0;
    const int nq = load_queries<QP>(a, dp, sq, sthr, &q0);

    const int dv = d / EV;
    const int lane = threadIdx.x & 31;
    const int s = lane & (G - 1);
    const int grp = lane / G;
    const int cpw = ROWS * (32 / G);
    const int64_t ntiles = (a.n_visit + cpw - 1) / cpw;
    const int64_t nwarps = static_cast<int64_t>(gridDim.x) * kScanWarps;
    const size_t row_bytes = static_cast<size_t>(d) * (BF16 ? 2 : 4);

    for (int64_t t = static_cast<int64_t>(blockIdx.x) * kScanWarps + (threadIdx.x >> 5); t < ntiles; t += nwarps) {
        const int64_t i0 = t * cpw + ROWS * grp;
        float x[ROWS][NV * EV];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int64_t i = i0 + r;
            const bool valid = i < a.n_visit;
            uint32_t v = 0;
            if (valid) v = a.cand ? __ldg(a.cand + i * a.stride) : static_cast<uint32_t>(i * a.stride);
            const uint4* row = reinterpret_cast<const uint4*>(static_cast<const char*>(a.g.vemb) + v * row_bytes);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const int vi = s + G * k;
                unpack_row<BF16>(valid && vi < dv ? __ldg(row + vi) : make_uint4(0u, 0u, 0u, 0u), x[r] + k * EV);
            }
        }
        const float4* q4 = reinterpret_cast<const float4*>(sq) + s * (EV / 4);
        for (int qi = 0; qi < nq; qi += QP, q4 += QP * (dp / 4)) {
            float2 acc[QP][ROWS];
#pragma unroll
            for (int q = 0; q < QP; ++q)
#pragma unroll
                for (int r = 0; r < ROWS; ++r) acc[q][r] = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < NV; ++k)
#pragma unroll
                for (int e4 = 0; e4 < EV / 4; ++e4)
#pragma unroll
                    for (int q = 0; q < QP; ++q) {
                        const float4 qq = q4[q * (dp / 4) + G * k * (EV / 4) + e4];
#pragma unroll
                        for (int r = 0; r < ROWS; ++r) {
                            const float* y = x[r] + k * EV + e4 * 4;
                            add_terms<TRANSE>(acc[q][r], make_float2(qq.x, qq.y), make_float2(y[0], y[1]));
                            add_terms<TRANSE>(acc[q][r], make_float2(qq.z, qq.w), make_float2(y[2], y[3]));
                        }
                    }
            float v[ROWS * QP];
#pragma unroll
            for (int q = 0; q < QP; ++q)
#pragma unroll
                for (int r = 0; r < ROWS; ++r) v[q * ROWS + r] = acc[q][r].x + acc[q][r].y;
            finish_rows<ROWS, QP, L, TRANSE>(a, v, s, G, i0, q0, qi, sthr, lane);
        }
    }
}

// rows of up to 32 * KX elements of any length: a warp per ROWS rows, lane s holds
// elements s, s + 32, ...
template <int KX, int ROWS, int QP, bool TRANSE>
__global__ void __launch_bounds__(kScanThreads, 2) k_tail_scan_el(const __grid_constant__ ScanArgs a) {
    extern __shared__ float4 smem4[];
    float* sq = reinterpret_cast<float*>(smem4);
    const int d = a.g.d;
    constexpr int dp = 32 * KX, L = ROWS * QP == 8 ? 3 : 1;
    static_assert(ROWS * QP == 8 || ROWS * QP == 2, "exchange steps for eight sums or two");
    float* sthr = sq + static_cast<int64_t>((a.chunk + QP - 1) / QP * QP) * dp;
    int q0;
    const int nq = load_queries<QP>(a, dp, sq, sthr, &q0);
    const int lane = threadIdx.x & 31;
    const int64_t ntiles = (a.n_visit + ROWS - 1) / ROWS;
    const int64_t nwarps = static_cast<int64_t>(gridDim.x) * kScanWarps;
    for (int64_t t = static_cast<int64_t>(blockIdx.x) * kScanWarps + (threadIdx.x >> 5); t < ntiles; t += nwarps) {
        const int64_t i0 = t * ROWS;
        float x[ROWS][KX];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int64_t i = i0 + r;
            const bool valid = i < a.n_visit;
            uint32_t v = 0;
            if (valid) v = a.cand ? __ldg(a.cand + i * a.stride) : static_cast<uint32_t>(i * a.stride);
#pragma unroll
            for (int k = 0; k < KX; ++k) {
                const int j = lane + 32 * k;
                x[r][k] = valid && j < d ? emb_f32(a.g.vemb, a.g.dtype, v, d, j) : 0.f;
            }
        }
        const float* sv = sq + lane;
        for (int qi = 0; qi < nq; qi += QP, sv += QP * dp) {
            float v[ROWS * QP];
#pragma unroll
            for (int j = 0; j < ROWS * QP; ++j) v[j] = 0.f;
#pragma unroll
            for (int k = 0; k < KX; ++k)
#pragma unroll
                for (int q = 0; q < QP; ++q) {
                    const float qq = sv[q * dp + 32 * k];
#pragma unroll
                    for (int r = 0; r < ROWS; ++r) {
                        float& c = v[q * ROWS + r];
                        if constexpr (TRANSE) c += fabsf(__fsub_rn(qq, x[r][k]));
                        else c += qq * x[r][k];
                    }
                }
            finish_rows<ROWS, QP, L, TRANSE>(a, v, lane, 32, i0, q0, qi, sthr, lane);
        }
    }
}

// a lane's sums of candidate v's row for Q queries from q, elements lane, lane + 32, ...
template <bool TRANSE, int Q>
__device__ __forceinline__ void any_terms(const DevGraph& g, uint32_t v, const float* q, int lane, float (&acc)[2]) {
    const int d = g.d;
    acc[0] = acc[1] = 0.f;
    auto run = [&](auto at) {
        constexpr int U = 8;  // elements in flight
        int j = lane;
        for (; j + 32 * (U - 1) < d; j += 32 * U) {
            float c[U];
#pragma unroll
            for (int u = 0; u < U; ++u) c[u] = at(j + 32 * u);
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int k = 0; k < Q; ++k) {
                    const float x = q[k * d + j + 32 * u];
                    if constexpr (TRANSE) acc[k] += fabsf(__fsub_rn(x, c[u]));
                    else acc[k] += x * c[u];
                }
        }
        for (; j < d; j += 32) {
            const float c = at(j);
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                const float x = q[k * d + j];
                if constexpr (TRANSE) acc[k] += fabsf(__fsub_rn(x, c));
                else acc[k] += x * c;
            }
        }
    };
    if (g.dtype == MHR_F32) {
        const float* row = static_cast<const float*>(g.vemb) + static_cast<int64_t>(v) * d;
        run([&](int j) { return __ldg(row + j); });
    } else {
        const uint16_t* row = static_cast<const uint16_t*>(g.vemb) + static_cast<int64_t>(v) * d;
        run([&](int j) { return bf16_to_f32(__ldg(row + j)); });
    }
}

// Longer rows: one warp per candidate, the row read again (from L1) for every two
// queries.  What bounds it is the latency of those loads and of each query's chain of
// additions, so eight elements of the row are in flight and two chains run side by side.
// 64 queries x 100,000 candidates of 1,000 fp32 values: DistMult 5.40 -> 3.85 ms, TransE
// 5.13 -> 3.84 ms.
template <bool TRANSE>
__global__ void __launch_bounds__(kScanThreads) k_tail_scan_any(const __grid_constant__ ScanArgs a) {
    extern __shared__ float4 smem4[];
    float* sq = reinterpret_cast<float*>(smem4);
    const int d = a.g.d;
    float* sthr = sq + static_cast<int64_t>(a.chunk) * d;
    int q0;
    const int nq = load_queries<1>(a, d, sq, sthr, &q0);
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = static_cast<int64_t>(gridDim.x) * kScanWarps;
    const float gamma32 = a.g.gamma32;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * kScanWarps + (threadIdx.x >> 5); i < a.n_visit; i += nwarps) {
        const int64_t pos = i * a.stride;
        const uint32_t v = a.cand ? __ldg(a.cand + pos) : static_cast<uint32_t>(pos);
        for (int qi = 0; qi < nq; qi += 2) {
            float acc[2];
            if (qi + 1 < nq) any_terms<TRANSE, 2>(a.g, v, sq + static_cast<int64_t>(qi) * d, lane, acc);
            else any_terms<TRANSE, 1>(a.g, v, sq + static_cast<int64_t>(qi) * d, lane, acc);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (qi + k == nq) break;
                for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
                emit(a, q0 + qi + k, lane == 0, TRANSE ? __fsub_rn(gamma32, acc[k]) : acc[k], i, lane, sthr[qi + k]);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// CTA-wide radix select: the k-th largest key (1-based), 8 bits per pass
// ---------------------------------------------------------------------------
struct SelectSmem {
    unsigned hist[256];
    int digit;
    unsigned krem;
    unsigned count;
};

// warp 0: the digit whose bin holds the krem-th largest remaining key, and the
// rank inside that bin (bins scanned from 255 down)
__device__ __forceinline__ void pick_digit(SelectSmem& sm, unsigned krem) {
    if (threadIdx.x < 32) {
        const int L = threadIdx.x;
        unsigned c[8], local = 0;
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            c[m] = sm.hist[255 - 8 * L - m];
            local += c[m];
        }
        const unsigned incl = warp_incl_scan<unsigned>(local);
        const unsigned excl = incl - local;
        if (excl < krem && krem <= incl) {
            unsigned acc = excl;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                if (acc + c[m] >= krem) {
                    sm.digit = 255 - 8 * L - m;
                    sm.krem = krem - acc;
                    break;
                }
                acc += c[m];
            }
        }
    }
}

// the order-preserving key of an fp64 score, +0 and -0 mapped together (the
// result order compares scores numerically)
__device__ __forceinline__ uint64_t score_key(double w) {
    if (w == 0.0) w = 0.0;
    const uint64_t b = static_cast<uint64_t>(__double_as_longlong(w));
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// k-th largest fp32 survivor score (1 <= k <= n)
__device__ float select_kth_score(const SurvRec* a, int64_t n, int64_t k, SelectSmem& sm) {
    uint32_t prefix = 0, mask = 0;
    unsigned krem = static_cast<unsigned>(k);
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int b = threadIdx.x; b < 256; b += blockDim.x) sm.hist[b] = 0u;
        __syncthreads();
        for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
            const uint32_t key = f2key(a[i].s);
            if ((key & mask) == prefix) atomicAdd(&sm.hist[(key >> shift) & 255u], 1u);
        }
        __syncthreads();
        pick_digit(sm, krem);
        __syncthreads();
        prefix |= static_cast<uint32_t>(sm.digit) << shift;
        mask |= 255u << shift;
        krem = sm.krem;
        __syncthreads();
    }
    return key2f(prefix);
}

// composite key of a band record: (score key, ~v), larger = earlier in the result
__device__ __forceinline__ unsigned band_digit(uint64_t hi, uint32_t lo, int p) {
    return p < 8 ? static_cast<unsigned>((hi >> (56 - 8 * p)) & 255u)
                 : static_cast<unsigned>((lo >> (24 - 8 * (p - 8))) & 255u);
}

// k-th largest composite key of n band records (1 <= k <= n); keys are distinct
__device__ void select_kth_band(const BandRec* a, int64_t n, int64_t k, SelectSmem& sm, uint64_t* khi,
                                uint32_t* klo) {
    uint64_t phi = 0, mhi = 0;
    uint32_t plo = 0, mlo = 0;
    unsigned krem = static_cast<unsigned>(k);
    for (int p = 0; p < 12; ++p) {
        for (int b = threadIdx.x; b < 256; b += blockDim.x) sm.hist[b] = 0u;
        __syncthreads();
        for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
            const uint64_t hi = score_key(a[i].w);
            const uint32_t lo = ~a[i].v;
            if ((hi & mhi) == phi && (lo & mlo) == plo) atomicAdd(&sm.hist[band_digit(hi, lo, p)], 1u);
        }
        __syncthreads();
        pick_digit(sm, krem);
        __syncthreads();
        const uint64_t dg = static_cast<uint64_t>(sm.digit);
        if (p < 8) {
            phi |= dg << (56 - 8 * p);
            mhi |= 255ull << (56 - 8 * p);
        } else {
            plo |= static_cast<uint32_t>(dg) << (24 - 8 * (p - 8));
            mlo |= 255u << (24 - 8 * (p - 8));
        }
        krem = sm.krem;
        __syncthreads();
    }
    *khi = phi;
    *klo = plo;
}

// ---------------------------------------------------------------------------
// sampling threshold: thr[q] = (K-th best sampled fp32 score) - 2E, rounded
// down; -inf when the sample holds fewer than K candidates
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kFinalThreads) k_tail_thr(const SurvRec* __restrict__ surv, int64_t cap,
                                                           const unsigned* __restrict__ cnt, int K, double E2,
                                                           float* __restrict__ thr) {
    __shared__ SelectSmem sm;
    const int q = blockIdx.x;
    const int64_t n = min(static_cast<int64_t>(cnt[q]), cap);
    if (n < K) {
        if (threadIdx.x == 0) thr[q] = -INFINITY;
        return;
    }
    const float kth = select_kth_score(surv + static_cast<int64_t>(q) * cap, n, K, sm);
    if (threadIdx.x == 0) thr[q] = __double2float_rd(__dsub_rd(static_cast<double>(kth), E2));
}

// ---------------------------------------------------------------------------
// per query: band, fp64 rescoring, the K best in order
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool ranks_before(const BandRec& x, const BandRec& y) {
    return x.w > y.w || (x.w == y.w && x.v < y.v);
}

constexpr int kQ64Max = 2048;  // rows up to this length use the shared fp64 query vector

template <bool TRANSE>
__device__ __forceinline__ double row_term64(double q, float c) {
    if constexpr (TRANSE) return fabs(__dsub_rn(q, static_cast<double>(c)));
    else return __dmul_rn(q, static_cast<double>(c));
}

// w(h, r, v) in the canonical order, with q64[j] = e_h[j] + w_r[j] (TransE)
// or e_h[j] * w_r[j] (DistMult) already formed in fp64: the same operations
// on the same values as the reference definition, j = 0..d-1 in order
template <bool TRANSE>
__device__ double rescore_row(const DevGraph& g, const double* q64, uint32_t v) {
    const int d = g.d;
    double acc = 0.0;
    if (g.dtype == MHR_F32 && (d & 3) == 0) {
        const float4* c4 = reinterpret_cast<const float4*>(static_cast<const float*>(g.vemb) + static_cast<int64_t>(v) * d);
#pragma unroll 4
        for (int j4 = 0; j4 < (d >> 2); ++j4) {
            const float4 c = __ldg(c4 + j4);
            const double* q = q64 + 4 * j4;
            acc = __dadd_rn(acc, row_term64<TRANSE>(q[0], c.x));
            acc = __dadd_rn(acc, row_term64<TRANSE>(q[1], c.y));
            acc = __dadd_rn(acc, row_term64<TRANSE>(q[2], c.z));
            acc = __dadd_rn(acc, row_term64<TRANSE>(q[3], c.w));
        }
    } else if (g.dtype == MHR_BF16 && (d & 7) == 0) {
        const uint4* c8 = reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(g.vemb) + static_cast<int64_t>(v) * d);
#pragma unroll 2
        for (int j8 = 0; j8 < (d >> 3); ++j8) {
            const uint4 w = __ldg(c8 + j8);
            const double* q = q64 + 8 * j8;
            acc = __dadd_rn(acc, row_term64<TRANSE>(q[0], bf_lo(w.x)));
            acc = __dadd_rn(acc, row_term64<TRANSE>(q[1], bf_hi(w.x)));
            acc = __dadd_rn(acc, row_term64<TRANSE>(q[2], bf_lo(w.y)));
            acc = __dadd_rn(acc, row_term64<TRANSE>(q[3], bf_hi(w.y)));
            acc = __dadd_rn(acc, row_term64<TRANSE>(q[4], bf_lo(w.z)));
            acc = __dadd_rn(acc, row_term64<TRANSE>(q[5], bf_hi(w.z)));
            acc = __dadd_rn(acc, row_term64<TRANSE>(q[6], bf_lo(w.w)));
            acc = __dadd_rn(acc, row_term64<TRANSE>(q[7], bf_hi(w.w)));
        }
    } else {
        for (int j = 0; j < d; ++j) acc = __dadd_rn(acc, row_term64<TRANSE>(q64[j], emb_f32(g.vemb, g.dtype, v, d, j)));
    }
    return TRANSE ? __dsub_rn(g.gamma, acc) : acc;
}

__global__ void __launch_bounds__(kFinalThreads)
    k_tail_final(DevGraph g, const uint32_t* __restrict__ h, const uint16_t* __restrict__ r,
                 const SurvRec* __restrict__ surv, int64_t cap, const unsigned* __restrict__ cnt,
                 BandRec* __restrict__ band, int K, double E2, mhr_tail* __restrict__ out,
                 int32_t* __restrict__ n_out, unsigned* __restrict__ band_cnt) {
    __shared__ SelectSmem sm;
    extern __shared__ __align__(16) BandRec sbuf[];  // kSortMax records, then the fp64 query vector
    double* q64 = reinterpret_cast<double*>(sbuf + kSortMax);
    const int q = blockIdx.x;
    if (static_cast<int64_t>(cnt[q]) > cap) return;  // overflowed: rescanned alone by the host
    const int64_t n = cnt[q];
    const SurvRec* a = surv + static_cast<int64_t>(q) * cap;
    BandRec* b = band + static_cast<int64_t>(q) * cap;
    const uint32_t hq = h[q], rq = r[q];
    const bool transe = g.fn == MHR_SCORE_TRANSE_L1;
    const bool shared_q = g.d <= kQ64Max;

    // 1. the band: survivors within 2E of the K-th best fp32 score
    double lo = -INFINITY;
    if (n > K) lo = __dsub_rd(static_cast<double>(select_kth_score(a, n, K, sm)), E2);
    if (threadIdx.x == 0) sm.count = 0u;
    bool bad = false;  // the query's own rows are no multiples of the integers' unit
    for (int j = threadIdx.x; j < g.d; j += blockDim.x) {
        const float e = emb_f32(g.vemb, g.dtype, hq, g.d, j), w = emb_f32(g.remb, g.dtype, rq, g.d, j);
        if (transe) add_fixed(add_fixed(0, e, false, g.qbits, bad), w, false, g.qbits, bad);
        if (!shared_q) continue;
        const double e64 = static_cast<double>(e), w64 = static_cast<double>(w);
        q64[j] = transe ? __dadd_rn(e64, w64) : __dmul_rn(e64, w64);
    }
    const bool whole = !__syncthreads_or(bad);
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        const SurvRec x = a[i];
        if (static_cast<double>(x.s) >= lo) {
            const unsigned p = atomicAdd(&sm.count, 1u);
            b[p].v = x.v;
        }
    }
    __syncthreads();
    const unsigned nb = sm.count;
    // fp64 rescoring.  TransE in integers, eight lanes per member and four members at a
    // time; a lane's share of a row is 32 coordinates' steps, so short rows of many
    // members, members the integers do not hold and DistMult go one per thread, over
    // dense warps.  200,000 members of 4 values: 2.1 ms by threads, 13 ms by a warp per
    // member; the whole call for 1,000 members: d = 16 157 and 155 us, 48 180 and 176, 64
    // 194 and 172, 128 252 and 189; for 40,000: d = 16 1.05 and 1.21 ms, 32 1.59 and
    // 1.20, 48 2.14 and 2.47, 64 2.68 and 1.85, 128 4.86 and 3.09; up to 128 members
    // the integers are never slower (threads, integers).
    const bool fixed = transe && whole && (nb <= 128u || g.d >= 64 || g.d % 32 == 0);
    __syncthreads();  // everyone has nb
    if (threadIdx.x == 0) sm.count = 0u;
    __syncthreads();
    if (fixed) {
        const int lane = threadIdx.x & 31;
        constexpr unsigned W = kFinalThreads / 32;
        const unsigned per = min(32u, (nb + 4 * W - 1) / (4 * W) * 4u);  // members of a warp's step
        for (unsigned b0 = (threadIdx.x >> 5) * per; b0 < nb; b0 += per * W) {
            const int m = static_cast<int>(min(per, nb - b0));
            bool left = lane < m;
            const uint32_t v = left ? b[b0 + lane].v : 0u;
            const double w = warp_w64_fixed_each(g, hq, rq, v, m, lane, left);
            if (lane < m) b[b0 + lane] = BandRec{w, v, left ? 1u : 0u};
            if (left) sm.count = 1u;
        }
        __syncthreads();
    }
    if (!fixed || sm.count) {
        for (unsigned p = threadIdx.x; p < nb; p += blockDim.x) {
            const uint32_t v = b[p].v;
            if (fixed && b[p].pad == 0u) continue;
            double w;
            if (!shared_q) w = edge_w64(g, hq, rq, v);
            else if (transe) w = rescore_row<true>(g, q64, v);
            else w = rescore_row<false>(g, q64, v);
            b[p] = BandRec{w, v, 0u};
        }
    }
    __syncthreads();

    // a short band: a record's place is the number of records before it
    if (nb <= static_cast<unsigned>(kRankMax)) {
        uint64_t* keys = reinterpret_cast<uint64_t*>(sbuf);  // (score key, vertex), two words a record
        for (unsigned i = threadIdx.x; i < nb; i += blockDim.x) {
            keys[2 * i] = score_key(b[i].w);
            keys[2 * i + 1] = b[i].v;
        }
        __syncthreads();
        for (unsigned i = threadIdx.x; i < nb; i += blockDim.x) {
            const uint64_t hi = keys[2 * i], v = keys[2 * i + 1];
            int rank = 0;
            for (unsigned j = 0; j < nb; ++j) {
                const ulonglong2 o = *reinterpret_cast<const ulonglong2*>(keys + 2 * j);
                rank += o.x > hi || (o.x == hi && o.y < v) ? 1 : 0;
            }
            if (rank < K) out[static_cast<int64_t>(q) * K + rank] = mhr_tail{b[i].w, static_cast<uint32_t>(v), 0u};
        }
        if (threadIdx.x == 0) {
            n_out[q] = static_cast<int32_t>(min(nb, static_cast<unsigned>(K)));
            band_cnt[q] = nb;
        }
        return;
    }

    // 2. the records to sort: the whole band, or exactly its K best
    unsigned m;
    if (nb <= static_cast<unsigned>(kSortMax)) {
        for (unsigned i = threadIdx.x; i < nb; i += blockDim.x) sbuf[i] = b[i];
        m = nb;
    } else {
        uint64_t khi;
        uint32_t klo;
        select_kth_band(b, nb, K, sm, &khi, &klo);
        if (threadIdx.x == 0) sm.count = 0u;
        __syncthreads();
        for (int64_t i = threadIdx.x; i < nb; i += blockDim.x) {
            const uint64_t hi = score_key(b[i].w);
            const uint32_t lw = ~b[i].v;
            if (hi > khi || (hi == khi && lw >= klo)) {
                const unsigned p = atomicAdd(&sm.count, 1u);
                if (p < static_cast<unsigned>(kSortMax)) sbuf[p] = b[i];
            }
        }
        __syncthreads();
        m = min(sm.count, static_cast<unsigned>(kSortMax));
    }
    unsigned P = 1;
    while (P < m) P <<= 1;
    for (unsigned i = m + threadIdx.x; i < P; i += blockDim.x) sbuf[i] = BandRec{-INFINITY, 0xffffffffu, 0u};
    __syncthreads();

    // 3. bitonic sort of P records, best first
    for (unsigned size = 2; size <= P; size <<= 1) {
        for (unsigned stride = size >> 1; stride > 0; stride >>= 1) {
            for (unsigned i = threadIdx.x; i < P; i += blockDim.x) {
                const unsigned j = i ^ stride;
                if (j > i) {
                    const BandRec x = sbuf[i], y = sbuf[j];
                    const bool best_first = (i & size) == 0;
                    if (best_first ? ranks_before(y, x) : ranks_before(x, y)) {
                        sbuf[i] = y;
                        sbuf[j] = x;
                    }
                }
            }
            __syncthreads();
        }
    }

    // 4. output
    const unsigned nout = min(m, static_cast<unsigned>(K));
    mhr_tail* o = out + static_cast<int64_t>(q) * K;
    for (unsigned i = threadIdx.x; i < nout; i += blockDim.x) {
        mhr_tail t;
        t.score = sbuf[i].w;
        t.v = sbuf[i].v;
        t.pad = 0u;
        o[i] = t;
    }
    if (threadIdx.x == 0) {
        n_out[q] = static_cast<int32_t>(nout);
        band_cnt[q] = nb;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

cudaError_t grow(void** p, size_t* have, size_t want) {
    if (*have >= want && *p) return cudaSuccess;
    if (*p) cudaFree(*p);
    *p = nullptr;
    *have = 0;
    cudaError_t e = cudaMalloc(p, want ? want : 16);
    if (e == cudaSuccess) *have = want;
    return e;
}

// scan kernel and launch shape for the graph's row format
struct ScanKernel {
    void (*fn)(ScanArgs) = nullptr;
    int G = 1;
    int dp = 0;    // floats of a query vector in shared memory
    int qp = 1;    // queries scored at a time
    int rows = 1;  // candidates a warp takes at a time
    int per_sm = 1;
};

template <int NV, int ROWS, int QP, int L, bool BF16>
void use_scan(ScanKernel& k, bool transe, int G) {
    k.fn = transe ? k_tail_scan<NV, ROWS, QP, L, BF16, true> : k_tail_scan<NV, ROWS, QP, L, BF16, false>;
    k.G = G;
    k.dp = G * NV * (BF16 ? 8 : 4);
    k.qp = QP;
    k.rows = ROWS * (32 / G);
}

template <int ROWS, int QP>
void use_scan_vec(ScanKernel& k, const DevGraph& dg) {
    constexpr int N = ROWS * QP, L = N == 8 ? 3 : 1;
    const bool transe = dg.fn == MHR_SCORE_TRANSE_L1, bf = dg.dtype == MHR_BF16;
    const int dv = dg.d / (bf ? 8 : 4), nvmax = bf ? 2 : 4;
    int G = 1;
    while ((dv + G - 1) / G > nvmax) G <<= 1;
    if (G == 1) {
        if (bf) use_scan<2, ROWS, QP, 0, true>(k, transe, G);
        else use_scan<4, ROWS, QP, 0, false>(k, transe, G);
    } else if (G == 2 || L == 1) {
        if (bf) use_scan<2, ROWS, QP, 1, true>(k, transe, G);
        else use_scan<4, ROWS, QP, 1, false>(k, transe, G);
    } else if (G == 4) {
        if (bf) use_scan<2, ROWS, QP, L == 3 ? 2 : L, true>(k, transe, G);
        else use_scan<4, ROWS, QP, L == 3 ? 2 : L, false>(k, transe, G);
    } else {
        if (bf) use_scan<2, ROWS, QP, L, true>(k, transe, G);
        else use_scan<4, ROWS, QP, L, false>(k, transe, G);
    }
}

template <int KX>
void use_scan_el(ScanKernel& k, bool transe, bool few) {
    if (few) k.fn = transe ? k_tail_scan_el<KX, 2, 1, true> : k_tail_scan_el<KX, 2, 1, false>;
    else k.fn = transe ? k_tail_scan_el<KX, 4, 2, true> : k_tail_scan_el<KX, 4, 2, false>;
    k.G = 32;
    k.dp = 32 * KX;
    k.qp = few ? 1 : 2;
    k.rows = few ? 2 : 4;
}

// Whole vectors where the rows have them: as few lanes per row as hold it in 16
// elements each.  Otherwise element by element, up to 16 per lane.  Up to four
// queries the rows' bandwidth bounds the scan, and two rows per group with more
// warps in flight read them faster (one query over 1M rows of 512 bytes: 77 us, four
// rows 89 us); beyond, eight sums at a time take a third fewer instructions.
ScanKernel pick_scan(const DevGraph& dg, int nq) {
    const bool transe = dg.fn == MHR_SCORE_TRANSE_L1, bf = dg.dtype == MHR_BF16;
    const int d = dg.d, ev = bf ? 8 : 4, nvmax = bf ? 2 : 4;
    const bool few = nq <= 4;
    ScanKernel k;
    if (d % ev == 0 && d / ev <= 32 * nvmax) {
        if (few) use_scan_vec<2, 1>(k, dg);
        else use_scan_vec<4, 2>(k, dg);
        return k;
    }
    if (d <= 32) use_scan_el<1>(k, transe, few);
    else if (d <= 64) use_scan_el<2>(k, transe, few);
    else if (d <= 128) use_scan_el<4>(k, transe, few);
    else if (d <= 256) use_scan_el<8>(k, transe, few);
    else if (d <= 512) use_scan_el<16>(k, transe, few);
    else {
        k.fn = transe ? k_tail_scan_any<true> : k_tail_scan_any<false>;
        k.G = 32;
        k.dp = d;
    }
    return k;
}

// shared memory of a block that takes n queries
size_t scan_smem(const ScanKernel& sk, int n) {
    const size_t whole = (n + sk.qp - 1) / sk.qp * sk.qp;
    return whole * sk.dp * 4 + (whole + sk.qp) * 4;
}

// most queries a block takes: their vectors fit the query buffer (one iteration's always do)
int scan_fit(const ScanKernel& sk) {
    const size_t n = kQueryBytes / (static_cast<size_t>(sk.dp) * 4 + 4);
    return static_cast<int>(std::max<size_t>(sk.qp, n / sk.qp * sk.qp));
}

// Host-side set-up of the scan kernel for launches of up to nq_max queries:
// the shared-memory attribute and the resident blocks per SM.  Done once per
// call, before any event is recorded, so event times cover device work only.
mhr_status scan_setup(ScanKernel& sk, int nq_max) {
    const size_t smem = scan_smem(sk, std::min(nq_max, scan_fit(sk)));
    MHR_CUDA_TRY(cudaFuncSetAttribute(sk.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
    int n = 0;
    MHR_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, sk.fn, kScanThreads, smem));
    sk.per_sm = std::max(1, n);
    return MHR_OK;
}

// a.nq <= the nq_max given to scan_setup.  The queries are cut into chunks until
// every resident warp has about eight units of a tile and a chunk (an uneven last
// one then costs a tenth at most), down to eight queries, whose arithmetic still
// covers loading the tile's rows once more per chunk.
mhr_status launch_scan(const mhr_graph* g, const ScanKernel& sk, const ScanArgs& a, cudaStream_t st) {
    if (a.nq <= 0 || a.n_visit <= 0) return MHR_OK;
    const int64_t ntiles = (a.n_visit + sk.rows - 1) / sk.rows;
    const int64_t blocks = int64_t(std::max(1, g->num_sms)) * sk.per_sm;
    int64_t chunks = std::min<int64_t>((8 * blocks * kScanWarps + ntiles - 1) / ntiles, (a.nq + 7) / 8);
    chunks = std::max<int64_t>({int64_t(1), chunks, (a.nq + scan_fit(sk) - 1) / scan_fit(sk)});
    ScanArgs b = a;
    b.G = sk.G;
    b.chunk = static_cast<int>((a.nq + chunks - 1) / chunks + sk.qp - 1) / sk.qp * sk.qp;
    chunks = (a.nq + b.chunk - 1) / b.chunk;
    const int64_t need = (ntiles + kScanWarps - 1) / kScanWarps;
    const dim3 grid(static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(need, blocks / chunks))),
                    static_cast<unsigned>(chunks));
    sk.fn<<<grid, kScanThreads, scan_smem(sk, b.chunk), st>>>(b);
    MHR_CUDA_TRY(cudaGetLastError());
    return MHR_OK;
}

mhr_status ensure_cands(mhr_graph* g, int type, cudaStream_t st) {
    TailCache* tc = g->tail;
    if (tc->cands[type]) return MHR_OK;
    const int64_t n = g->dg.n;
    const int nb = kCompactBlocks;
    const int64_t per_block = (n + nb - 1) / nb;
    int64_t* counts = nullptr;
    MHR_CUDA_TRY(cudaMalloc(&counts, sizeof(int64_t) * (nb + 1)));
    auto bail = [&](mhr_status s) {
        cudaFree(counts);
        return s;
    };
    k_type_count<<<nb, 1024, 0, st>>>(g->dg.vtypes, n, type, per_block, counts);
    k_type_offsets<<<1, 1024, 0, st>>>(counts, nb);
    int64_t total = 0;
    cudaError_t e = cudaMemcpyAsync(&total, counts + nb, sizeof total, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return bail(cuda_fail(e, "candidate count"));
    uint32_t* ids = nullptr;
    e = cudaMalloc(&ids, sizeof(uint32_t) * std::max<int64_t>(1, total));
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaMalloc (candidate list)"));
    k_type_write<<<nb, 1024, 0, st>>>(g->dg.vtypes, n, type, per_block, counts, ids);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaFree(ids);
        return bail(cuda_fail(e, "candidate list"));
    }
    tc->cands[type] = ids;
    tc->ncand[type] = total;
    return bail(MHR_OK);
}

}  // namespace
}  // namespace mhr

using namespace mhr;

extern "C" mhr_status mhr_tail_topk(const mhr_graph* gc, int32_t nq, const uint32_t* h, const uint16_t* r,
                                    int32_t cand_type, int32_t K, mhr_tail* out, int32_t* n_out, mhr_mem mem,
                                    mhr_stats* stats, void* cuda_stream) {
    const auto t_start = std::chrono::steady_clock::now();
    MHR_TRY(check_graph(gc));
    mhr_graph* g = const_cast<mhr_graph*>(gc);
    if (nq < 0) return fail(MHR_EINVAL, "nq must be >= 0");
    if (K < 1) return fail(MHR_EINVAL, "K must be >= 1");
    if (K > MHR_TAIL_K_MAX) return fail(MHR_ERANGE, "K exceeds MHR_TAIL_K_MAX");
    if (cand_type < -1 || cand_type > 255) return fail(MHR_EINVAL, "cand_type must be in [-1, 255]");
    if (mem != MHR_MEM_HOST && mem != MHR_MEM_DEVICE) return fail(MHR_EINVAL, "unknown mem kind");
    const int d = g->dg.d;
    if (static_cast<size_t>(d) * 4 + 4 > kQueryBytes) return fail(MHR_ERANGE, "dim exceeds 16383 for tail prediction");
    if (stats) *stats = mhr_stats{};
    if (nq == 0) return MHR_OK;
    if (!h || !r || !out || !n_out) return fail(MHR_EINVAL, "NULL array");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);

    if (!g->tail) g->tail = new TailCache();
    TailCache* tc = g->tail;
    if (!tc->pinned) MHR_CUDA_TRY(cudaMallocHost(reinterpret_cast<void**>(&tc->pinned), kPinned));
    if (stats)
        for (cudaEvent_t& e : tc->ev)
            if (!e) MHR_CUDA_TRY(cudaEventCreate(&e));

    // validate the queries on the host (a short copy when they live on the device)
    std::vector<uint32_t> vh;
    std::vector<uint16_t> vr;
    const uint32_t* hh = h;
    const uint16_t* hr = r;
    if (mem == MHR_MEM_DEVICE) {
        uint32_t* ph = reinterpret_cast<uint32_t*>(tc->pinned);
        uint16_t* pr = reinterpret_cast<uint16_t*>(ph + nq);
        if (6ull * nq > kPinned) {
            vh.resize(nq);
            vr.resize(nq);
            ph = vh.data();
            pr = vr.data();
        }
        MHR_CUDA_TRY(cudaMemcpyAsync(ph, h, 4ull * nq, cudaMemcpyDeviceToHost, st));
        MHR_CUDA_TRY(cudaMemcpyAsync(pr, r, 2ull * nq, cudaMemcpyDeviceToHost, st));
        MHR_CUDA_TRY(cudaStreamSynchronize(st));
        hh = ph;
        hr = pr;
    }
    for (int i = 0; i < nq; ++i) {
        if (static_cast<int64_t>(hh[i]) >= g->dg.n) return fail(MHR_EINVAL, "head out of range");
        if (static_cast<int32_t>(hr[i]) >= g->dg.R) return fail(MHR_EINVAL, "relation out of range");
    }

    const uint32_t* cand = nullptr;
    int64_t Nc = g->dg.n;
    if (cand_type >= 0) {
        MHR_TRY(ensure_cands(g, cand_type, st));
        cand = tc->cands[cand_type];
        Nc = tc->ncand[cand_type];
    }

    // sizes: sample M, survivor capacity per query, queries per launch
    const int64_t M = std::min<int64_t>(Nc, std::max<int64_t>({int64_t(8192), int64_t(32) * K, Nc / 256}));
    const bool one_pass = M >= Nc;
    const int64_t ratio = one_pass ? 1 : (Nc + M - 1) / M;
    const int64_t capB = one_pass ? Nc : std::min<int64_t>(Nc, int64_t(8) * K * ratio + 8192);
    const int64_t capA = one_pass ? 0 : M;
    const size_t per_query = static_cast<size_t>(capA) * sizeof(SurvRec) +
                             static_cast<size_t>(capB) * (sizeof(SurvRec) + sizeof(BandRec)) + 64;
    int QB = static_cast<int>(std::min<int64_t>({static_cast<int64_t>(nq), int64_t(kMaxBatch),
                                                 static_cast<int64_t>(kQueryBytes / (static_cast<size_t>(d) * 4 + 4))}));
    QB = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(QB, static_cast<int64_t>(kScratchBudget / per_query))));

    // scratch layout
    size_t off = 0;
    auto carve = [&](size_t bytes) {
        const size_t o = off;
        off = align_up(off + bytes, 256);
        return o;
    };
    const size_t o_h = carve(4ull * nq), o_r = carve(2ull * nq), o_out = carve(sizeof(mhr_tail) * nq * K),
                 o_nout = carve(4ull * nq), o_thr = carve(4ull * QB), o_cnt = carve(4ull * QB * 3),
                 o_sa = carve(sizeof(SurvRec) * QB * capA),
                 o_sb = carve(sizeof(SurvRec) * QB * capB), o_band = carve(sizeof(BandRec) * QB * capB);
    MHR_CUDA_TRY(grow(&tc->scratch, &tc->scratch_bytes, off));
    char* base = static_cast<char*>(tc->scratch);
    uint32_t* d_h = reinterpret_cast<uint32_t*>(base + o_h);
    uint16_t* d_r = reinterpret_cast<uint16_t*>(base + o_r);
    mhr_tail* d_out = reinterpret_cast<mhr_tail*>(base + o_out);
    int32_t* d_nout = reinterpret_cast<int32_t*>(base + o_nout);
    float* d_thr = reinterpret_cast<float*>(base + o_thr);
    unsigned* d_cnt = reinterpret_cast<unsigned*>(base + o_cnt);  // [QB] sample, [QB] full pass, [QB] band
    unsigned* d_bc = d_cnt + 2 * QB;
    SurvRec* d_sa = reinterpret_cast<SurvRec*>(base + o_sa);
    SurvRec* d_sb = reinterpret_cast<SurvRec*>(base + o_sb);
    BandRec* d_band = reinterpret_cast<BandRec*>(base + o_band);
    if (mem == MHR_MEM_HOST) {
        MHR_CUDA_TRY(cudaMemcpyAsync(d_h, h, 4ull * nq, cudaMemcpyHostToDevice, st));
        MHR_CUDA_TRY(cudaMemcpyAsync(d_r, r, 2ull * nq, cudaMemcpyHostToDevice, st));
    } else {
        d_h = const_cast<uint32_t*>(h);
        d_r = const_cast<uint16_t*>(r);
        d_out = out;
        d_nout = n_out;
    }

    const double E2 = 2.0 * (g->eps32_edge + g->eps64_edge) * (1.0 + 1e-6);
    ScanKernel sk = pick_scan(g->dg, std::min(QB, nq));
    const size_t final_smem = sizeof(BandRec) * kSortMax + (d <= kQ64Max ? sizeof(double) * d : 0);
    MHR_CUDA_TRY(cudaFuncSetAttribute(k_tail_final, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(final_smem)));
    MHR_TRY(scan_setup(sk, std::min(QB, nq)));

    int64_t n_pairs = 0, n_surv = 0, n_band = 0, n_rescan = 0;
    double ms_scan = 0.0;
    if (stats) MHR_CUDA_TRY(cudaEventRecord(tc->ev[0], st));
    static_assert(sizeof(unsigned) * 2 * kMaxBatch <= kPinned, "a batch's counts fit the pinned buffer");
    unsigned* hc = reinterpret_cast<unsigned*>(tc->pinned);  // survivors, then band sizes
    unsigned* hb = hc + QB;
    for (int c0 = 0; c0 < nq && Nc > 0; c0 += QB) {
        const int qb = std::min(QB, nq - c0);
        MHR_CUDA_TRY(cudaMemsetAsync(d_cnt, 0, 4ull * QB * 2, st));
        ScanArgs a{};
        a.g = g->dg;
        a.h = d_h + c0;
        a.r = d_r + c0;
        a.nq = qb;
        a.cand = cand;
        unsigned* cntB = d_cnt + QB;
        if (!one_pass) {
            a.n_visit = M;
            a.stride = Nc / M;
            a.thr = nullptr;
            a.surv = d_sa;
            a.cap = capA;
            a.cnt = d_cnt;
            MHR_TRY(launch_scan(g, sk, a, st));
            k_tail_thr<<<qb, kFinalThreads, 0, st>>>(d_sa, capA, d_cnt, K, E2, d_thr);
            MHR_CUDA_TRY(cudaGetLastError());
            n_pairs += static_cast<int64_t>(qb) * M;
        }
        a.n_visit = Nc;
        a.stride = 1;
        a.thr = one_pass ? nullptr : d_thr;
        a.surv = d_sb;
        a.cap = capB;
        a.cnt = cntB;
        if (stats) MHR_CUDA_TRY(cudaEventRecord(tc->ev[2], st));
        MHR_TRY(launch_scan(g, sk, a, st));
        if (stats) MHR_CUDA_TRY(cudaEventRecord(tc->ev[3], st));
        n_pairs += static_cast<int64_t>(qb) * Nc;
        k_tail_final<<<qb, kFinalThreads, final_smem, st>>>(g->dg, d_h + c0, d_r + c0, d_sb, capB, cntB, d_band, K, E2,
                                                            d_out + static_cast<int64_t>(c0) * K, d_nout + c0, d_bc);
        MHR_CUDA_TRY(cudaGetLastError());
        MHR_CUDA_TRY(cudaMemcpyAsync(hc, cntB, 4ull * (QB + qb), cudaMemcpyDeviceToHost, st));
        MHR_CUDA_TRY(cudaStreamSynchronize(st));
        if (stats) {
            float ms = 0.f;
            MHR_CUDA_TRY(cudaEventElapsedTime(&ms, tc->ev[2], tc->ev[3]));
            ms_scan += ms;
        }
        for (int i = 0; i < qb; ++i) {
            if (static_cast<int64_t>(hc[i]) <= capB) {
                n_surv += hc[i];
                n_band += hb[i];
                continue;
            }
            // survivors overflowed the sized buffer: rescan this query alone with
            // room for every candidate
            const size_t o_bs = align_up(sizeof(SurvRec) * Nc, 256);
            const size_t need = o_bs + sizeof(BandRec) * Nc + 256;
            MHR_CUDA_TRY(grow(&tc->big, &tc->big_bytes, need));
            SurvRec* bs = static_cast<SurvRec*>(tc->big);
            BandRec* bb = reinterpret_cast<BandRec*>(static_cast<char*>(tc->big) + o_bs);
            unsigned* bcnt = d_cnt;  // the sample counts are no longer needed
            MHR_CUDA_TRY(cudaMemsetAsync(bcnt, 0, 4, st));
            ScanArgs b = a;
            b.h = d_h + c0 + i;
            b.r = d_r + c0 + i;
            b.nq = 1;
            b.thr = one_pass ? nullptr : d_thr + i;
            b.surv = bs;
            b.cap = Nc;
            b.cnt = bcnt;
            MHR_TRY(launch_scan(g, sk, b, st));
            k_tail_final<<<1, kFinalThreads, final_smem, st>>>(g->dg, d_h + c0 + i, d_r + c0 + i, bs, Nc, bcnt, bb, K, E2,
                                                               d_out + static_cast<int64_t>(c0 + i) * K, d_nout + c0 + i,
                                                               d_bc + i);
            MHR_CUDA_TRY(cudaGetLastError());
            unsigned c1 = 0, b1 = 0;
            MHR_CUDA_TRY(cudaMemcpyAsync(&c1, bcnt, 4, cudaMemcpyDeviceToHost, st));
            MHR_CUDA_TRY(cudaMemcpyAsync(&b1, d_bc + i, 4, cudaMemcpyDeviceToHost, st));
            MHR_CUDA_TRY(cudaStreamSynchronize(st));
            n_pairs += Nc;
            n_surv += c1;
            n_band += b1;
            ++n_rescan;
        }
    }
    // every batch ended with a synchronisation; wait for what came after
    bool wait = stats != nullptr;
    if (Nc == 0) {
        MHR_CUDA_TRY(cudaMemsetAsync(d_nout, 0, 4ull * nq, st));
        wait = true;
    }
    if (stats) MHR_CUDA_TRY(cudaEventRecord(tc->ev[1], st));
    if (mem == MHR_MEM_HOST) {
        MHR_CUDA_TRY(cudaMemcpyAsync(out, d_out, sizeof(mhr_tail) * nq * K, cudaMemcpyDeviceToHost, st));
        MHR_CUDA_TRY(cudaMemcpyAsync(n_out, d_nout, 4ull * nq, cudaMemcpyDeviceToHost, st));
        wait = true;
    }
    if (wait) MHR_CUDA_TRY(cudaStreamSynchronize(st));
    if (stats) {
        float ms_dev = 0.f;
        MHR_CUDA_TRY(cudaEventElapsedTime(&ms_dev, tc->ev[0], tc->ev[1]));
        stats->edges_scanned = n_pairs;
        stats->candidates = n_surv;
        stats->rescored = n_band;
        stats->dense_queries = n_rescan;
        stats->ms_device = ms_dev;
        stats->ms_join = ms_scan;
        stats->ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t_start).count();
    }
    return MHR_OK;
}
