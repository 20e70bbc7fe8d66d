// Graph residency: upload, validation, reverse CSR, error bounds, edge scores.
//
// The graph is the paper's three inputs (Sec. 3.1): the (h, r, t) edge list
// as a CSR by head, the entity embedding table and the relation embedding
// table.  Per-relation edge tables and hash-table embedding stores of the
// CPU design (Alg. 1, Sec. 3.3) become one CSR with a relation id per edge,
// its transpose, and dense row-major embedding arrays.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <string>

#include "mhr_exact.cuh"
#include "mhr_internal.cuh"
#include "mhr_score.cuh"
#include "mhr_sort.cuh"
#include "mhr_util.cuh"
#include <cuda_bf16.h>

static_assert(sizeof(mhr_graph_desc) == 104, "mhr_graph_desc layout");
static_assert(sizeof(mhr_path) == 24, "mhr_path layout");
static_assert(sizeof(mhr_query_opts) == 48, "mhr_query_opts layout");
static_assert(sizeof(mhr_constraints) == 40, "mhr_constraints layout");
static_assert(sizeof(mhr_graph_info) == 80, "mhr_graph_info layout");
static_assert(sizeof(mhr_mlp) == 32, "mhr_mlp layout");
static_assert(sizeof(mhr_stats) == 88, "mhr_stats layout");

namespace mhr {

static thread_local std::string g_last_error;

void set_error(const std::string& msg) { g_last_error = msg; }

mhr_status fail(mhr_status st, const std::string& msg) {
    g_last_error = msg;
    return st;
}

mhr_status cuda_fail(cudaError_t e, const char* what) {
    g_last_error = std::string("CUDA error in ") + what + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? MHR_ENOMEM : MHR_ECUDA;
}

int device_sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return sms;
}

mhr_status check_graph(const mhr_graph* g) {
    if (!g) return fail(MHR_EINVAL, "graph handle is NULL");
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != g->device)
        return fail(MHR_EINVAL, "the graph was loaded on another device than the current one");
    return MHR_OK;
}

// ---------------------------------------------------------------------------
// validation kernels (flags, never traps)
// ---------------------------------------------------------------------------
enum {
    kErrOffsets = 0,
    kErrColRange = 1,
    kErrRelRange = 2,
    kErrRowOrder = 3,
    kErrSelfLoop = 4,
    kErrNonFinite = 5,
    kErrCount = 8
};

__global__ void k_validate_offsets(const int64_t* __restrict__ off, int64_t n, int64_t E,
                                   int* __restrict__ err) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t u = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; u < n; u += stride)
        if (off[u] > off[u + 1]) err[kErrOffsets] = 1;
    if (blockIdx.x == 0 && threadIdx.x == 0 && (off[0] != 0 || off[n] != E)) err[kErrOffsets] = 1;
}

// Checks every edge and writes its source.  Each warp walks consecutive edges
// (the rows of the next 32 are found among the row starts after the last one),
// so short and empty rows cost what long ones do: 20 M edges in 0.1 ms (a warp
// per row took 1.26 ms).
__global__ void k_validate_edges(const int64_t* __restrict__ off, const uint32_t* __restrict__ col,
                                 const uint16_t* __restrict__ rel, int64_t n, int64_t E, int32_t R,
                                 uint32_t* __restrict__ src, int* __restrict__ err) {
    const int lane = threadIdx.x & 31;
    const int64_t warp_id = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
    const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    const int64_t steps = (E + 31) >> 5;
    const int64_t s0 = steps * warp_id / nwarps, s1 = steps * (warp_id + 1) / nwarps;
    if (s0 >= s1) return;  // warp-uniform
    int64_t row = warp_row_search(off, n, s0 * 32, lane);
    for (int64_t st = s0; st < s1; ++st) {
        const int64_t p = st * 32 + lane;
        const int64_t u = warp_rows_from(off, n, row, min(p, E - 1), lane);
        row = __shfl_sync(0xffffffffu, u, 31);
        if (p >= E) continue;
        const uint32_t c = col[p];
        const uint32_t r = rel[p];
        src[p] = static_cast<uint32_t>(u);
        if (c >= static_cast<uint64_t>(n)) err[kErrColRange] = 1;
        if (r >= static_cast<uint32_t>(R)) err[kErrRelRange] = 1;
        if (c == static_cast<uint64_t>(u)) err[kErrSelfLoop] = 1;
        if (p > off[u]) {
            const uint32_t pc = col[p - 1];
            const uint32_t pr = rel[p - 1];
            if (!(pc < c || (pc == c && pr < r))) err[kErrRowOrder] = 1;
        }
    }
}

__global__ void k_validate_finite(const void* __restrict__ tab, int dtype, int64_t count,
                                  int* __restrict__ err) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < count; i += stride) {
        float x = dtype == MHR_F32 ? static_cast<const float*>(tab)[i]
                                   : bf16_to_f32(static_cast<const uint16_t*>(tab)[i]);
        if (!isfinite(x)) err[kErrNonFinite] = 1;
    }
}

// ---------------------------------------------------------------------------
// reverse CSR
// ---------------------------------------------------------------------------
__global__ void k_count_in(const uint32_t* __restrict__ col, int64_t E, uint32_t* __restrict__ indeg) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t p = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; p < E; p += stride)
        atomicAdd(&indeg[col[p]], 1u);
}

__device__ __forceinline__ int64_t row_of_edge(const int64_t* __restrict__ off, int64_t n, int64_t p) {
    // largest u with off[u] <= p (rows may be empty)
    int64_t lo = 0, hi = n;  // answer in [0, n)
    while (lo + 1 < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (off[mid] <= p) lo = mid;
        else hi = mid;
    }
    return lo;
}

// edge[i]: the CSR edges sorted by destination (stable, so a row is in
// (source, relation) order)
__global__ void k_fill_reverse(const uint32_t* __restrict__ edge, int64_t E, const uint32_t* __restrict__ src,
                               const uint16_t* __restrict__ rel, const float* __restrict__ w,
                               uint32_t* __restrict__ rcol, uint16_t* __restrict__ rrel, float* __restrict__ rw) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < E; i += stride) {
        const uint32_t p = edge[i];
        rcol[i] = src[p];
        rrel[i] = rel[p];
        if (rw) rw[i] = w[p];
    }
}

// ---------------------------------------------------------------------------
// weight index: rows sorted by fp32 edge weight, descending
// ---------------------------------------------------------------------------
__global__ void k_weight_keys(const float* __restrict__ w, int64_t E, uint32_t* __restrict__ key) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < E; i += stride)
        key[i] = ~f2key(w[i]);
}

// key[i] = end[edge[i]]: the row (source or destination) of the i-th edge
__global__ void k_row_keys(const uint32_t* __restrict__ edge, int64_t E, const uint32_t* __restrict__ end,
                           uint32_t* __restrict__ key, uint32_t* __restrict__ copy) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < E; i += stride) {
        const uint32_t e = edge[i];
        key[i] = end[e];
        copy[i] = e;
    }
}

__global__ void k_fill_sorted(const uint32_t* __restrict__ edge, int64_t E, const uint32_t* __restrict__ far,
                              const uint16_t* __restrict__ rel, const float* __restrict__ w, uint2* __restrict__ se,
                              uint16_t* __restrict__ sr) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < E; i += stride) {
        const uint32_t e = edge[i];
        se[i] = make_uint2(far[e], __float_as_uint(w[e]));
        sr[i] = rel[e];
    }
}

__global__ void k_fill_records(const int64_t* __restrict__ off, int64_t n, const uint2* __restrict__ se,
                               VertexRec* __restrict__ v, unsigned long long* __restrict__ sums) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride) {
        const int64_t lo = off[i], m = off[i + 1] - lo;
        VertexRec r;
        r.deg = static_cast<uint32_t>(m);
        r.maxw = m > 0 ? __uint_as_float(se[lo].y) : 0.f;
        r.row = static_cast<uint32_t>(lo);
        r.maxp_key = 0u;
        const int64_t at[4] = {4, 32, 256, 2048};
#pragma unroll
        for (int k = 0; k < 4; ++k) r.rank[k] = __uint_as_float(m > at[k] ? se[lo + at[k]].y : 0xff800000u);
        v[i] = r;
        sums[i] = 0ull;
    }
}

// p of every edge in row order, each row's largest p and the degrees summed over
// it (one atomic per run of lanes in a row)
__global__ void k_fill_potentials(const int64_t* __restrict__ off, int64_t n, int64_t E,
                                  const uint32_t* __restrict__ col, const float* __restrict__ w, VertexRec* v,
                                  float* __restrict__ p, unsigned long long* __restrict__ sums) {
    const int lane = threadIdx.x & 31;
    const int64_t warp_id = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
    const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    const int64_t steps = (E + 31) >> 5;
    const int64_t s0 = steps * warp_id / nwarps, s1 = steps * (warp_id + 1) / nwarps;
    if (s0 >= s1) return;  // warp-uniform
    int64_t row = warp_row_search(off, n, s0 * 32, lane);
    for (int64_t st = s0; st < s1; ++st) {
        const int64_t i = st * 32 + lane;
        const int64_t u = warp_rows_from(off, n, row, min(i, E - 1), lane);
        row = __shfl_sync(0xffffffffu, u, 31);
        uint32_t deg = 0u, key = 0u;
        if (i < E) {
            const uint2 f = *reinterpret_cast<const uint2*>(v + col[i]);  // deg and maxw
            deg = f.x;
            const float x = deg ? __fadd_rn(w[i], __uint_as_float(f.y)) : __int_as_float(0xff800000);
            p[i] = x;
            key = f2key(x);
        }
        const unsigned peers = __match_any_sync(0xffffffffu, i < E ? static_cast<uint32_t>(u) : 0xffffffffu);
        const uint32_t km = __reduce_max_sync(peers, key);
        const unsigned long long tot = (static_cast<unsigned long long>(__reduce_add_sync(peers, deg >> 16)) << 16) +
                                       __reduce_add_sync(peers, deg & 0xffffu);
        if (i < E && lane == __ffs(peers) - 1) {
            atomicMax(&v[u].maxp_key, km);
            if (tot) atomicAdd(&sums[u], tot);
        }
    }
}

// ---------------------------------------------------------------------------
// norms behind the fp32 error bound
// ---------------------------------------------------------------------------
// The largest ||x||_1 and the largest ||x||_2^2 (or ||x||_inf) over the rows, in fp64.
// Summing every row in fp64 is bound by its pipe (1.0 ms for 1 M rows of 128 fp32
// values), so a first pass, a warp per row, sums in fp32 rounded up at every step
// and only the rows whose sum can still be the largest are summed again.  That is a
// handful of rows, or, when all rows have the same norm, every one at the old cost.
__global__ void __launch_bounds__(256) k_row_norms(const void* __restrict__ tab, int dtype, int64_t rows, int d,
                                                   float2* __restrict__ sums, unsigned* __restrict__ top,
                                                   int aux_is_inf) {
    __shared__ float s1[8], s2[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float m1 = 0.f, m2 = 0.f;
    const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    for (int64_t r = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5; r < rows; r += nwarps) {
        float l1 = 0.f, aux = 0.f;
        for (int j = lane; j < d; j += 32) {
            const float x = fabsf(emb_f32(tab, dtype, r, d, j));
            l1 = __fadd_ru(l1, x);
            aux = aux_is_inf ? fmaxf(aux, x) : __fadd_ru(aux, __fmul_ru(x, x));
        }
        for (int o = 16; o > 0; o >>= 1) {
            l1 = __fadd_ru(l1, __shfl_xor_sync(0xffffffffu, l1, o));
            const float y = __shfl_xor_sync(0xffffffffu, aux, o);
            aux = aux_is_inf ? fmaxf(aux, y) : __fadd_ru(aux, y);
        }
        if (lane == 0) sums[r] = make_float2(l1, aux);
        m1 = fmaxf(m1, l1);
        m2 = fmaxf(m2, aux);
    }
    if (lane == 0) {
        s1[wid] = m1;
        s2[wid] = m2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < static_cast<int>(blockDim.x >> 5); ++w) {
            m1 = fmaxf(m1, s1[w]);
            m2 = fmaxf(m2, s2[w]);
        }
        // non-negative floats compare like their bit patterns
        atomicMax(top + 0, __float_as_uint(m1));
        atomicMax(top + 1, __float_as_uint(m2));
    }
}

// The candidates of k_row_norms in fp64, j = 0 .. d-1, a thread per row.  A rounded-up
// sum is at most d / 32 + 6 steps of 2^-23 above the exact one, and 2^-149 more per
// element whose square underflows.
__global__ void __launch_bounds__(256) k_row_norms64(const void* __restrict__ tab, int dtype, int64_t rows, int d,
                                                     const float2* __restrict__ sums, const unsigned* __restrict__ top,
                                                     unsigned long long* __restrict__ max_l1,
                                                     unsigned long long* __restrict__ max_aux, int aux_is_inf) {
    const double keep = 1.0 - (d / 32 + 8) * 0x1p-23, tiny = d * 0x1p-149;
    const double lo1 = static_cast<double>(__uint_as_float(top[0])) * keep - tiny;
    const double lo2 = static_cast<double>(__uint_as_float(top[1])) * keep - tiny;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t r = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; r < rows; r += stride) {
        const float2 s = sums[r];
        if (!(s.x >= lo1 || s.y >= lo2)) continue;
        double l1 = 0.0, aux = 0.0;
#pragma unroll 8
        for (int j = 0; j < d; ++j) {
            const double x = fabs(static_cast<double>(emb_f32(tab, dtype, r, d, j)));
            l1 += x;
            aux = aux_is_inf ? fmax(aux, x) : aux + x * x;
        }
        // non-negative doubles compare like their bit patterns
        atomicMax(max_l1, static_cast<unsigned long long>(__double_as_longlong(l1)));
        atomicMax(max_aux, static_cast<unsigned long long>(__double_as_longlong(aux)));
    }
}

static double gam(double n, double u) { return n * u / (1.0 - n * u); }

// Bound on |S32 - S64| for one path (three edges), valid for any summation
// order of the fp32 screening arithmetic:
//   TransE: |fl32(w) - w| <= |gamma - fl32(gamma)| + g_{d+4}(2^-24) (N + |gamma| + 1)
//           with N = 2 max ||e||_1 + max ||w_r||_1 bounding sum |a|+|b|+|c|
//   DistMult: <= g_{d+3}(2^-24) M with M = max ||w_r||_inf * max ||e||_2^2
//           bounding sum |a b c| (Cauchy-Schwarz)
//   the same with 2^-53 for the fp64 value, plus the two path additions.
// Also Q of the integer route of exact weights: the sum's bound N < 2^(53 - Q), and
// at most 149: every binary32 value is a multiple of 2^-149, and a finer unit would
// shift subnormal coordinates past 32 bits.
static void compute_bounds(mhr_graph* g) {
    const double u32 = std::ldexp(1.0, -24), u64 = std::ldexp(1.0, -53);
    const int d = g->dg.d;
    const double gamma = g->dg.gamma;
    double eps32, eps64, wmax;
    if (g->fn == MHR_SCORE_TRANSE_L1) {
        const double N = 2.0 * g->max_l1 + g->max_rel_l1;
        int e = 0;
        std::frexp(N, &e);  // N < 2^e
        g->dg.qbits = std::min(149, 53 - (e + 1));
        const double gerr = std::fabs(gamma - static_cast<double>(static_cast<float>(gamma)));
        eps32 = gerr + gam(d + 4, u32) * (N + std::fabs(gamma) + 1.0);
        eps64 = gam(d + 4, u64) * (N + std::fabs(gamma) + 1.0);
        wmax = std::fabs(gamma) + N;
    } else {
        const double M = g->max_rel_inf * g->max_l2sq;
        eps32 = gam(d + 3, u32) * M;
        eps64 = gam(d + 3, u64) * M;
        wmax = M;
    }
    g->eps32_edge = eps32;
    g->eps64_edge = eps64;
    const double path = 3.0 * (eps32 + eps64) +
                        (gam(2, u32) + gam(2, u64)) * 3.0 * (wmax + eps32 + eps64);
    g->err_path = path * (1.0 + 1e-6) + 1e-300;
    // Tensor-core middle-edge screen (DistMult): p_j = fl32(e_u[j] e_v[j]) is
    // split p = p_hi + p_lo + r with bf16 parts, |r| <= 2^-16 |p|; w_r likewise;
    // the products p_hi w_hi + p_hi w_lo + p_lo w_hi are exact in fp32 and the
    // dropped p_lo w_lo is <= 2^-16 |p w|, so each term is within
    // (2^-24 + 4 * 2^-16) |e_u e_v w| of the exact one.  The tensor-core fp32
    // accumulation (3 products per term, order unspecified) is bounded with a
    // unit roundoff of 2^-22 to allow for its alignment truncation.
    if (g->fn == MHR_SCORE_DISTMULT) {
        const double M = g->max_rel_inf * g->max_l2sq;
        const double term = std::ldexp(1.0, -24) + 4.0 * std::ldexp(1.0, -16);
        const double epstc = (term + gam(3.0 * d + 3, std::ldexp(1.0, -22)) * (1.0 + term)) * M;
        g->epstc_edge = epstc;
        const double ptc = 2.0 * eps32 + epstc + 3.0 * eps64 +
                           (gam(2, u32) + gam(2, u64)) * 3.0 * (wmax + epstc + eps32 + eps64);
        g->err_path_tc = ptc * (1.0 + 1e-6) + 1e-300;
    }
}

// bf16 hi / lo split of the relation table (tensor-core middle-edge screen)
__global__ void k_split_rel(const void* __restrict__ remb, int dtype, int64_t count, uint16_t* __restrict__ hi,
                            uint16_t* __restrict__ lo) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < count; i += stride) {
        const float w = dtype == MHR_F32 ? static_cast<const float*>(remb)[i]
                                         : bf16_to_f32(static_cast<const uint16_t*>(remb)[i]);
        const __nv_bfloat16 h = __float2bfloat16_rn(w);
        hi[i] = __bfloat16_as_ushort(h);
        lo[i] = __bfloat16_as_ushort(__float2bfloat16_rn(w - __bfloat162float(h)));
    }
}

// ---------------------------------------------------------------------------
// edge scores
// ---------------------------------------------------------------------------
// fp32 weights of m edges: the given triples, or (src == NULL) consecutive
// CSR edges.  Each warp owns a contiguous range of the edges and walks it 32 at a
// time, so one row search at the range's start replaces a search per edge: the
// rows of the next 32 edges are found among the row starts that follow the last
// one (warp_rows_from).  Scoring 20 M edges of 512-byte rows (d = 128 fp32)
// takes 1.75 ms, 5.9 TB/s of gathered tail rows through L2, which bounds it; a
// 20-step search and a generic scorer in every lane (536 instructions per edge)
// took 18.7 ms.  G = 0: rows that warp_score_v does not take.  Every weight is summed
// in the order of edge_w32_group with the width score_group_width gives.
// FEW: a warp takes `per` < 32 edges at a time, when 32 would leave warps idle.
// With kout / kin the edges' order keys are also reduced to per-vertex maxima
// (one atomic per run of lanes with the same source) and, with kout_r / kin_r,
// to per (vertex, relation) maxima.
// Resident blocks per SM: three with four rounds of rows in flight, eight for the one
// row in flight of G = 0 (400,000 edges of 513 fp32 values: 0.69 ms at three, 0.44).
constexpr int edge_blocks(int G) { return G ? 3 : 8; }
template <int G, bool FEW>
__global__ void __launch_bounds__(256, edge_blocks(G))
    k_edge_w32(DevGraph g, const uint32_t* __restrict__ src, const uint16_t* __restrict__ rel,
               const uint32_t* __restrict__ dst, int64_t m, int per, int width, float* __restrict__ out,
               uint32_t* __restrict__ kout, uint32_t* __restrict__ kin, uint32_t* __restrict__ kout_r,
               uint32_t* __restrict__ kin_r) {
    if (!FEW) per = 32;
    const int lane = threadIdx.x & 31;
    const int64_t warp_id = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
    const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    const int64_t steps = (m + per - 1) / per;
    const int64_t s0 = steps * warp_id / nwarps, s1 = steps * (warp_id + 1) / nwarps;
    if (s0 >= s1) return;  // warp-uniform
    int64_t row = src ? 0 : warp_row_search(g.off, g.n, s0 * per, lane);
    for (int64_t st = s0; st < s1; ++st) {
        const int64_t i = st * per + lane;
        const bool live = (!FEW || lane < per) && i < m;
        uint32_t u = 0, r = 0, v = 0;  // dead lanes score vertex 0's rows
        if (src) {
            if (live) {
                u = src[i];
                r = rel[i];
                v = dst[i];
            }
        } else {
            const int64_t mine = warp_rows_from(g.off, g.n, row, min(i, m - 1), lane);
            row = __shfl_sync(0xffffffffu, mine, per - 1);
            if (live) {
                u = static_cast<uint32_t>(mine);
                r = g.rel[i];
                v = g.col[i];
            }
        }
        float w;
        if constexpr (G > 0) w = warp_score_v<G, G < 32, FEW>(g, u, v, (r << 1) | 1u, lane, per);
        else w = warp_score_any(g, u, r, v, width, lane);
        if (live && out) out[i] = w;
        if (kout) {
            const uint32_t k = f2key(w);
            const unsigned peers = __match_any_sync(0xffffffffu, live ? u : 0xffffffffu);
            const uint32_t km = __reduce_max_sync(peers, k);
            if (live) {
                if (lane == __ffs(peers) - 1) atomicMax(&kout[u], km);
                atomicMax(&kin[v], k);
                if (kout_r) {
                    atomicMax(&kout_r[static_cast<int64_t>(u) * g.R + r], k);
                    atomicMax(&kin_r[static_cast<int64_t>(v) * g.R + r], k);
                }
            }
        }
    }
}

// Triples whose rows warp_score_v does not take: a group of `width` lanes per triple,
// all resident warps at once.  A warp of the kernel above goes through 32 of them in
// turn: 512,000 triples of 513 fp32 values 0.56 ms, here 0.28; 100 of them 122 us, 30.
__global__ void __launch_bounds__(256) k_triple_w32(DevGraph g, const uint32_t* __restrict__ src,
                                                    const uint16_t* __restrict__ rel, const uint32_t* __restrict__ dst,
                                                    int64_t m, int width, float* __restrict__ out) {
    const int sub = threadIdx.x & (width - 1), per = blockDim.x / width;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * per;
    const int64_t ends = (m + per - 1) / per * per;  // every lane of a warp takes the same steps
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * per + threadIdx.x / width; i < ends; i += stride) {
        const int64_t e = min(i, m - 1);
        const float w = edge_w32_group(g, src[e], rel[e], dst[e], sub, width);
        if (sub == 0 && i < m) out[i] = w;
    }
}

// launch of k_edge_w32 with the graph's scorer
using EdgeKernel = void (*)(DevGraph, const uint32_t*, const uint16_t*, const uint32_t*, int64_t, int, int, float*,
                            uint32_t*, uint32_t*, uint32_t*, uint32_t*);
template <bool FEW>
static EdgeKernel edge_kernel(int G) {
    switch (G) {
        case 1: return k_edge_w32<1, FEW>;
        case 2: return k_edge_w32<2, FEW>;
        case 4: return k_edge_w32<4, FEW>;
        case 8: return k_edge_w32<8, FEW>;
        case 16: return k_edge_w32<16, FEW>;
        default: return k_edge_w32<32, FEW>;
    }
}

static cudaError_t launch_edge_w32(const DevGraph& g, const uint32_t* src, const uint16_t* rel, const uint32_t* dst,
                                   int64_t m, float* out, uint32_t* kout, uint32_t* kin, uint32_t* kout_r,
                                   uint32_t* kin_r, int sms, cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    const int G = hit_group_width(g.d, g.dtype, 2), width = score_group_width(g.d, g.dtype);
    const bool vec = score_vec2(g, G);
    if (!vec && src && !kout) {
        const int64_t blocks = std::min<int64_t>(static_cast<int64_t>(sms) * 8, (m * width + 255) / 256);
        k_triple_w32<<<static_cast<unsigned>(blocks), 256, 0, st>>>(g, src, rel, dst, m, width, out);
        return cudaGetLastError();
    }
    // one resident wave, and steps of as many edges as still give every warp one
    const int64_t wave = static_cast<int64_t>(sms) * edge_blocks(vec ? G : 0);
    const int least = vec ? 32 / G * std::min(G, kScoreRounds) : 32;  // edges a warp scores together
    int per = 32;
    while (per > least && (m + per - 1) / per < wave * 8) per >>= 1;
    const EdgeKernel fn = !vec ? k_edge_w32<0, false> : (per < 32 ? edge_kernel<true>(G) : edge_kernel<false>(G));
    const int64_t blocks = std::min<int64_t>(wave, ((m + per - 1) / per + 7) / 8);
    fn<<<static_cast<unsigned>(blocks), 256, 0, st>>>(g, src, rel, dst, m, per, width, out, kout, kin, kout_r, kin_r);
    return cudaGetLastError();
}

// fp64 weights, one thread per edge
__global__ void k_edge_scores64(DevGraph g, const uint32_t* __restrict__ src,
                                const uint16_t* __restrict__ rel, const uint32_t* __restrict__ dst,
                                int64_t m, double* __restrict__ out) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < m; i += stride) {
        uint32_t u, r, v;
        if (src) {
            u = src[i];
            r = rel[i];
            v = dst[i];
        } else {
            u = static_cast<uint32_t>(row_of_edge(g.off, g.n, i));
            r = g.rel[i];
            v = g.col[i];
        }
        out[i] = edge_w64(g, u, r, v);
    }
}

// fp64 weights, a warp per 32 consecutive edges: TransE in integers, eight lanes per
// edge, the few edges that leaves and DistMult in fp64 sums of terms staged through
// shared memory (mhr_exact.cuh).  What bounds it: TransE the integer issue, DistMult
// the fp64 pipe (one addition per coordinate).  A thread per edge fetches 16 bytes of
// 96 rows per step and runs three fp64 operations and three conversions per
// coordinate: for 2M edges of 128 fp32 values 2.82 ms, now 0.82 ms (TransE) and 1.16
// ms (DistMult); of 16 values 0.36 ms against 0.23 and 0.26; of 8 values 0.19 ms both.
// Shorter rows than kEdge64Warp keep it: a step covers 32 coordinates, filled or not.
// As above, `per` is less than 32 (a multiple of four) for few edges.
constexpr int kEdge64Warps = 4;
constexpr int kEdge64Warp = 16;
__global__ void __launch_bounds__(kEdge64Warps * 32) k_edge_scores64_warp(DevGraph g, const uint32_t* __restrict__ src,
                                                                         const uint16_t* __restrict__ rel,
                                                                         const uint32_t* __restrict__ dst, int64_t m,
                                                                         int per, double* __restrict__ out) {
    __shared__ double stage[kEdge64Warps][32 * 33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t warp_id = blockIdx.x * static_cast<int64_t>(kEdge64Warps) + w;
    const int64_t nwarps = static_cast<int64_t>(gridDim.x) * kEdge64Warps;
    const int64_t steps = (m + per - 1) / per;
    const int64_t s0 = steps * warp_id / nwarps, s1 = steps * (warp_id + 1) / nwarps;
    if (s0 >= s1) return;  // warp-uniform; no block-wide step below
    int64_t row = src ? 0 : warp_row_search(g.off, g.n, s0 * per, lane);
    for (int64_t st = s0; st < s1; ++st) {
        const int64_t i = st * per + lane;
        const bool live = lane < per && i < m;
        uint32_t u = 0, r = 0, v = 0;
        if (src) {
            if (live) {
                u = src[i];
                r = rel[i];
                v = dst[i];
            }
        } else {
            const int64_t mine = warp_rows_from(g.off, g.n, row, min(i, m - 1), lane);
            row = __shfl_sync(0xffffffffu, mine, per - 1);
            if (live) {
                u = static_cast<uint32_t>(mine);
                r = g.rel[i];
                v = g.col[i];
            }
        }
        double mine = 0.0;
        bool left = live;
        if (g.fn == MHR_SCORE_TRANSE_L1) {
            const int n = static_cast<int>(min(static_cast<int64_t>(per), m - st * per));
            mine = warp_w64_fixed_each(g, u, r, v, n, lane, left);
        }
        if (__any_sync(0xffffffffu, left)) {
            const double x = warp_w64_staged(g, u, r, v, left, stage[w], lane);
            if (left) mine = x;
        }
        if (live) out[i] = mine;
    }
}

// keys -> fp32 upper bounds: + slack (two fp32 evaluations of one edge in
// different summation orders differ by at most 2 * eps32), rounded up
__global__ void k_maxw_finish(uint32_t* __restrict__ a, int64_t n, double slack) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride) {
        const uint32_t k = a[i];
        float f;
        if (k == 0u) f = __int_as_float(0xff800000);
        else f = __double2float_ru(__dadd_ru(static_cast<double>(key2f(k)), slack));
        a[i] = __float_as_uint(f);
    }
}

}  // namespace mhr

using namespace mhr;

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
namespace {

struct Scoped {
    std::vector<void*> ptrs;
    ~Scoped() {
        for (void* p : ptrs) cudaFree(p);
    }
    template <typename T>
    cudaError_t alloc(T** p, size_t bytes) {
        cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), bytes ? bytes : 1);
        if (e == cudaSuccess) ptrs.push_back(*p);
        return e;
    }
};

void free_graph(mhr_graph* g);

// Device-memory cap of a resident graph (bytes), from MHR_GRAPH_MEMORY_CAP_BYTES;
// 0 = none.  Read at every load.
size_t graph_memory_cap() {
    const char* v = std::getenv("MHR_GRAPH_MEMORY_CAP_BYTES");
    if (!v || !*v) return 0;
    char* end = nullptr;
    const unsigned long long c = std::strtoull(v, &end, 10);
    return (end && *end == '\0') ? static_cast<size_t>(c) : 0;
}

mhr_status graph_alloc(mhr_graph* g, void** p, size_t bytes) {
    const size_t want = bytes ? bytes : 16;
    if (g->memory_cap && g->alloc_bytes + want > g->memory_cap) {
        *p = nullptr;
        return fail(MHR_ENOMEM, "graph device memory would exceed MHR_GRAPH_MEMORY_CAP_BYTES (" +
                                    std::to_string(g->memory_cap) + " bytes)");
    }
    cudaError_t e = cudaMalloc(p, want);
    if (e != cudaSuccess) {
        *p = nullptr;
        return cuda_fail(e, "cudaMalloc (graph)");
    }
    g->allocations.push_back(*p);
    g->alloc_bytes += want;
    return MHR_OK;
}

// Device arrays of the weight index (36 bytes per edge and 80 per vertex)
struct IndexArrays {
    float *w, *rw, *p, *rp;
    uint2 *se, *rse;
    uint16_t *sr, *rsr;
    VertexRec *vout, *vin;
    unsigned long long *sout, *sin;
};

// bytes of the split relation table
size_t split_bytes(const mhr_graph* g) {
    return g->fn == MHR_SCORE_DISTMULT ? sizeof(uint16_t) * 2 * static_cast<size_t>(g->dg.R) * g->dg.d : 0;
}

// The index is kept when it fits: within the graph's memory cap, and within
// half of the device memory that is free once the graph itself is resident (the
// rest stays for query plans).  A graph without one runs the joins that weigh
// every hit.
void alloc_index(mhr_graph* g, int64_t n, int64_t E, IndexArrays* ix) {
    if (!E) return;
    auto round = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t e2 = round(sizeof(uint16_t) * E), e4 = round(sizeof(uint32_t) * E), e8 = round(sizeof(uint2) * E),
                 n8 = round(sizeof(unsigned long long) * n), nr = round(sizeof(VertexRec) * n);
    const size_t total = 2 * (e2 + 2 * e4 + e8 + n8 + nr);
    // still to come: the reverse adjacency and DistMult's split relation table, and
    // (released later) a list of the sort
    const size_t later = static_cast<size_t>(E) * 6 + sizeof(int64_t) * (n + 1) + split_bytes(g);
    if (g->memory_cap && g->alloc_bytes + total + later > g->memory_cap) return;
    size_t avail = 0, all = 0;
    if (cudaMemGetInfo(&avail, &all) != cudaSuccess || avail < later + static_cast<size_t>(E) * 4 ||
        total > (avail - later - static_cast<size_t>(E) * 4) / 2) {
        cudaGetLastError();
        return;
    }
    char* p = nullptr;
    if (cudaMalloc(reinterpret_cast<void**>(&p), total) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    g->allocations.push_back(p);
    g->alloc_bytes += total;
    auto take = [&](size_t bytes) {
        char* q = p;
        p += bytes;
        return static_cast<void*>(q);
    };
    ix->w = static_cast<float*>(take(e4));
    ix->rw = static_cast<float*>(take(e4));
    ix->p = static_cast<float*>(take(e4));
    ix->rp = static_cast<float*>(take(e4));
    ix->se = static_cast<uint2*>(take(e8));
    ix->rse = static_cast<uint2*>(take(e8));
    ix->sr = static_cast<uint16_t*>(take(e2));
    ix->rsr = static_cast<uint16_t*>(take(e2));
    ix->vout = static_cast<VertexRec*>(take(nr));
    ix->vin = static_cast<VertexRec*>(take(nr));
    ix->sout = static_cast<unsigned long long*>(take(n8));
    ix->sin = static_cast<unsigned long long*>(take(n8));
}

mhr_status load_impl(const mhr_graph_desc* desc, mhr_graph* g, cudaStream_t st) {
    const int64_t n = desc->n_vertices, E = desc->n_edges;
    const int R = desc->n_relations, d = desc->dim;
    const bool host = desc->mem == MHR_MEM_HOST;
    const cudaMemcpyKind kind = host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
    const size_t esz = desc->emb_dtype == MHR_F32 ? 4 : 2;
    g->num_sms = device_sm_count();
    const int grid = std::max(1, g->num_sms) * 8;

    int64_t* off;
    uint32_t* col;
    uint16_t* rel;
    uint8_t* vt;
    void *vemb, *remb;
    MHR_TRY(graph_alloc(g, reinterpret_cast<void**>(&off), sizeof(int64_t) * (n + 1)));
    MHR_TRY(graph_alloc(g, reinterpret_cast<void**>(&col), sizeof(uint32_t) * E));
    MHR_TRY(graph_alloc(g, reinterpret_cast<void**>(&rel), sizeof(uint16_t) * E));
    MHR_TRY(graph_alloc(g, reinterpret_cast<void**>(&vt), n));
    MHR_TRY(graph_alloc(g, &vemb, esz * n * d));
    MHR_TRY(graph_alloc(g, &remb, esz * R * d));
    MHR_CUDA_TRY(cudaMemcpyAsync(off, desc->offsets, sizeof(int64_t) * (n + 1), kind, st));
    if (E) {
        MHR_CUDA_TRY(cudaMemcpyAsync(col, desc->cols, sizeof(uint32_t) * E, kind, st));
        MHR_CUDA_TRY(cudaMemcpyAsync(rel, desc->rels, sizeof(uint16_t) * E, kind, st));
    }
    if (desc->vtypes) MHR_CUDA_TRY(cudaMemcpyAsync(vt, desc->vtypes, n, kind, st));
    else MHR_CUDA_TRY(cudaMemsetAsync(vt, 0, n, st));
    MHR_CUDA_TRY(cudaMemcpyAsync(vemb, desc->vertex_emb, esz * n * d, kind, st));
    MHR_CUDA_TRY(cudaMemcpyAsync(remb, desc->rel_emb, esz * R * d, kind, st));

    // --- validation
    Scoped tmp;
    int* err;
    MHR_CUDA_TRY(tmp.alloc(&err, sizeof(int) * kErrCount));
    MHR_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int) * kErrCount, st));
    k_validate_offsets<<<grid, 256, 0, st>>>(off, n, E, err);
    int herr[kErrCount];
    MHR_CUDA_TRY(cudaMemcpyAsync(herr, err, sizeof herr, cudaMemcpyDeviceToHost, st));
    MHR_CUDA_TRY(cudaStreamSynchronize(st));
    if (herr[kErrOffsets])
        return fail(MHR_EINVAL, "offsets must start at 0, be non-decreasing and end at n_edges");
    // scratch, one allocation (for a small graph they are a good part of the load): the
    // norms' maxima, scan lengths and sums, in-degrees; the reverse sort, and the source
    // of every edge
    uint32_t *src = nullptr, *indeg;
    unsigned long long* mx;  // four maxima in fp64, then the four of the first pass in fp32
    int64_t *n_dev, *partials;
    SortScratch ss{};
    const size_t tiles = sort_tiles(static_cast<uint64_t>(E)), nc = 256 * tiles;
    const size_t eb = (sizeof(uint32_t) * E + 255) / 256 * 256, cb = (sizeof(int64_t) * (nc + 1) + 255) / 256 * 256;
    const size_t pb = (sizeof(int64_t) * kScanPartials + 255) / 256 * 256, nb = (sizeof(uint32_t) * n + 255) / 256 * 256;
    char* mem;
    MHR_CUDA_TRY(tmp.alloc(&mem, 3 * 256 + pb + nb + (E ? 5 * eb + 2 * cb : 0)));
    mx = reinterpret_cast<unsigned long long*>(mem);
    n_dev = reinterpret_cast<int64_t*>(mem + 256);
    ss.n_counts = reinterpret_cast<int64_t*>(mem + 512);
    ss.partials = partials = reinterpret_cast<int64_t*>(mem + 768);  // left zero by every scan
    indeg = reinterpret_cast<uint32_t*>(mem + 768 + pb);
    mem += 768 + pb + nb;
    MHR_CUDA_TRY(cudaMemsetAsync(mx, 0, sizeof(unsigned long long) * 6, st));
    MHR_CUDA_TRY(cudaMemsetAsync(partials, 0, pb + nb, st));  // and the in-degrees
    if (E) {
        src = reinterpret_cast<uint32_t*>(mem);
        for (int i = 0; i < 2; ++i) {
            ss.key[i] = reinterpret_cast<uint32_t*>(mem + (1 + i) * eb);
            ss.val[i] = reinterpret_cast<uint32_t*>(mem + (3 + i) * eb);
        }
        mem += 5 * eb;
        ss.counts = reinterpret_cast<uint32_t*>(mem);
        ss.offsets = reinterpret_cast<int64_t*>(mem + cb);
        const int64_t nch = static_cast<int64_t>(nc);
        MHR_CUDA_TRY(cudaMemcpyAsync(ss.n_counts, &nch, sizeof nch, cudaMemcpyHostToDevice, st));
        k_validate_edges<<<grid, 256, 0, st>>>(off, col, rel, n, E, R, src, err);
    }
    k_validate_finite<<<grid, 256, 0, st>>>(vemb, desc->emb_dtype, n * d, err);
    k_validate_finite<<<grid, 256, 0, st>>>(remb, desc->emb_dtype, static_cast<int64_t>(R) * d, err);
    MHR_CUDA_TRY(cudaGetLastError());
    MHR_CUDA_TRY(cudaMemcpyAsync(herr, err, sizeof herr, cudaMemcpyDeviceToHost, st));
    MHR_CUDA_TRY(cudaStreamSynchronize(st));
    if (herr[kErrColRange]) return fail(MHR_EINVAL, "a destination id is >= n_vertices");
    if (herr[kErrRelRange]) return fail(MHR_EINVAL, "a relation id is >= n_relations");
    if (herr[kErrSelfLoop]) return fail(MHR_EINVAL, "self loops are not allowed");
    if (herr[kErrRowOrder])
        return fail(MHR_EINVAL, "each row must be sorted by (col, rel) without repeated (col, rel)");
    if (herr[kErrNonFinite]) return fail(MHR_EINVAL, "an embedding value is NaN or infinite");

    DevGraph& dg = g->dg;
    dg.n = n;
    dg.E = E;
    dg.R = R;
    dg.d = d;
    dg.dtype = desc->emb_dtype;
    dg.fn = desc->score_fn;
    dg.gamma = desc->gamma;
    dg.gamma32 = static_cast<float>(desc->gamma);
    dg.off = off;
    dg.col = col;
    dg.rel = rel;
    dg.vtypes = vt;
    dg.vemb = vemb;
    dg.remb = remb;
    g->fn = desc->score_fn;

    // --- fp32 edge weights: per-vertex maxima (pruning bounds), and the weights
    // themselves when the index is kept
    uint32_t *kout, *kin, *kout_r = nullptr, *kin_r = nullptr;
    MHR_TRY(graph_alloc(g, reinterpret_cast<void**>(&kout), sizeof(uint32_t) * n));
    MHR_TRY(graph_alloc(g, reinterpret_cast<void**>(&kin), sizeof(uint32_t) * n));
    MHR_CUDA_TRY(cudaMemsetAsync(kout, 0, sizeof(uint32_t) * n, st));
    MHR_CUDA_TRY(cudaMemsetAsync(kin, 0, sizeof(uint32_t) * n, st));
    IndexArrays ix{};
    alloc_index(g, n, E, &ix);
    const int64_t nr = n * static_cast<int64_t>(R);
    if (!ix.w && nr <= kMaxRelBoundEntries) {
        // per (vertex, relation) bounds: the joins without an index weigh every hit
        MHR_TRY(graph_alloc(g, reinterpret_cast<void**>(&kout_r), sizeof(uint32_t) * nr));
        MHR_TRY(graph_alloc(g, reinterpret_cast<void**>(&kin_r), sizeof(uint32_t) * nr));
        MHR_CUDA_TRY(cudaMemsetAsync(kout_r, 0, sizeof(uint32_t) * nr, st));
        MHR_CUDA_TRY(cudaMemsetAsync(kin_r, 0, sizeof(uint32_t) * nr, st));
    }
    MHR_CUDA_TRY(launch_edge_w32(dg, nullptr, nullptr, nullptr, E, ix.w, kout, kin, kout_r, kin_r,
                                 std::max(1, g->num_sms), st));

    // --- reverse CSR (in-edges of each vertex, rows sorted by (source, relation))
    int64_t* roff;
    uint32_t* rcol;
    uint16_t* rrel;
    MHR_TRY(graph_alloc(g, reinterpret_cast<void**>(&roff), sizeof(int64_t) * (n + 1)));
    MHR_TRY(graph_alloc(g, reinterpret_cast<void**>(&rcol), sizeof(uint32_t) * E));
    MHR_TRY(graph_alloc(g, reinterpret_cast<void**>(&rrel), sizeof(uint16_t) * E));
    {
        MHR_CUDA_TRY(cudaMemcpyAsync(n_dev, &n, sizeof(int64_t), cudaMemcpyHostToDevice, st));
        if (E) k_count_in<<<grid, 256, 0, st>>>(col, E, indeg);
        MHR_CUDA_TRY(device_excl_scan<uint32_t>(indeg, n_dev, partials, roff, st));
        if (E) {
            int bits = 1;
            while (((n - 1) >> bits) != 0) ++bits;
            uint32_t* edge;
            MHR_CUDA_TRY(radix_sort_pairs(col, nullptr, static_cast<uint32_t>(E), bits, ss, &edge, st));
            k_fill_reverse<<<grid, 256, 0, st>>>(edge, E, src, rel, ix.w, rcol, rrel, ix.rw);
            MHR_CUDA_TRY(cudaGetLastError());
            if (ix.w) {
                // All edges by weight, then (stable) by row: every row ends up in
                // weight order, in both directions.
                uint32_t* copy;
                MHR_CUDA_TRY(tmp.alloc(&copy, sizeof(uint32_t) * E));
                const uint32_t m = static_cast<uint32_t>(E);
                k_weight_keys<<<grid, 256, 0, st>>>(ix.w, E, ss.key[0]);
                MHR_CUDA_TRY(radix_sort_pairs(ss.key[0], nullptr, m, 32, ss, &edge, st));
                uint32_t* key = edge == ss.val[0] ? ss.key[0] : ss.key[1];
                k_row_keys<<<grid, 256, 0, st>>>(edge, E, src, key, copy);
                MHR_CUDA_TRY(radix_sort_pairs(key, edge, m, bits, ss, &edge, st));
                k_fill_sorted<<<grid, 256, 0, st>>>(edge, E, col, rel, ix.w, ix.se, ix.sr);
                k_row_keys<<<grid, 256, 0, st>>>(copy, E, col, ss.key[0], ss.val[0]);
                MHR_CUDA_TRY(radix_sort_pairs(ss.key[0], ss.val[0], m, bits, ss, &edge, st));
                k_fill_sorted<<<grid, 256, 0, st>>>(edge, E, src, rel, ix.w, ix.rse, ix.rsr);
                k_fill_records<<<grid, 256, 0, st>>>(off, n, ix.se, ix.vout, ix.sout);
                k_fill_records<<<grid, 256, 0, st>>>(roff, n, ix.rse, ix.vin, ix.sin);
                k_fill_potentials<<<grid, 256, 0, st>>>(off, n, E, col, ix.w, ix.vout, ix.p, ix.sout);
                k_fill_potentials<<<grid, 256, 0, st>>>(roff, n, E, rcol, ix.rw, ix.vin, ix.rp, ix.sin);
                MHR_CUDA_TRY(cudaGetLastError());
            }
        }
        // the scan wrote n_dev-long output plus the total at roff[n]
        MHR_CUDA_TRY(cudaStreamSynchronize(st));
    }

    // --- host copies of row starts (query sizing)
    g->h_off.resize(n + 1);
    g->h_roff.resize(n + 1);
    MHR_CUDA_TRY(cudaMemcpyAsync(g->h_off.data(), off, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToHost, st));
    MHR_CUDA_TRY(cudaMemcpyAsync(g->h_roff.data(), roff, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToHost, st));

    // --- norms
    unsigned* top = reinterpret_cast<unsigned*>(mx + 4);
    float2* sums = reinterpret_cast<float2*>(src);  // the sort is done with its scratch
    const int64_t most = std::max<int64_t>(n, R);
    if (!src || 5 * E < 2 * most) MHR_CUDA_TRY(tmp.alloc(&sums, sizeof(float2) * most));
    const int rgrid = std::max(1, std::min(grid, (R + 7) / 8));
    k_row_norms<<<grid, 256, 0, st>>>(vemb, desc->emb_dtype, n, d, sums, top, 0);
    k_row_norms64<<<grid, 256, 0, st>>>(vemb, desc->emb_dtype, n, d, sums, top, mx + 0, mx + 1, 0);
    k_row_norms<<<rgrid, 256, 0, st>>>(remb, desc->emb_dtype, R, d, sums, top + 2, 1);
    k_row_norms64<<<rgrid, 256, 0, st>>>(remb, desc->emb_dtype, R, d, sums, top + 2, mx + 2, mx + 3, 1);
    MHR_CUDA_TRY(cudaGetLastError());
    unsigned long long hm[4];
    MHR_CUDA_TRY(cudaMemcpyAsync(hm, mx, sizeof hm, cudaMemcpyDeviceToHost, st));
    MHR_CUDA_TRY(cudaStreamSynchronize(st));
    double dm[4];
    std::memcpy(dm, hm, sizeof dm);
    g->max_l1 = dm[0];
    g->max_l2sq = dm[1];
    g->max_rel_l1 = dm[2];
    g->max_rel_inf = dm[3];
    if (g->h_roff[n] != E) return fail(MHR_ECUDA, "reverse CSR construction is inconsistent");
    for (int64_t u = 0; u < n; ++u) {
        g->max_out_deg = std::max(g->max_out_deg, g->h_off[u + 1] - g->h_off[u]);
        g->max_in_deg = std::max(g->max_in_deg, g->h_roff[u + 1] - g->h_roff[u]);
    }

    dg.roff = roff;
    dg.rcol = rcol;
    dg.rrel = rrel;
    dg.w = ix.w;
    dg.rw = ix.rw;
    dg.se = ix.se;
    dg.sr = ix.sr;
    dg.rse = ix.rse;
    dg.rsr = ix.rsr;
    dg.p = ix.p;
    dg.rp = ix.rp;
    dg.vout = ix.vout;
    dg.vin = ix.vin;
    dg.sout = ix.sout;
    dg.sin = ix.sin;
    compute_bounds(g);
    if (g->fn == MHR_SCORE_DISTMULT) {
        const int64_t cnt = static_cast<int64_t>(R) * d;
        MHR_TRY(graph_alloc(g, reinterpret_cast<void**>(&g->wsplit), split_bytes(g)));
        k_split_rel<<<std::max(1, std::min(grid, static_cast<int>((cnt + 255) / 256))), 256, 0, st>>>(
            remb, desc->emb_dtype, cnt, g->wsplit, g->wsplit + cnt);
        MHR_CUDA_TRY(cudaGetLastError());
    }
    // per-vertex (and, without the index, per (vertex, relation)) bounds on the
    // fp32 weight of adjacent edges, for bound pruning
    {
        k_maxw_finish<<<grid, 256, 0, st>>>(kout, n, 2.0 * g->eps32_edge);
        k_maxw_finish<<<grid, 256, 0, st>>>(kin, n, 2.0 * g->eps32_edge);
        if (kout_r) {
            k_maxw_finish<<<grid, 256, 0, st>>>(kout_r, nr, 2.0 * g->eps32_edge);
            k_maxw_finish<<<grid, 256, 0, st>>>(kin_r, nr, 2.0 * g->eps32_edge);
        }
        MHR_CUDA_TRY(cudaGetLastError());
        MHR_CUDA_TRY(cudaStreamSynchronize(st));
        dg.maxw_out = reinterpret_cast<const float*>(kout);
        dg.maxw_in = reinterpret_cast<const float*>(kin);
        dg.maxw_out_r = reinterpret_cast<const float*>(kout_r);
        dg.maxw_in_r = reinterpret_cast<const float*>(kin_r);
    }
    const double big = 1e30;
    if (!(g->max_l1 < big && g->max_rel_l1 < big && g->max_l2sq < big && g->max_rel_inf < big &&
          g->err_path < 1e20))
        return fail(MHR_EINVAL, "embedding magnitudes are too large for fp32 screening");
    return MHR_OK;
}

void free_graph(mhr_graph* g);

}  // namespace

namespace mhr {

// A load that keeps the index leaves these out (8 bytes per vertex and relation and 0.3
// ms of its time at 1 M vertices and 16 relations) since only the pruned join reads
// them: 256 queries of 256 fp32 values, its counters, 4.1 ms without and 3.5 with.
void build_rel_bounds(mhr_graph* g, cudaStream_t st) {
    const int64_t n = g->dg.n, nr = n * static_cast<int64_t>(g->dg.R);
    const size_t bytes = sizeof(uint32_t) * static_cast<size_t>(nr);
    if (g->rel_bounds_tried) return;
    g->rel_bounds_tried = true;
    if (g->dg.maxw_out_r || nr > kMaxRelBoundEntries) return;
    if (g->memory_cap && g->alloc_bytes + 2 * bytes > g->memory_cap) return;
    Scoped tmp;
    uint32_t *k = nullptr, *ko = nullptr;  // per-vertex maxima, not kept; both tables
    cudaError_t e = tmp.alloc(&k, sizeof(uint32_t) * 2 * n);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&ko), 2 * bytes);
    if (e == cudaSuccess) e = cudaMemsetAsync(k, 0, sizeof(uint32_t) * 2 * n, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(ko, 0, 2 * bytes, st);
    if (e == cudaSuccess)
        e = launch_edge_w32(g->dg, nullptr, nullptr, nullptr, g->dg.E, nullptr, k, k + n, ko, ko + nr,
                            std::max(1, g->num_sms), st);
    if (e == cudaSuccess) {
        k_maxw_finish<<<std::max(1, g->num_sms) * 8, 256, 0, st>>>(ko, 2 * nr, 2.0 * g->eps32_edge);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        if (ko) cudaFree(ko);
        return;
    }
    g->allocations.push_back(ko);
    g->alloc_bytes += 2 * bytes;
    g->dg.maxw_out_r = reinterpret_cast<const float*>(ko);
    g->dg.maxw_in_r = reinterpret_cast<const float*>(ko + nr);
}

void destroy_plans(mhr_graph* g);  // mhr_query.cu
void destroy_tail(mhr_graph* g);   // mhr_tail.cu
void destroy_beam(mhr_graph* g);   // mhr_beam.cu
}

namespace {
void free_graph(mhr_graph* g) {
    if (!g) return;
    mhr::destroy_plans(g);
    mhr::destroy_tail(g);
    mhr::destroy_beam(g);
    for (void* p : g->allocations) cudaFree(p);
    delete g;
}
}  // namespace

extern "C" mhr_status mhr_graph_load(const mhr_graph_desc* desc, mhr_graph** out, void* cuda_stream) {
    if (!out) return fail(MHR_EINVAL, "out is NULL");
    *out = nullptr;
    if (!desc) return fail(MHR_EINVAL, "desc is NULL");
    if (desc->n_vertices < 1 || desc->n_vertices >= (1ll << 32))
        return fail(MHR_EINVAL, "n_vertices must be in [1, 2^32)");
    if (desc->n_edges < 0 || desc->n_edges >= (1ll << 32)) return fail(MHR_EINVAL, "n_edges must be in [0, 2^32)");
    if (desc->n_relations < 1 || desc->n_relations > 65536) return fail(MHR_EINVAL, "n_relations must be in [1, 65536]");
    if (desc->dim < 1 || desc->dim > 65536) return fail(MHR_EINVAL, "dim must be in [1, 65536]");
    if (desc->emb_dtype != MHR_F32 && desc->emb_dtype != MHR_BF16) return fail(MHR_EINVAL, "unknown emb_dtype");
    if (desc->mem != MHR_MEM_HOST && desc->mem != MHR_MEM_DEVICE) return fail(MHR_EINVAL, "unknown mem kind");
    if (desc->score_fn != MHR_SCORE_TRANSE_L1 && desc->score_fn != MHR_SCORE_DISTMULT)
        return fail(MHR_EINVAL, "unknown score_fn");
    if (!std::isfinite(desc->gamma)) return fail(MHR_EINVAL, "gamma must be finite");
    if (!desc->offsets || (desc->n_edges && (!desc->cols || !desc->rels)) || !desc->vertex_emb || !desc->rel_emb)
        return fail(MHR_EINVAL, "a required array pointer is NULL");
    if (desc->mem == MHR_MEM_HOST) {
        const int64_t* o = desc->offsets;
        if (o[0] != 0 || o[desc->n_vertices] != desc->n_edges)
            return fail(MHR_EINVAL, "offsets must start at 0 and end at n_edges");
    }
    mhr_graph* g = new (std::nothrow) mhr_graph();
    if (!g) return fail(MHR_ENOMEM, "host allocation failed");
    if (cudaGetDevice(&g->device) != cudaSuccess) {
        delete g;
        return fail(MHR_ECUDA, "no CUDA device");
    }
    g->memory_cap = graph_memory_cap();
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    mhr_status rc = load_impl(desc, g, st);
    if (rc != MHR_OK) {
        cudaStreamSynchronize(st);
        std::string keep = mhr_last_error();
        free_graph(g);
        set_error(keep);
        return rc;
    }
    *out = g;
    return MHR_OK;
}

extern "C" mhr_status mhr_graph_free(mhr_graph* g) {
    if (!g) return MHR_OK;
    cudaDeviceSynchronize();
    free_graph(g);
    return MHR_OK;
}

extern "C" mhr_status mhr_edge_scores(const mhr_graph* g, const uint32_t* src, const uint16_t* rel,
                                      const uint32_t* dst, int64_t n, int32_t precision, void* out,
                                      mhr_mem mem, void* cuda_stream) {
    MHR_TRY(check_graph(g));
    if (n < 0) return fail(MHR_EINVAL, "n must be >= 0");
    if (precision != 0 && precision != 2) return fail(MHR_EINVAL, "precision must be 0 (fp32) or 2 (fp64)");
    if (!out && n) return fail(MHR_EINVAL, "out is NULL");
    if (!src != !rel || !src != !dst) return fail(MHR_EINVAL, "src, rel and dst must all be given or all NULL");
    if (!src && n != g->dg.E) return fail(MHR_EINVAL, "with src == NULL, n must equal n_edges");
    if (mem != MHR_MEM_HOST && mem != MHR_MEM_DEVICE) return fail(MHR_EINVAL, "unknown mem kind");
    if (n == 0) return MHR_OK;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const size_t osz = precision == 0 ? 4 : 8;
    Scoped tmp;
    const uint32_t *ds = src, *dd = dst;
    const uint16_t* dr = rel;
    void* dout = out;
    if (mem == MHR_MEM_HOST) {
        if (src) {
            uint32_t *a, *c;
            uint16_t* b;
            MHR_CUDA_TRY(tmp.alloc(&a, 4 * n));
            MHR_CUDA_TRY(tmp.alloc(&b, 2 * n));
            MHR_CUDA_TRY(tmp.alloc(&c, 4 * n));
            MHR_CUDA_TRY(cudaMemcpyAsync(a, src, 4 * n, cudaMemcpyHostToDevice, st));
            MHR_CUDA_TRY(cudaMemcpyAsync(b, rel, 2 * n, cudaMemcpyHostToDevice, st));
            MHR_CUDA_TRY(cudaMemcpyAsync(c, dst, 4 * n, cudaMemcpyHostToDevice, st));
            ds = a;
            dr = b;
            dd = c;
        }
        void* o;
        MHR_CUDA_TRY(tmp.alloc(&o, osz * n));
        dout = o;
    }
    // ids must be in range: checked on the device copy is costly; validate host
    // arrays here when they are on the host
    if (mem == MHR_MEM_HOST && src) {
        for (int64_t i = 0; i < n; ++i)
            if (src[i] >= g->dg.n || dst[i] >= g->dg.n || rel[i] >= g->dg.R)
                return fail(MHR_EINVAL, "edge id out of range");
    }
    const int sms = std::max(1, g->num_sms);
    if (precision == 0) {
        MHR_CUDA_TRY(launch_edge_w32(g->dg, ds, dr, dd, n, static_cast<float*>(dout), nullptr, nullptr, nullptr,
                                     nullptr, sms, st));
    } else {
        if (g->dg.d >= kEdge64Warp) {
            const int64_t wave = int64_t(sms) * 6;
            int per = 32;
            while (per > 4 && (n + per - 1) / per < wave * kEdge64Warps) per >>= 1;
            const int64_t blocks = std::min<int64_t>(wave, ((n + per - 1) / per + kEdge64Warps - 1) / kEdge64Warps);
            k_edge_scores64_warp<<<static_cast<unsigned>(blocks), kEdge64Warps * 32, 0, st>>>(g->dg, ds, dr, dd, n, per,
                                                                                             static_cast<double*>(dout));
        } else
            k_edge_scores64<<<sms * 16, 128, 0, st>>>(g->dg, ds, dr, dd, n, static_cast<double*>(dout));
    }
    MHR_CUDA_TRY(cudaGetLastError());
    if (mem == MHR_MEM_HOST) {
        MHR_CUDA_TRY(cudaMemcpyAsync(out, dout, osz * n, cudaMemcpyDeviceToHost, st));
        MHR_CUDA_TRY(cudaStreamSynchronize(st));
    }
    return MHR_OK;
}

extern "C" mhr_status mhr_graph_get_info(const mhr_graph* g, mhr_graph_info* out) {
    MHR_TRY(check_graph(g));
    if (!out) return fail(MHR_EINVAL, "out is NULL");
    out->n_vertices = g->dg.n;
    out->n_edges = g->dg.E;
    out->n_relations = g->dg.R;
    out->dim = g->dg.d;
    out->max_out_degree = g->max_out_deg;
    out->max_in_degree = g->max_in_deg;
    out->eps32_edge = g->eps32_edge;
    out->eps64_edge = g->eps64_edge;
    out->err_path = g->err_path;
    out->epstc_edge = g->epstc_edge;
    out->err_path_tc = g->err_path_tc;
    return MHR_OK;
}

extern "C" const char* mhr_last_error(void) { return g_last_error.c_str(); }

extern "C" const char* mhr_version(void) { return "mhr-gb300 0.1 (sm_103a)"; }
