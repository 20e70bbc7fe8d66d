// Warp-cooperative fp32 edge weights: 32 edges per warp, one per lane, scored
// by groups of G lanes with 16-byte vector loads; and the row of a CSR
// position for warps that walk consecutive edges.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mhr_internal.cuh"

namespace mhr {

__device__ __forceinline__ int64_t upper_bound_i64(const int64_t* __restrict__ a, int64_t n, int64_t x) {
    // first index i in [0, n) with a[i] > x (n if none)
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (a[mid] <= x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// The last j with offs[j] <= x, for offs[0] <= x, found by the whole warp with
// a 32-ary search over offs[0 .. n] (x is warp-uniform).
__device__ __forceinline__ int64_t warp_row_search(const int64_t* __restrict__ offs, int64_t n, int64_t x, int lane) {
    int64_t lo = 0, span = n + 1;  // offs[lo] <= x < offs[lo + span] (or the end)
    while (span > 32) {
        const int64_t step = (span + 31) >> 5;
        const int64_t j = lane * step;
        const bool le = j < span && offs[lo + j] <= x;
        const int64_t c = __popc(__ballot_sync(0xffffffffu, le));  // >= 1: offs[lo] <= x
        const int64_t nlo = (c - 1) * step;
        span = min(step, span - nlo);
        lo += nlo;
    }
    const bool le = lane < span && offs[lo + lane] <= x;
    return lo + __popc(__ballot_sync(0xffffffffu, le)) - 1;
}

// Row of position x >= offs[lo] of each lane, given a row lo at or before the
// warp's first one: each lane counts the row starts after lo that are <= x
// among the next 32 (five shuffle steps); a lane with more than 31 of them
// (empty rows) searches on its own.  All lanes call.
__device__ __forceinline__ int64_t warp_rows_from(const int64_t* __restrict__ offs, int64_t n, int64_t lo, int64_t x,
                                                  int lane) {
    const int64_t j = lo + 1 + lane;
    const int64_t b = j <= n ? offs[j] : INT64_MAX;
    int own = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
        const int64_t pv = __shfl_sync(0xffffffffu, b, own + step - 1);
        if (pv <= x) own += step;
    }
    const int64_t b31 = __shfl_sync(0xffffffffu, b, 31);
    if (b31 <= x) return upper_bound_i64(offs, n + 1, x) - 1;
    return lo + own;
}

// fp32 weights of 32 edges, one per lane, for rows of at most two 16-byte
// vectors per lane of a G-lane group (bf16 with d % 8 == 0 and d / 8 <= 2G,
// fp32 with d % 4 == 0 and d / 4 <= 2G).  An edge joins `fixv` and `rndv`; bit
// 0 of rsa says whether fixv is its head, the other bits hold the relation.
// The rows of the random side (rndv) of up to four rounds of 32 / G edges are
// loaded before any arithmetic, so a warp keeps up to four rows per group in
// flight instead of one; the fixed side and the relation row are the same few
// rows for many edges and come from L1.  The group sums of RB rounds are
// reduced together: plain xor steps down to RB lanes, then a butterfly in which
// each step halves the rounds a lane carries, so lane `sub` ends with round
// (sub mod RB): RB - 1 shuffles for the last log2(RB) steps of RB rounds
// instead of RB log2(RB).  Every lane still adds its own partial to its
// partner's at each step of the same xor tree, and fp32 addition is
// commutative, so with the same per-element expression and the same order
// within a lane the weights are those edge_w32_group computes for width G.  SPLIT:
// a lane's two vectors are summed each by itself and then added, the first step of the
// tree of a group twice as wide, so the weights are those of width 2G: sums of 4 or 8
// terms before the tree instead of 8 or 16, a smaller error (20 M edges of 128 fp32
// values: relative 3.53e-8 against 3.60e-8).
// Four rounds at a time and three 256-thread blocks per SM (80 registers)
// measured fastest on the frontier expansion of 38.6 M edges with 256-byte rows
// (3.31 ms; eight rounds at two blocks per SM 3.88 ms; two rounds at four
// blocks 3.32 ms).
constexpr int kScoreRounds = 4;
// FEW: only the edges of lanes 0 .. n-1 are wanted, n a multiple of the edges of a batch.
template <int G, bool SPLIT = false, bool FEW = false>
__device__ __forceinline__ float warp_score_v(const DevGraph& g, uint32_t fixv, uint32_t rndv, uint32_t rsa, int lane,
                                              int n = 32) {
    constexpr int H = 32 / G;
    constexpr int RB = G < kScoreRounds ? G : kScoreRounds;  // rounds loaded and reduced together
    const unsigned FULL = 0xffffffffu;
    const int sub = lane & (G - 1);
    const bool f32 = g.dtype == MHR_F32;
    const bool transe = g.fn == MHR_SCORE_TRANSE_L1;
    const int nvec = f32 ? (g.d >> 2) : (g.d >> 3);  // 16-byte vectors per row
    const bool h0 = sub < nvec, h1 = sub + G < nvec;
    const uint4* E = static_cast<const uint4*>(g.vemb);
    const uint4* Rw = static_cast<const uint4*>(g.remb);
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    float wmine = 0.f;
#pragma unroll
    for (int rb = 0; rb < G; rb += RB) {
        if (FEW && rb * H >= n) break;
        uint4 C0[RB], C1[RB];
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int src = (rb + i) * H + lane / G;
            const int64_t v = __shfl_sync(FULL, rndv, src);
            C0[i] = h0 ? __ldg(E + v * nvec + sub) : z;
            C1[i] = h1 ? __ldg(E + v * nvec + sub + G) : z;
        }
        float acc[RB];
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const int src = (rb + i) * H + lane / G;
            const uint32_t q2 = __shfl_sync(FULL, rsa, src);
            const int64_t rr = q2 >> 1;
            const bool sa = (q2 & 1u) != 0u;
            const int64_t fv = __shfl_sync(FULL, fixv, src);
            const uint4 F0 = h0 ? __ldg(E + fv * nvec + sub) : z, B0 = h0 ? __ldg(Rw + rr * nvec + sub) : z;
            const uint4 F1 = h1 ? __ldg(E + fv * nvec + sub + G) : z, B1 = h1 ? __ldg(Rw + rr * nvec + sub + G) : z;
            // fixed head: the edge (fixv, r, rndv); fixed tail: (rndv, r, fixv)
            const uint4 As[2] = {sa ? F0 : C0[i], sa ? F1 : C1[i]};
            const uint4 Cs[2] = {sa ? C0[i] : F0, sa ? C1[i] : F1};
            const uint4 Bs[2] = {B0, B1};
            float a_ = 0.f;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (k == 0 && !h0) break;
                if (k == 1 && !h1) break;
                const uint32_t a[4] = {As[k].x, As[k].y, As[k].z, As[k].w};
                const uint32_t b[4] = {Bs[k].x, Bs[k].y, Bs[k].z, Bs[k].w};
                const uint32_t c[4] = {Cs[k].x, Cs[k].y, Cs[k].z, Cs[k].w};
                float p_ = SPLIT ? 0.f : a_;
                if (f32) {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        p_ += term_tr(__uint_as_float(a[e]), __uint_as_float(b[e]), __uint_as_float(c[e]), transe);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        p_ += term_tr(bf_lo(a[e]), bf_lo(b[e]), bf_lo(c[e]), transe);
                        p_ += term_tr(bf_hi(a[e]), bf_hi(b[e]), bf_hi(c[e]), transe);
                    }
                }
                a_ = SPLIT && k == 1 ? a_ + p_ : p_;
            }
            acc[i] = a_;
        }
        // xor steps G/2 .. RB: every round's sum over lanes that differ in those bits
#pragma unroll
        for (int off = G >> 1; off >= RB; off >>= 1)
#pragma unroll
            for (int i = 0; i < RB; ++i) acc[i] += __shfl_xor_sync(FULL, acc[i], off, G);
        // butterfly over the low log2(RB) bits: keep the half of the rounds
        // selected by this lane's bit, send the other half to the partner
#pragma unroll
        for (int off = RB >> 1; off > 0; off >>= 1) {
            const bool hi = (sub & off) != 0;
#pragma unroll
            for (int j = 0; j < off; ++j) {
                const float send = hi ? acc[j] : acc[j + off];
                const float keep = hi ? acc[j + off] : acc[j];
                acc[j] = keep + __shfl_xor_sync(FULL, send, off, G);
            }
        }
        // lane sub of group gi now holds round rb + (sub mod RB) of edge (round) * H + gi
        const float w = transe ? __fsub_rn(g.gamma32, acc[0]) : acc[0];
        const int rd = lane / H;
        const float tw = __shfl_sync(FULL, w, (lane & (H - 1)) * G + (rd & (RB - 1)));
        if (rd >= rb && rd < rb + RB) wmine = tw;
    }
    return wmine;
}

// The same for rows of any length: groups of `G` lanes (a power of two <= 32)
// score 32 / G edges at a time.
__device__ __forceinline__ float warp_score_any(const DevGraph& g, uint32_t hu, uint32_t r, uint32_t tv, int G,
                                                int lane) {
    const int H = 32 / G, sub = lane & (G - 1);
    float wmine = 0.f;
    for (int rd = 0; rd < G; ++rd) {
        const int src = rd * H + lane / G;
        const uint32_t a = __shfl_sync(0xffffffffu, hu, src);
        const uint32_t rr = __shfl_sync(0xffffffffu, r, src);
        const uint32_t b = __shfl_sync(0xffffffffu, tv, src);
        const float w = edge_w32_group(g, a, rr, b, sub, G);
        const float tw = __shfl_sync(0xffffffffu, w, ((lane - rd * H) & (H - 1)) * G);
        if (lane / H == rd) wmine = tw;
    }
    return wmine;
}

// Whether warp_score_v<G> takes the graph's rows
__host__ __device__ inline bool score_vec2(const DevGraph& g, int G) {
    return g.dtype == MHR_F32 ? ((g.d & 3) == 0 && (g.d >> 2) <= 2 * G) : ((g.d & 7) == 0 && (g.d >> 3) <= 2 * G);
}

// lanes that score one edge together: about `per` 16-byte vectors per lane per row
inline int hit_group_width(int d, int dtype, int per) {
    const int vec = (dtype == MHR_F32) ? ((d & 3) == 0 ? d / 4 : d) : ((d & 7) == 0 ? d / 8 : d);
    const int want = (vec + per - 1) / per;
    int w = 1;
    while (w < want && w < 32) w <<= 1;
    return w;
}

}  // namespace mhr
