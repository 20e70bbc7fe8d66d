// fp64 edge weights in the canonical operation order (j = 0 .. d-1, each
// operation rounded to nearest), computed by a warp.
//
// GB300's fp64 pipe takes 16 cycles of an SM per warp instruction, and the
// canonical sum is one chain of d additions.  A TransE weight needs neither: its
// terms |(a + b) - c| and their partial sums are exact in fp64 whenever every
// coordinate is a multiple of 2^-Q and the sum stays below 2^(53 - Q), and then
// the rounded operations, in any order, are integer additions.  Q follows from
// the graph's largest norms (the sum's bound N < 2^(53 - Q)), so only the first
// condition is checked, per value: of fp32 coordinates drawn from N(0, 0.09),
// one edge in two thousand has a value too small for it; bf16 coordinates never
// fail.  Failing edges, and DistMult (products of three values do not fit), take the
// fp64 route: terms formed by all lanes, one lane per edge adds them in order.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mhr_internal.cuh"

namespace mhr {

// Exact binary32 -> binary64 widening done with integer operations (the value
// is finite: the graph load rejects NaN and infinity), keeping the slow fp64
// pipe for the arithmetic: sign and mantissa move over, the exponent is
// re-biased (1023 - 127 = 896), and a subnormal is first normalised.
__device__ __forceinline__ double widen(float f) {
    const uint32_t u = __float_as_uint(f);
    const uint64_t sign = static_cast<uint64_t>(u >> 31) << 63;
    uint32_t e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
    if (e == 0u) {
        if (m == 0u) return __longlong_as_double(static_cast<long long>(sign));
        const int sh = __clz(m) - 8;  // moves the top set bit to position 23
        m = (m << sh) & 0x7fffffu;
        e = static_cast<uint32_t>(1 - sh);
    }
    const uint64_t bits = sign | (static_cast<uint64_t>(e + 896u) << 52) | (static_cast<uint64_t>(m) << 29);
    return __longlong_as_double(static_cast<long long>(bits));
}

__device__ __forceinline__ double term64(float a, float b, float c, bool transe) {
    const double x = widen(a), y = widen(b), z = widen(c);
    return transe ? fabs(__dsub_rn(__dadd_rn(x, y), z)) : __dmul_rn(__dmul_rn(x, y), z);
}

// x in units of 2^-Q; bad is set when x is no multiple of one.  |x| < 2^(53 - Q).
__device__ __forceinline__ int64_t to_fixed(float x, int Q, bool& bad) {
    const uint32_t u = __float_as_uint(x);
    uint32_t e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
    if (e) m |= 0x800000u;
    else e = 1u;
    // m * 2^(e - 150) = v * 2^-Q  with  v = (m << 29) >> r
    const int r = min(63, 179 - Q - static_cast<int>(e));
    const uint64_t o = static_cast<uint64_t>(m) << 29, v = o >> r;
    bad |= (v << r) != o;
    const int64_t s = static_cast<int64_t>(static_cast<int32_t>(u) >> 31);
    return (static_cast<int64_t>(v) ^ s) - s;
}

// coordinates j .. j+3 of a row
__device__ __forceinline__ float4 row4(const void* tab, int dtype, int64_t row, int d, int j) {
    if (dtype == MHR_F32) {
        const float* p = static_cast<const float*>(tab) + row * d + j;
        if ((d & 3) == 0) return __ldg(reinterpret_cast<const float4*>(p));
        return make_float4(j < d ? p[0] : 0.f, j + 1 < d ? p[1] : 0.f, j + 2 < d ? p[2] : 0.f, j + 3 < d ? p[3] : 0.f);
    }
    const uint16_t* p = static_cast<const uint16_t*>(tab) + row * d + j;
    if ((d & 3) == 0) {
        const uint2 x = __ldg(reinterpret_cast<const uint2*>(p));
        return make_float4(bf_lo(x.x), bf_hi(x.x), bf_lo(x.y), bf_hi(x.y));
    }
    return make_float4(j < d ? bf16_to_f32(p[0]) : 0.f, j + 1 < d ? bf16_to_f32(p[1]) : 0.f,
                       j + 2 < d ? bf16_to_f32(p[2]) : 0.f, j + 3 < d ? bf16_to_f32(p[3]) : 0.f);
}

// TransE weight of edge (h, r, t) by the warp, in integers; *ok is false (and the
// value unusable) when a coordinate is no multiple of 2^-Q.  All lanes call with
// the same edge and get the same result.
__device__ __forceinline__ double warp_w64_fixed(const DevGraph& g, uint32_t h, uint32_t r, uint32_t t, int lane, bool* ok) {
    const int Q = g.qbits, d = g.d;
    int64_t acc = 0;
    bool bad = false;
    for (int j = 4 * lane; j < d; j += 128) {
        const float4 a = row4(g.vemb, g.dtype, h, d, j), b = row4(g.remb, g.dtype, r, d, j), c = row4(g.vemb, g.dtype, t, d, j);
        const float x[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.x, b.y, b.z, b.w}, z[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t v = to_fixed(x[k], Q, bad) + to_fixed(y[k], Q, bad) - to_fixed(z[k], Q, bad);
            acc += v < 0 ? -v : v;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    *ok = __ballot_sync(0xffffffffu, bad) == 0u;
    // acc <= 2^53 and a power of two: both steps are exact
    const double sum = __dmul_rn(__ll2double_rn(acc), __longlong_as_double(static_cast<long long>(1023 - Q) << 52));
    return __dsub_rn(g.gamma, sum);
}

// fp64 weights of up to 32 edges, one per lane (live lanes), in the canonical
// order: each 32-coordinate chunk is read row by row (whole 128-byte lines), all
// lanes form its terms into `stage` (32 x 33 doubles of the warp's shared memory),
// then each lane adds its edge's terms in order.  A lane per edge straight from
// the rows fetched every line eight times (16 bytes of 96 rows per step do not
// stay in L1).  All lanes call.
__device__ __forceinline__ double warp_w64_staged(const DevGraph& g, uint32_t h, uint32_t r, uint32_t t, bool live,
                                                  double* stage, int lane) {
    const int d = g.d;
    const bool transe = g.fn == MHR_SCORE_TRANSE_L1;
    const unsigned mask = __ballot_sync(0xffffffffu, live);
    const int n = 32 - __clz(mask);  // edges 0 .. n-1 cover the live ones
    const int sub = lane & 7, row = lane >> 3;  // eight lanes per edge, four edges at a time
    double acc = 0.0;
    for (int j0 = 0; j0 < d; j0 += 32) {
        const int j = j0 + 4 * sub;
#pragma unroll 4
        for (int e0 = 0; e0 < n; e0 += 4) {
            const int e = e0 + row;
            const uint32_t eh = __shfl_sync(0xffffffffu, h, e & 31), er = __shfl_sync(0xffffffffu, r, e & 31),
                           et = __shfl_sync(0xffffffffu, t, e & 31);
            if (e < n && ((mask >> e) & 1u) && j < d) {
                const float4 a = row4(g.vemb, g.dtype, eh, d, j), b = row4(g.remb, g.dtype, er, d, j),
                             c = row4(g.vemb, g.dtype, et, d, j);
                double* s = stage + e * 33 + 4 * sub;
                s[0] = term64(a.x, b.x, c.x, transe);
                s[1] = term64(a.y, b.y, c.y, transe);
                s[2] = term64(a.z, b.z, c.z, transe);
                s[3] = term64(a.w, b.w, c.w, transe);
            }
        }
        __syncwarp();
        if (live) {
            const int m = min(32, d - j0);
            const double* s = stage + lane * 33;
            if (m == 32) {
#pragma unroll 8
                for (int k = 0; k < 32; ++k) acc = __dadd_rn(acc, s[k]);
            } else {
                for (int k = 0; k < m; ++k) acc = __dadd_rn(acc, s[k]);
            }
        }
        __syncwarp();
    }
    return transe ? __dsub_rn(g.gamma, acc) : acc;
}

}  // namespace mhr
