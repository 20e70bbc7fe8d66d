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
// fail.  Failing edges, and DistMult (whose partial sums round), take the fp64 route:
// terms formed by all lanes, one lane per edge adds them in order.  A DistMult term
// rounds once (the product of two binary32 values is exact in binary64), so it is
// formed in integers too (mul3_rn), which leaves one fp64 operation per coordinate
// of three.
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

// The binary64 product a * b * c of finite binary32 values, rounded to nearest even
// (once: a * b has 48 bits and is exact; no product of three leaves binary64's normal
// range).  The 72-bit product of the significands is cut to its top 53 bits, half
// of the last place and ties decided by the bits below.  A zero factor gives +0,
// which adds like -0 to any sum that starts at +0.
__host__ __device__ __forceinline__ uint64_t mul3_bits(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t ea = (a >> 23) & 0xffu, eb = (b >> 23) & 0xffu, ec = (c >> 23) & 0xffu;
    uint32_t ma = (a & 0x7fffffu) | 0x800000u, mb = (b & 0x7fffffu) | 0x800000u, mc = (c & 0x7fffffu) | 0x800000u;
    int e = static_cast<int>(ea + eb + ec);
    if (ea == 0u || eb == 0u || ec == 0u) {  // a zero or a subnormal: normalise
        uint32_t* m[3] = {&ma, &mb, &mc};
        const uint32_t ex[3] = {ea, eb, ec};
        for (int i = 0; i < 3; ++i) {
            if (ex[i]) continue;
            *m[i] &= 0x7fffffu;
            if (*m[i] == 0u) return 0ull;
            e += 1;
            while (!(*m[i] & 0x800000u)) {
                *m[i] <<= 1;
                e -= 1;
            }
        }
    }
    const uint64_t p = static_cast<uint64_t>(ma) * mb;  // 47 or 48 bits
    const uint64_t lo = static_cast<uint64_t>(static_cast<uint32_t>(p)) * mc;
    const uint64_t hi = static_cast<uint64_t>(static_cast<uint32_t>(p >> 32)) * mc + (lo >> 32);  // bits 32 .. 71
    const uint32_t x0 = static_cast<uint32_t>(lo), top = static_cast<uint32_t>(hi >> 32);       // 32 <= top < 256
    const uint32_t k = 17u + (top >= 64u ? 1u : 0u) + (top >= 128u ? 1u : 0u);                    // bits below the top 53
    const uint64_t r = (hi << (32u - k)) | (x0 >> k);
    const uint32_t rem = x0 & ((1u << k) - 1u), half = 1u << (k - 1u);
    const uint64_t up = rem + (static_cast<uint32_t>(r) & 1u) > half ? 1u : 0u;
    // the leading one of r adds the last unit of the exponent, a carry another
    const uint64_t ex = static_cast<uint64_t>(e - 450 + 1023 + 52 - 1 + static_cast<int>(k));
    return (static_cast<uint64_t>((a ^ b ^ c) >> 31) << 63) | ((ex << 52) + r + up);
}
__device__ __forceinline__ double mul3_rn(float a, float b, float c) {
    return __longlong_as_double(
        static_cast<long long>(mul3_bits(__float_as_uint(a), __float_as_uint(b), __float_as_uint(c))));
}

__device__ __forceinline__ double term64(float a, float b, float c, bool transe) {
    return transe ? fabs(__dsub_rn(__dadd_rn(widen(a), widen(b)), widen(c))) : mul3_rn(a, b, c);
}

// acc + sign * x in units of 2^-Q, sign = 1 or -1; bad is set when x is no multiple of
// one.  x = m 2^(e - 150) is m shifted left by e - 150 + Q places, one multiply-add into
// the 64-bit sum, or right by a few when it is small.  The shift stays below 30: a
// normal x has 2^23 <= m and |x| < 2^(53 - Q); a subnormal one has e = 1 and Q <= 149.
__device__ __forceinline__ int64_t add_fixed(int64_t acc, float x, bool minus, int Q, bool& bad) {
    const uint32_t u = __float_as_uint(x);
    const uint32_t e = (u >> 23) & 0xffu;
    uint32_t m = (u & 0x7fffffu) | (e ? 0x800000u : 0u);
    int sh = static_cast<int>(max(e, 1u)) - 150 + Q;
    if (sh < 0) {
        const int k = min(-sh, 31);
        bad |= (m & ((1u << k) - 1u)) != 0u;
        m >>= k;
        sh = 0;
    }
    const int32_t sm = ((static_cast<int32_t>(u) < 0) != minus) ? -static_cast<int32_t>(m) : static_cast<int32_t>(m);
    return acc + static_cast<int64_t>(sm) * static_cast<int32_t>(1u << sh);
}

// |a + b - c| in units of 2^-Q
__device__ __forceinline__ int64_t abs_fixed(float a, float b, float c, int Q, bool& bad) {
    const int64_t v = add_fixed(add_fixed(add_fixed(0, a, false, Q, bad), b, false, Q, bad), c, true, Q, bad);
    return v < 0 ? -v : v;
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
            acc += abs_fixed(x[k], y[k], z[k], Q, bad);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    *ok = __ballot_sync(0xffffffffu, bad) == 0u;
    // acc <= 2^53 and a power of two: both steps are exact
    const double sum = __dmul_rn(__ll2double_rn(acc), __longlong_as_double(static_cast<long long>(1023 - Q) << 52));
    return __dsub_rn(g.gamma, sum);
}

// The same for the edges of lanes 0 .. n-1, four at a time by eight lanes each: the
// same conversions as a warp per edge with an eighth of the reduction's shuffles per
// edge, for many edges.  `left` stays set on the lanes whose edge does not fit.
__device__ __forceinline__ double warp_w64_fixed_each(const DevGraph& g, uint32_t h, uint32_t r, uint32_t t, int n,
                                                      int lane, bool& left) {
    const int Q = g.qbits, d = g.d;
    const int sub = lane & 7, grp = lane >> 3;
    int64_t mine = 0;
    for (int b = 0; b < n; b += 4) {
        const int src = min(b + grp, 31);
        const uint32_t eh = __shfl_sync(0xffffffffu, h, src), er = __shfl_sync(0xffffffffu, r, src),
                       et = __shfl_sync(0xffffffffu, t, src);
        int64_t acc = 0;
        bool bad = false;
#pragma unroll 2
        for (int j = 4 * sub; j < d; j += 32) {
            const float4 a = row4(g.vemb, g.dtype, eh, d, j), e = row4(g.remb, g.dtype, er, d, j), c = row4(g.vemb, g.dtype, et, d, j);
            const float x[4] = {a.x, a.y, a.z, a.w}, y[4] = {e.x, e.y, e.z, e.w}, z[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                acc += abs_fixed(x[k], y[k], z[k], Q, bad);
            }
        }
        if (bad) acc = -1;  // sums are not negative: the top bit survives the additions below as a marker
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            const int64_t other = __shfl_xor_sync(0xffffffffu, acc, o);
            acc = (acc < 0 || other < 0) ? -1 : acc + other;
        }
        const int64_t got = __shfl_sync(0xffffffffu, acc, (lane & 3) * 8);
        if ((lane >> 2) == (b >> 2)) mine = got;
    }
    if (lane < n && mine >= 0) left = false;
    // mine <= 2^53 and a power of two: both steps are exact
    const double sum = __dmul_rn(__ll2double_rn(mine), __longlong_as_double(static_cast<long long>(1023 - Q) << 52));
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
