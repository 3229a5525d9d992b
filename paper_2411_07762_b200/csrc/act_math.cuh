// Arithmetic shared by the activation kernels: the smoothing divide, the int8 codes and the
// storage of T (Sec. 4.2 smoothing, Sec. 5.1 per-token round-to-nearest, Sec. 4.1 projection).
#pragma once
#include "aser_common.cuh"

namespace aser {

struct RawChunk {  // 8 activations and their 8 smoothing divisors
    uint4 x;
    float4 s0, s1;
};

__device__ __forceinline__ RawChunk load_raw(const __half* xrow, const float* s, int col, bool ok) {
    RawChunk rc;
    rc.x = ok ? *reinterpret_cast<const uint4*>(xrow + col) : make_uint4(0, 0, 0, 0);
    if (s) {
        rc.s0 = *reinterpret_cast<const float4*>(s + col);
        rc.s1 = *reinterpret_cast<const float4*>(s + col + 4);
    } else {
        rc.s0 = make_float4(1.f, 1.f, 1.f, 1.f);
        rc.s1 = rc.s0;
    }
    return rc;
}

// x~ = fp32(x) / s, one IEEE division each.  Dividing by 1 is the identity, and s is 1 on all
// but the few outlier channels, so the (long) division sequence is skipped for such groups.
__device__ __forceinline__ void smooth8(const RawChunk& rc, float (&v)[8]) {
    const __half* h = reinterpret_cast<const __half*>(&rc.x);
    const bool ones = rc.s0.x == 1.f && rc.s0.y == 1.f && rc.s0.z == 1.f && rc.s0.w == 1.f &&
                      rc.s1.x == 1.f && rc.s1.y == 1.f && rc.s1.z == 1.f && rc.s1.w == 1.f;
    if (ones) {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = __half2float(h[i]);
        return;
    }
    v[0] = __fdiv_rn(__half2float(h[0]), rc.s0.x); v[1] = __fdiv_rn(__half2float(h[1]), rc.s0.y);
    v[2] = __fdiv_rn(__half2float(h[2]), rc.s0.z); v[3] = __fdiv_rn(__half2float(h[3]), rc.s0.w);
    v[4] = __fdiv_rn(__half2float(h[4]), rc.s1.x); v[5] = __fdiv_rn(__half2float(h[5]), rc.s1.y);
    v[6] = __fdiv_rn(__half2float(h[6]), rc.s1.z); v[7] = __fdiv_rn(__half2float(h[7]), rc.s1.w);
}

// T element(s) -> memory.  `lo_off` == 0: T[j] = bf16(t).  Otherwise T is stored as a PAIR of
// bf16 numbers, T[j] = bf16(t) and T[j + lo_off] = bf16(t - T[j]), whose sum carries 16
// significant bits; a linear kernel given the up projection twice, [L_B | L_B], then adds both.
__device__ __forceinline__ void store_t(__nv_bfloat16* row, int j, float t, int lo_off) {
    const __nv_bfloat16 hi = __float2bfloat16_rn(t);
    row[j] = hi;
    if (lo_off) row[j + lo_off] = __float2bfloat16_rn(t - __bfloat162float(hi));
}
__device__ __forceinline__ void store_t2(__nv_bfloat16* row, int j, float t0, float t1, int lo_off) {
    const __nv_bfloat162 hi = __floats2bfloat162_rn(t0, t1);
    *reinterpret_cast<__nv_bfloat162*>(row + j) = hi;
    if (lo_off)
        *reinterpret_cast<__nv_bfloat162*>(row + j + lo_off) =
            __floats2bfloat162_rn(t0 - __low2float(hi), t1 - __high2float(hi));
}

// The factor that stands in for the division by a row's scale: 0 for a row of zeros, and where 1 / sc may overflow.  Then
// every undivided element is zero (the smallest fp16 magnitude over 127 is 4.7e-10); what smoothing divided goes by exact codes.
__device__ __forceinline__ float code_rcp(float sc) { return sc > 0x1p-127f ? __frcp_rn(sc) : 0.f; }

// Exact codes for eight values (the definition: IEEE quotient, round half to even, clamp).
static __device__ __noinline__ uint2 quant8_exact(float v0, float v1, float v2, float v3, float v4, float v5,
                                           float v6, float v7, float sc, float qmax) {
    const float v[8] = {v0, v1, v2, v3, v4, v5, v6, v7};
    uint32_t w[2] = {0, 0};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int q = rne_clamp(__fdiv_rn(v[i], sc), -qmax, qmax);
        w[i >> 2] |= (uint32_t)(q & 0xFF) << (8 * (i & 3));
    }
    return make_uint2(w[0], w[1]);
}
// The same codes, with rcp = code_rcp(sc), on packed fp32 pairs: t = x~ * (1 / sc), rounded by adding
// 1.5 * 2^23 (the low byte of the sum is the code); the distance of t to that integer tells the
// near-ties, and a group with one takes the exact path as a whole.
__device__ __forceinline__ uint2 quant8_pairs(const float (&v)[8], float sc, float rcp, float qmax) {
    const float kMagic = 12582912.0f;
    const float2 r2 = make_float2(rcp, rcp), m2 = make_float2(kMagic, kMagic);
    const float2 nm2 = make_float2(-kMagic, -kMagic), neg1 = make_float2(-1.f, -1.f);
    uint32_t q[8];
    float far = 0.f;        // largest distance of a product to its rounded integer (branch-free)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 t = __fmul2_rn(make_float2(v[2 * i], v[2 * i + 1]), r2);
        const float2 u = __fadd2_rn(t, m2);
        const float2 w = __fadd2_rn(u, nm2);            // the rounded integer
        const float2 d = __ffma2_rn(w, neg1, t);        // t - w, exact
        q[2 * i] = __float_as_uint(u.x);
        q[2 * i + 1] = __float_as_uint(u.y);
        far = fmaxf(far, fmaxf(fabsf(d.x), fabsf(d.y)));
    }
    if (far > 0.4999f || (rcp == 0.f && sc > 0.f)) return quant8_exact(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], sc, qmax);
    const uint32_t a01 = __byte_perm(q[0], q[1], 0x0040), a23 = __byte_perm(q[2], q[3], 0x0040);
    const uint32_t a45 = __byte_perm(q[4], q[5], 0x0040), a67 = __byte_perm(q[6], q[7], 0x0040);
    return make_uint2(__byte_perm(a01, a23, 0x5410), __byte_perm(a45, a67, 0x5410));
}

// Eight codes of a row whose divisors are all 1: fp16 pairs widened by the conversion unit, then on
// packed fp32 pairs su = x * (1 / sc) + 1.5 * 2^23 (one rounding: the low byte of su is the code),
// -w = 1.5 * 2^23 - su (exact) and d = x * (1 / sc) - w, the distance of the product to its integer.
// rne(x / sc) can differ from that integer only where the product is within 3.1e-5 of a tie (by so much the quotient
// and the product differ at most): a group with an element within 4e-5 (one in 1600) sets *tie and needs the exact division.
__device__ __forceinline__ uint2 codes8_try(const uint4& x, float rcp, bool* tie) {
    const float kMagic = 12582912.0f;
    const float2 m2 = make_float2(kMagic, kMagic), neg1 = make_float2(-1.f, -1.f), r2 = make_float2(rcp, rcp);
    const uint32_t xw[4] = {x.x, x.y, x.z, x.w};
    uint32_t u[8];
    float far = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&xw[i]));
        const float2 su = __ffma2_rn(f, r2, m2);
        const float2 nw = __ffma2_rn(su, neg1, m2);
        const float2 d = __ffma2_rn(f, r2, nw);
        u[2 * i] = __float_as_uint(su.x);
        u[2 * i + 1] = __float_as_uint(su.y);
        far = max3_abs(far, d.x, d.y);
    }
    *tie = far > 0.49996f;
    const uint32_t a01 = __byte_perm(u[0], u[1], 0x0040), a23 = __byte_perm(u[2], u[3], 0x0040);
    const uint32_t a45 = __byte_perm(u[4], u[5], 0x0040), a67 = __byte_perm(u[6], u[7], 0x0040);
    return make_uint2(__byte_perm(a01, a23, 0x5410), __byte_perm(a45, a67, 0x5410));
}
__device__ __forceinline__ uint2 codes8_exact(const uint4& x, float sc, float qmax) {
    const __half2* h = reinterpret_cast<const __half2*>(&x);
    const float2 a = __half22float2(h[0]), b = __half22float2(h[1]), c = __half22float2(h[2]), d = __half22float2(h[3]);
    return quant8_exact(a.x, a.y, b.x, b.y, c.x, c.y, d.x, d.y, sc, qmax);
}
__device__ __forceinline__ uint2 codes8_unit(const uint4& x, float sc, float rcp, float qmax) {
    bool tie;
    const uint2 q = codes8_try(x, rcp, &tie);
    return tie ? codes8_exact(x, sc, qmax) : q;
}

// ---------------------------------------------------------------------------
// Whole rows in registers: the row maxima, the scales and the codes of R token rows by one CTA.
// ---------------------------------------------------------------------------
// A thread has the same CPT 8-column chunks of every row (chunk threadIdx.x + i * blockDim.x), so X is read once and the
// smoothing divisors once for all rows.  The divisors are 1 on all but the ~1 % outlier channels, and testing for them per
// element costs a quarter of the pass: each thread makes a mask of its chunks (0x7fff per undivided column, which also
// takes the magnitude) and lists the divided columns of the CTA; the maximum of the undivided ones is one AND and one half2
// maximum per pair, the codes are made as if nothing were divided, and the listed columns are done apart, one (row, column)
// per thread, with IEEE divisions.  More listed columns than the list holds: the general loop, which divides wherever
// a divisor is not 1.  The maximum does not depend on the order, so scales and codes have the same bits by every path.
constexpr int kRowsList = 512;
template <int R>
struct RowsShared {
    unsigned rowmax[R];         // bits of a non-negative float: ordered like the floats
    int n_list;
    int list_col[kRowsList];
};

// (Codes of a NaN are unspecified: -1 by the fast path, -qmax by the exact one.)
template <int CPT, int R>
__device__ __forceinline__ void quantize_rows(const __half* __restrict__ X, const float* __restrict__ s, int nrows, int K,
                                              int8_t* __restrict__ Xq, float* __restrict__ a_scale, float qmax,
                                              RowsShared<R>& sh) {
    const int TH = blockDim.x, tid = threadIdx.x, lane = tid & 31, chunks = K / 8;
    uint4 x[R][CPT];
#pragma unroll
    for (int i = 0; i < CPT; ++i) {
        const int c = tid + i * TH;
#pragma unroll
        for (int rr = 0; rr < R; ++rr)
            x[rr][i] = (rr < nrows && c < chunks) ? *reinterpret_cast<const uint4*>(X + (size_t)rr * K + c * 8)
                                                  : make_uint4(0, 0, 0, 0);
    }
    uint32_t mask[CPT][4];
#pragma unroll
    for (int i = 0; i < CPT; ++i)
#pragma unroll
        for (int w = 0; w < 4; ++w) mask[i][w] = 0x7fff7fffu;
    if (tid == 0) sh.n_list = 0;
    if (tid < R) sh.rowmax[tid] = 0u;
    __syncthreads();
    if (s) {
#pragma unroll
        for (int i = 0; i < CPT; ++i) {
            const int c = tid + i * TH;
            if (c >= chunks) continue;
            const float4 s0 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c);
            const float4 s1 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c + 1);
            const float sv[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (sv[e] != 1.f) {
                    mask[i][e >> 1] &= (e & 1) ? 0x0000ffffu : 0xffff0000u;
                    const int at = atomicAdd(&sh.n_list, 1);
                    if (at < kRowsList) sh.list_col[at] = c * 8 + e;
                }
        }
    }
    __syncthreads();
    const int listed = sh.n_list;
    if (listed <= kRowsList) {
        for (int e = tid; e < listed * R; e += TH) {
            const int rr = e % R, col = sh.list_col[e / R];
            if (rr >= nrows) continue;
            const float f = __fdiv_rn(__half2float(X[(size_t)rr * K + col]), __ldg(s + col));
            atomicMax(&sh.rowmax[rr], __float_as_uint(fmaxf(fabsf(f), 0.f)));       // a NaN does not count
        }
#pragma unroll
        for (int rr = 0; rr < R; ++rr) {
            __half2 h = __float2half2_rn(0.f);
#pragma unroll
            for (int i = 0; i < CPT; ++i) {
                const uint32_t xw[4] = {x[rr][i].x, x[rr][i].y, x[rr][i].z, x[rr][i].w};
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const uint32_t v = xw[w] & mask[i][w];
                    h = __hmax2(h, *reinterpret_cast<const __half2*>(&v));
                }
            }
            const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(__low2float(h), __high2float(h))));
            if (lane == 0) atomicMax(&sh.rowmax[rr], m);
        }
    } else {
#pragma unroll
        for (int rr = 0; rr < R; ++rr) {
            float m = 0.f;
#pragma unroll
            for (int i = 0; i < CPT; ++i) {
                const int c = tid + i * TH;
                if (c >= chunks) continue;
                RawChunk rc;
                rc.x = x[rr][i];
                rc.s0 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c);
                rc.s1 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c + 1);
                float v[8];
                smooth8(rc, v);
#pragma unroll
                for (int e = 0; e < 8; ++e) m = fmaxf(m, fabsf(v[e]));
            }
            const unsigned u = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
            if (lane == 0) atomicMax(&sh.rowmax[rr], u);
        }
    }
    __syncthreads();
    float sc[R], rcp[R];
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
        sc[rr] = __fdiv_rn(__uint_as_float(sh.rowmax[rr]), qmax);
        rcp[rr] = code_rcp(sc[rr]);
    }
#pragma unroll
    for (int rr = 0; rr < R; ++rr)
        if (tid == rr && rr < nrows) a_scale[rr] = sc[rr];
    if (listed <= kRowsList) {
#pragma unroll
        for (int i = 0; i < CPT; ++i) {
            const int c = tid + i * TH;
#pragma unroll
            for (int rr = 0; rr < R; ++rr) {
                const uint2 q = codes8_unit(x[rr][i], sc[rr], rcp[rr], qmax);
                if (rr < nrows && c < chunks) *reinterpret_cast<uint2*>(Xq + (size_t)rr * K + c * 8) = q;
            }
        }
        __syncthreads();            // orders the stores above before the single bytes below
        for (int e = tid; e < listed * R; e += TH) {
            const int rr = e % R, col = sh.list_col[e / R];
            if (rr >= nrows) continue;
            const float scale = __fdiv_rn(__uint_as_float(sh.rowmax[rr]), qmax);
            const float xt = __fdiv_rn(__half2float(X[(size_t)rr * K + col]), __ldg(s + col));
            const float quot = scale > 0.f ? __fdiv_rn(xt, scale) : xt * 0.f;
            const int code = quot != quot ? -1 : rne_clamp(quot, -qmax, qmax);
            Xq[(size_t)rr * K + col] = (int8_t)code;
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < CPT; ++i) {
        const int c = tid + i * TH;
        if (c >= chunks) continue;
#pragma unroll
        for (int rr = 0; rr < R; ++rr) {
            if (rr >= nrows) continue;
            RawChunk rc;
            rc.x = x[rr][i];
            rc.s0 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c);
            rc.s1 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c + 1);
            float v[8];
            smooth8(rc, v);
            *reinterpret_cast<uint2*>(Xq + (size_t)rr * K + c * 8) = quant8_pairs(v, sc[rr], rcp[rr], qmax);
        }
    }
}

}  // namespace aser
