// Offline weight path: smoothing multiply, per-output-channel int4 round-to-nearest,
// nibble packing (Sec. 4.2 Eq. 10/12 Q(W_s); Sec. 5.1 per-channel RTN), plus the
// permutation between the canonical packed form and the tensor-core kernel's layout.
#include "aser_common.cuh"

namespace aser {

namespace {

// Low nibbles of four words, one after the other in sixteen bits.
__device__ __forceinline__ uint32_t nibbles4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    uint32_t x = __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410) & 0x0F0F0F0Fu;
    x = (x | (x >> 4)) & 0x00FF00FFu;
    return (x | (x >> 8)) & 0x0000FFFFu;
}

// A CTA quantizes whole rows, one after the other; thread t takes the chunks t, t + TH, ... of a row, s
// stays in shared memory, so W is read once and s once per CTA.  The next row is loaded before the current one
// is reduced; the products w s are kept in registers between the maximum and the codes.  Codes: one fused multiply-add
// v * (1 / scale) + 1.5 * 2^23 on packed fp32 pairs (the low nibble is the code), two more give the distance of the product
// to its integer.  v * (1 / scale) is within 4e-6 of the quotient (|quotient| <= 7), so its rounding is that of the
// IEEE quotient unless it lies within 1e-5 of a tie; such chunks (one in ten thousand), and those with a NaN, are
// divided, as are rows with a scale whose reciprocal is not safely a normal number.
// What bounds it is instruction issue as much as HBM (2 K bytes in, K / 2 out per row): 28672 x 8192 246 us with two
// passes over the row, 134 with the row and s in registers, every step on single floats and the products made twice,
// 123 now (4.8 TB/s); 4096 x 4096 14.0 -> 12.4.
template <int TH, int V>
__global__ void __launch_bounds__(TH)
pack_w4_kernel(const __half* __restrict__ W, const float* __restrict__ s, int N, int K,
               uint8_t* __restrict__ Wq, float* __restrict__ w_scale) {
    extern __shared__ float4 s_sm[];          // [K / 4]
    __shared__ float red[2][TH / 32];
    const int chunks = K / 8, tid = threadIdx.x;
    uint4 next[V];
    auto load = [&](int n) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int c = tid + v * TH;
            next[v] = make_uint4(0, 0, 0, 0);
            if (n < N && c < chunks) next[v] = __ldcs(reinterpret_cast<const uint4*>(W + (size_t)n * K) + c);
        }
    };
    load(blockIdx.x);
    // Up to two chunks per thread s stays in registers (one barrier and one trip through shared memory less, which counts
    // where a CTA has two rows: 1024 x 4096 6.5 -> 5.6 us), above that in shared memory (the two float4s of a chunk lie K / 8
    // apart: consecutive threads read consecutive ones).
    constexpr bool kKeepS = V <= 2;
    float4 kept[kKeepS ? V : 1][2];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int c = tid + v * TH;
        float4 s0 = make_float4(1.f, 1.f, 1.f, 1.f), s1 = s0;
        if (s && c < chunks) {
            s0 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c);
            s1 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c + 1);
        }
        if (kKeepS) { kept[kKeepS ? v : 0][0] = s0; kept[kKeepS ? v : 0][1] = s1; }
        else if (c < chunks) { s_sm[c] = s0; s_sm[chunks + c] = s1; }
    }
    if (!kKeepS) __syncthreads();
    int buf = 0;
    for (int n = blockIdx.x; n < N; n += gridDim.x, buf ^= 1) {
        float2 x[V][4];
        float amax = 0.f;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int c = tid + v * TH;
            float4 s0 = make_float4(1.f, 1.f, 1.f, 1.f), s1 = s0;
            if (kKeepS) { s0 = kept[kKeepS ? v : 0][0]; s1 = kept[kKeepS ? v : 0][1]; }
            else if (c < chunks) { s0 = s_sm[c]; s1 = s_sm[chunks + c]; }
            const float2 sv[4] = {make_float2(s0.x, s0.y), make_float2(s0.z, s0.w), make_float2(s1.x, s1.y), make_float2(s1.z, s1.w)};
            const __half2* h = reinterpret_cast<const __half2*>(&next[v]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                x[v][i] = __fmul2_rn(__half22float2(h[i]), sv[i]);          // s == NULL: times 1, exact
                amax = max3_abs(amax, x[v][i].x, x[v][i].y);
            }
        }
        load(n + gridDim.x);
        amax = warp_max(amax);
        if ((tid & 31) == 0) red[buf][tid >> 5] = amax;
        __syncthreads();
        amax = red[buf][0];
#pragma unroll
        for (int i = 1; i < TH / 32; ++i) amax = fmaxf(amax, red[buf][i]);
        const float sc = __fdiv_rn(amax, 7.0f);
        if (tid == 0) w_scale[n] = sc;
        const bool divide = !(sc > 1e-30f && sc < 1e30f);
        const float inv = __fdiv_rn(1.f, sc);
        const float2 inv2 = make_float2(inv, inv), m2 = make_float2(12582912.f, 12582912.f), neg1 = make_float2(-1.f, -1.f);
        uint32_t* out = reinterpret_cast<uint32_t*>(Wq + (size_t)n * (K / 2));
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int c = tid + v * TH;
            uint32_t u[8];
            float far = 0.f;                                                // largest distance to a code
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 su = __ffma2_rn(x[v][i], inv2, m2);
                const float2 d = __ffma2_rn(x[v][i], inv2, __ffma2_rn(su, neg1, m2));
                far = max3_abs_nan(far, d.x, d.y);
                u[2 * i] = __float_as_uint(su.x);
                u[2 * i + 1] = __float_as_uint(su.y);
            }
            uint32_t word = nibbles4(u[0], u[1], u[2], u[3]) | (nibbles4(u[4], u[5], u[6], u[7]) << 16);
            if (divide || !(far < 0.49999f)) {
                word = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float f = i & 1 ? x[v][i >> 1].y : x[v][i >> 1].x;
                    const int q = amax > 0.f ? rne_clamp(__fdiv_rn(f, sc), -8.f, 7.f) : 0;
                    word |= (uint32_t)(q & 0xF) << (4 * i);
                }
            }
            if (c < chunks) out[c] = word;
        }
    }
}

// The eight codes of a canonical word (column i in nibble i) to a word of the blocked layout (columns
// 0..3 in the low nibbles of its bytes, 4..7 in the high ones), and back.
__device__ __forceinline__ uint32_t spread_nibbles(uint32_t x) {
    x = (x | (x << 8)) & 0x00FF00FFu;
    return (x | (x << 4)) & 0x0F0F0F0Fu;
}
__device__ __forceinline__ uint32_t gather_nibbles(uint32_t x) {
    x = (x | (x >> 4)) & 0x00FF00FFu;
    return (x | (x >> 8)) & 0x0000FFFFu;
}
template <bool INVERSE>
__device__ __forceinline__ uint32_t reorder(uint32_t w) {
    if (INVERSE) return gather_nibbles(w & 0x0F0F0F0Fu) | (gather_nibbles((w >> 4) & 0x0F0F0F0Fu) << 16);
    return spread_nibbles(w & 0xFFFFu) | (spread_nibbles(w >> 16) << 4);
}

// Canonical [N, K/2] <-> blocked layout (see aser_common.cuh).  A CTA moves the 128 rows of up to
// kRepackBlocks adjacent column blocks in 16-byte pieces: four lanes take the 64 bytes of a row that
// one block covers, eight rows per warp, so both sides move whole 32-byte sectors (64 contiguous
// bytes on the canonical side, 128 on the blocked one) and a thread has eight pieces in flight.
// Rows >= N of the last block are zero codes.  28672 x 8192: 117 us with a 4-byte word per thread, 45 us now
// (5.2 TB/s).
constexpr int kRepackThreads = 256, kRepackBlocks = 4;
template <bool INVERSE>
__global__ void __launch_bounds__(kRepackThreads)
repack_w4_kernel(uint8_t* __restrict__ Wq, int N, int K, uint8_t* __restrict__ Wk) {
    const int kblocks = K / kWkCols, nb = blockIdx.x, kb0 = blockIdx.y * kRepackBlocks;
    const int sub = threadIdx.x & 3, r0 = threadIdx.x >> 2;       // 64 rows per round
    constexpr int kRounds = kWkRows * 4 / kRepackThreads;
    uint4 v[kRepackBlocks][kRounds];
#pragma unroll
    for (int b = 0; b < kRepackBlocks; ++b)
#pragma unroll
        for (int i = 0; i < kRounds; ++i) {
            const int kb = kb0 + b, row = r0 + i * (kRepackThreads / 4), n = nb * kWkRows + row;
            v[b][i] = make_uint4(0, 0, 0, 0);
            if (kb >= kblocks || n >= N) continue;
            const uint8_t* src = INVERSE
                ? Wk + ((size_t)nb * kblocks + kb) * kWkBlockBytes + sub * (kWkRows * 16) + row * 16
                : Wq + (size_t)n * (K / 2) + kb * (kWkCols / 2) + sub * 16;
            v[b][i] = __ldcs(reinterpret_cast<const uint4*>(src));
        }
#pragma unroll
    for (int b = 0; b < kRepackBlocks; ++b)
#pragma unroll
        for (int i = 0; i < kRounds; ++i) {
            const int kb = kb0 + b, row = r0 + i * (kRepackThreads / 4), n = nb * kWkRows + row;
            if (kb >= kblocks || (INVERSE && n >= N)) continue;
            const uint4 x = v[b][i];
            uint8_t* dst = INVERSE
                ? Wq + (size_t)n * (K / 2) + kb * (kWkCols / 2) + sub * 16
                : Wk + ((size_t)nb * kblocks + kb) * kWkBlockBytes + sub * (kWkRows * 16) + row * 16;
            *reinterpret_cast<uint4*>(dst) =
                make_uint4(reorder<INVERSE>(x.x), reorder<INVERSE>(x.y), reorder<INVERSE>(x.z), reorder<INVERSE>(x.w));
        }
}

template <int TH, int V>
int launch_pack_cfg(const __half* W, const float* s, int N, int K, uint8_t* Wq, float* w_scale, cudaStream_t st) {
    static int resident[kMaxDevices] = {0};       // CTAs that fit the device at once
    int dev = 0, sms = 0;
    int rc = current_device(&dev);
    if (rc == ASER_OK) rc = device_sm_count(&sms);
    if (rc != ASER_OK) return rc;
    if (resident[dev] == 0) {
        int per_sm = 0;
        const int most = V <= 2 ? 0 : TH * V * 32;       // for the longest rows of this configuration: shared memory holds s
        cudaError_t e = cudaFuncSetAttribute(pack_w4_kernel<TH, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pack_w4_kernel<TH, V>, TH, most);
        if (e != cudaSuccess || per_sm < 1) return record_cuda_error(e, "pack_w4 occupancy");
        resident[dev] = per_sm * sms;
    }
    const int grid = N < resident[dev] ? N : resident[dev];
    pack_w4_kernel<TH, V><<<grid, TH, V <= 2 ? 0 : (size_t)K * 4, st>>>(W, s, N, K, Wq, w_scale);
    return check_launch("pack_w4_kernel");
}

}  // namespace

// Threads per row by its length, four chunks per thread at most up to 16384 columns: fewer threads
// per row mean more rows in flight per SM, which is what hides the reduction (28672 x 8192: 135 us
// with 256 threads, 150 with 512; 8192 x 16384: 86 with 512, 98 with 1024).
int launch_pack_w4(const __half* W, const float* s, int N, int K, uint8_t* Wq, float* w_scale,
                   cudaStream_t st) {
    if (N == 0) return ASER_OK;
    const int per256 = (K / 8 + 255) / 256;
    if (per256 <= 1) return launch_pack_cfg<256, 1>(W, s, N, K, Wq, w_scale, st);
    if (per256 <= 2) return launch_pack_cfg<256, 2>(W, s, N, K, Wq, w_scale, st);
    if (per256 <= 3) return launch_pack_cfg<256, 3>(W, s, N, K, Wq, w_scale, st);
    if (per256 <= 4) return launch_pack_cfg<256, 4>(W, s, N, K, Wq, w_scale, st);
    if (per256 <= 6) return launch_pack_cfg<512, 3>(W, s, N, K, Wq, w_scale, st);
    if (per256 <= 8) return launch_pack_cfg<512, 4>(W, s, N, K, Wq, w_scale, st);
    if (per256 <= 12) return launch_pack_cfg<512, 6>(W, s, N, K, Wq, w_scale, st);
    return launch_pack_cfg<512, 8>(W, s, N, K, Wq, w_scale, st);
}

// `inverse` false: reads Wq, writes Wk.  true: reads Wk, writes Wq.
int launch_repack_w4(const uint8_t* Wq, int N, int K, uint8_t* Wk, bool inverse, cudaStream_t st) {
    if (N == 0) return ASER_OK;
    const int kblocks = K / kWkCols, nblocks = (N + kWkRows - 1) / kWkRows;
    const dim3 grid(nblocks, (kblocks + kRepackBlocks - 1) / kRepackBlocks);
    if (inverse) repack_w4_kernel<true><<<grid, kRepackThreads, 0, st>>>(const_cast<uint8_t*>(Wq), N, K, Wk);
    else repack_w4_kernel<false><<<grid, kRepackThreads, 0, st>>>(const_cast<uint8_t*>(Wq), N, K, Wk);
    return check_launch("repack_w4_kernel");
}

}  // namespace aser
