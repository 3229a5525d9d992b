// Offline weight path: smoothing multiply, per-output-channel int4 round-to-nearest,
// nibble packing (Sec. 4.2 Eq. 10/12 Q(W_s); Sec. 5.1 per-channel RTN), plus the
// permutation between the canonical packed form and the tensor-core kernel's layout.
#include "aser_common.cuh"

namespace aser {

namespace {

// A CTA quantizes whole rows, one after the other; thread t keeps the chunks t, t + TH, ... of a row
// and their smoothing factors in registers, so W is read once and s once per CTA.  The next row is
// loaded before the current one is reduced.  Codes: v * (1 / scale) is within 4e-6 of the quotient
// (|quotient| <= 7), so its rounding is that of the IEEE quotient unless it lies within 1e-5 of a
// tie; such chunks (one in ten thousand) are divided, as are rows with a scale whose reciprocal is
// not safely a normal number.
// HBM-bound by design: 2 K bytes in, K / 2 out per row.  28672 x 8192: 246 us with two passes over
// the row, both multiplying by s from L1 and one dividing every element; 135 us now (4.3 TB/s).
template <int TH, int V>
__global__ void __launch_bounds__(TH)
pack_w4_kernel(const __half* __restrict__ W, const float* __restrict__ s, int N, int K,
               uint8_t* __restrict__ Wq, float* __restrict__ w_scale) {
    __shared__ float red[2][TH / 32];
    const int chunks = K / 8, tid = threadIdx.x;
    constexpr bool kKeepS = V <= 4;           // else (rows above 16384) s is read again, from L1
    float kept[kKeepS ? V : 1][8];
    auto load_s = [&](int v, float (&f)[8]) {
        const int c = tid + v * TH;
#pragma unroll
        for (int i = 0; i < 8; ++i) f[i] = 1.f;
        if (s && c < chunks) {
            const float4 s0 = __ldg(reinterpret_cast<const float4*>(s + c * 8)), s1 = __ldg(reinterpret_cast<const float4*>(s + c * 8 + 4));
            f[0] = s0.x; f[1] = s0.y; f[2] = s0.z; f[3] = s0.w;
            f[4] = s1.x; f[5] = s1.y; f[6] = s1.z; f[7] = s1.w;
        }
    };
    if constexpr (kKeepS) {
#pragma unroll
        for (int v = 0; v < V; ++v) load_s(v, kept[v]);
    }
    auto get_s = [&](int v, float (&f)[8]) {
        if (!kKeepS) { load_s(v, f); return; }
#pragma unroll
        for (int i = 0; i < 8; ++i) f[i] = kept[kKeepS ? v : 0][i];
    };
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
    int buf = 0;
    for (int n = blockIdx.x; n < N; n += gridDim.x, buf ^= 1) {
        uint4 raw[V];
        float amax = 0.f;
#pragma unroll
        for (int v = 0; v < V; ++v) raw[v] = next[v];
        load(n + gridDim.x);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const __half2* h = reinterpret_cast<const __half2*>(&raw[v]);
            float sv[8];
            get_s(v, sv);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 w = __half22float2(h[i]);          // s == NULL: times 1, exact
                amax = fmaxf(amax, fmaxf(fabsf(__fmul_rn(w.x, sv[2 * i])), fabsf(__fmul_rn(w.y, sv[2 * i + 1]))));
            }
        }
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
        uint32_t* out = reinterpret_cast<uint32_t*>(Wq + (size_t)n * (K / 2));
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int c = tid + v * TH;
            const __half2* h = reinterpret_cast<const __half2*>(&raw[v]);
            float sv[8];
            get_s(v, sv);
            constexpr float kMagic = 12582912.f;                // 1.5 * 2^23: rounds to an integer in the low bits
            uint32_t word = 0;
            bool near = true;                                   // every element within 0.49999 of its code (false for NaN)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 w = __half22float2(h[i]);
                const float a = __fmul_rn(__fmul_rn(w.x, sv[2 * i]), inv), b = __fmul_rn(__fmul_rn(w.y, sv[2 * i + 1]), inv);
                const float ra = __fadd_rn(a, kMagic), rb = __fadd_rn(b, kMagic);
                near = near && fabsf(a - __fsub_rn(ra, kMagic)) < 0.49999f && fabsf(b - __fsub_rn(rb, kMagic)) < 0.49999f;
                word |= (__float_as_uint(ra) & 0xFu) << (8 * i);         // column 2j -> low nibble of byte j
                word |= (__float_as_uint(rb) & 0xFu) << (8 * i + 4);
            }
            if (divide || !near) {
                word = 0;
                const __half* e = reinterpret_cast<const __half*>(&raw[v]);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float x = __fmul_rn(__half2float(e[i]), sv[i]);
                    const int q = amax > 0.f ? rne_clamp(__fdiv_rn(x, sc), -8.f, 7.f) : 0;
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
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pack_w4_kernel<TH, V>, TH, 0);
        if (e != cudaSuccess || per_sm < 1) return record_cuda_error(e, "pack_w4 occupancy");
        resident[dev] = per_sm * sms;
    }
    const int grid = N < resident[dev] ? N : resident[dev];
    pack_w4_kernel<TH, V><<<grid, TH, 0, st>>>(W, s, N, K, Wq, w_scale);
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
