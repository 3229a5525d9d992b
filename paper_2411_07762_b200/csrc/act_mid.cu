// Activation step of 33 to a few hundred tokens in one launch without scratch memory (Sec. 4.2 smoothing, Sec. 5.1
// per-token round-to-nearest, Sec. 4.1 projection T = X~ L_A^T).
//
// At these sizes neither bytes nor products take long (101 x 8192: 2.5 MB, under 1 us of either); what bounds the step
// is its longest chain of dependent steps.  The codes need nothing of T and T nothing of the codes, so they are made
// by different CTAs of one grid, each with the shortest chain there is:
//  * a quantizing CTA takes whole rows into registers (quantize_rows): one round trip, a maximum, the codes;
//  * a projecting cluster takes 32 tokens x 32 rows of L_A, its CTAs' warps 64 columns of K at a time.  mma.sync m16n8k16:
//    an inner product does not care about the order of k, so a thread's k positions are the 8 columns that one 16-byte
//    load brings, the same for X and L_A, and neither goes through shared memory.  X is divided where the divisor is
//    not 1 (fp32, then fp16, as in the other kernels).  The warps' sums meet in shared memory, the CTAs' in distributed
//    shared memory, both in a fixed order; the order depends on K alone, not on the number of tokens.
#include "act_math.cuh"
#include "aser_common.cuh"
#include "sm100_ptx.cuh"

namespace aser {

namespace {

constexpr int kMThreads = 256, kMWarps = kMThreads / 32;
constexpr int kMTok = 32, kMRank = 32;              // tile of a projecting cluster
constexpr int kMAcc = kMTok * kMRank / 32;          // sums per thread

__device__ __forceinline__ void mid_mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Grid: t_tiles * CL projecting CTAs (clusters of CL along K), then the quantizing CTAs, R rows each.
// A sum (register 4 (4 mt + nt) + e of lane 4 g + t) is token 16 mt + g + 8 (e / 2), L_A row 8 nt + 2 t + e % 2.
template <int CPT, int R>
__global__ void __launch_bounds__(kMThreads, 2)
quant_act_mid_kernel(const __half* __restrict__ X, const float* __restrict__ s, const __half* __restrict__ LA, int M, int K,
                     int r, int t_tiles, int CL, int8_t* __restrict__ Xq, float* __restrict__ a_scale,
                     __nv_bfloat16* __restrict__ T, int ldt, int lo_off, float qmax) {
    // As in the few-token kernel: the wait comes first, dependents may start once everything before this kernel is done.
    grid_dep_wait();
    grid_dep_launch();
    __shared__ union {
        RowsShared<R> rows;
        float red[kMWarps][kMAcc][32];
    } sh;
    __shared__ float part[kMAcc][32];
    if ((int)blockIdx.x >= t_tiles * CL) {
        const int row0 = ((int)blockIdx.x - t_tiles * CL) * R, nrows = M - row0 < R ? M - row0 : R;
        if (nrows > 0)
            quantize_rows<CPT, R>(X + (size_t)row0 * K, s, nrows, K, Xq + (size_t)row0 * K, a_scale + row0, qmax, sh.rows);
        return;         // clusters take one role or the other, so no peer waits for this CTA
    }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int tile = (int)blockIdx.x / CL, rank = (int)blockIdx.x % CL;
    const int j_tiles = (r + kMRank - 1) / kMRank, j0 = tile % j_tiles * kMRank, m0 = tile / j_tiles * kMTok;
    float acc[2][4][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[mt][nt][e] = 0.f;
    const __half* xp[4];
    const __half* lp[4];
    bool x_ok[4], l_ok[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {           // token rows g + 8 i, L_A rows g + 8 i
        x_ok[i] = m0 + g + 8 * i < M;
        l_ok[i] = j0 + g + 8 * i < r;
        xp[i] = X + (size_t)(x_ok[i] ? m0 + g + 8 * i : 0) * K + t * 8;
        lp[i] = LA + (size_t)(l_ok[i] ? j0 + g + 8 * i : 0) * K + t * 8;
    }
    for (int u = rank * kMWarps + warp; u < K / 64; u += CL * kMWarps) {
        uint4 xv[2][4], lv[2][4];
        float4 s0[2], s1[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = u * 64 + h * 32;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                xv[h][i] = x_ok[i] ? *reinterpret_cast<const uint4*>(xp[i] + c) : make_uint4(0, 0, 0, 0);
                lv[h][i] = l_ok[i] ? __ldg(reinterpret_cast<const uint4*>(lp[i] + c)) : make_uint4(0, 0, 0, 0);
            }
            s0[h] = s1[h] = make_float4(1.f, 1.f, 1.f, 1.f);
            if (s) {
                s0[h] = __ldg(reinterpret_cast<const float4*>(s + c + t * 8));
                s1[h] = __ldg(reinterpret_cast<const float4*>(s + c + t * 8) + 1);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float sv[8] = {s0[h].x, s0[h].y, s0[h].z, s0[h].w, s1[h].x, s1[h].y, s1[h].z, s1[h].w};
            uint32_t xw[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { xw[i][0] = xv[h][i].x; xw[i][1] = xv[h][i].y; xw[i][2] = xv[h][i].z; xw[i][3] = xv[h][i].w; }
            bool ones = true;
#pragma unroll
            for (int e = 0; e < 8; ++e) ones = ones && sv[e] == 1.f;
            if (!ones) {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    if (sv[e] == 1.f) continue;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t word = xw[i][e >> 1];
                        const __half hv = __ushort_as_half((unsigned short)((e & 1) ? (word >> 16) : (word & 0xffffu)));
                        const uint32_t hb = (uint32_t)__half_as_ushort(__float2half_rn(__fdiv_rn(__half2float(hv), sv[e])));
                        xw[i][e >> 1] = (e & 1) ? ((word & 0x0000ffffu) | (hb << 16)) : ((word & 0xffff0000u) | hb);
                    }
                }
            }
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                const uint4 l = lv[h][nt];
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    mid_mma(acc[mt][nt], xw[2 * mt][0], xw[2 * mt + 1][0], xw[2 * mt][1], xw[2 * mt + 1][1], l.x, l.y);
                    mid_mma(acc[mt][nt], xw[2 * mt][2], xw[2 * mt + 1][2], xw[2 * mt][3], xw[2 * mt + 1][3], l.z, l.w);
                }
            }
        }
    }
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) sh.red[warp][(mt * 4 + nt) * 4 + e][lane] = acc[mt][nt][e];
    __syncthreads();
    for (int i = tid; i < kMAcc * 32; i += kMThreads) {
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < kMWarps; ++w) v += sh.red[w][i >> 5][i & 31];
        part[i >> 5][i & 31] = v;
    }
    if (CL > 1) { cluster_arrive(); cluster_wait(); }
    else __syncthreads();
    const int per = kMAcc * 32 / CL;        // sums that this CTA finishes
    const uint32_t mine = smem_u32(&part[0][0]);
    for (int i = rank * per + tid; i < (rank + 1) * per; i += kMThreads) {
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = q < CL ? (CL > 1 ? ld_cluster_f32(map_to_rank(mine + 4u * i, q)) : part[i >> 5][i & 31]) : 0.f;
        float sum = v[0];
#pragma unroll
        for (int q = 1; q < 8; ++q) sum += v[q];
        const int reg = i >> 5, ln = i & 31;
        const int m = m0 + (reg >> 4) * 16 + (ln >> 2) + 8 * ((reg >> 1) & 1), j = j0 + ((reg >> 2) & 3) * 8 + (ln & 3) * 2 + (reg & 1);
        if (m < M && j < r) store_t(T + (size_t)m * ldt, j, sum, lo_off);
    }
    if (CL > 1) { cluster_arrive(); cluster_wait(); }       // nobody leaves while a peer may still read its sums
}

// CTAs of a projecting cluster: 64 columns for every warp, where K has them.
int mid_cluster(int K) { return K >= 4096 ? 8 : K >= 2048 ? 4 : K >= 1024 ? 2 : 1; }

template <typename Kernel>
int launch_mid_cfg(Kernel* kernel, int R, const __half* X, const float* s, const __half* LA, int M, int K, int r, int8_t* Xq,
                   float* a_scale, __nv_bfloat16* T, int ldt, int lo_off, float qmax, cudaStream_t st) {
    const int CL = mid_cluster(K);
    const int t_tiles = (M + kMTok - 1) / kMTok * ((r + kMRank - 1) / kMRank), rows = (M + R - 1) / R;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(t_tiles * CL + (rows + CL - 1) / CL * CL, 1, 1);
    cfg.blockDim = dim3(kMThreads, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = CL; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, X, s, LA, M, K, r, t_tiles, CL, Xq, a_scale, T,
                                             ldt, lo_off, qmax);
    if (e != cudaSuccess) return record_cuda_error(e, "quant_act_mid_kernel");
    return check_launch("quant_act_mid_kernel");
}

}  // namespace

namespace {
// Rows of a quantizing CTA: one while the rows are few (the shortest chain), more where they would be several waves of CTAs
// (1000 x 1024, rank 32, us with one / two / four: 9.8 / 8.3 / 7.2; 333 x 8192: 11.7 / 9.0), as far as registers go.
int mid_rows(int M, int K) { return K > 8192 || M <= 128 ? 1 : M > 512 && K <= 2048 ? 4 : 2; }
}  // namespace

// The CTAs of this kernel are short and two are resident on an SM; the cluster kernel's step hardly depends on the
// number of tokens until its clusters no longer fit at once.  Measured, this kernel | the cluster kernel, us: rank 32: 64 x 4096 4.5 |
// 9.7, 448 x 4096 (336 CTAs) 9.2 | 10.2, 101 x 8192 7.7 | 12.7, 333 x 8192 (254) 9.0 | 13.1, 448 x 8192 (336) 14.3 | 13.0, 333 x 14336
// (421) 17.5 | 17.8; rank 128: 200 x 4096 (324) 10.0 | 10.8, 333 x 4096 (518) 12.2 | 10.9, 200 x 8192 (324) 14.1 | 16.1, 333 x 8192 (518)
// 17.0 | 16.4, 200 x 14336 (424) 19.2 | 23.3; short rows: 1000 x 1024, rank 128 (506, four rows each) 10.0 | 10.1, rank 32 (314) 7.2 |
// 9.5, 448 x 2048, rank 128 (448) 9.0 | 9.6, 1000 x 3072, rank 32 (628) 12.1 | 15.0, rank 128 (1012) 21.1 | 17.7.
bool quant_act_mid_prefers(int M, int K, int r) {
    const int rows = mid_rows(M, K);
    const int ctas = (M + rows - 1) / rows + mid_cluster(K) * ((M + kMTok - 1) / kMTok) * ((r + kMRank - 1) / kMRank);
    return ctas <= (rows == 4 ? 450 : K < 4096 ? 630 : K <= 8192 ? 340 : 424);
}

int launch_quant_act_mid(const __half* X, const float* s, const __half* LA, int M, int K, int r, int8_t* Xq, float* a_scale,
                         __nv_bfloat16* T, int ldt, int lo_off, float qmax, cudaStream_t st) {
    // chunks of eight columns per thread by the row length, one, two or four rows per quantizing CTA
    const int chunks = (K / 8 + kMThreads - 1) / kMThreads, rows = mid_rows(M, K);
    auto go = [&](auto* kernel) { return launch_mid_cfg(kernel, rows, X, s, LA, M, K, r, Xq, a_scale, T, ldt, lo_off, qmax, st); };
    if (rows == 4) return go(quant_act_mid_kernel<1, 4>);        // up to 2048 columns
    if (chunks <= 1) return rows == 2 ? go(quant_act_mid_kernel<1, 2>) : go(quant_act_mid_kernel<1, 1>);
    if (chunks <= 2) return rows == 2 ? go(quant_act_mid_kernel<2, 2>) : go(quant_act_mid_kernel<2, 1>);
    if (chunks <= 4) return rows == 2 ? go(quant_act_mid_kernel<4, 2>) : go(quant_act_mid_kernel<4, 1>);
    if (chunks <= 8) return go(quant_act_mid_kernel<8, 1>);
    return go(quant_act_mid_kernel<16, 1>);
}

}  // namespace aser
