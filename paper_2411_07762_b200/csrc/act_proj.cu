// Activation path for many tokens when the caller provides scratch memory: two kernels.
//
//   act_proj_kernel    T.  A CTA owns 128 tokens and one slice of K; TMA streams the slice of X
//                      through a shared-memory ring together with the matching columns of L_A.  The consumer
//                      warps write x / s back as fp16 where s != 1, one thread issues tcgen05.mma
//                      (kind::f16) with L_A on the M side (up to four groups of 128 rows, so the
//                      down projections of several layers that share X are computed in one pass)
//                      and the 128 tokens on the N side.  The slices' partial T are summed in order and rounded to bf16.
//   act_rows_kernel    up to 8192 columns (see below), and without a projection (then it is the only kernel): scales and codes of
//                      whole rows, beside act_proj_kernel.
//   act_quant_kernel   otherwise: the scale from row maxima that act_proj_kernel left in the scratch, the codes, and T
//                      from the partial T beside them.
//
// Which of the two (beside_from): running beside each other the kernels take little more than the longer one while X, which both
// read, comes from L2 for the second; they move X twice and L_A once per 128 tokens to the SMs, at 4.5 TB/s (each alone, cold,
// has L2 15 % and HBM 20 % busy: latency of the loads in flight).  Rows of more than 8192 columns exceed L2 at a few thousand tokens and both streams come from
// HBM; many rows of L_A at 8192 columns are bound by their own traffic already.  Few tokens: beside, a tile has at most eight
// slices of K, so with few tiles the projection is the longer chain the more rows of L_A there are.  The activation step, us, beside |
// after each other: rank 128: 33 x 4096 12.4 | 11.9, 64 x 4096 12.3 | 12.5, 600 x 4096 12.7 | 14.1, 4096 x 4096 24.3 | 28.9, 33 x 3072 11.0 |
// 12.3, 64 x 6144 14.8 | 13.9, 128 x 6144 14.0 | 14.8; rank 64: 300 x 8192 16.7 | 16.6, 449 x 8192 16.6 | 17.3, 4096 x 8192 45.8 | 46.7; rank 128:
// 1500 x 14336 46 | 41, 4096 x 14336 100 | 85; rank 256: 64 x 4096 17.3 | 15.5, 449 x 4096 17.8 | 17.0, 800 x 4096 18.7 | 19.3, 4096 x 4096 30.6 |
// 36.7, 100 x 2048 14.2 | 14.2, 600 x 2048 14.9 | 15.4, 600 x 8192 28.2 | 22.2; rank 384: 64 x 4096 22.3 | 17.6, 800 x 4096 24.1 | 22.8, 1600 x 4096 26.4 |
// 26.4, 4096 x 4096 36.8 | 43.3, 600 x 2048 19.7 | 18.2, 300 x 512 17.8 | 18.0, 200 x 3584 22.0 | 23.9.  (Rank 512 would gain from 2500 tokens on.)
//
// (Sec. 4.2 smoothing M^-1 X of Eq. 10, Sec. 5.1 per-token round-to-nearest, Sec. 4.1 projection
// V_r^T S^-1 of the reconstruction branch.)  All kernels are deterministic: no atomics on global memory.
// Every mbarrier wait is bounded; a CTA that gives up makes its tokens' partial T, and row maxima, NaN.
#include "act_math.cuh"
#include "aser_common.cuh"
#include "sm100_ptx.cuh"

namespace aser {

namespace {

constexpr int kPTok = 128;                  // tokens per CTA (the MMA's N)
constexpr int kPCols = 64;                  // columns per stage: one 128-byte swizzled tile row
constexpr int kPConsumerWarps = 8;
constexpr int kPWarpLa = 2 + kPConsumerWarps;           // producer of the L_A tiles
constexpr int kPThreads = (3 + kPConsumerWarps) * 32;   // X producer, MMA issuer, consumers, L_A producer
constexpr int kPTileBytes = kPTok * 128;    // 128 rows x 64 fp16 (an X tile or one L_A group tile)
constexpr int kPMaxGroups = 4;              // 128-row groups of L_A: r <= 512
constexpr int kProjPlanSms = 148;           // chunks and slices are planned for this many SMs (the
                                            // scratch size must not depend on the device)
constexpr long long kPWaitLimitClocks = 400000000ll;   // about 0.2 s of SM clocks per wait
// Tokens from which the kernels run beside each other (see above).
constexpr int kNever = 0x7fffffff;
constexpr int beside_from(int K, int r) {
    if (K > 8192 || r > 384) return kNever;
    if (K > 4096) return r > 128 ? kNever : K < 8192 ? 100 : 400;
    if (r <= 128) return K < 4096 ? 0 : 64;
    if (r <= 256) return K <= 3584 ? 100 : 600;
    return K < 1024 || (K > 2048 && K <= 3584) ? 100 : 1600;
}
constexpr bool rows_beside(int M, int K, int r) { return M >= beside_from(K, r); }
constexpr int kPMaxCluster = 8;             // CTAs of a cluster
constexpr int kPCacheUnits = 254;           // 8-column units with a divisor whose divisors are kept in shared memory
constexpr int kPUncached = 255;             // tag of such a unit beyond the cache: its divisors are read from global memory

// Stages of the ring.  Beside act_rows_kernel they leave room on the SM for two CTAs of act_rows_kernel (K bytes of mask, 4.2
// KB, and a KB per resident CTA); at least the 128 KB that later stage the partial T.
__host__ __device__ constexpr int proj_stages(int groups, int K, bool beside) {
    const int per_stage = kPTileBytes * (1 + groups);
    int ns = (beside ? 213 * 1024 - 2 * (K + 5300) : 208 * 1024) / per_stage;
    const int least = (131072 + per_stage - 1) / per_stage;
    ns = ns < least ? least : ns;
    return ns > 8 ? 8 : ns;                 // 6, 4, 3, 2 stages for 1..4 groups; 5 beside rows of 8192 columns (one group)
}

__device__ __noinline__ bool pj_wait_slow(uint32_t bar, uint32_t parity, volatile int* flag) {
    uint32_t spins = 0;
    long long t0 = 0;
    while (!mbar_try_wait(bar, parity)) {
        if ((++spins & 255u) == 0) {
            if (*flag) return false;
            if (t0 == 0) {
                t0 = clock64();
            } else if (clock64() - t0 > kPWaitLimitClocks) {
                *flag = 1;
                return false;
            }
        }
    }
    return true;
}
__device__ __forceinline__ bool pj_wait(uint32_t bar, uint32_t parity, volatile int* flag) {
    if (mbar_try_wait(bar, parity)) return true;
    return pj_wait_slow(bar, parity, flag);
}
__device__ __forceinline__ bool pj_warp_wait(uint32_t bar, uint32_t parity, volatile int* flag, int lane) {
    int ok = 1;
    if (lane == 0) ok = pj_wait(bar, parity, flag) ? 1 : 0;
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}
__device__ __forceinline__ uint4 pj_lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void pj_sts128(uint32_t addr, uint4 v) {
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// A group's partial sums, tensor memory -> `buf` as [token][128 rows of the group].  A warp reaches the 32 lanes (rows j) of
// its quarter, warp % 4; the two warps of a quarter take 64 tokens each.  gave_up: NaN instead.
__device__ __forceinline__ void pj_stage_t(uint32_t tmem, int g, uint32_t buf, int cw, int warp, int lane, bool gave_up) {
    const int q = warp & 3, half = cw >> 2;
#pragma unroll 1
    for (int c0 = half * 64; c0 < half * 64 + 64; c0 += 16) {
        uint32_t v[16];
        tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(g * 128 + c0), v);
        tmem_wait_ld(v);
#pragma unroll
        for (int e = 0; e < 16; ++e)
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(buf + (uint32_t)(c0 + e) * 512u + (uint32_t)(q * 32 + lane) * 4u), "r"(gave_up ? 0x7fc00000u : v[e]) : "memory");
    }
}

// grid = (KS slices, token tiles).
// MAXIMA: the row maxima of |x~| over the slice and the partial T go to the scratch,
//   amax_part [KS][M]               fp32 (NaN: the CTA gave up)
//   t_part    [KS][groups][M][128]  fp32, by 128-row group of L_A (rows past r: unspecified; NaN: the CTA gave up)
// otherwise the slices of a tile are a cluster that sums the partial T through distributed shared memory and writes T.
// map_x: X as fp16 [K / 64 blocks][M][64], box 1 block x 128 rows, 128-byte swizzle (rows past
// M read as zero).  map_la: L_A as fp16 [K / 64 blocks][r][64], box 1 block x r rows (r / 2 rows
// above 256).
template <bool MAXIMA>
__global__ void __launch_bounds__(kPThreads, 1)
act_proj_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_la,
                const float* __restrict__ s, int M, int K, int r, float* __restrict__ amax_part,
                float* __restrict__ t_part, __nv_bfloat16* __restrict__ T, int ldt, int lo_off) {
    // The r rows of L_A arrive as one box (r <= 256, the largest box) or as two boxes of r / 2
    // rows; in shared memory the rows follow one another, 128 bytes each, so group g is the 16 KB
    // at g * 16 KB whatever the boxes.  Where r is not a multiple of 128 the last group's MMA also
    // reads the stale rows behind row r; their accumulator rows are never read.
    const int la_boxes = r <= 256 ? 1 : 2;
    const int la_box_rows = r / la_boxes;
    const uint32_t la_stage_bytes = (uint32_t)r * 128u;
    extern __shared__ uint8_t smem_raw[];
    // A programmatic dependent of whatever precedes it.  The signal must stay behind the wait: act_quant_kernel reads X
    // and s, and the linear kernel after it the weights, before waits of their own, which is sound because neither
    // starts until everything before this kernel is done.
    grid_dep_wait();
    grid_dep_launch();
    const uint32_t sraw = smem_u32(smem_raw);
    const uint32_t sb = (sraw + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (sb - sraw);
    const int groups = (r + 127) / 128;
    const int NS = proj_stages(groups, K, !MAXIMA);
    const int stage_bytes = kPTileBytes * (1 + groups);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ks = blockIdx.x, tile = blockIdx.y;
    const int blk0 = K / kPCols * ks / (int)gridDim.x, nst = K / kPCols * (ks + 1) / (int)gridDim.x - blk0;    // the slice
    const int k0 = blk0 * kPCols, Kc = nst * kPCols;
    const int row0 = tile * kPTok;                  // first token of the tile inside the chunk
    // after the ring: barriers, flags, the per-warp row maxima
    uint8_t* tail = smem + NS * stage_bytes;
    const uint32_t bars = sb + NS * stage_bytes;
    auto bar_full = [&](int st) { return bars + st * 8; };
    auto bar_ready = [&](int st) { return bars + (8 + st) * 8; };
    auto bar_free = [&](int st) { return bars + (16 + st) * 8; };
    const uint32_t bar_acc = bars + 24 * 8;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tail + 25 * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 25 * 8 + 8);
    volatile int* never_flag = abort_flag + 1;                      // stays 0: waits of the wind-down
    // per 8 columns of the slice: 0 = all divisors are 1, else 1 + the unit's place in s_cache (or kPUncached)
    uint8_t* unit_tag = tail + 256;
    float* s_cache = reinterpret_cast<float*>(tail + 256 + ((Kc / 8 + 15) & ~15));  // [kPCacheUnits][8] divisors
    float* amax_w = s_cache + kPCacheUnits * 8;                     // MAXIMA: [8 warps][128 rows]
    int* n_cached = reinterpret_cast<int*>(tail + 25 * 8 + 16);
    const uint32_t tmem_cols = groups <= 1 ? 128u : groups == 2 ? 256u : 512u;

    if (warp == 0) {
        if (lane == 0) {
            for (int st = 0; st < 8; ++st) {
                mbar_init(bar_full(st), 2);                  // the X producer and the L_A producer
                mbar_init(bar_ready(st), kPConsumerWarps);
                mbar_init(bar_free(st), 1);
            }
            mbar_init(bar_acc, 1);
            *abort_flag = 0;
            *never_flag = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            fence_proxy_async_smem();
            prefetch_tensormap(&map_x);
            prefetch_tensormap(&map_la);
            // The first round of the ring is requested before the other warps are ready: it needs
            // only the barriers set up above.
            for (int i = 0; i < NS && i < nst; ++i) {
                mbar_arrive_expect_tx(bar_full(i), (uint32_t)kPTileBytes);
                tma_load_3d(sb + i * stage_bytes, &map_x, 0, row0, (k0 + i * kPCols) / kPCols, bar_full(i));
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else if (warp < kPWarpLa) {
        // The smoothing divisors are 1 on all but the few outlier channels.  A unit that has one
        // keeps its eight divisors in shared memory, so that the streaming loop below never waits
        // for global memory.
        if (tid == 64) *n_cached = 0;
        named_bar_sync(1, kPConsumerWarps * 32);
        for (int g = tid - 64; g < Kc / 8; g += kPConsumerWarps * 32) {
            int tag = 0;
            if (s) {
                const float4 a = __ldg(reinterpret_cast<const float4*>(s + k0 + g * 8));
                const float4 b = __ldg(reinterpret_cast<const float4*>(s + k0 + g * 8) + 1);
                const bool one = a.x == 1.f && a.y == 1.f && a.z == 1.f && a.w == 1.f &&
                                 b.x == 1.f && b.y == 1.f && b.z == 1.f && b.w == 1.f;
                if (!one) {
                    const int at = atomicAdd(n_cached, 1);
                    tag = kPUncached;
                    if (at < kPCacheUnits) {
                        tag = at + 1;
                        *reinterpret_cast<float4*>(s_cache + at * 8) = a;
                        *reinterpret_cast<float4*>(s_cache + at * 8 + 4) = b;
                    }
                }
            }
            unit_tag[g] = (uint8_t)tag;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ================= TMA producer =================
        if (lane == 0) {
            bool ok = true;
            int issued = (NS < nst) ? NS : nst;
            for (int i = issued; i < nst && ok; ++i) {
                const int st = i % NS;
                ok = pj_wait(bar_free(st), (uint32_t)(i / NS - 1) & 1u, abort_flag);
                if (!ok) break;
                const uint32_t dst = sb + st * stage_bytes;
                const int kblk = (k0 + i * kPCols) / kPCols;
                mbar_arrive_expect_tx(bar_full(st), (uint32_t)kPTileBytes);
                tma_load_3d(dst, &map_x, 0, row0, kblk, bar_full(st));
                ++issued;
            }
            if (*abort_flag) {      // let copies already issued land before the shared memory goes away
                for (int i = (issued > NS ? issued - NS : 0); i < issued; ++i)
                    pj_wait(bar_full(i % NS), (uint32_t)(i / NS) & 1u, never_flag);
            }
        }
    } else if (warp == kPWarpLa) {
        // ================= L_A producer: one box of up to 256 rows (two groups) per copy =================
        if (lane == 0) {
            bool ok = true;
            int issued = 0;
            for (int i = 0; i < nst && ok; ++i) {
                const int st = i % NS;
                if (i >= NS) ok = pj_wait(bar_free(st), (uint32_t)(i / NS - 1) & 1u, abort_flag);
                if (!ok) break;
                const uint32_t dst = sb + st * stage_bytes + kPTileBytes;
                const int kblk = (k0 + i * kPCols) / kPCols;
                mbar_arrive_expect_tx(bar_full(st), la_stage_bytes);
                for (int b = 0; b < la_boxes; ++b)
                    tma_load_3d(dst + b * la_box_rows * 128, &map_la, 0, b * la_box_rows, kblk, bar_full(st));
                ++issued;
            }
            if (*abort_flag) {
                for (int i = (issued > NS ? issued - NS : 0); i < issued; ++i)
                    pj_wait(bar_full(i % NS), (uint32_t)(i / NS) & 1u, never_flag);
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer =================
        if (lane == 0) {
            const uint32_t idesc = make_idesc(1u, 0u, 128u, (uint32_t)kPTok);
            bool ok = true;
            for (int i = 0; i < nst && ok; ++i) {
                const int st = i % NS;
                ok = pj_wait(bar_ready(st), (uint32_t)(i / NS) & 1u, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint64_t bdesc = smem_desc_sw128(sb + st * stage_bytes);
                for (int g = 0; g < groups; ++g) {
                    const uint64_t adesc = smem_desc_sw128(sb + st * stage_bytes + (1 + g) * kPTileBytes);
#pragma unroll
                    for (int kk = 0; kk < kPCols / 16; ++kk)
                        mma_f16_ss(tmem + g * 128, adesc + 2 * kk, bdesc + 2 * kk, idesc, (i != 0 || kk != 0) ? 1u : 0u);
                }
                tc_commit(bar_free(st));
            }
            tc_commit(bar_acc);     // arrives when every MMA issued above has completed
            if (!ok) pj_wait(bar_acc, 0u, never_flag);      // giving up: let them finish before leaving
        }
    } else if (warp < kPWarpLa) {
        // ================= consumers =================
        // Warp cw owns the 16-byte piece cw (8 columns) of every row; lane = rows lane, +32, +64, +96.
        const int cw = warp - 2;
        float amax[4] = {0.f, 0.f, 0.f, 0.f};
        __half2 hmax[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) hmax[q] = __float2half2_rn(0.f);
        bool ok = true;
        for (int i = 0; i < nst; ++i) {
            const int st = i % NS;
            ok = pj_warp_wait(bar_full(st), (uint32_t)(i / NS) & 1u, abort_flag, lane);
            if (!ok) break;
            const uint32_t base = sb + st * stage_bytes;
            const int tag = unit_tag[i * 8 + cw];
            if (MAXIMA || tag != 0) {
                uint32_t addr[4], wd[4][4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int row = lane + 32 * q;
                    addr[q] = base + (uint32_t)row * 128u + (uint32_t)((cw ^ (row & 7)) << 4);
                    const uint4 v = pj_lds128(addr[q]);
                    wd[q][0] = v.x; wd[q][1] = v.y; wd[q][2] = v.z; wd[q][3] = v.w;
                }
                uint32_t zd[4][4];              // without the divided columns: what the half-precision maximum sees
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int w = 0; w < 4; ++w) zd[q][w] = wd[q][w];
                if (tag != 0) {
                    const float4* sp = (tag != kPUncached) ? reinterpret_cast<const float4*>(s_cache + (tag - 1) * 8)
                                                           : reinterpret_cast<const float4*>(s + k0 + i * kPCols + cw * 8);
                    const float4 s0 = sp[0], s1 = sp[1];
                    const float sv[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
                    // Only the columns with a divisor (the same for every lane: lanes are rows) are divided and
                    // written back as fp16(x~); their maximum is taken in fp32.
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        if (sv[e] != 1.f) {
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const uint32_t word = wd[q][e >> 1];
                                const __half hv = __ushort_as_half((unsigned short)((e & 1) ? (word >> 16) : (word & 0xffffu)));
                                const float f = __fdiv_rn(__half2float(hv), sv[e]);
                                if (MAXIMA) amax[q] = fmaxf(amax[q], fabsf(f));
                                const uint32_t hb = (uint32_t)__half_as_ushort(__float2half_rn(f));
                                wd[q][e >> 1] = (e & 1) ? ((word & 0x0000ffffu) | (hb << 16)) : ((word & 0xffff0000u) | hb);
                                zd[q][e >> 1] &= (e & 1) ? 0x0000ffffu : 0xffff0000u;
                            }
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) pj_sts128(addr[q], make_uint4(wd[q][0], wd[q][1], wd[q][2], wd[q][3]));
                    fence_proxy_async_smem();       // the MMA reads these through the async proxy
                }
                if (MAXIMA) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int w = 0; w < 4; ++w)
                            hmax[q] = __hmax2(hmax[q], __habs2(*reinterpret_cast<const __half2*>(&zd[q][w])));
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_ready(st));
        }
        if (MAXIMA) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                amax_w[cw * kPTok + lane + 32 * q] = fmaxf(amax[q], fmaxf(__low2float(hmax[q]), __high2float(hmax[q])));
            named_bar_sync(1, kPConsumerWarps * 32);
            const int row = tid - 64;
            if (row < kPTok && row0 + row < M) {
                float a = amax_w[row];
#pragma unroll
                for (int w = 1; w < kPConsumerWarps; ++w) a = fmaxf(a, amax_w[w * kPTok + row]);
                if (*abort_flag) a = __int_as_float(0x7fc00000);        // not all columns were seen
                amax_part[(size_t)ks * M + row0 + row] = a;
            }
        }
        if (ok) ok = pj_warp_wait(bar_acc, 0u, abort_flag, lane);
        tc_fence_after();
        if (MAXIMA) {
            // ---- partial T: tensor memory -> shared memory as [token][128 rows of the group] -> one
            // bulk copy per group into the scratch, where a group's tile is contiguous.  The ring is idle by
            // now (every MMA has completed) and serves as two 64 KB staging buffers. ----
            const int rows_valid = (M - row0 < kPTok) ? (M - row0) : kPTok;
            for (int g = 0; g < groups; ++g) {
                const uint32_t buf = sb + (uint32_t)(g & 1) * 65536u;
                if (g >= 2) {               // the copy that last read this buffer must be done with it
                    if (tid == 64) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    named_bar_sync(1, kPConsumerWarps * 32);
                }
                pj_stage_t(tmem, g, buf, cw, warp, lane, false);
                fence_proxy_async_smem();
                named_bar_sync(1, kPConsumerWarps * 32);
                float* dst = t_part + (((size_t)ks * groups + g) * M + row0) * 128;
                if (*abort_flag) {          // a wait gave up: these tokens' T, and with it their outputs, become NaN
                    for (int e = tid - 64; e < rows_valid * 128; e += kPConsumerWarps * 32) dst[e] = __int_as_float(0x7fc00000);
                } else if (tid == 64) {
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                                 ::"l"(dst), "r"(buf), "r"((uint32_t)rows_valid * 512u) : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
            }
            if (tid == 64) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
            tc_fence_before();
        }
    }
    if (!MAXIMA) {
        // ---- T: every CTA of the cluster stages its partial sums of a group as [token][128 rows], then finishes its share
        // of the tokens from everybody's, in slice order.  (The ring is idle: every MMA of this CTA has completed.) ----
        __syncthreads();        // also the copies of a CTA that gave up have landed
        const int cw = warp - 2;
        const int share0 = kPTok * 32 * ks / (int)gridDim.x, share1 = kPTok * 32 * (ks + 1) / (int)gridDim.x;   // float4s of a group
        for (int g = 0; g < groups; ++g) {
            if (warp >= 2 && warp < kPWarpLa) pj_stage_t(tmem, g, sb, cw, warp, lane, *abort_flag != 0);
            cluster_arrive();
            cluster_wait();
            for (int e = share0 + tid; e < share1; e += kPThreads) {
                const int m = row0 + (e >> 5), j = g * 128 + (e & 31) * 4;
                if (m >= M || j >= r) continue;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
                for (int q0 = 0; q0 < (int)gridDim.x; q0 += 4) {        // four loads in flight (registers: see act_rows_kernel's)
                    float4 a[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        a[q] = q0 + q < (int)gridDim.x ? ld_cluster_f32x4(map_to_rank(sb + (uint32_t)e * 16u, (uint32_t)(q0 + q)))
                                                       : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int q = 0; q < 4; ++q) { v.x += a[q].x; v.y += a[q].y; v.z += a[q].z; v.w += a[q].w; }
                }
                store_t2(T + (size_t)m * ldt, j, v.x, v.y, lo_off);
                store_t2(T + (size_t)m * ldt, j + 2, v.z, v.w, lo_off);
            }
            cluster_arrive();           // nobody overwrites its sums, or leaves, while a peer may still read them
            cluster_wait();
        }
        tc_fence_before();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
    }
}

// Where the kernels run one after the other.  grid = ceil(M / kQRows), 256 threads; a CTA takes kQRows token rows, several
// 16-byte loads per thread are in flight, and the per-row scales are computed once per CTA (one
// warp per row).  The kernel is bound by instruction issue, not by bytes, so the common case is
// kept free of per-column work: the CTA first lists the columns whose divisor is not 1 (the few
// outlier channels); the main loop then treats every column as undivided, and the listed columns
// are redone afterwards, one (row, column) per thread, with both IEEE divisions.  A smoothing
// vector with more such columns than the list holds takes the general loop, which tests every
// group of eight divisors.
// Launched as a programmatic dependent of act_proj_kernel: the list and the first loads of X
// (inputs of the whole step, not products of that kernel; written before it started, see its signal) are
// done before the dependency wait.
constexpr int kQRows = 4;
__global__ void __launch_bounds__(256, 4)
act_quant_kernel(const __half* __restrict__ X, const float* __restrict__ s, int M, int K,
                 int r, int KS, const float* amax_part, const float* t_part,
                 int8_t* __restrict__ Xq, float* __restrict__ a_scale, __nv_bfloat16* __restrict__ T,
                 int ldt, int lo_off, float qmax) {
    __shared__ float sc_sm[kQRows], rcp_sm[kQRows];
    __shared__ int n_list;
    __shared__ int list_col[kRowsList];
    grid_dep_launch();      // a dependent linear kernel may start streaming its weights
    const int row0 = blockIdx.x * kQRows;
    const int nrows = (M - row0 < kQRows) ? (M - row0) : kQRows;
    const int chunks = K / 8;
    const int groups = (r + 127) / 128;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const __half* xbase = X + (size_t)(row0) * K;
    uint4 x[kQRows];
    int c = threadIdx.x;
    auto load_x = [&](int cc) {
#pragma unroll
        for (int rr = 0; rr < kQRows; ++rr)
            x[rr] = (rr < nrows && cc < chunks) ? *reinterpret_cast<const uint4*>(xbase + (size_t)rr * K + cc * 8)
                                                : make_uint4(0, 0, 0, 0);
    };
    load_x(c);
    // ---- columns with a divisor (any order; entries past the capacity are only counted) ----
    if (threadIdx.x == 0) n_list = 0;
    __syncthreads();
    if (s) {
        for (int g = threadIdx.x; g < K / 4; g += 256) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(s) + g);
            const float sv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (sv[e] != 1.f) {
                    const int at = atomicAdd(&n_list, 1);
                    if (at < kRowsList) list_col[at] = g * 4 + e;
                }
            }
        }
    }
    grid_dep_wait();        // the partial maxima and the partial T come from act_proj_kernel
    // ---- scales: warp w takes row w ----
    if (warp < nrows) {
        float v = (lane < KS) ? amax_part[(size_t)lane * M + row0 + warp] : 0.f;
        for (int ks = lane + 32; ks < KS; ks += 32) {
            const float u = amax_part[(size_t)ks * M + row0 + warp];
            v = (u != u || v != v) ? __int_as_float(0x7fc00000) : fmaxf(v, u);
        }
        const bool bad = __any_sync(0xffffffffu, v != v);
        float a = warp_max(v);
        if (bad) a = __int_as_float(0x7fc00000);
        if (lane == 0) {
            const float sc = __fdiv_rn(a, qmax);
            sc_sm[warp] = sc;
            rcp_sm[warp] = code_rcp(sc);
            a_scale[row0 + warp] = sc;
        }
    } else if (warp < kQRows && lane == 0) {
        sc_sm[warp] = 0.f;
        rcp_sm[warp] = 0.f;
    }
    // ---- T of these rows: the slices' partials summed in slice order ----
    for (int e = threadIdx.x; e < nrows * r; e += 256) {
        const int rr = e / r, j = e - rr * r;
        const float* tp = t_part + ((size_t)(j >> 7) * M + row0 + rr) * 128 + (j & 127);
        const size_t slice = (size_t)groups * M * 128;
        float t = 0.f;
        int ks = 0;
        for (; ks + 4 <= KS; ks += 4) {         // four loads in flight, summed in slice order
            const float a0 = tp[ks * slice], a1 = tp[(ks + 1) * slice];
            const float a2 = tp[(ks + 2) * slice], a3 = tp[(ks + 3) * slice];
            t += a0; t += a1; t += a2; t += a3;
        }
        for (; ks < KS; ++ks) t += tp[ks * slice];
        store_t(T + (size_t)(row0 + rr) * ldt, j, t, lo_off);
    }
    __syncthreads();
    const int listed = n_list;
    float scr[kQRows], rc1[kQRows];
#pragma unroll
    for (int rr = 0; rr < kQRows; ++rr) {
        scr[rr] = sc_sm[rr];
        rc1[rr] = rcp_sm[rr];
    }
    if (listed <= kRowsList) {
        // ---- codes, every column taken as undivided ----
        for (; c < chunks; c += 256) {
            uint2 q[kQRows];
#pragma unroll
            for (int rr = 0; rr < kQRows; ++rr) {
                q[rr] = codes8_unit(x[rr], scr[rr], rc1[rr], qmax);
                if (!(scr[rr] > 0.f)) q[rr] = make_uint2(0u, 0u);      // zero row, or a poisoned scale
            }
            load_x(c + 256);        // the next iteration's loads are in flight during the stores
#pragma unroll
            for (int rr = 0; rr < kQRows; ++rr)
                if (rr < nrows) *reinterpret_cast<uint2*>(Xq + (size_t)(row0 + rr) * K + c * 8) = q[rr];
        }
        // ---- the listed columns again, with their divisors ----
        __syncthreads();            // orders the stores above before the single bytes below
        for (int e = threadIdx.x; e < listed * kQRows; e += 256) {
            const int rr = e & (kQRows - 1), col = list_col[e / kQRows];
            if (rr >= nrows) continue;
            const float sc = sc_sm[rr];
            int code = 0;
            if (sc > 0.f) {
                const float xt = __fdiv_rn(__half2float(xbase[(size_t)rr * K + col]), __ldg(s + col));
                code = rne_clamp(__fdiv_rn(xt, sc), -qmax, qmax);
            }
            Xq[(size_t)(row0 + rr) * K + col] = (int8_t)code;
        }
        return;
    }
    // ---- general loop: many columns have a divisor ----
    for (; c < chunks; c += 256) {
        const float4 s0 = __ldg(reinterpret_cast<const float4*>(s + c * 8));
        const float4 s1 = __ldg(reinterpret_cast<const float4*>(s + c * 8) + 1);
        const float sv[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
        uint2 q[kQRows];
#pragma unroll
        for (int rr = 0; rr < kQRows; ++rr) {
            const __half* h = reinterpret_cast<const __half*>(&x[rr]);
            float f[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {       // x~ = x / s, IEEE division, only where the divisor is not 1
                f[e] = __half2float(h[e]);
                if (sv[e] != 1.f) f[e] = __fdiv_rn(f[e], sv[e]);
            }
            q[rr] = (scr[rr] > 0.f) ? quant8_pairs(f, scr[rr], rc1[rr], qmax) : make_uint2(0u, 0u);
        }
        load_x(c + 256);
#pragma unroll
        for (int rr = 0; rr < kQRows; ++rr)
            if (rr < nrows) *reinterpret_cast<uint2*>(Xq + (size_t)(row0 + rr) * K + c * 8) = q[rr];
    }
}

// The codes and scales need nothing from act_proj_kernel, so the two kernels run beside each other.  Without a projection
// it is the only kernel of the pass and waits for what precedes it first.
//
// A row belongs to W warps (one up to 2048 columns, two up to 4096), a lane has at most C 8-column chunks of it in registers: all loads
// of a row leave together, its maximum is one warp reduction, and no block-wide barrier ties the warps of an SM together, so
// some load while others compute.  (A block per two or four rows with two chunks per thread spent 155 instructions per chunk, two
// thirds of them per-group overhead.)
// The divisors are 1 on all but the ~1 % outlier channels: once per CTA a mask of the undivided columns (a byte each) and a
// list of the divided ones are made; the maximum of the undivided columns is taken through the mask, the codes as if
// nothing were divided, and the listed columns are done apart, one per lane, with IEEE divisions.  A CTA with more
// divided columns than the list holds tests every divisor.
constexpr int kRThreads = 256, kRWarps = kRThreads / 32;
constexpr int kRItems = 2;              // listed columns of a lane that are loaded with the row

template <int C, int W>
__global__ void __launch_bounds__(kRThreads, C <= 8 ? 3 : 2)
act_rows_kernel(const __half* __restrict__ X, const float* __restrict__ s, int M, int K, bool beside,
                int8_t* __restrict__ Xq, float* __restrict__ a_scale, float qmax) {
    extern __shared__ uint2 mask[];         // [K / 8]: 0xff per undivided column
    __shared__ unsigned part[2][kRWarps];   // row maxima of the warps of a row
    __shared__ int n_list;
    __shared__ int list_col[kRowsList];
    __shared__ float list_s[kRowsList];     // their divisors
    if (!beside) grid_dep_wait();
    grid_dep_launch();      // a dependent linear kernel may start streaming its weights
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, chunks = K / 8;
    constexpr int per = kRWarps / W, cs = W * 32;                    // rows at a time; chunks between a lane's
    const int sub = warp / W, c0 = warp % W * 32 + lane;             // this warp's row of them, this lane's first chunk
    const int row_step = gridDim.x * per;
    int m = blockIdx.x * per + sub;
    uint4 x[C];
    auto load = [&](int row) {
        const uint4* p = reinterpret_cast<const uint4*>(X + (size_t)row * K) + c0;
#pragma unroll
        for (int i = 0; i < C; ++i) x[i] = c0 + i * cs < chunks ? p[i * cs] : make_uint4(0, 0, 0, 0);
    };
    if (m < M) load(m);
    if (tid == 0) n_list = 0;
    __syncthreads();
    const float4* s4 = reinterpret_cast<const float4*>(s);
    for (int cc = tid; cc < chunks; cc += 2 * kRThreads) {          // two chunks' divisors in flight
        float4 sv4[2][2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = cc + h * kRThreads;
            sv4[h][0] = sv4[h][1] = make_float4(1.f, 1.f, 1.f, 1.f);
            if (s && c < chunks) { sv4[h][0] = __ldg(s4 + 2 * c); sv4[h][1] = __ldg(s4 + 2 * c + 1); }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = cc + h * kRThreads;
            if (c >= chunks) continue;
            const float sv[8] = {sv4[h][0].x, sv4[h][0].y, sv4[h][0].z, sv4[h][0].w, sv4[h][1].x, sv4[h][1].y, sv4[h][1].z, sv4[h][1].w};
            uint32_t b[2] = {0xffffffffu, 0xffffffffu};
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (sv[e] != 1.f) {
                    b[e >> 2] &= ~(0xffu << (8 * (e & 3)));
                    const int at = atomicAdd(&n_list, 1);
                    if (at < kRowsList) { list_col[at] = c * 8 + e; list_s[at] = sv[e]; }
                }
            mask[c] = make_uint2(b[0], b[1]);
        }
    }
    __syncthreads();
    const int listed = n_list;
    const bool general = listed > kRowsList;
    auto row_sync = [&]() {                 // the warps of a row
        if (W == 1) __syncwarp();
        else named_bar_sync(1 + sub, W * 32);
    };
    // this lane's first listed columns: the same in every row
    int col[kRItems];
    float sd[kRItems], xt[kRItems];
#pragma unroll
    for (int k = 0; k < kRItems; ++k) {
        const int e = c0 + k * cs;
        col[k] = (!general && e < listed) ? list_col[e] : -1;
        sd[k] = col[k] >= 0 ? list_s[e] : 1.f;
    }
    for (int flip = 0; m < M; m += row_step, flip ^= 1) {
        const __half* xrow = X + (size_t)m * K;
        int8_t* out = Xq + (size_t)m * K;
#pragma unroll
        for (int k = 0; k < kRItems; ++k) xt[k] = col[k] >= 0 ? __half2float(xrow[col[k]]) : 0.f;
        float big = 0.f;
        if (!general) {
            __half2 h = __float2half2_rn(0.f);
#pragma unroll
            for (int i = 0; i < C; ++i) {
                if (c0 + i * cs >= chunks) continue;
                const uint2 b = mask[c0 + i * cs];
                const uint32_t xw[4] = {x[i].x, x[i].y, x[i].z, x[i].w};
                const uint32_t bw[4] = {__byte_perm(b.x, 0, 0x1100), __byte_perm(b.x, 0, 0x3322), __byte_perm(b.y, 0, 0x1100), __byte_perm(b.y, 0, 0x3322)};
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const uint32_t v = xw[w] & bw[w] & 0x7fff7fffu;
                    h = __hmax2(h, *reinterpret_cast<const __half2*>(&v));
                }
            }
            big = fmaxf(__low2float(h), __high2float(h));
#pragma unroll
            for (int k = 0; k < kRItems; ++k)
                if (col[k] >= 0) {
                    xt[k] = __fdiv_rn(xt[k], sd[k]);
                    big = fmaxf(big, fabsf(xt[k]));
                }
            for (int e = c0 + kRItems * cs; e < listed; e += cs)
                big = fmaxf(big, fabsf(__fdiv_rn(__half2float(xrow[list_col[e]]), list_s[e])));
        } else {
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const int c = c0 + i * cs;
                if (c >= chunks) continue;
                RawChunk rc;
                rc.x = x[i];
                rc.s0 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c);
                rc.s1 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c + 1);
                float v[8];
                smooth8(rc, v);
#pragma unroll
                for (int e = 0; e < 8; ++e) big = fmaxf(big, fabsf(v[e]));
            }
        }
        unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(big));       // non-negative floats are ordered like their bits
        if (W > 1) {
            if (lane == 0) part[flip][warp] = top;
            row_sync();
            for (int w = 0; w < W; ++w) top = max(top, part[flip][sub * W + w]);
        }
        const float sc = __fdiv_rn(__uint_as_float(top), qmax), rcp = code_rcp(sc);
        if (c0 == 0) a_scale[m] = sc;
        if (!(sc > 0.f)) {
#pragma unroll
            for (int i = 0; i < C; ++i)
                if (c0 + i * cs < chunks) reinterpret_cast<uint2*>(out)[c0 + i * cs] = make_uint2(0u, 0u);
        } else if (!general) {
            unsigned ties = 0;
#pragma unroll
            for (int i = 0; i < C; ++i) {
                if (c0 + i * cs >= chunks) continue;
                bool tie;
                reinterpret_cast<uint2*>(out)[c0 + i * cs] = codes8_try(x[i], rcp, &tie);
                if (tie) ties |= 1u << i;
            }
            while (ties) {          // a product next to a tie: the chunk once more, divided
                const int c = c0 + (__ffs(ties) - 1) * cs;
                ties &= ties - 1;
#pragma unroll 1
                for (int e = 0; e < 8; ++e)
                    out[c * 8 + e] = (int8_t)rne_clamp(__fdiv_rn(__half2float(xrow[c * 8 + e]), sc), -qmax, qmax);
            }
            if (listed > 0) {
                row_sync();         // orders the stores above before the single bytes below
#pragma unroll
                for (int k = 0; k < kRItems; ++k)
                    if (col[k] >= 0) out[col[k]] = (int8_t)rne_clamp(__fdiv_rn(xt[k], sc), -qmax, qmax);
                for (int e = c0 + kRItems * cs; e < listed; e += cs) {
                    const int cc = list_col[e];
                    out[cc] = (int8_t)rne_clamp(__fdiv_rn(__fdiv_rn(__half2float(xrow[cc]), list_s[e]), sc), -qmax, qmax);
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const int c = c0 + i * cs;
                if (c >= chunks) continue;
                RawChunk rc;
                rc.x = x[i];
                rc.s0 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c);
                rc.s1 = __ldg(reinterpret_cast<const float4*>(s) + 2 * c + 1);
                float v[8];
                smooth8(rc, v);
                reinterpret_cast<uint2*>(out)[c] = quant8_pairs(v, sc, rcp, qmax);
            }
        }
        if (m + row_step < M) load(m + row_step);
    }
    // This kernel is not over before act_proj_kernel is: who waits for it waits for both.  (One CTA is enough; the others
    // make room for the linear kernel.)
    if (beside && blockIdx.x == 0) grid_dep_wait();
}

// W warps per row and C chunks per lane: the fewest warps that need at most eight chunks; sixteen where eight warps do not
// suffice (rows above 16384).
int launch_rows(cudaLaunchConfig_t cfg, const __half* X, const float* s, int M, int K, bool beside, int8_t* Xq,
                float* a_scale, float qmax) {
    auto go = [&](auto* kernel, int W) {
        const int per = kRWarps / W, groups = (M + per - 1) / per, most = (beside || K > 16384 ? 2 : 3) * kProjPlanSms;
        cfg.gridDim = dim3(groups < most ? groups : most, 1, 1);
        cfg.blockDim = dim3(kRThreads, 1, 1);
        cfg.dynamicSmemBytes = (size_t)K;               // the mask, 8 bytes per chunk: at most 32 KB
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, X, s, M, K, beside, Xq, a_scale, qmax);
        return e == cudaSuccess ? (int)ASER_OK : record_cuda_error(e, "act_rows_kernel");
    };
    if (K <= 1024) return go(act_rows_kernel<4, 1>, 1);
    if (K <= 2048) return go(act_rows_kernel<8, 1>, 1);
    if (K <= 4096) return go(act_rows_kernel<8, 2>, 2);
    if (K <= 8192) return go(act_rows_kernel<8, 4>, 4);
    if (K <= 16384) return go(act_rows_kernel<8, 8>, 8);
    return go(act_rows_kernel<16, 8>, 8);
}

// Slices of K, of at least four 64-column stages.  Beside act_rows_kernel the slices are one cluster: the size of at most eight that
// gives the most CTAs while all clusters fit at once (a GPC has 16 to 20 SMs; 2048 x 4096, rank 64: 16 clusters of eight took
// two waves, 24 us); how many fit is written down for a part of 148 SMs rather than asked for, since the slices decide the order of
// T's sums, which should not depend on the device.  Otherwise as many equal slices as keep the grid within one wave.
// Cutting long inputs into chunks of tokens whose X stays in L2 for the second kernel cost more in fixed time per
// launch pair than the L2 hits saved (4096 x 14336 at rank 128: 140 us in three chunks, 95 us in one).
int proj_slices(int M, int K, bool beside, int num_sms) {
    const int blocks = K / kPCols;
    const int tiles = (M + kPTok - 1) / kPTok;
    int ks_best = 1;
    if (beside) {
        constexpr int fit[kPMaxCluster + 1] = {0, kProjPlanSms, 72, 44, 32, 24, 20, 14, 14};
        for (int ks = 2; ks <= kPMaxCluster && ks <= blocks / 4; ++ks)
            if (tiles <= fit[ks]) ks_best = ks;
        return ks_best;
    }
    for (int ks = 1; ks <= blocks / 4 && tiles * ks <= num_sms; ++ks)
        if (blocks % ks == 0) ks_best = ks;
    return ks_best;
}

// Floats of the row-maxima part of the scratch, padded so that the partial T behind it starts on
// a 128-byte boundary (it is written by bulk copies, which need 16-byte alignment).
size_t proj_amax_floats(int M, int slices) { return ((size_t)slices * M + 31) & ~(size_t)31; }

// What M tokens leave in the scratch, one kernel after the other.
size_t proj_scratch_bytes(int M, int r, int slices) {
    return (proj_amax_floats(M, slices) + (size_t)slices * M * ((r + 127) / 128) * 128) * sizeof(float);
}

}  // namespace

// Enough for any pass of up to M tokens where the two orders meet, so that a caller may size it for his largest: nothing goes through the
// scratch from beside_from tokens on; below, the slices of all tiles are at most one wave.
size_t quant_act_ws_scratch_bytes(int M, int K, int r) {
    if (M <= 32 || r == 0) return 0;
    const int from = beside_from(K, r);
    if (from == kNever) return proj_scratch_bytes(M, r, proj_slices(M, K, false, kProjPlanSms));
    const int few = M < from ? M : from - 1;
    if (few <= 32) return 0;
    const int most = K / kPCols / 4 > 1 ? K / kPCols / 4 : 1;            // slices of a pass
    const long long rows = (long long)most * few;
    return proj_scratch_bytes((int)(rows < (long long)kProjPlanSms * kPTok ? rows : (long long)kProjPlanSms * kPTok), r, 1);
}

int quant_act_ws_launches(int M, int K) { return M <= 32 ? 1 : 2; }

int launch_quant_act_ws(const __half* X, const float* s, const __half* LA, int M, int K, int r,
                        int8_t* Xq, float* a_scale, __nv_bfloat16* T, void* scratch, size_t scratch_bytes,
                        cudaStream_t st, int act_bits, bool t_pair, int M_pass) {
    const float qmax = (float)((1 << (act_bits - 1)) - 1);
    const int ldt = t_pair ? 2 * r : r, lo_off = t_pair ? r : 0;
    const int groups = (r + 127) / 128;
    if (groups > kPMaxGroups) return record_error(ASER_ERR_SHAPE, "quant_act: r beyond 512");
    if (M_pass == 0) M_pass = M;
    const bool beside = r > 0 && rows_beside(M_pass, K, r);
    const int KS = proj_slices(M_pass, K, beside, kProjPlanSms);
    if (scratch == nullptr || misaligned16(scratch) || (r > 0 && !beside && scratch_bytes < proj_scratch_bytes(M, r, KS)))
        return record_error(ASER_ERR_WORKSPACE, "quant_act: scratch missing or too small");
    float* amax_part = static_cast<float*>(scratch);
    float* t_part = amax_part + proj_amax_floats(M, KS);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaSuccess;
    if (r > 0) {
        const int Kc = (K / kPCols + KS - 1) / KS * kPCols, NS = proj_stages(groups, K, beside);       // the longest slice
        // the ring (at least 128 KB: it later stages the partial T) and the tail
        const size_t smem = (size_t)NS * kPTileBytes * (1 + groups) + 256 + ((Kc / 8 + 15) & ~15) +
                            kPCacheUnits * 8 * sizeof(float) + (beside ? 0 : kPConsumerWarps * kPTok * sizeof(float)) + 1024;
        auto* kernel = beside ? act_proj_kernel<false> : act_proj_kernel<true>;
        static size_t configured_all[2][kMaxDevices] = {{0}};
        size_t* configured = configured_all[beside ? 0 : 1];
        int dev = 0;
        int rc = current_device(&dev);
        if (rc != ASER_OK) return rc;
        if (smem > configured[dev]) {
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            // all of the SM's shared memory, not only what this kernel needs: act_rows_kernel has to find room beside it
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
            if (e != cudaSuccess) return record_cuda_error(e, "act_proj smem attribute");
            configured[dev] = smem;
        }
        CUtensorMap mx, mla;
        rc = encode_map_blocks(&mx, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, X, M, K, kPTok, 1);
        if (rc != ASER_OK) return rc;
        rc = encode_map_blocks(&mla, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, LA, r, K, r <= 256 ? r : r / 2, 1);
        if (rc != ASER_OK) return rc;
        cudaLaunchAttribute pattr[2] = {attr[0], {}};
        pattr[1].id = cudaLaunchAttributeClusterDimension;
        pattr[1].val.clusterDim.x = beside ? KS : 1; pattr[1].val.clusterDim.y = 1; pattr[1].val.clusterDim.z = 1;
        cudaLaunchConfig_t pcfg = cfg;
        pcfg.attrs = pattr;
        pcfg.numAttrs = 2;
        pcfg.gridDim = dim3(KS, (M + kPTok - 1) / kPTok, 1);
        pcfg.blockDim = dim3(kPThreads, 1, 1);
        pcfg.dynamicSmemBytes = smem;
        e = cudaLaunchKernelEx(&pcfg, kernel, mx, mla, s, M, K, r, amax_part, t_part, T, ldt, lo_off);
        if (e != cudaSuccess) return record_cuda_error(e, "act_proj_kernel");
    }
    if (r > 0 && !beside) {
        cfg.gridDim = dim3((M + kQRows - 1) / kQRows, 1, 1);
        cfg.blockDim = dim3(256, 1, 1);
        e = cudaLaunchKernelEx(&cfg, act_quant_kernel, X, s, M, K, r, KS, (const float*)amax_part, (const float*)t_part, Xq,
                               a_scale, T, ldt, lo_off, qmax);
        return e == cudaSuccess ? (int)ASER_OK : record_cuda_error(e, "act_quant_kernel");
    }
    return launch_rows(cfg, X, s, M, K, r > 0, Xq, a_scale, qmax);
}

}  // namespace aser
