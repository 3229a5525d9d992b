// Tensor-core kernel of the ASER linear for 17 to 512 tokens (Sec. 4.2, "W_q X + L_A L_B X"), every tile split along
// K over a cluster:
//   acc = Xq Wq^T (int8 x int4 -> int32),  Y = fp16(acc * a_scale[m] * w_scale[n] + T L_B^T).
//
// At these sizes a layer has fewer tiles than the part has SMs and a launch lasts little longer than its fixed costs, so what
// bounds it is the length of a CTA's chain: start-up, its share of K, the exchange of partial sums, the epilogue.
//  * One item per CTA: a tile of 128 channels x up to 128 tokens, computed transposed (D[n, token]) as in linear_tc.cu, and
//    a slice of K.  The S slices of a tile are a cluster.  Nothing is carried from item to item, so there is one
//    accumulator, and tensor memory holds eight A blocks beside it and the low-rank accumulator.
//  * The packed weights do not go through shared memory: sixteen warps load them straight into registers (two blocks of
//    8 KB per group of four warps ahead, the first before anything else, while the activation kernel still runs), turn them
//    into int8 (value 16 q) and write them to tensor memory.  Shared memory carries the activations alone.
//  * A stage is two blocks: their activations in one copy, one barrier that counts the copy's bytes and the eight warps that
//    unpack, one commit that frees both operands.  One thread issues all integer products: those of one thread into the same
//    sums run in order, those of two only if each waits for the other's issue.
//  * Partial sums: each CTA stages its int32 sums as [token][128 channels] where the activations were and sends every peer
//    the tokens that this peer finishes, one bulk copy each into a buffer of its own (16 n tokens per CTA).  Integer sums:
//    the order does not matter.
//  * The low-rank product of the tokens that a CTA finishes has sums and an issuing thread of its own; two warps load and
//    convert its operands (T bf16 -> fp16, exact in the fp16 normal range).  Chunks of 64 in order: the same sums as in the
//    other kernels.
//  * The sixteen warps are the epilogue as well; outputs leave through shared memory as tensor stores of 16 tokens.
// Every wait is bounded: on expiry the CTA sets the status word and winds down.
//
// Measured against linear_tc_kernel (or linear_pair_kernel, whichever the shape had), the linear step alone in graphs on one box
// (tokens x channels x K, us): 17 x 4096 x 4096 13.2 -> 8.4; 32 x 14336 x 4096 20.4 -> 10.0; 64 x 4096 x 14336 21.1 -> 12.8;
// 101 x 8192 x 8192 26.5 -> 16.7; 128 x 14336 x 4096 20.9 -> 14.3; 200 x 8192 x 2048 14.7 -> 10.5; 400 x 4096 x 4096 19.6 -> 13.3;
// 256 x 4096 x 14336 32.4 -> 20.2.  (Repeats of one call: the weights come from L2.)  What bounds it is latency: at 101 x 8192 x
// 8192, cold, L2 is 18 % busy, HBM 22, the SM 22; set-up takes 1.2 us, exchange and outputs 3, and between them a stage brings 44 KB
// to every SM (activations are read once per 128 channels).
#include "aser_common.cuh"
#include "sm100_ptx.cuh"

namespace aser {

namespace {

constexpr int kUnpackWarps = 16, kThreads = (kUnpackWarps + 5) * 32;   // + activation producer, issuers of the integer and of the low-rank products, two of the low-rank operands
constexpr int kWarpIssue = kUnpackWarps + 1, kWarpLr = kUnpackWarps + 3;
constexpr int kSlots = 8, kStages = kSlots / 2;  // A blocks in tensor memory = activation blocks in shared memory, two to a stage
constexpr int kMaxTok = 128, kMaxSplit = 8;
constexpr int kLbBytes = 128 * 128;
constexpr long long kWaitClocks = 400000000ll;   // about 0.2 s of SM clocks per wait

constexpr int B_FULL = 0, B_FREE = B_FULL + kStages, B_ACC = B_FREE + kStages, B_RECV = B_ACC + 1,
              B_LR_FULL = B_RECV + 1, B_LR_CONV = B_LR_FULL + 2, B_LR_FREE = B_LR_CONV + 2, B_LR_DONE = B_LR_FREE + 2,
              kNumBars = B_LR_DONE + 1;
static_assert(kNumBars * 8 + 8 <= 256, "barrier area");

struct Params {
    const uint8_t* Wk;
    const float* a_scale;
    const float* w_scale;
    int32_t* acc_debug;
    uint32_t* status;
    int M, N, r, KB;
    int tok, own;          // tokens of a tile, tokens that a CTA of the cluster finishes (multiples of 16)
    int TT;                // token tiles
    CatSplit cat;
};

// Shared memory behind a 1024-byte boundary: activation ring (later the staged sums and outputs), received sums, low-rank
// operands (two sets), barriers, the scales of the tokens that this CTA finishes.
struct Smem {
    int x_block, recv, lr, lr_set, bars, scales, total;
};
__host__ __device__ inline Smem smem_of(int tok, int own, int S) {
    Smem m;
    m.x_block = tok * 128;
    m.recv = kSlots * m.x_block;         // twice what the staged sums take
    m.lr = (m.recv + (S - 1) * own * 512 + 1023) & ~1023;
    m.lr_set = kLbBytes + own * 128;
    m.bars = m.lr + 2 * m.lr_set;
    m.scales = m.bars + 256;
    m.total = m.scales + own * 4 + 1024;
    return m;
}

struct Stop {
    volatile int* flag;    // shared
    uint32_t* status;      // global
};

__device__ __noinline__ bool wait_slow(uint32_t bar, uint32_t parity, volatile int* flag, uint32_t* status) {
    uint32_t spins = 0;
    long long t0 = 0;
    while (!mbar_try_wait(bar, parity)) {
        if ((++spins & 255u) == 0) {
            if (*flag) return false;
            const long long now = clock64();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > kWaitClocks) {
                *flag = 1;
                atomicOr(status, 1u);
                if (atomicCAS(status + 1, 0u, 0x40000000u | threadIdx.x) == 0u) {    // which wait it was
                    status[2] = blockIdx.x;
                    status[3] = (bar & 255u) >> 3;
                    status[4] = parity;
                }
                return false;
            }
        }
    }
    return true;
}
__device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity, const Stop& stop) {
    if (mbar_try_wait(bar, parity)) return true;
    return wait_slow(bar, parity, stop.flag, stop.status);
}
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, const Stop& stop, int lane) {
    int ok = 1;
    if (lane == 0) ok = wait(bar, parity, stop) ? 1 : 0;
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}
// Copies in flight, to peers too, land before a CTA that gave up lets go of its shared memory.
__device__ __forceinline__ void let_copies_land() {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000) {}
}
__device__ __forceinline__ uint4 ld_weights(const uint8_t* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// Shared memory of this CTA -> shared memory of a peer, counted on a barrier of the peer.
__device__ __forceinline__ void send(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}

// Grid: S * NT * TT CTAs in clusters of S; cluster = nt * TT + tt.
__global__ void __launch_bounds__(kThreads, 1)
linear_split_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_lb,
                    const __grid_constant__ CUtensorMap map_t, const __grid_constant__ CUtensorMap map_y,
                    const Params p, const int S) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sb = smem_u32(smem);
    const Smem L = smem_of(p.tok, p.own, S);
    auto bar = [&](int i) { return sb + (uint32_t)L.bars + 8u * i; };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L.bars + kNumBars * 8);
    volatile int* stop_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const Stop stop{stop_flag, p.status};
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)blockIdx.x % S, tile = (int)blockIdx.x / S, nt = tile / p.TT, tt = tile % p.TT;
    const int n0 = nt * 128, tok0 = tt * p.tok;
    const int kb0 = p.KB * rank / S, nkb = p.KB * (rank + 1) / S - kb0, stages = (nkb + 1) / 2;
    const int own0 = rank * p.own;                       // this CTA's tokens of the tile: [own0, own0 + owned)
    const int owned = p.tok - own0 < p.own ? (p.tok - own0 > 0 ? p.tok - own0 : 0) : p.own;
    const int chunks = owned > 0 ? (p.r + 63) / 64 : 0;

    // unpack warps: the first two blocks' weights are on their way before anything else
    const int q = warp & 3, group = warp >> 2, row = q * 32 + lane;
    const uint8_t* wsrc = p.Wk + ((size_t)nt * p.KB + kb0) * kWkBlockBytes + row * 16;
    uint4 raw[2][4];
    auto fetch = [&](int b, uint4 (&to)[4]) {
#pragma unroll
        for (int s4 = 0; s4 < 4; ++s4) to[s4] = ld_weights(wsrc + (size_t)b * kWkBlockBytes + s4 * 2048);
    };
    if (warp < kUnpackWarps) {
        if (group < nkb) fetch(group, raw[0]);
        if (group + 4 < nkb) fetch(group + 4, raw[1]);
    } else if (warp == kUnpackWarps) {
        for (int i = lane; i < kNumBars; i += 32) {
            uint32_t count = 1;
            if (i < B_FREE) count = 9;                   // eight warps' A rows and the copy
            if (i >= B_LR_CONV && i < B_LR_FREE) count = 2;
            mbar_init(bar(i), count);
        }
        if (lane == 0) *stop_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
            if (S > 1 && owned > 0) mbar_arrive_expect_tx(bar(B_RECV), (uint32_t)((S - 1) * owned * 512));
            prefetch_tensormap(&map_x);
            prefetch_tensormap(&map_y);
        }
    } else if (warp == kWarpIssue) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else if (warp == kWarpLr && lane == 0 && chunks > 0) {
        prefetch_tensormap(&map_lb);
        prefetch_tensormap(&map_t);
    }
    tc_fence_before();
    __syncthreads();
    if (S > 1) cluster_arrive();         // the peers' barriers are in place: waited for before sums are sent
    tc_fence_after();
    const uint32_t tmem = *tmem_slot, tm_lr = tmem + kMaxTok, tm_a = tmem + 2 * kMaxTok;

    // The next activation kernel may be set up meanwhile: it waits for the end of this kernel before it reads anything, and
    // lets its own dependents start only then.
    if (threadIdx.x == 0) grid_dep_launch();
    if (warp == kUnpackWarps) {
        // =================== activation producer ===================
        if (lane == 0) {
            grid_dep_wait();             // Xq comes from the kernel launched before this one
            // Two blocks to a copy: a copy costs its thread 500 cycles whatever its size.  (The second block of the last copy
            // may lie past the slice or past K.)
            bool ok = true;
            for (int st = 0; st < stages && ok; ++st) {
                const int s = st % kStages;
                if (st >= kStages) ok = wait(bar(B_FREE + s), (uint32_t)(st / kStages - 1) & 1u, stop);
                if (!ok) break;
                mbar_arrive_expect_tx(bar(B_FULL + s), 2u * (uint32_t)L.x_block);
                tma_load_3d(sb + 2 * s * L.x_block, &map_x, 0, tok0, kb0 + 2 * st, bar(B_FULL + s));
            }
            if (!ok || *stop_flag) let_copies_land();
        }
    } else if (warp == kWarpIssue) {
        // =================== integer products ===================
        // The whole warp goes through the loop and one lane is elected around the products (the same one every time), which
        // keeps their operands in uniform registers: in a branch of lane 0 the same loop took 10 to 40 % longer, and two
        // such threads with alternate blocks 11 %.
        const uint32_t idesc = make_idesc(2, 1, 128, (uint32_t)p.tok);
        bool ok = true;
        for (int st = 0; st < stages; ++st) {
            const int s = st % kStages;
            ok = wait(bar(B_FULL + s), (uint32_t)(st / kStages) & 1u, stop);
            ok = __all_sync(0xffffffffu, ok) != 0;
            if (!ok) break;
            tc_fence_after();
            const uint64_t xdesc = smem_desc_sw128(sb + 2 * s * L.x_block);
            const uint32_t a = tm_a + s * 64;
            if (elect_one()) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (2 * st + h < nkb)
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            mma_i8_ts(tmem, a + h * 32 + kk * 8, xdesc + (uint64_t)(h * (L.x_block >> 4) + 2 * kk), idesc,
                                      (st | h | kk) != 0 ? 1u : 0u);
                tc_commit(bar(B_FREE + s));
            }
            __syncwarp();
        }
        if (ok && elect_one()) tc_commit(bar(B_ACC));
        __syncwarp();
    } else if (warp == kWarpIssue + 1) {
        // =================== low-rank products ===================
        const uint32_t idesc = make_idesc(1, 0, 128, (uint32_t)p.own);
        bool ok = true;
        for (int c = 0; c < chunks; ++c) {
            ok = wait(bar(B_LR_CONV + (c & 1)), (uint32_t)(c >> 1) & 1u, stop);
            ok = __all_sync(0xffffffffu, ok) != 0;
            if (!ok) break;
            tc_fence_after();
            const uint32_t set = sb + (uint32_t)(L.lr + (c & 1) * L.lr_set);
            const uint64_t ad = smem_desc_sw128(set), bd = smem_desc_sw128(set + kLbBytes);
            const int steps = p.r - c * 64 >= 64 ? 4 : (p.r - c * 64) / 16;
            if (elect_one()) {
                for (int kk = 0; kk < steps; ++kk)
                    mma_f16_ss(tm_lr, ad + 2 * kk, bd + 2 * kk, idesc, (c | kk) != 0 ? 1u : 0u);
                tc_commit(bar(B_LR_FREE + (c & 1)));
            }
            __syncwarp();
        }
        if (ok && chunks > 0 && elect_one()) tc_commit(bar(B_LR_DONE));
        __syncwarp();
    } else if (warp >= kWarpLr) {
        // =================== low-rank operands ===================
        const int w = warp - kWarpLr;
        bool ok = true;
        int loaded = 0;
        auto load_lb = [&](int c) {
            const uint32_t set = sb + (uint32_t)(L.lr + (c & 1) * L.lr_set);
            mbar_arrive_expect_tx(bar(B_LR_FULL + (c & 1)), (uint32_t)L.lr_set);
            tma_load_2d(set, &map_lb, c * 64, n0, bar(B_LR_FULL + (c & 1)));
        };
        auto load_t = [&](int c) {
            tma_load_2d(sb + (uint32_t)(L.lr + (c & 1) * L.lr_set + kLbBytes), &map_t, c * 64 + cat_layer(p.cat, n0) * p.r,
                        tok0 + own0, bar(B_LR_FULL + (c & 1)));
        };
        if (w == 0 && lane == 0 && chunks > 0) {         // L_B does not wait for the activation kernel
            for (int c = 0; c < chunks && c < 2; ++c) load_lb(c);
            grid_dep_wait();
            for (int c = 0; c < chunks && c < 2; ++c) load_t(c);
            loaded = chunks < 2 ? chunks : 2;
        }
        for (int c = 0; c < chunks && ok; ++c) {
            if (w == 0 && lane == 0 && c >= 2) {
                ok = wait(bar(B_LR_FREE + (c & 1)), (uint32_t)((c >> 1) - 1) & 1u, stop);
                if (ok) { load_lb(c); load_t(c); ++loaded; }
            }
            __syncwarp();
            if (ok) ok = wait(bar(B_LR_FULL + (c & 1)), (uint32_t)(c >> 1) & 1u, stop);
            ok = __all_sync(0xffffffffu, ok) != 0;
            if (!ok) break;
            uint4* t = reinterpret_cast<uint4*>(smem + L.lr + (c & 1) * L.lr_set + kLbBytes);
            for (int i = w * 32 + lane; i < p.own * 8; i += 64) {
                const uint4 v = t[i];
                const uint32_t in[4] = {v.x, v.y, v.z, v.w};
                uint32_t out[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const __half2 h = __floats2half2_rn(__uint_as_float(in[k] << 16), __uint_as_float(in[k] & 0xFFFF0000u));
                    out[k] = *reinterpret_cast<const uint32_t*>(&h);
                }
                t[i] = make_uint4(out[0], out[1], out[2], out[3]);
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_LR_CONV + (c & 1)));
        }
        if ((!ok || *stop_flag) && w == 0 && lane == 0 && loaded > 0) let_copies_land();
    } else {
        // =================== unpack: int4 -> int8 (x16) into tensor memory ===================
        bool ok = true;
        auto block = [&](int b, uint4 (&w)[4]) {
            const int s = b % kSlots;
            if (b >= kSlots) ok = warp_wait(bar(B_FREE + s / 2), (uint32_t)(b / kSlots - 1) & 1u, stop, lane);
            if (!ok) return;
            if (b == nkb) {              // the half of the last stage that is not there
                if (lane == 0) mbar_arrive(bar(B_FULL + s / 2));
                return;
            }
            tc_fence_after();
            const uint32_t a = tm_a + s * 32 + ((uint32_t)(q * 32) << 16);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t v[16];
#pragma unroll
                for (int s4 = 0; s4 < 2; ++s4) {
                    const uint32_t xs[4] = {w[2 * h + s4].x, w[2 * h + s4].y, w[2 * h + s4].z, w[2 * h + s4].w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        v[s4 * 8 + 2 * e] = (xs[e] << 4) & 0xF0F0F0F0u;      // columns c0 .. c0+3
                        v[s4 * 8 + 2 * e + 1] = xs[e] & 0xF0F0F0F0u;         // columns c0+4 .. c0+7
                    }
                }
                tmem_st16(a + h * 16, v);
            }
            if (b + 8 < nkb) fetch(b + 8, w);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_FULL + s / 2));
        };
        for (int b = group; b < 2 * stages && ok; b += 8) {
            block(b, raw[0]);
            if (ok && b + 4 < 2 * stages) block(b + 4, raw[1]);
        }

        // =================== epilogue ===================
        grid_dep_wait();                 // a_scale comes from the kernel launched before this one
        float* scales = reinterpret_cast<float*>(smem + L.scales);
        if ((int)threadIdx.x < owned) {
            const int m = tok0 + own0 + (int)threadIdx.x;
            scales[threadIdx.x] = m < p.M ? __ldg(p.a_scale + m) : 0.f;
        }
        const int n = n0 + row;
        const float ws16 = (n < p.N ? __ldg(p.w_scale + n) : 0.f) * 0.0625f;          // the sums hold 16 q x
        if (ok) ok = warp_wait(bar(B_ACC), 0u, stop, lane);
        tc_fence_after();
        const uint32_t lanes = (uint32_t)(q * 32) << 16;
        if (S > 1) {
            // the sums that peers finish, staged as [token][128 channels] (the ring is idle: all products are complete)
            for (int c = group * 16; c < p.tok; c += 64) {
                if (c >= own0 && c < own0 + owned) continue;
                uint32_t v[16];
                tmem_ld16(tmem + lanes + (uint32_t)c, v);
                tmem_wait_ld(v);
#pragma unroll
                for (int e = 0; e < 16; ++e)
                    asm volatile("st.shared.b32 [%0], %1;" ::"r"(sb + (uint32_t)((c + e) * 512 + row * 4)), "r"(v[e]) : "memory");
            }
            fence_proxy_async_smem();
            cluster_wait();              // (arrived on by every thread at the start)
        }
        named_bar_sync(1, kUnpackWarps * 32);        // staged, and the scales are there
        if (S > 1) {
            if (threadIdx.x == 0 && !*stop_flag) {
                for (int d = 1; d < S; ++d) {            // each CTA starts with another peer
                    const int to = (rank + d) % S, first = to * p.own;
                    const int count = p.tok - first < p.own ? p.tok - first : p.own;
                    if (count <= 0) continue;
                    const int slot = rank < to ? rank : rank - 1;
                    send(map_to_rank(sb + (uint32_t)(L.recv + slot * count * 512), (uint32_t)to), sb + (uint32_t)(first * 512),
                         (uint32_t)(count * 512), map_to_rank(bar(B_RECV), (uint32_t)to));
                }
            }
            if (ok && owned > 0) ok = warp_wait(bar(B_RECV), 0u, stop, lane);
        }
        if (chunks > 0 && ok) {
            ok = warp_wait(bar(B_LR_DONE), 0u, stop, lane);
            tc_fence_after();
        }
        if (ok) {
            for (int c = group * 8; c < owned; c += 32) {
                uint32_t v[8], f[8];
                tmem_ld8(tmem + lanes + (uint32_t)(own0 + c), v);
                tmem_wait_ld8(v);
                if (chunks > 0) {
                    tmem_ld8(tm_lr + lanes + (uint32_t)c, f);
                    tmem_wait_ld8(f);
                }
                for (int src = 0; src < S - 1; ++src) {
                    const int* rp = reinterpret_cast<const int*>(smem + L.recv) + (src * owned + c) * 128 + row;
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] += (uint32_t)rp[e * 128];
                }
                const int m0 = tok0 + own0 + c;
                // outputs as [token][128 channels]: where this CTA's own sums would be staged (nobody sends those)
                uint16_t* out = reinterpret_cast<uint16_t*>(smem + (size_t)own0 * 512) + c * 128 + row;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float y = fmaf((float)(int)v[e], scales[c + e] * ws16, chunks > 0 ? __uint_as_float(f[e]) : 0.f);
                    out[e * 128] = __half_as_ushort(__float2half_rn(y));
                    if (p.acc_debug && m0 + e < p.M && n < p.N) p.acc_debug[(size_t)(m0 + e) * p.N + n] = (int)v[e] >> 4;
                }
            }
        }
        fence_proxy_async_smem();
        ok = named_bar_all(1, kUnpackWarps * 32, ok);
        if (threadIdx.x == 0 && ok) {
            for (int c = 0; c < owned; c += 16)
                if (tok0 + own0 + c < p.M) tma_store_2d_tile(&map_y, n0, tok0 + own0 + c, sb + (uint32_t)(own0 * 512 + c * 256));
            bulk_store_commit();
            bulk_store_wait_read();      // (the stores themselves are complete when the kernel is)
        }
        if (threadIdx.x == 0 && !ok) let_copies_land();
        tc_fence_before();
    }

    // =================== teardown ===================
    __syncwarp();
    tc_fence_before();
    if (S > 1 && warp >= kUnpackWarps) cluster_wait();
    __syncthreads();
    if (S > 1) {                         // nobody leaves while a peer still reads from or writes to its shared memory
        cluster_arrive();
        cluster_wait();
    }
    if (warp == kWarpIssue) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// Opts the kernel in to its largest shared memory, once per device.
int configure() {
    static int done[kMaxDevices] = {0};
    int dev = 0;
    const int rc = current_device(&dev);
    if (rc != ASER_OK) return rc;
    if (!done[dev]) {
        const cudaError_t e = cudaFuncSetAttribute(linear_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return record_cuda_error(e, "linear_split smem attribute");
        done[dev] = 1;
    }
    return ASER_OK;
}

// Clusters of S CTAs of this kernel (one CTA per SM) that are resident at once.
int active_clusters(int S) {
    static int cached[kMaxDevices][kMaxSplit + 1];       // 0: not asked yet
    int dev = 0;
    if (current_device(&dev) != ASER_OK) return 0;
    if (cached[dev][S] == 0) {
        if (configure() != ASER_OK) return 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(S, 1, 1);
        cfg.blockDim = dim3(kThreads, 1, 1);
        cfg.dynamicSmemBytes = 227 * 1024;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = S; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, linear_split_kernel, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
        cached[dev][S] = n > 0 ? n : -1;
    }
    return cached[dev][S] > 0 ? cached[dev][S] : 0;
}

struct Plan { int NT, TT, tok, S, own; };

// The largest split with which all tiles are resident at once (S = 0: the tiles alone are too many).
Plan make_plan(int M, int N, int K) {
    Plan c = {};
    c.NT = (N + 127) / 128;
    c.TT = (M + kMaxTok - 1) / kMaxTok;
    c.tok = ((M + c.TT - 1) / c.TT + 15) / 16 * 16;
    const long long tiles = (long long)c.NT * c.TT;
    for (int S = 1; S <= kMaxSplit && S <= K / kWkCols / 2; ++S) {
        const int own = ((c.tok + S - 1) / S + 15) / 16 * 16;
        if (tiles <= active_clusters(S) && smem_of(c.tok, own, S).total <= 227 * 1024) { c.S = S; c.own = own; }
    }
    return c;
}

}  // namespace

// Up to 16 tokens the streaming kernel has the shorter chain; above 512, or where the tiles are more than one wave, a kernel
// that stays for several items; with fewer than eight column blocks or four channel tiles there is little to split.
bool linear_split_prefers(int M, int N, int K) {
    if (M <= kLinearDecodeMaxTokens || M > 512 || K < 1024 || N < 512) return false;
    return make_plan(M, N, K).S > 0;
}

int launch_linear_split(const int8_t* Xq, const float* a_scale, const uint8_t* Wk, const float* w_scale,
                        const __nv_bfloat16* T, const __half* LB, int M, int N, int K, int r, __half* Y,
                        int32_t* acc_debug, void* workspace, cudaStream_t st, bool overlap_prev, int ldt, CatSplit cat) {
    const Plan plan = make_plan(M, N, K);
    if (plan.S == 0) return record_error(ASER_ERR_SHAPE, "linear_split: too many tiles");
    int rc = configure();
    if (rc != ASER_OK) return rc;
    CUtensorMap mx, mlb, mt, my;
    rc = encode_map_2d(&my, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, Y, M, N, 16, 128, CU_TENSOR_MAP_SWIZZLE_NONE);
    if (rc != ASER_OK) return rc;
    rc = encode_map_blocks(&mx, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Xq, M, K, plan.tok, 2);
    if (rc != ASER_OK) return rc;
    if (r > 0) {
        rc = encode_map_2d(&mlb, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, LB, N, r, 128, 64, CU_TENSOR_MAP_SWIZZLE_128B);
        if (rc != ASER_OK) return rc;
        rc = encode_map_2d_ld(&mt, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, T, M, r * cat.layers, ldt > 0 ? ldt : r * cat.layers,
                              plan.own, 64, CU_TENSOR_MAP_SWIZZLE_128B);
        if (rc != ASER_OK) return rc;
    } else {
        mlb = mx;
        mt = mx;
    }
    Params p = {};
    p.Wk = Wk; p.a_scale = a_scale; p.w_scale = w_scale; p.acc_debug = acc_debug;
    p.status = static_cast<uint32_t*>(workspace);
    p.M = M; p.N = N; p.r = r; p.KB = K / kWkCols;
    p.tok = plan.tok; p.own = plan.own; p.TT = plan.TT;
    p.cat = cat;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(plan.S * plan.NT * plan.TT, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem_of(plan.tok, plan.own, plan.S).total;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = plan.S; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap_prev ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, linear_split_kernel, mx, mlb, mt, my, p, plan.S);
    if (e != cudaSuccess) return record_cuda_error(e, "linear_split_kernel");
    return check_launch("linear_split_kernel");
}

}  // namespace aser
