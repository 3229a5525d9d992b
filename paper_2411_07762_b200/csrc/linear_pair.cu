// Tensor-core kernel of the ASER linear for many tokens (Sec. 4.2, "W_q X + L_A L_B X"), on pairs of CTAs:
//   acc = Xq Wq^T (int8 x int4 -> int32),  Y = fp16(acc * a_scale[m] * w_scale[n] + T L_B^T).
//
// As in linear_tc.cu the tile is computed transposed, D[n, token]: packed int4 weights are streamed to
// shared memory, turned into int8 (value 16 q) in registers and written to TENSOR MEMORY as the A
// operand; the int8 activations are the B operand in shared memory.  What bounds that kernel at many
// tokens is not arithmetic (tensor pipe busy 41 to 55 %) but the hand-over of A blocks: they are unpacked
// for 128 tokens at a time, two accumulators and the fp32 low-rank accumulator leave tensor memory for
// four of them, and a 128 x 128 tile asks 192 bytes of shared memory per cycle at full rate.  Here:
//  * two CTAs share a tile of 256 output channels x 256 tokens (cta_group::2): each holds 128 rows of
//    A and of D, and half the tokens' activations.  An A block serves 256 tokens instead of 128, an SM
//    loads 24 KB per 128 columns of K for twice the products, 96 bytes of shared memory per cycle;
//  * the tile's tokens are two halves, each with an accumulator of 128 columns and a thread of its own
//    in the leader CTA that issues the half's MMAs.  The other 256 columns of tensor memory are EIGHT A
//    blocks, in four stages of two;
//  * there is no low-rank accumulator.  When a half's integer sums are complete the epilogue takes them
//    into registers (64 per thread) and hands the columns back at once; the half's low-rank product
//    (kind::f16) is computed into THE SAME columns, read and added to the scaled sums.  One half's
//    turn-around is covered by the other half's MMAs;
//  * A blocks and activations of a stage share one barrier each way, so an issuer waits once and commits
//    once per eight MMAs (75 cycles each; a wait or a commit costs as much as one to four of them);
//  * the packed words of a group's next stage are in registers before its slot is free;
//  * both halves' outputs stay in registers as fp16 until both accumulators are free, then leave through
//    shared memory as tensor stores (two-byte stores, 64 bytes per warp and token, took 4300 cycles a half
//    and held up the other half's turn-around);
//  * arrivals on the other CTA's barriers are plain arrivals: with .release.cluster each cost its thread
//    a cluster-wide fence, in the unpack groups' loop of all places (4096 x 4096 x 14336: 229 -> 178 us);
//  * warpgroups of their own register budget (setmaxnreg): one of producers and issuers, two that
//    unpack (alternate stages), two of epilogue.
//
// Work: whole tiles, dealt round robin to the pairs; a remainder of at most half a wave is dealt as half
// tiles (one half each, the other issuer only hands slots on).  No tile is shared, so there are no
// partial sums and no workspace beyond the status word.
// Every wait is bounded: on expiry the CTA sets the status word and winds down.
//
// Measured against linear_tc_kernel<128>, the linear step alone, both in graphs on one box (tokens x channels x K, rank 64;
// us): 2048 x 14336 x 4096 133 -> 110; 4096 x 14336 x 4096 242 -> 197; 4096 x 4096 x 14336 204 -> 163; 4096 x 8192 x 8192
// 236 -> 181; 1500 x 4096 x 4096 37.6 -> 33.3; 1024 x 4096 x 4096 28.4 -> 23.7; 333 x 14336 x 4096 36.0 -> 32.6; 4096 x 28672 x
// 8192 at rank 256, under the power cap, 1173 -> 777.  A stage takes 1230 cycles
// against 1024 of MMAs (4096 x 4096 x 14336, rank 0); a tile of K = 4096 pays 5000 more for its turn-around, 11000
// with a low-rank term.  Sixteen epilogue warps (72 registers at launch) or both halves' sums read at once cost
// more in spilled registers than they saved there (gate projection 116 -> 122 ... 139 us).
#include "aser_common.cuh"
#include "sm100_ptx.cuh"

namespace aser {

namespace {

constexpr int kThreads = 640;                  // five warpgroups
constexpr int kRegsLaunch = 96;                // per thread at launch: 640 x 96 = 128 x (48 + 2 x 72 + 2 x 144)
constexpr int kKS = 2;                         // 128-column blocks per stage
constexpr int kNS = 4, kNW = 2;                // stages of the operand ring (A blocks and activations) and of the weight ring
constexpr int kHalf = 128, kHw = kHalf / 2;    // tokens per half; a CTA holds half of them
constexpr int kWStage = kKS * kWkBlockBytes;
constexpr int kXStage = kKS * kHalf * 128;  // a CTA holds half of each half's tokens
constexpr int kLbBytes = 128 * 128, kTBytes = (kHalf / 2) * 128;
constexpr int kYRow = 256;                     // bytes of a staged output row: 128 channels
constexpr int kOffX = 0, kOffW = kOffX + kNS * kXStage, kOffLr = kOffW + kNW * kWStage,
              kOffT = kOffLr + 2 * kLbBytes,             // T chunks: [half][slot]
              kOffBar = kOffT + 4 * kTBytes, kOffScale = kOffBar + 256;
constexpr int kSmemBytes = kOffScale + 2 * kHalf * 4 + 1024;
static_assert(2 * kHalf * kYRow <= kOffBar - kOffLr, "the outputs of a tile are staged where its low-rank operands were");
static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
constexpr long long kWaitClocks = 400000000ll; // about 0.2 s of SM clocks per wait

// Barriers.  "leader": waited on by the leader CTA's issuers, arrived on from both CTAs; "pair": arrived
// on in both CTAs by a commit of the leader's issuers; the others are local to a CTA.
//   W_FULL, W_FREE[s]    weight bytes landed -> unpack; in registers (count 4) -> weight producer
//   FULL[s]              leader, count 3: both CTAs' activation bytes landed, both CTAs' A blocks written -> issuers
//   FREE[s]              pair, count 2: both halves' MMAs of the stage retired -> unpack, activation producer
//   ACC_FULL[h]          pair: integer sums complete -> epilogue
//   D_READ[h]            leader: integer sums in registers -> issuer (the low-rank product may overwrite them)
//   LR_DONE[h]           pair: low-rank product complete -> epilogue
//   ACC_EMPTY[h]         leader: everything read -> issuer (next tile)
//   LR_FULL              a set of low-rank operands landed -> epilogue (converts T)
//   LR_CONV              leader, count 2: set converted in both CTAs -> issuers
//   LR_PART              pair: first of two sets multiplied by a half -> epilogue (loads the next set)
constexpr int B_W_FULL = 0, B_W_FREE = B_W_FULL + kNW, B_FULL = B_W_FREE + kNW, B_FREE = B_FULL + kNS,
              B_ACC_FULL = B_FREE + kNS, B_D_READ = B_ACC_FULL + 2, B_LR_DONE = B_D_READ + 2,
              B_ACC_EMPTY = B_LR_DONE + 2, B_LR_FULL = B_ACC_EMPTY + 2, B_LR_CONV = B_LR_FULL + 1,
              B_LR_PART = B_LR_CONV + 1, kNumBars = B_LR_PART + 1;
static_assert(kNumBars * 8 + 8 <= 256, "barrier area");
constexpr int kEpiWarps = 8, kEpiThreads = 256;

struct Params {
    LinearGroup g;         // one layer, or (GROUP) several of one rank
    int tile0[kMaxGroup];  // first tile of 256 rows of each layer
    const float* a_scale;
    int32_t* acc_debug;
    uint32_t* status;
    int M, r;
    int KB;                // 128-column blocks
    int NT, TT;            // tiles of 256 rows, whole token columns (see Plan)
    int full, cut, items;  // items [0, full): whole tiles; [full, full + 2 cut): the halves of further tiles; then the short ones
    int tt_outer;          // tile numbering: 1 = token tile outer
    CatSplit cat;
};

struct Maps { CUtensorMap lb[kMaxGroup], y[kMaxGroup]; };

// `step` tokens lie between the rows of the two CTAs: a whole tile's tokens are [CTA][half][rows], a
// single half's [CTA][rows].
// nt is the tile inside its layer.
struct Item { int nt, tok0, halves, step, layer; };

template <bool GROUP>
__device__ __forceinline__ Item get_item(const Params& p, int i) {
    Item w;
    int tt, part = 0;
    bool single = i >= p.full;
    if (i >= p.full + 2 * p.cut) {          // the last, short column of tokens
        w.nt = i - p.full - 2 * p.cut;
        tt = p.TT;
    } else {
        int tile = i;
        if (single) { tile = p.full + ((i - p.full) >> 1); part = (i - p.full) & 1; }
        if (p.tt_outer) { tt = tile / p.NT; w.nt = tile - tt * p.NT; }
        else { w.nt = tile / p.TT; tt = tile - w.nt * p.TT; }
    }
    w.tok0 = (2 * tt + part) * kHalf;
    w.halves = single ? 1 : 2;
    w.step = single ? kHw : kHalf;
    w.layer = 0;
    if (GROUP) {
#pragma unroll
        for (int l = 1; l < kMaxGroup; ++l)
            if (l < p.g.layers && w.nt >= p.tile0[l]) w.layer = l;
        w.nt -= p.tile0[w.layer];
    }
    return w;
}

struct Stop {
    volatile int* flag;    // shared
    uint32_t* status;      // global
};

// Bounded wait on a barrier phase: false after the limit or when another role of this CTA gave up.
// (In line: a call would keep the compiler from giving each warpgroup its register budget.)
__device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity, const Stop& stop) {
    uint32_t spins = 0;
    long long t0 = 0;
    while (!mbar_try_wait(bar, parity)) {
        if ((++spins & 255u) == 0) {
            if (*stop.flag) return false;
            const long long now = clock64();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > kWaitClocks) {
                *stop.flag = 1;
                atomicOr(stop.status, 1u);
                if (atomicCAS(stop.status + 1, 0u, 0x80000000u | threadIdx.x) == 0u) {    // which wait it was
                    stop.status[2] = blockIdx.x;
                    stop.status[3] = (bar & 1023u) >> 3;
                    stop.status[4] = parity;
                }
                return false;
            }
        }
    }
    return true;
}

__device__ __forceinline__ bool group_wait(uint32_t bar, uint32_t parity, const Stop& stop, bool leader, int group) {
    bool ok = true;
    if (leader) ok = wait(bar, parity, stop);
    return group == 0 ? named_bar_all(3, 128, ok) : named_bar_all(4, 128, ok);
}

// Copies in flight land before a CTA that gave up lets go of its shared memory.
__device__ __forceinline__ void let_copies_land() {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000) {}
}

template <bool DEBUG_ACC, bool GROUP>
__global__ void __launch_bounds__(kThreads, 1)
linear_pair_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_t,
                   const __grid_constant__ Maps maps, const __grid_constant__ Params p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = smem_u32(smem), bar0 = sbase + kOffBar;
    auto bar = [&](int i) { return bar0 + 8u * i; };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffBar + kNumBars * 8);
    volatile int* stop_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const Stop stop{stop_flag, p.status};
    const int chunks = (p.r + 63) / 64;
    const int stages = (p.KB + kKS - 1) / kKS;      // per item

    auto weights_of = [&](int item) {
        const Item w = get_item<GROUP>(p, item);
        const int NB = (p.g.N[w.layer] + kWkRows - 1) / kWkRows;
        int nb = 2 * w.nt + (int)rank;
        if (nb >= NB) nb = NB - 1;                 // rows past N: any weights, the results are dropped
        return p.g.Wk[w.layer] + (size_t)nb * p.KB * kWkBlockBytes;
    };
    auto load_weights = [&](const uint8_t* src, int kb, uint32_t s) {
        const uint32_t bytes = (p.KB - kb < kKS ? p.KB - kb : kKS) * kWkBlockBytes;
        mbar_arrive_expect_tx(bar(B_W_FULL + s), bytes);
        bulk_copy_g2s(sbase + kOffW + s * kWStage, src + (size_t)kb * kWkBlockBytes, bytes, bar(B_W_FULL + s));
    };

    if (warp == 0) {
        for (int i = lane; i < kNumBars; i += 32) {
            uint32_t count = 1;
            if (i >= B_W_FREE && i < B_FULL) count = 4;
            if (i >= B_FULL && i < B_FREE) count = 3;
            if ((i >= B_FREE && i < B_ACC_FULL) || i == B_LR_CONV) count = 2;
            if ((i >= B_D_READ && i < B_LR_DONE) || (i >= B_ACC_EMPTY && i < B_LR_FULL)) count = 2 * kEpiWarps;
            mbar_init(bar(i), count);
        }
        if (lane == 0) *stop_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {           // the first stages of weights leave before tensor memory is there
            const uint8_t* src = weights_of(pair);
            for (int c = 0; c < kNW && c < stages; ++c) load_weights(src, c * kKS, c);
        }
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    if (warp == 1 && lane == 0) {
        prefetch_tensormap(&map_x);
        prefetch_tensormap(&maps.y[0]);
        if (p.r > 0) { prefetch_tensormap(&maps.lb[0]); prefetch_tensormap(&map_t); }
    }
    tc_fence_before();
    __syncthreads();
    cluster_arrive();          // both CTAs' barriers are in place before anything is sent across
    cluster_wait();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t tm_a = tmem + 2 * kHalf;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
        if (warp == 0 && lane == 0) {
            // =================== weight producer ===================
            uint32_t c = 0;
            bool ok = true;
            for (int i = pair; i < p.items && ok; i += pairs) {
                const uint8_t* src = weights_of(i);
                for (int kb = 0; kb < p.KB; kb += kKS, ++c) {
                    if (i == pair && kb < kNW * kKS) continue;     // already on its way
                    ok = wait(bar(B_W_FREE + c % kNW), ((c / kNW) & 1) ^ 1, stop);
                    if (!ok) break;
                    load_weights(src, kb, c % kNW);
                }
            }
            if (!ok || *stop_flag) let_copies_land();
        } else if (warp == 1 && lane == 0) {
            // =================== activation producer ===================
            grid_dep_wait();       // Xq comes from the kernel launched before this one
            const uint32_t full0 = map_to_rank(bar(B_FULL), 0);
            uint32_t c = 0;
            bool ok = true;
            for (int i = pair; i < p.items && ok; i += pairs) {
                const Item w = get_item<GROUP>(p, i);
                for (int kb = 0; kb < p.KB; kb += kKS, ++c) {
                    const uint32_t s = c % kNS;
                    ok = wait(bar(B_FREE + s), ((c / kNS) & 1) ^ 1, stop);
                    if (!ok) break;
                    // both CTAs' bytes are counted on the leader's barrier; blocks past K and tokens past M read as zero
                    if (rank == 0) mbar_arrive_expect_tx(bar(B_FULL + s), 2 * kKS * kHalf * 128);
                    tma_load_3d_pair(sbase + kOffX + s * kXStage, &map_x, 0, w.tok0 + (int)rank * w.step, kb, full0 + 8u * s);
                }
            }
            if (!ok || *stop_flag) let_copies_land();
        } else if (warp >= 2 && lane == 0 && rank == 0) {
            // =================== MMA issuer of one half (leader CTA) ===================
            const int h = warp - 2;
            const uint32_t d = tmem + h * kHalf;
            constexpr uint32_t idesc_i8 = make_idesc(2, 1, 256, kHalf), idesc_f16 = make_idesc(1, 0, 256, kHalf);
            constexpr uint32_t xblock = (kHalf * 128) >> 4;                 // descriptor step between a stage's blocks
            const uint32_t xoff = h * (kHw) * 128;
            uint32_t ca = 0, done = 0, conv = 0;
            bool ok = true, ready = false;     // ready: stage ca was seen complete already
            // the chunks [c0, c1) of the set that occupies the slots
            auto multiply = [&](int c0, int c1, bool fresh) {
                tc_fence_after();
                for (int c = c0; c < c1; ++c) {
                    const uint64_t ad = smem_desc_sw128(sbase + kOffLr + (c & 1) * kLbBytes);
                    const uint64_t bd = smem_desc_sw128(sbase + kOffT + (h * 2 + (c & 1)) * kTBytes);
                    int steps = (p.r - c * 64) / 16;
                    if (steps > 4) steps = 4;
                    for (int kk = 0; kk < steps; ++kk)
                        mma_f16_ss_pair(d, ad + 2 * kk, bd + 2 * kk, idesc_f16, (fresh && c == c0 && kk == 0) ? 0u : 1u);
                }
            };
            for (int i = pair; i < p.items && ok; i += pairs) {
                const Item w = get_item<GROUP>(p, i);
                const bool mine = h < w.halves;
                if (mine) ok = wait(bar(B_ACC_EMPTY + h), (done & 1) ^ 1, stop);
                if (!ok) break;
                for (int kb = 0; kb < p.KB; kb += kKS, ++ca) {
                    const int s = ca % kNS, s1 = (ca + 1) % kNS;
                    if (!ready) ok = wait(bar(B_FULL + s), (ca / kNS) & 1, stop);
                    if (!ok) break;
                    ready = false;
                    if (mine) {
                        tc_fence_after();
                        const uint64_t xdesc = smem_desc_sw128(sbase + kOffX + s * kXStage + xoff);
                        const uint32_t a = tm_a + s * (kKS * 32);
                        if (kb + kKS <= p.KB) {
                            ready = mma_i8_stage_pair(d, a, xdesc, xblock, idesc_i8, kb != 0 ? 1u : 0u, bar(B_FULL + s1),
                                                      ((ca + 1) / kNS) & 1);
                        } else {
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk)
                                mma_i8_ts_pair(d, a + kk * 8, xdesc + 2 * kk, idesc_i8, (kb | kk) != 0 ? 1u : 0u);
                        }
                    }
                    tc_commit_pair(bar(B_FREE + s));       // a half without tokens only hands the slot on
                }
                if (!ok) break;
                if (mine) {
                    tc_commit_pair(bar(B_ACC_FULL + h));
                    if (chunks > 0) {
                        // The low-rank product into the same columns, once their sums are in registers.  Up to two chunks
                        // are one set for both halves; more are two sets for each half in turn, so that every half
                        // adds its chunks in order (the same sums as linear_tc.cu, whichever kernel serves a shape).
                        const uint32_t first = conv + (chunks > 2 ? 2 * h : 0);
                        // one set: converted long ago, so it is looked at while the epilogue reads the sums.  (With more
                        // sets a half skips phases of LR_CONV, and only D_READ says that those are over.)
                        if (chunks <= 2) ok = wait(bar(B_LR_CONV), first & 1, stop);
                        ok = ok && wait(bar(B_D_READ + h), done & 1, stop);
                        if (chunks > 2) ok = ok && wait(bar(B_LR_CONV), first & 1, stop);
                        if (!ok) break;
                        multiply(0, chunks < 2 ? chunks : 2, true);
                        if (chunks > 2) {
                            tc_commit_pair(bar(B_LR_PART));
                            ok = wait(bar(B_LR_CONV), (first + 1) & 1, stop);
                            if (!ok) break;
                            multiply(2, chunks, false);
                        }
                        tc_commit_pair(bar(B_LR_DONE + h));
                    }
                    ++done;
                }
                if (chunks > 0) conv += chunks <= 2 ? 1 : 2 * w.halves;      // sets per item
            }
        }
    } else if (warp < 12) {
        // =================== unpack: int4 -> int8 (x16) into tensor memory ===================
        asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
        const int q = warp & 3, row = q * 32 + lane, group = (warp - 4) >> 2;
        const bool leader = (threadIdx.x & 127) == 0;
        const uint32_t full0 = map_to_rank(bar(B_FULL), 0);
        const int items = (p.items - pair + pairs - 1) / pairs;
        const uint32_t total = (uint32_t)items * (uint32_t)stages;
        // the packed words of this group's next stage are fetched while the MMAs still use its slot
        uint4 raw[kKS][4];
        auto fetch = [&](uint32_t c) {
            const uint32_t s = c % kNW;                     // = group
            if (!group_wait(bar(B_W_FULL + s), (c / kNW) & 1, stop, leader, group)) return false;
            const uint8_t* src = smem + kOffW + s * kWStage + row * 16;
#pragma unroll
            for (int j = 0; j < kKS; ++j)                   // a ragged stage's second block: whatever is there
#pragma unroll
                for (int s4 = 0; s4 < 4; ++s4) raw[j][s4] = *reinterpret_cast<const uint4*>(src + j * kWkBlockBytes + s4 * 2048);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_W_FREE + s));
            return true;
        };
        bool ok = (uint32_t)group < total ? fetch(group) : true;
        for (uint32_t c = group; c < total && ok; c += 2) {
            const uint32_t s = c % kNS;
            const uint32_t a = tm_a + s * (kKS * 32) + ((uint32_t)(q * 32) << 16);
            ok = group_wait(bar(B_FREE + s), ((c / kNS) & 1) ^ 1, stop, leader, group);
            if (!ok) break;
            tc_fence_after();
#pragma unroll
            for (int j = 0; j < 2 * kKS; ++j) {              // 64 columns at a time
                uint32_t v[16];
#pragma unroll
                for (int s4 = 0; s4 < 2; ++s4) {
                    const uint4 x = raw[j >> 1][(j & 1) * 2 + s4];
                    const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        v[s4 * 8 + 2 * e] = (xs[e] << 4) & 0xF0F0F0F0u;      // columns c0 .. c0+3
                        v[s4 * 8 + 2 * e + 1] = xs[e] & 0xF0F0F0F0u;         // columns c0+4 .. c0+7
                    }
                }
                tmem_st16(a + j * 16, v);
            }
            tmem_wait_st();
            tc_fence_before();
            if (group == 0) named_bar_sync(3, 128);
            else named_bar_sync(4, 128);
            if (leader) mbar_arrive_cluster(full0 + 8u * s);
            if (c + 2 < total) ok = fetch(c + 2);
        }
    } else {
        // =================== epilogue ===================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 144;");
        const int q = warp & 3, side = (warp - 12) >> 2;      // side: the CTA whose tokens this warp's columns are
        const int et = threadIdx.x - 12 * 32;
        const uint32_t lane_sel = (uint32_t)(q * 32) << 16;
        const uint32_t dread0 = map_to_rank(bar(B_D_READ), 0), empty0 = map_to_rank(bar(B_ACC_EMPTY), 0),
                       conv0 = map_to_rank(bar(B_LR_CONV), 0);
        float* scales = reinterpret_cast<float*>(smem + kOffScale);
        uint32_t done = 0, sets = 0, parts = 0;               // done: bit h = parity of the half's items
        bool ok = true;
        grid_dep_wait();           // a_scale and T come from the kernel launched before this one
        // a set of low-rank operands: chunks [c0, c1), T of the halves in the mask (one thread)
        auto load_set = [&](const Item& w, int c0, int c1, int mask) {
            const int row0 = (2 * w.nt + (int)rank) * 128, t_col = p.g.t_col[w.layer] + cat_layer(p.cat, w.nt * 256) * p.r;
            mbar_arrive_expect_tx(bar(B_LR_FULL), (c1 - c0) * (kLbBytes + ((mask & 1) + (mask >> 1)) * kHw * 128));
            for (int c = c0; c < c1; ++c) {
                tma_load_2d(sbase + kOffLr + (c & 1) * kLbBytes, &maps.lb[w.layer], c * 64, row0, bar(B_LR_FULL));
                for (int h = 0; h < 2; ++h)
                    if (mask >> h & 1)
                        tma_load_2d(sbase + kOffT + (h * 2 + (c & 1)) * kTBytes, &map_t, c * 64 + t_col,
                                    w.tok0 + (int)rank * w.step + h * kHw, bar(B_LR_FULL));
            }
        };
        // ... of an item's first set
        auto load_first = [&](const Item& w) {
            if (chunks <= 2) load_set(w, 0, chunks, w.halves == 2 ? 3 : 1);
            else load_set(w, 0, 2, 1);
        };
        // T of the set just landed: bf16 -> fp16 in place (exact in the fp16 normal range)
        auto convert_set = [&](int c0, int c1, int mask) {
            bool landed = true;
            if (et == 0) landed = wait(bar(B_LR_FULL), sets & 1, stop);
            ++sets;
            if (!named_bar_all(1, kEpiThreads, landed)) return false;
            for (int h = 0; h < 2; ++h) {
                if (!(mask >> h & 1)) continue;
                for (int i = et; i < (c1 - c0) * kHw * 8; i += kEpiThreads) {
                    const int c = i >= kHw * 8 ? 1 : 0, e = i - c * kHw * 8;
                    uint4* t = reinterpret_cast<uint4*>(smem + kOffT + (h * 2 + c) * kTBytes) + e;
                    const uint4 raw = *t;
                    const uint32_t in[4] = {raw.x, raw.y, raw.z, raw.w};
                    uint32_t out[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const __half2 v = __floats2half2_rn(__uint_as_float(in[k] << 16), __uint_as_float(in[k] & 0xFFFF0000u));
                        out[k] = *reinterpret_cast<const uint32_t*>(&v);
                    }
                    *t = make_uint4(out[0], out[1], out[2], out[3]);
                }
            }
            fence_proxy_async_smem();
            named_bar_sync(1, kEpiThreads);
            if (et == 0) mbar_arrive_cluster(conv0);
            return true;
        };
        int i = pair;
        Item w = {};
        if (i < p.items) w = get_item<GROUP>(p, i);
        if (chunks > 0 && i < p.items && et == 0) load_first(w);
        while (i < p.items && ok) {
            // the item after this one (its first operands are loaded as soon as their place is free)
            const int i_next = i + pairs;
            Item next = {};
            if (i_next < p.items) next = get_item<GROUP>(p, i_next);
            const int n0 = (2 * w.nt + (int)rank) * 128, n = n0 + q * 32 + lane, N = p.g.N[w.layer];
            const float ws16 = (n < N ? __ldg(p.g.w_scale[w.layer] + n) : 0.f) * 0.0625f;      // the sums hold 16 q x
            {   // token scales in the order of the accumulator's columns: [half][CTA][rows]
                const int h = et >= kHalf ? 1 : 0, col = et - h * kHalf, cta = col >= kHw ? 1 : 0;
                const int tok = w.tok0 + cta * w.step + h * kHw + (col - cta * kHw);
                if (et < 2 * kHalf) scales[et] = (h < w.halves && tok < p.M) ? __ldg(p.a_scale + tok) : 0.f;
            }
            if (chunks > 0) ok = convert_set(0, chunks < 2 ? chunks : 2, chunks <= 2 && w.halves == 2 ? 3 : 1);
            else named_bar_sync(1, kEpiThreads);          // the scales are there
            if (!ok) break;
            uint32_t y[2][4][8];           // fp16 pairs of both halves: stored when both accumulators are free
            // A warp whose wait gave up does no more work but still takes part in every barrier of the item, which
            // ends with all warps going on or giving up together.
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h >= w.halves) continue;
                const uint32_t d = tmem + h * kHalf + lane_sel + side * kHw;
                if (h == 1 && chunks > 2) {
                    const bool converted = convert_set(0, 2, 2);
                    ok = ok && converted;
                }
                if (ok) {
                    if (lane == 0) ok = wait(bar(B_ACC_FULL + h), (done >> h) & 1, stop);
                    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                }
                uint32_t v[4][16];
                if (ok) {
                    tc_fence_after();
#pragma unroll
                    for (int c = 0; c < 4; ++c) tmem_ld16(d + c * 16, v[c]);
                    tmem_wait_ld_all();
#pragma unroll
                    for (int c = 0; c < 4; ++c) tmem_use(v[c]);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster((chunks > 0 ? dread0 : empty0) + 8u * h);
                    if (DEBUG_ACC) {
                        const int tok = w.tok0 + side * w.step + h * kHw;
#pragma unroll
                        for (int c = 0; c < 4; ++c)
#pragma unroll
                            for (int j = 0; j < 16; ++j)
                                if (tok + c * 16 + j < p.M && n < N)
                                    p.acc_debug[(size_t)(tok + c * 16 + j) * N + n] = ((int)v[c][j]) >> 4;
                    }
                }
                if (chunks > 2) {
                    // the half's second set
                    bool free = ok;
                    if (et == 0 && free) {
                        free = wait(bar(B_LR_PART), parts & 1, stop);
                        if (free) load_set(w, 2, chunks, 1 << h);
                    }
                    ++parts;
                    ok = named_bar_all(1, kEpiThreads, free);
                    if (ok) ok = convert_set(2, chunks, 1 << h);
                }
                if (chunks > 0 && ok) {
                    if (lane == 0) ok = wait(bar(B_LR_DONE + h), (done >> h) & 1, stop);
                    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                    tc_fence_after();
                    // the first half is through: the second half's first set
                    if (ok && chunks > 2 && h == 0 && w.halves == 2 && et == 0) load_set(w, 0, 2, 2);
                }
                if (!ok) continue;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t f[16];
                    if (chunks > 0) {
                        tmem_ld16(d + c * 16, f);
                        tmem_wait_ld(f);
                    }
                    const float4* ap = reinterpret_cast<const float4*>(scales + h * kHalf + side * kHw + c * 16);
#pragma unroll
                    for (int j4 = 0; j4 < 4; ++j4) {
                        const float4 a4 = ap[j4];
                        const float as[4] = {a4.x, a4.y, a4.z, a4.w};
                        float o[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            o[j] = fmaf((float)(int)v[c][4 * j4 + j], as[j] * ws16, chunks > 0 ? __uint_as_float(f[4 * j4 + j]) : 0.f);
                        const __half2 h0 = __floats2half2_rn(o[0], o[1]), h1 = __floats2half2_rn(o[2], o[3]);
                        y[h][c][2 * j4] = *reinterpret_cast<const uint32_t*>(&h0);
                        y[h][c][2 * j4 + 1] = *reinterpret_cast<const uint32_t*>(&h1);
                    }
                }
                if (chunks > 0) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(empty0 + 8u * h);
                }
                done ^= 1u << h;
            }
            // The outputs, [half][CTA][token][128 channels], are staged where the low-rank operands were: every warp
            // has seen the item's last low-rank product retire.  They leave as tensor stores, which clip at M and N.
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h >= w.halves || !ok) continue;
                uint16_t* stage = reinterpret_cast<uint16_t*>(smem + kOffLr) + ((h * 2 + side) * kHw) * (kYRow / 2) + q * 32 + lane;
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        stage[(c * 16 + 2 * j) * (kYRow / 2)] = (uint16_t)(y[h][c][j] & 0xFFFFu);
                        stage[(c * 16 + 2 * j + 1) * (kYRow / 2)] = (uint16_t)(y[h][c][j] >> 16);
                    }
            }
            fence_proxy_async_smem();
            ok = named_bar_all(1, kEpiThreads, ok);
            if (!ok) break;
            if (et == 0) {
                if (n0 < N) {
                    for (int b = 0; b < 2 * w.halves; ++b) {
                        const int tok = w.tok0 + (b & 1) * w.step + (b >> 1) * kHw;
                        if (tok < p.M) tma_store_2d_tile(&maps.y[w.layer], n0, tok, sbase + kOffLr + b * kHw * kYRow);
                    }
                    bulk_store_commit();
                    bulk_store_wait_read();
                }
                if (chunks > 0 && i_next < p.items) load_first(next);
            }
            if (chunks == 0) named_bar_sync(1, kEpiThreads);      // the staging area has been read
            w = next;
            i = i_next;
        }
        if (et == 0) {
            bulk_store_wait_all();
            if (!ok || *stop_flag) let_copies_land();
        }
    }

    // =================== teardown ===================
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    cluster_arrive();          // nothing is sent to a CTA that has left
    cluster_wait();
    if (warp == 2) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// The deal of the work.  A column of 256 tokens is whole when it has more than 128, the last may be short:
// short columns give single halves, and the tiles of the last, incomplete wave may be cut into single
// halves.  Items go to the pairs round robin, whole tiles first.  The cost is the load of the busiest pair in
// cycles per stage of 256 columns: 1500 for a whole tile, 1300 for a single half (measured, the epilogue
// spread over the stages; narrower tiles, bound by the unpacking, cost no less).
struct Plan { int NT, TT, full, cut, items; long long cost; };

Plan make_plan(int M, int NT, int pairs) {
    constexpr long long whole = 1500, single = 1300;
    const int columns = (M + 2 * kHalf - 1) / (2 * kHalf), last = M - (columns - 1) * 2 * kHalf;
    const int TT = last <= kHalf ? columns - 1 : columns, tiles = NT * TT;
    const int shorts = last <= kHalf ? NT : 0;
    Plan best = {};
    for (int cut = 0; cut <= 1; ++cut) {
        Plan c;
        c.NT = NT; c.TT = TT;
        c.cut = cut ? tiles % pairs : 0;
        c.full = tiles - c.cut;
        c.items = c.full + 2 * c.cut + shorts;
        // all pairs have full / pairs whole tiles, the first full % pairs one more; singles are dealt on from there
        const int rest = c.full % pairs, singles = c.items - c.full, free_pairs = pairs - rest;
        const int second = singles > free_pairs ? (singles - free_pairs + pairs - 1) / pairs : 0;
        const long long with_extra = rest > 0 ? whole + second * single : 0;
        const long long without = (singles > 0 ? 1 + (singles > pairs ? (singles - 1) / pairs : 0) : 0) * single;
        c.cost = (long long)(c.full / pairs) * whole + (with_extra > without ? with_extra : without);
        if (cut == 0 || c.cost < best.cost) best = c;
    }
    return best;
}

// Whether the kernel can run as it was built: the warpgroups' budgets add up to what the block is launched with and to
// nothing else, so a compiler that gives a thread another number of registers leaves every shape to linear_tc.
template <bool DEBUG_ACC, bool GROUP>
bool configure(int dev) {
    static int state[kMaxDevices] = {0};         // 1: ready, 2: not usable
    if (state[dev] == 0) {
        cudaFuncAttributes a;
        cudaError_t e = cudaFuncGetAttributes(&a, linear_pair_kernel<DEBUG_ACC, GROUP>);
        const bool fits = e == cudaSuccess && a.numRegs == kRegsLaunch;
        if (fits) e = cudaFuncSetAttribute(linear_pair_kernel<DEBUG_ACC, GROUP>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        if (e != cudaSuccess) (void)cudaGetLastError();
        state[dev] = fits && e == cudaSuccess ? 1 : 2;
    }
    return state[dev] == 1;
}

}  // namespace

// The estimates were fitted to whole forward passes (M 48 ... 2048, seven layer shapes): pairs win from about
// 600 tokens on nearly everywhere and below that where they fill the part or where linear_tc would have to
// share its tiles (linear step, 333 x 2048 x 2048: 14.0 against 25.5 us, 160 x 28672 x 8192: 70 / 77), linear_tc where few long
// tiles have to be split over the part (256 x 4096 x 14336: 31 us; the whole pass was 10 us longer with pairs),
// which pairs do not do.  Looked at again on 920 points (18 layer shapes of 1152 to 28672 columns, 65 to 4096 tokens drawn,
// ranks 0, 64 and 128; linear step in a graph): 1.153 times as fast as linear_tc alone in the geometric mean, four points slower
// by more than 1.5 %, the worst 6 % (1027 x 8192 x 28672: a short column of three tokens costs a pass over its weights).
bool linear_pair_prefers(int M, int N, int K, const CatSplit& cat) {
    if (M < kLinearPairMinTokens) return false;
    if (cat.layers > 1 && ((cat.b1 | (cat.layers > 2 ? cat.b2 : 0) | (cat.layers > 3 ? cat.b3 : 0)) & 255)) return false;
    int num_sms = 0, dev = 0;
    if (device_sm_count(&num_sms) != ASER_OK || num_sms < 2 || current_device(&dev) != ASER_OK) return false;
    const long long stages = (K / kWkCols + kKS - 1) / kKS;
    if (make_plan(M, (N + 255) / 256, num_sms / 2).cost * stages + 12000 >= linear_tc_estimate(M, N, K, num_sms)) return false;
    return configure<false, false>(dev) && configure<true, false>(dev);
}

// Layers that would each be served by this kernel, of one rank: one launch deals the tiles of all of them (two layers of 14336 x
// 4096, 333 tokens: 56 whole and 56 half tiles each on 74 pairs, so a whole and a half for the busiest pair, twice; together
// 112 and 112, three items at most).
bool linear_pair_groups(const LinearGroup& g, int M, int K) {
    int dev = 0;
    if (g.layers < 2 || g.layers > kMaxGroup || current_device(&dev) != ASER_OK) return false;
    for (int l = 0; l < g.layers; ++l)
        if (g.r[l] != g.r[0] || g.N[l] <= 0 || linear_split_prefers(M, g.N[l], K) || !linear_pair_prefers(M, g.N[l], K, CatSplit()))
            return false;
    return configure<false, true>(dev);
}

int launch_linear_pair_group(const int8_t* Xq, const float* a_scale, const __nv_bfloat16* T, int M, int K, const LinearGroup& g,
                             int32_t* acc_debug, void* workspace, cudaStream_t st, bool overlap_prev, int ldt, CatSplit cat) {
    if (g.layers > 1 && (acc_debug || cat.layers > 1))
        return record_error(ASER_ERR_SHAPE, "linear_pair: neither accumulators nor fused layers of a group");
    int num_sms = 0;
    int rc = device_sm_count(&num_sms);
    if (rc != ASER_OK) return rc;
    const int pairs = num_sms / 2 > 0 ? num_sms / 2 : 1, r = g.r[0];
    Params p = {};
    p.g = g;
    int NT = 0, t_cols = 0;
    long long rows = 0;
    for (int l = 0; l < g.layers; ++l) {
        p.tile0[l] = NT;
        NT += (g.N[l] + 255) / 256;
        rows += g.N[l];
        if (g.t_col[l] + r * cat.layers > t_cols) t_cols = g.t_col[l] + r * cat.layers;
    }
    const Plan plan = make_plan(M, NT, pairs);
    CUtensorMap mx, mt;
    Maps maps;
    rc = encode_map_blocks(&mx, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Xq, M, K, kHalf, kKS);
    if (rc != ASER_OK) return rc;
    mt = mx;
    if (r > 0) {
        rc = encode_map_2d_ld(&mt, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, T, M, t_cols, ldt > 0 ? ldt : t_cols, kHw, 64,
                              CU_TENSOR_MAP_SWIZZLE_128B);
        if (rc != ASER_OK) return rc;
    }
    for (int l = 0; l < kMaxGroup; ++l) {
        if (l >= g.layers) { maps.y[l] = maps.y[0]; maps.lb[l] = maps.lb[0]; continue; }
        rc = encode_map_2d(&maps.y[l], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, g.Y[l], M, g.N[l], kHw, 128, CU_TENSOR_MAP_SWIZZLE_NONE);
        if (rc != ASER_OK) return rc;
        maps.lb[l] = mx;
        if (r > 0) rc = encode_map_2d(&maps.lb[l], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, g.LB[l], g.N[l], r, 128, 64, CU_TENSOR_MAP_SWIZZLE_128B);
        if (rc != ASER_OK) return rc;
    }
    p.a_scale = a_scale; p.acc_debug = acc_debug;
    p.status = static_cast<uint32_t*>(workspace);
    p.M = M; p.r = r;
    p.KB = K / kWkCols;
    p.NT = plan.NT; p.TT = plan.TT; p.full = plan.full; p.cut = plan.cut; p.items = plan.items;
    // the smaller of the two operand sets stays in L2 while the other is streamed (as in linear_tc.cu)
    p.tt_outer = ((long long)M * K > rows * K / 2) ? 1 : 0;
    p.cat = cat;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (plan.items < pairs ? plan.items : pairs), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap_prev ? 2 : 1;
    const cudaError_t e = g.layers > 1 ? cudaLaunchKernelEx(&cfg, linear_pair_kernel<false, true>, mx, mt, maps, p)
                          : acc_debug  ? cudaLaunchKernelEx(&cfg, linear_pair_kernel<true, false>, mx, mt, maps, p)
                                       : cudaLaunchKernelEx(&cfg, linear_pair_kernel<false, false>, mx, mt, maps, p);
    if (e != cudaSuccess) return record_cuda_error(e, "linear_pair_kernel");
    return check_launch("linear_pair_kernel");
}

int launch_linear_pair(const int8_t* Xq, const float* a_scale, const uint8_t* Wk, const float* w_scale,
                       const __nv_bfloat16* T, const __half* LB, int M, int N, int K, int r, __half* Y,
                       int32_t* acc_debug, void* workspace, cudaStream_t st, bool overlap_prev, int ldt, CatSplit cat) {
    LinearGroup g = {};
    g.layers = 1;
    g.Wk[0] = Wk; g.w_scale[0] = w_scale; g.LB[0] = LB; g.Y[0] = Y;
    g.N[0] = N; g.r[0] = r;
    return launch_linear_pair_group(Xq, a_scale, T, M, K, g, acc_debug, workspace, st, overlap_prev, ldt, cat);
}

}  // namespace aser
