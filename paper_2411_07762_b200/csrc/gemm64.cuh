// fp64 matrix products for the offline construction step, on the fp64 tensor-core instruction.
//
//   C[m, n] = a0 * A[m, k] B + a1 * X1 + a2 * X2,   B given as [n, k] (TB) or as [k, n] rows
//
// The products of the construction are a tall or wide matrix (the weight error, 4096 x 4608 at the
// usual sizes) against 48 to 384 vectors.  What bounds them is the fp64 rate of the part (37 TFLOP/s
// measured for mma.sync f64 with operands in registers, 32 for fma); 96 rows against 134 MB of fp64
// are 87 us of arithmetic and 21 us of HBM.  So:
//  * a CTA owns 16 MT x 128 results (MT up to 6: all the vectors of a rank-64 layer), eight warps
//    take 16 columns each and hold the whole column strip of accumulators, so a fragment of B is
//    loaded once and a fragment of A is shared by two instructions;
//  * four stages of 16 k-columns arrive by cp.async; rows are padded to 20 (or 132) doubles, which
//    makes the 8-byte fragment loads of a half warp hit 32 different banks;
//  * k is split over CTAs where the tiles alone do not fill the part; the pieces are summed in order
//    by a second kernel, which also applies a1 X1 + a2 X2 (the result does not depend on timing).
// Measured, 96 x 4608 x 4096 and its transpose: 130 us (28 TFLOP/s); the 64 x 64 fma kernel, which
// one CTA per 64 columns left most SMs without, took 1500 us.
#pragma once
#include "aser_common.cuh"

namespace aser {
namespace gemm64 {

constexpr int kTN = 128, kTK = 16, kStages = 4, kThreads = 256;
constexpr int kLdK = kTK + 4;        // row pitch of a k-contiguous tile, in doubles
constexpr int kLdN = kTN + 4;        // row pitch of an n-contiguous tile

struct Args {
    const double *A, *B, *B2;        // batch 1 (apply a factor to two matrices) reads B2, writes C2
    double *C, *C2;
    long long lda, ldb, ldc;
    int m, n, k;
    int k_per_split;                 // a multiple of kTK
    int splits;                      // > 1: C is [splits][m][n], the raw sums
    const double *X1, *X2;           // [m, n] with pitch ldc, or null
    double a0, a1, a2;
    const double* a0_div;            // a0 is divided by *a0_div (or null)
    bool side;                       // the launch after this one may run beside it
    bool beside;                     // launched to run beside a side launch, and not over before that one is
};

template <int MT, bool TB>
constexpr int smem_bytes() {
    return kStages * (16 * MT * kLdK + (TB ? kTN * kLdK : kTK * kLdN)) * 8;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const double* src, bool ok) {
    const int bytes = ok ? 16 : 0;   // 0: the destination is filled with zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

template <int MT, bool TB>
__global__ void __launch_bounds__(kThreads, 1) gemm_kernel(const Args g) {
    constexpr int TM = 16 * MT;
    constexpr int kAElems = TM * kLdK, kBElems = TB ? kTN * kLdK : kTK * kLdN;
    extern __shared__ __align__(16) double sm[];
    if (g.side) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    const int n0 = blockIdx.x * kTN, m0 = blockIdx.y * TM;
    const int split = g.splits > 1 ? (int)blockIdx.z : 0;
    const bool second = g.splits == 1 && blockIdx.z == 1;
    const double* Bp = second ? g.B2 : g.B;
    const int k_begin = split * g.k_per_split;
    const int k_end = (k_begin + g.k_per_split < g.k) ? k_begin + g.k_per_split : g.k;
    const int steps = k_end > k_begin ? (k_end - k_begin + kTK - 1) / kTK : 0;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sm);

    auto load = [&](int st, int slot) {
        const int k0 = k_begin + st * kTK;
        const uint32_t sa = sbase + (uint32_t)(slot * (kAElems + kBElems)) * 8u, sb = sa + kAElems * 8u;
#pragma unroll
        for (int i = tid; i < TM * (kTK / 2); i += kThreads) {
            const int r = i / (kTK / 2), c = (i % (kTK / 2)) * 2;
            const bool ok = m0 + r < g.m && k0 + c < k_end;
            cp_async16(sa + (uint32_t)(r * kLdK + c) * 8u, ok ? g.A + (long long)(m0 + r) * g.lda + k0 + c : g.A, ok);
        }
        if (TB) {
#pragma unroll
            for (int i = tid; i < kTN * (kTK / 2); i += kThreads) {
                const int r = i / (kTK / 2), c = (i % (kTK / 2)) * 2;
                const bool ok = n0 + r < g.n && k0 + c < k_end;
                cp_async16(sb + (uint32_t)(r * kLdK + c) * 8u, ok ? Bp + (long long)(n0 + r) * g.ldb + k0 + c : Bp, ok);
            }
        } else {
#pragma unroll
            for (int i = tid; i < kTK * (kTN / 2); i += kThreads) {
                const int r = i / (kTN / 2), c = (i % (kTN / 2)) * 2;
                const bool ok = k0 + r < k_end && n0 + c < g.n;
                cp_async16(sb + (uint32_t)(r * kLdN + c) * 8u, ok ? Bp + (long long)(k0 + r) * g.ldb + n0 + c : Bp, ok);
            }
        }
    };

    double acc[MT][2][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.0;

#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) {
        if (s < steps) load(s, s);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int st = 0; st < steps; ++st) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
        __syncthreads();             // stage st has landed for all, stage st - 1 has been read by all
        if (st + kStages - 1 < steps) load(st + kStages - 1, (st + kStages - 1) % kStages);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const double* As = sm + (st % kStages) * (kAElems + kBElems);
        const double* Bs = As + kAElems;
#pragma unroll
        for (int kk = 0; kk < kTK; kk += 8) {
            double b[2][2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int col = warp * 16 + j * 8 + gq;
                b[j][0] = TB ? Bs[col * kLdK + kk + tq] : Bs[(kk + tq) * kLdN + col];
                b[j][1] = TB ? Bs[col * kLdK + kk + tq + 4] : Bs[(kk + tq + 4) * kLdN + col];
            }
#pragma unroll
            for (int i = 0; i < MT; ++i) {
                const double* ap = As + (i * 16 + gq) * kLdK + kk + tq;
                const double a0 = ap[0], a1 = ap[8 * kLdK], a2 = ap[4], a3 = ap[8 * kLdK + 4];
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    asm volatile(
                        "mma.sync.aligned.m16n8k8.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                        "{%0,%1,%2,%3};"
                        : "+d"(acc[i][j][0]), "+d"(acc[i][j][1]), "+d"(acc[i][j][2]), "+d"(acc[i][j][3])
                        : "d"(a0), "d"(a1), "d"(a2), "d"(a3), "d"(b[j][0]), "d"(b[j][1]));
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");

    const double a0 = g.splits > 1 ? 1.0 : (g.a0_div ? g.a0 / *g.a0_div : g.a0);
    double* Cp = second ? g.C2 : g.C;
    const long long ldc = g.splits > 1 ? g.n : g.ldc;
    if (g.splits > 1) Cp += (long long)split * g.m * g.n;
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = m0 + i * 16 + gq + 8 * h, c = n0 + warp * 16 + j * 8 + 2 * tq;
                if (r >= g.m || c >= g.n) continue;            // n is even
                double2 v = make_double2(a0 * acc[i][j][2 * h], a0 * acc[i][j][2 * h + 1]);
                const long long o = (long long)r * ldc + c;
                if (g.splits == 1 && g.X1) {
                    const double2 x = *reinterpret_cast<const double2*>(g.X1 + o);
                    v.x = fma(g.a1, x.x, v.x); v.y = fma(g.a1, x.y, v.y);
                }
                if (g.splits == 1 && g.X2) {
                    const double2 x = *reinterpret_cast<const double2*>(g.X2 + o);
                    v.x = fma(g.a2, x.x, v.x); v.y = fma(g.a2, x.y, v.y);
                }
                *reinterpret_cast<double2*>(Cp + o) = v;
            }
    if (g.beside && (blockIdx.x | blockIdx.y | blockIdx.z) == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// C = a0 * (sum of the pieces, in order) + a1 X1 + a2 X2; C and X1, X2 have the pitch ldc.
__global__ void __launch_bounds__(256) reduce_kernel(const double* __restrict__ part, const Args g) {
    const long long pairs = (long long)g.m * g.n / 2, e = (long long)blockIdx.x * 256 + threadIdx.x;
    if (e >= pairs) return;
    const double2* p = reinterpret_cast<const double2*>(part) + e;
    double2 s = p[0];
#pragma unroll 4
    for (int i = 1; i < g.splits; ++i) {
        const double2 v = p[(long long)i * pairs];
        s.x += v.x; s.y += v.y;
    }
    const double a0 = g.a0_div ? g.a0 / *g.a0_div : g.a0;
    const long long o = (2 * e) / g.n * g.ldc + (2 * e) % g.n;
    s.x *= a0; s.y *= a0;
    if (g.X1) {
        const double2 x = *reinterpret_cast<const double2*>(g.X1 + o);
        s.x = fma(g.a1, x.x, s.x); s.y = fma(g.a1, x.y, s.y);
    }
    if (g.X2) {
        const double2 x = *reinterpret_cast<const double2*>(g.X2 + o);
        s.x = fma(g.a2, x.x, s.x); s.y = fma(g.a2, x.y, s.y);
    }
    *reinterpret_cast<double2*>(g.C + o) = s;
}

// Rows of a CTA: the fewest row tiles of at most 96, then as few 16-row strips as cover them.
inline int row_strips(int m) {
    const int tiles = (m + 95) / 96, strips = ((m + 15) / 16 + tiles - 1) / tiles;
    return strips < 3 ? 3 : strips;
}

// Pieces that k is cut into: the estimate counts whole waves of CTAs (one per SM) in 16-column
// steps, a fixed cost of about eight steps per CTA, and the traffic of the pieces.
inline int split_count(int m, int n, int k, int num_sms) {
    const int mt = row_strips(m);
    const long long tiles = (long long)((m + 16 * mt - 1) / (16 * mt)) * ((n + kTN - 1) / kTN);
    const int steps = (k + kTK - 1) / kTK;
    int best = 1;
    double best_cost = 1e30;
    for (int s = 1; s <= 64 && (s == 1 || steps / s >= 4); ++s) {
        const long long waves = (tiles * s + num_sms - 1) / num_sms;
        const double cost = (double)waves * ((steps + s - 1) / s + 8) + (s > 1 ? 8.0 + 0.004 * (double)tiles * s : 0.0);
        if (cost < best_cost) { best_cost = cost; best = s; }
    }
    return best;
}

inline size_t partial_bytes(int m, int n, int k, int num_sms) {
    if (m <= 0 || n <= 0) return 0;
    const int s = split_count(m, n, k, num_sms);
    return s > 1 ? (size_t)s * m * n * 8 : 0;
}

template <int MT, bool TB>
int launch_mt(const Args& g, int batch, cudaStream_t st) {
    static bool configured[kMaxDevices] = {false};
    int dev = 0;
    const int rc = current_device(&dev);
    if (rc != ASER_OK) return rc;
    if (!configured[dev]) {
        const cudaError_t e = cudaFuncSetAttribute(gemm_kernel<MT, TB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   smem_bytes<MT, TB>());
        if (e != cudaSuccess) return record_cuda_error(e, "gemm64 smem attribute");
        configured[dev] = true;
    }
    const dim3 grid((g.n + kTN - 1) / kTN, (g.m + 16 * MT - 1) / (16 * MT), g.splits > 1 ? g.splits : batch);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem_bytes<MT, TB>();
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g.beside ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, gemm_kernel<MT, TB>, g);
    return e == cudaSuccess ? (int)ASER_OK : record_cuda_error(e, "gemm64");
}

template <bool TB>
int launch_tb(const Args& g, int batch, cudaStream_t st) {
    switch (row_strips(g.m)) {
        case 3: return launch_mt<3, TB>(g, batch, st);
        case 4: return launch_mt<4, TB>(g, batch, st);
        case 5: return launch_mt<5, TB>(g, batch, st);
        default: return launch_mt<6, TB>(g, batch, st);
    }
}

// C = A B^T in `pieces` parts of k, raw, one after the other at `part` (pieces * m * n doubles): who reads them sums them in order.
inline int run_pieces(Args g, double* part, int pieces, cudaStream_t st) {
    const int steps = (g.k + kTK - 1) / kTK;
    g.splits = pieces;
    g.k_per_split = (steps + pieces - 1) / pieces * kTK;
    g.C = part;
    return launch_tb<true>(g, 1, st);
}

// Their sum, [m, n] (n even).
inline int sum_pieces(const double* part, int m, int n, int pieces, double* C, long long ldc, cudaStream_t st) {
    Args g = {};
    g.C = C; g.ldc = ldc; g.m = m; g.n = n; g.splits = pieces; g.a0 = 1.0;
    const long long pairs = (long long)m * n / 2;
    reduce_kernel<<<(unsigned)((pairs + 255) / 256), 256, 0, st>>>(part, g);
    return check_launch("gemm64 sum");
}

// n, k, all pitches even; pointers 16-byte aligned; `part` holds partial_bytes(m, n, k).  With
// B2 (and C2) the same A is applied to two matrices and k is not split.
inline int run(Args g, bool tb, double* part, int num_sms, cudaStream_t st) {
    if (g.m <= 0 || g.n <= 0) return ASER_OK;
    const int batch = g.B2 ? 2 : 1;
    g.splits = batch == 2 ? 1 : split_count(g.m, g.n, g.k, num_sms);
    const int steps = (g.k + kTK - 1) / kTK;
    g.k_per_split = (steps + g.splits - 1) / g.splits * kTK;
    if (g.splits == 1) return tb ? launch_tb<true>(g, batch, st) : launch_tb<false>(g, batch, st);
    Args p = g;
    p.C = part;
    const int rc = tb ? launch_tb<true>(p, 1, st) : launch_tb<false>(p, 1, st);
    if (rc != ASER_OK) return rc;
    const long long pairs = (long long)g.m * g.n / 2;
    reduce_kernel<<<(unsigned)((pairs + 255) / 256), 256, 0, st>>>(part, g);
    return check_launch("gemm64 reduce");
}

}  // namespace gemm64
}  // namespace aser
