// Device-side construction of the error-reconstruction factors of one layer (Algorithm 1 body;
// Sec. 4.1 Eq. 5-6 and the factor split below Eq. 8; Sec. 4.2 Eq. 10 for the smoothed operands):
//   E   = W diag(s) - dequant(Q4(W diag(s)))                     [N, K]
//   G   = X~^T X~ + lambda I,  X~ = X_cal diag(s)^-1,  lambda = damping * trace / K   (the paper's X X^T)
//   S   = lower Cholesky factor of G                              (whitening, Eq. 5)
//   A   = E S,  A ~ U_r Sigma_r V_r^T                             (truncated SVD, Eq. 6)
//   L_B = U_r Sigma_r  [N, r],   L_A = V_r^T S^-1  [r, K]
// All in fp64.
//
// S is not needed for the factors.  With u a left singular vector of A, sigma its value,
//   A A^T = E G E^T = F F^T,  F = [ sqrt(lambda) E | E X~^T ]   [N, K + tokens],
// so F has the singular values and left vectors of A, and since A = E S,
//   v^T S^-1 = sigma^-1 u^T A S^-1 = sigma^-1 u^T E:  L_A = Sigma_r^-1 U_r^T E.
// With no more tokens than channels F takes the place of A: no Gram matrix, no Cholesky factor, no
// triangular solve (4096 x 4096 with 512 tokens: 17 GFLOP instead of 180).  The factor S is computed
// when the caller asks for it, when there are more tokens than channels (then A is the smaller
// matrix), and when lambda is so small that the damped Gram matrix may turn out singular, which
// the Cholesky factorisation has to report.
//
// The r leading left vectors come from subspace iteration on F F^T with p = r + oversampling
// vectors as rows (Ut [p, N]): Y = Ut F, Z = Y F^T, normalised by the Cholesky factor of Z Z^T.
// After two plain steps the steps follow the Chebyshev recurrence T' = 2 (2/b F F^T - I) T - T"
// on [0, b], b the smallest Ritz value (from below an estimate of sigma_p^2, so nothing wanted is
// damped): the recurrence is linear in the rows, so both of its terms may be multiplied by the
// inverse Cholesky factor after every step and it keeps its accuracy whatever the spread of the
// spectrum (the first step, from vectors that mix the whole of it, is normalised in two stages).  b is estimated anew every dozen steps.  With x = sigma_r^2 / sigma_p^2, a step of the
// recurrence gains exp(acosh(2 x - 1)), a plain one x: at x = 1.2 ... 1.6, where quantization errors
// lie, 22 steps reach what 60 to 90 plain ones would.  Measured against the exact triplets (2048 x
// 2048, 512 tokens, r = 64): product 5e-5 after 18 such steps, 9e-5 after 48 plain ones.
// The final Rayleigh-Ritz step works on the p x p Cholesky factor L of (Ut F)(Ut F)^T: one-sided
// Jacobi rotations of its rows until they are orthogonal; their norms are the singular values.
//
// 4096 x 4096, 512 tokens, r = 64 took 236.8 ms with plain iteration on A, a 64 x 64 fma product
// (157 ms), one thread per column in the triangular solves (46 ms) and one launch per Jacobi round
// (11 ms); then 11.0 ms: Y and Z 5.8 (at 28 of 37 TFLOP/s), Cholesky factors 1.1, Jacobi 1.4; with the Gram matrix and its
// factorisation beside the products of the next step, and a Jacobi round that keeps up the norms of its rows
// instead of summing them, 9.8 ms (2000 x 1536, r = 16: 2.84 -> 2.51, 3000 x 3840, r = 48: 7.90 -> 6.71).  2048 x
// 1024, r = 256: 784 -> 47 ms.
#include "aser_common.cuh"
#include "gemm64.cuh"

namespace aser {

namespace {

// ---------------------------------------------------------------------------
// C[i,j] = beta * C[i,j] + alpha * sum_k A(i,k) B(k,j), all fp64, element (i,k) of A at
// A[i * ai + k * ak] (so a transposed operand is a pair of swapped strides), C row-major with
// leading dimension ldc.  64 x 64 x 16 tiles, 256 threads, 4 x 4 results per thread.
// ---------------------------------------------------------------------------
constexpr int kGT = 64, kGK = 16;

__global__ void __launch_bounds__(256)
dgemm_kernel(int m, int n, int k, double alpha, const double* __restrict__ A, long long ai, long long ak,
             const double* __restrict__ B, long long bk, long long bj, double beta, double* __restrict__ C,
             long long ldc) {
    __shared__ double As[kGK][kGT + 1];
    __shared__ double Bs[kGK][kGT + 1];
    const int tid = threadIdx.x;
    const int i0 = blockIdx.y * kGT, j0 = blockIdx.x * kGT;
    const int ti = (tid / 16) * 4, tj = (tid % 16) * 4;
    double acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
    for (int k0 = 0; k0 < k; k0 += kGK) {
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            const int t = tid + l * 256;
            int ii, kk;
            if (ak == 1) { kk = t % kGK; ii = t / kGK; } else { ii = t % kGT; kk = t / kGT; }
            As[kk][ii] = (i0 + ii < m && k0 + kk < k) ? A[(long long)(i0 + ii) * ai + (long long)(k0 + kk) * ak] : 0.0;
            int jj, kb;
            if (bj == 1) { jj = t % kGT; kb = t / kGT; } else { kb = t % kGK; jj = t / kGK; }
            Bs[kb][jj] = (j0 + jj < n && k0 + kb < k) ? B[(long long)(k0 + kb) * bk + (long long)(j0 + jj) * bj] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < kGK; ++kk) {
            double a[4], b[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) { a[x] = As[kk][ti + x]; b[x] = Bs[kk][tj + x]; }
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[x][y] = fma(a[x], b[y], acc[x][y]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const int i = i0 + ti + x, j = j0 + tj + y;
            if (i < m && j < n) {
                double* c = C + (long long)i * ldc + j;
                *c = (beta == 0.0 ? 0.0 : beta * *c) + alpha * acc[x][y];
            }
        }
}

int dgemm(cudaStream_t st, int m, int n, int k, double alpha, const double* A, long long ai, long long ak,
          const double* B, long long bk, long long bj, double beta, double* C, long long ldc) {
    if (m <= 0 || n <= 0) return ASER_OK;
    dim3 grid((n + kGT - 1) / kGT, (m + kGT - 1) / kGT);
    dgemm_kernel<<<grid, 256, 0, st>>>(m, n, k, alpha, A, ai, ak, B, bk, bj, beta, C, ldc);
    return check_launch("dgemm_kernel");
}

// ---------------------------------------------------------------------------
// Cholesky, lower, in place, blocked by 64 columns: factor the diagonal block (one CTA), solve
// the panel below it row by row against that block, update the trailing matrix with a GEMM.
// A non-positive pivot sets *fail (the factor is then unusable).
// ---------------------------------------------------------------------------
constexpr int kCB = 64;

__global__ void __launch_bounds__(kCB)
potrf_diag_kernel(double* __restrict__ A, long long lda, int nb, int* __restrict__ fail) {
    __shared__ double T[kCB][kCB + 1];
    const int t = threadIdx.x;
    for (int i = 0; i < nb; ++i) T[i][t] = (t < nb) ? A[(long long)i * lda + t] : 0.0;
    __syncthreads();
    for (int j = 0; j < nb; ++j) {
        if (t == j) {
            double d = T[j][j];
            if (!(d > 0.0)) { *fail = 1; d = 1.0; }
            T[j][j] = sqrt(d);
        }
        __syncthreads();
        if (t > j && t < nb) T[t][j] /= T[j][j];
        __syncthreads();
        if (t > j && t < nb)
            for (int c = j + 1; c <= t; ++c) T[t][c] -= T[t][j] * T[c][j];
        __syncthreads();
    }
    for (int i = 0; i < nb; ++i)
        if (t < nb) A[(long long)i * lda + t] = (t <= i) ? T[i][t] : 0.0;    // the strict upper part is zeroed
}

// Rows of the panel P [rows, nb] (leading dimension ld): P <- P L^-T with L the nb x nb lower
// block; one thread per row (forward substitution along the row).
__global__ void __launch_bounds__(128)
panel_solve_kernel(double* __restrict__ P, long long ld, int rows, const double* __restrict__ L, long long ldl, int nb) {
    __shared__ double Ls[kCB][kCB + 1];
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) Ls[e / nb][e % nb] = L[(long long)(e / nb) * ldl + e % nb];
    __syncthreads();
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= rows) return;
    double x[kCB];
    double* p = P + (long long)row * ld;
#pragma unroll 1
    for (int j = 0; j < nb; ++j) {
        double v = p[j];
        for (int i = 0; i < j; ++i) v -= x[i] * Ls[j][i];
        x[j] = v / Ls[j][j];
        p[j] = x[j];
    }
}

int potrf_lower(cudaStream_t st, double* A, long long lda, int n, int* fail) {
    for (int j = 0; j < n; j += kCB) {
        const int nb = (n - j < kCB) ? (n - j) : kCB;
        double* Ajj = A + (long long)j * lda + j;
        potrf_diag_kernel<<<1, kCB, 0, st>>>(Ajj, lda, nb, fail);
        const int rest = n - j - nb;
        if (rest > 0) {
            double* P = A + (long long)(j + nb) * lda + j;
            panel_solve_kernel<<<(rest + 127) / 128, 128, 0, st>>>(P, lda, rest, Ajj, lda, nb);
            // trailing update: A22 -= P P^T
            int rc = dgemm(st, rest, rest, nb, -1.0, P, lda, 1, P, 1, lda, 1.0, A + (long long)(j + nb) * lda + (j + nb), lda);
            if (rc != ASER_OK) return rc;
        }
    }
    return check_launch("potrf");
}

// Zero the strict upper triangle (the blocked factorisation leaves the original entries there).
__global__ void zero_upper_kernel(double* __restrict__ A, long long lda, int n) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)n * n) return;
    const int i = (int)(e / n), j = (int)(e % n);
    if (j > i) A[(long long)i * lda + j] = 0.0;
}

// ---------------------------------------------------------------------------
// operands
// ---------------------------------------------------------------------------
// E = fp32(W) * s (one fp32 multiply, as the quantizer sees it) - q * w_scale, in fp64, times *mul
// (or 1); eight columns per thread, rows of E ld apart.
__global__ void __launch_bounds__(256)
build_error_kernel(const __half* __restrict__ W, const float* __restrict__ s, const uint8_t* __restrict__ Wq,
                   const float* __restrict__ w_scale, int N, int K, double* __restrict__ E, long long ld,
                   const double* __restrict__ mul) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)N * (K / 8)) return;
    const int n = (int)(e / (K / 8)), k = (int)(e % (K / 8)) * 8;
    const uint4 raw = *reinterpret_cast<const uint4*>(W + (long long)n * K + k);
    const uint32_t codes = *reinterpret_cast<const uint32_t*>(Wq + (long long)n * (K / 2) + k / 2);
    const __half* h = reinterpret_cast<const __half*>(&raw);
    const double sc = (double)w_scale[n], f = mul ? *mul : 1.0;
    double v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float ws = __fmul_rn(__half2float(h[i]), s ? s[k + i] : 1.f);
        const int q = (int)(((codes >> (4 * i)) & 0xF) ^ 8) - 8;        // sign-extend the nibble
        v[i] = ((double)ws - (double)q * sc) * f;
    }
    double2* o = reinterpret_cast<double2*>(E + (long long)n * ld + k);
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = make_double2(v[2 * i], v[2 * i + 1]);
}

// Copy of W with the columns of the outlier set zeroed: what the quantizer sees under the outlier
// split of Sec. 4.2 (Eq. 12), where those columns are carried by the factors alone.
__global__ void mask_columns_kernel(const __half* __restrict__ W, int N, int K, const int* __restrict__ idx,
                                    int n_idx, __half* __restrict__ Wm) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)N * K) return;
    const int k = (int)(e % K);
    bool out = false;
    for (int i = 0; i < n_idx; ++i) out = out || (idx[i] == k);
    Wm[e] = out ? __float2half(0.f) : W[e];
}

// X~ = fp32(X) / s (one fp32 division), in fp64; rows past T (up to the grid) are zero.  The sum of
// squares of each row goes to row_sq.
__global__ void __launch_bounds__(256)
build_xs_kernel(const __half* __restrict__ X, const float* __restrict__ s, int T, int K, double* __restrict__ Xs,
                double* __restrict__ row_sq) {
    __shared__ double red[256];
    const int row = blockIdx.x;
    double sum = 0.0;
    for (int k = threadIdx.x; k < K; k += 256) {
        double v = 0.0;
        if (row < T) {
            const float x = __half2float(X[(long long)row * K + k]);
            v = (double)(s ? __fdiv_rn(x, s[k]) : x);
        }
        Xs[(long long)row * K + k] = v;
        sum = fma(v, v, sum);
    }
    red[threadIdx.x] = sum;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) row_sq[row] = red[0];
}

// lambda = damping * trace(X~^T X~) / K, its root and the root's inverse.  A trace that is zero or
// not finite has no positive definite damped Gram matrix.
__global__ void lambda_kernel(const double* __restrict__ row_sq, int rows, int K, double damping,
                              double* __restrict__ out, int* __restrict__ fail) {
    double t = 0.0;
    for (int i = threadIdx.x; i < rows; i += 32) t += row_sq[i];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x != 0) return;
    double lam = damping * t / K;
    if (!(lam > 0.0) || !(lam < 1e300)) { *fail = 1; lam = 1.0; }
    out[0] = lam; out[1] = sqrt(lam); out[2] = 1.0 / sqrt(lam);
}

// G += lambda I with lambda = damping * trace(G) / K; one CTA (the trace is summed in a fixed order).
__global__ void __launch_bounds__(256) damp_kernel(double* __restrict__ G, int K, double damping) {
    __shared__ double red[256];
    double t = 0.0;
    for (int i = threadIdx.x; i < K; i += 256) t += G[(long long)i * K + i];
    red[threadIdx.x] = t;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    const double lam = damping * red[0] / K;
    for (int i = threadIdx.x; i < K; i += 256) G[(long long)i * K + i] += lam;
}

// Start vectors: a fixed hash of the index mapped to (-1, 1) (any full-rank start works).
__global__ void init_basis_kernel(double* __restrict__ Qt, long long n) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    unsigned long long z = (unsigned long long)e * 0x9E3779B97F4A7C15ull + 0x243F6A8885A308D3ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    Qt[e] = (double)(z >> 11) * (2.0 / 9007199254740992.0) - 1.0;
}

// ---------------------------------------------------------------------------
// One round of one-sided Jacobi: CTA b rotates rows (i, j) = pairs[b] of Bt [p, N] so that they
// become orthogonal, and applies the same rotation to rows i, j of Qt [p, K].  For more vectors than
// one CTA's shared memory holds.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
jacobi_round_kernel(double* __restrict__ Bt, int N, double* __restrict__ Qt, int K, int p, int round) {
    // round-robin tournament over p (even) players: player p-1 stays, the others rotate
    const int b = blockIdx.x, m = p - 1;
    int i = (b == 0) ? m : (round + b) % m;
    int j = (round + m - b) % m;
    if (b == 0) { i = round % m; j = m; }
    if (i > j) { const int t = i; i = j; j = t; }
    double* bi = Bt + (long long)i * N;
    double* bj = Bt + (long long)j * N;
    __shared__ double red[3][256];
    double a = 0.0, bb = 0.0, g = 0.0;
    for (int k = threadIdx.x; k < N; k += 256) {
        const double x = bi[k], y = bj[k];
        a = fma(x, x, a); bb = fma(y, y, bb); g = fma(x, y, g);
    }
    red[0][threadIdx.x] = a; red[1][threadIdx.x] = bb; red[2][threadIdx.x] = g;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            red[0][threadIdx.x] += red[0][threadIdx.x + o];
            red[1][threadIdx.x] += red[1][threadIdx.x + o];
            red[2][threadIdx.x] += red[2][threadIdx.x + o];
        }
        __syncthreads();
    }
    a = red[0][0]; bb = red[1][0]; g = red[2][0];
    if (fabs(g) <= 1e-300 || fabs(g) <= 1e-17 * sqrt(a * bb)) return;      // already orthogonal
    const double zeta = (bb - a) / (2.0 * g);
    const double t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
    const double c = 1.0 / sqrt(1.0 + t * t), s = c * t;
    for (int k = threadIdx.x; k < N; k += 256) {
        const double x = bi[k], y = bj[k];
        bi[k] = c * x - s * y;
        bj[k] = s * x + c * y;
    }
    double* qi = Qt + (long long)i * K;
    double* qj = Qt + (long long)j * K;
    for (int k = threadIdx.x; k < K; k += 256) {
        const double x = qi[k], y = qj[k];
        qi[k] = c * x - s * y;
        qj[k] = s * x + c * y;
    }
}

// ---------------------------------------------------------------------------
// Small matrices (p <= kMaxP), one CTA with everything in registers or shared memory.
// ---------------------------------------------------------------------------
constexpr int kMaxP = 112;

// H [p, p] symmetric (or `pieces` that add up to it, contiguous) -> Linv = L^-1 (lower, zeros above) with H = L L^T, and L itself if G is given.
// 16 x 16 threads hold the matrix cyclically (row ti + 16 a, column tj + 16 b).  Elimination step j
// needs row j alone (the multipliers of column j are its entries, by symmetry): its owners write it to
// shared memory, then every thread updates its T x T entries; columns below j, done with, hold the
// rows of the inverse instead.  One barrier per step: 40 us for p = 96 (one thread per row and three
// barriers took 74 for each block of 64, and the inverse another 310).
template <int T>
__global__ void __launch_bounds__(256)
chol_inverse_kernel(const double* __restrict__ H, long long ldh, int p, int pieces, double* __restrict__ Linv, long long ldl,
                    double* __restrict__ G, long long ldg, int* __restrict__ fail) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");      // (only a launch made for it makes use of this)
    __shared__ double row[2][16 * T];
    __shared__ double piv[16 * T];
    const int ti = threadIdx.x >> 4, tj = threadIdx.x & 15;
    double w[T][T];
#pragma unroll
    for (int a = 0; a < T; ++a)
#pragma unroll
        for (int b = 0; b < T; ++b) {
            const int i = ti + 16 * a, j = tj + 16 * b;
            w[a][b] = (i < p && j < p) ? H[(long long)i * ldh + j] : (i == j ? 1.0 : 0.0);
        }
    for (int q = 1; q < pieces; ++q)         // H is the sum of its pieces, p * p apart
#pragma unroll
        for (int a = 0; a < T; ++a)
#pragma unroll
            for (int b = 0; b < T; ++b) {
                const int i = ti + 16 * a, j = tj + 16 * b;
                if (i < p && j < p) w[a][b] += H[(long long)q * p * p + (long long)i * ldh + j];
            }
    bool bad = false;
#pragma unroll
    for (int ja = 0; ja < T; ++ja) {
#pragma unroll 1
        for (int jj = 0; jj < 16; ++jj) {
            const int j = 16 * ja + jj, buf = jj & 1;
            if (ti == jj) {
#pragma unroll
                for (int b = 0; b < T; ++b) row[buf][tj + 16 * b] = w[ja][b];
            }
            __syncthreads();
            double d = row[buf][j];
            if (!(d > 0.0)) { bad = true; d = 1.0; }
            if (threadIdx.x == 0) piv[j] = d;
            const double inv = 1.0 / d;
            double v[T];
#pragma unroll
            for (int b = 0; b < T; ++b) v[b] = (tj + 16 * b == j) ? 1.0 : row[buf][tj + 16 * b];
#pragma unroll
            for (int a = ja; a < T; ++a) {
                const int i = ti + 16 * a;
                if (i <= j) continue;
                const double l = row[buf][i] * inv;
#pragma unroll
                for (int b = 0; b < T; ++b) {
                    if (tj + 16 * b == j) w[a][b] = 0.0;
                    w[a][b] = fma(-l, v[b], w[a][b]);
                }
            }
        }
    }
    __syncthreads();
    if (bad && threadIdx.x == 0) *fail = 1;
    if (threadIdx.x < 16 * T) piv[threadIdx.x] = 1.0 / sqrt(piv[threadIdx.x]);
    __syncthreads();
#pragma unroll
    for (int a = 0; a < T; ++a)
#pragma unroll
        for (int b = 0; b < T; ++b) {
            const int i = ti + 16 * a, j = tj + 16 * b;
            if (i >= p || j >= p) continue;
            Linv[(long long)i * ldl + j] = (j < i) ? w[a][b] * piv[i] : (j == i ? piv[i] : 0.0);
            if (G) {        // row i froze at step i: its entries right of the diagonal are d_i l_ji
                G[(long long)j * ldg + i] = (j >= i) ? w[a][b] * piv[i] : 0.0;
            }
        }
}

// *b = the smallest eigenvalue of H = L L^T, from above, by twelve inverse iterations with L^-1.
__global__ void __launch_bounds__(1024)
smallest_eigenvalue_kernel(const double* __restrict__ Linv, long long ldl, int p, double* __restrict__ b) {
    __shared__ double v[512], u[512], red[32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto sum_squares = [&](const double* x) {
        double s = 0.0;
        for (int i = tid; i < p; i += 1024) s = fma(x[i], x[i], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) red[warp] = s;
        __syncthreads();
        s = 0.0;
        for (int i = 0; i < 32; ++i) s += red[i];
        __syncthreads();
        return s;
    };
    for (int i = tid; i < p; i += 1024) v[i] = 1.0;
    __syncthreads();
    double last = 1.0;
    for (int it = 0; it < 12; ++it) {
        const double nv = 1.0 / sqrt(sum_squares(v));
        for (int i = warp; i < p; i += 32) {                 // u = Linv v / |v|
            double s = 0.0;
            for (int j = lane; j <= i; j += 32) s = fma(Linv[(long long)i * ldl + j], v[j], s);
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) u[i] = s * nv;
        }
        __syncthreads();
        last = sum_squares(u);                               // v^T H^-1 v / v^T v
        // v = Linv^T u: 32 columns per warp, the rows dealt over the warps of a column group
        const int groups = (p + 31) / 32, per = 32 / groups, grp = warp % groups, part = warp / groups;
        const int j = grp * 32 + lane;
        double s = 0.0;
        if (part < per && j < p)
            for (int i = j + part; i < p; i += per) s = fma(Linv[(long long)i * ldl + j], u[i], s);
        __shared__ double acc[32][33];
        acc[warp][lane] = s;
        __syncthreads();
        if (warp < groups && j < p) {
            double t = 0.0;
            for (int q = 0; q < per; ++q) t += acc[q * groups + warp][lane];
            v[j] = t;
        }
        __syncthreads();
    }
    if (tid == 0) *b = 1.0 / last;
}

// One-sided Jacobi on the rows of G [p, p], the rotations applied to V (the identity at first):
// V G has orthogonal rows.  All rounds in one CTA, rows in shared memory, half a warp per pair; ends
// with the first sweep that finds every pair orthogonal to rounding.  The tangent of an angle is
// taken in fp32 from an fp64 quotient (its error only leaves the pair for a later sweep), cosine and sine in fp64, so the
// rotations are orthogonal to fp64 rounding.  The squared norms of the rows are summed when a sweep begins and then follow the
// rotations, in fp64 and for the angle as it was taken: good to a few roundings of the larger norm of a pair.
// A sweep that rotates nothing, which ends the loop, has only seen norms that were summed in it.
constexpr int kJacobiThreads = 896;          // kMaxP / 2 half warps
static_assert(kJacobiThreads / 16 >= kMaxP / 2, "a half warp per pair");
__global__ void __launch_bounds__(kJacobiThreads)
jacobi_kernel(double* __restrict__ G, double* __restrict__ V, int p) {
    extern __shared__ __align__(16) double jsm[];
    double* g = jsm;
    double* v = jsm + p * p;
    __shared__ double sq[kMaxP];             // squared norms of the rows: summed at the start of a sweep, then kept up
    __shared__ int rotated;
    const int pair = threadIdx.x >> 4, lane = threadIdx.x & 15;
    for (int e = threadIdx.x; e < p * p; e += kJacobiThreads) { g[e] = G[e]; v[e] = (e / p == e % p) ? 1.0 : 0.0; }
    const int m = p - 1;
    for (int sweep = 0; sweep < 20; ++sweep) {
        __syncthreads();
        if (threadIdx.x == 0) rotated = 0;
        for (int i0 = 0; i0 < p; i0 += kJacobiThreads / 16) {
            const int i = i0 + pair;
            double a = 0.0;
            if (i < p)
                for (int k = lane; k < p; k += 16) a = fma(g[i * p + k], g[i * p + k], a);
            for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (i < p && lane == 0) sq[i] = a;
        }
        __syncthreads();
        for (int round = 0; round < m; ++round) {
            // round-robin tournament over p (even) players: player p - 1 stays, the others rotate
            const int i = (pair == 0) ? round : (round + pair) % m;
            const int j = (pair == 0) ? m : (round + m - pair) % m;
            const bool have = pair < p / 2;
            double* gi = g + i * p;
            double* gj = g + j * p;
            // Both norms are read before the shuffles: every lane of the warp has them when one of its pairs writes new ones.
            const double a = have ? sq[i] : 0.0, b = have ? sq[j] : 0.0;
            double c = 0.0;
            if (have)
                for (int k = lane; k < p; k += 16) c = fma(gi[k], gj[k], c);
            for (int o = 8; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
            __syncwarp();
            if (have && c * c > 1e-28 * a * b) {
                const float zeta = (float)((b - a) / (2.0 * c)), z = fabsf(zeta);
                const float tf = z > 1e9f ? 0.5f / z : 1.f / (z + sqrtf(1.f + z * z));
                const double t = zeta >= 0.f ? (double)tf : -(double)tf;
                const double cs = rsqrt(1.0 + t * t), sn = cs * t;
                if (lane == 0) {            // the norms of the rows as they are rotated, whatever the angle
                    rotated = 1;
                    sq[i] = fmax(cs * cs * fma(t, fma(t, b, -2.0 * c), a), 0.0);
                    sq[j] = fmax(cs * cs * fma(t, fma(t, a, 2.0 * c), b), 0.0);
                }
                double* vi = v + i * p;
                double* vj = v + j * p;
                for (int k = lane; k < p; k += 16) {
                    const double x = gi[k], y = gj[k], w = vi[k], u = vj[k];
                    gi[k] = cs * x - sn * y; gj[k] = sn * x + cs * y;
                    vi[k] = cs * w - sn * u; vj[k] = sn * w + cs * u;
                }
            }
            __syncthreads();
        }
        if (!rotated) break;
    }
    for (int e = threadIdx.x; e < p * p; e += kJacobiThreads) { G[e] = g[e]; V[e] = v[e]; }
}

__global__ void identity_kernel(double* __restrict__ V, int p) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < p * p) V[e] = (e / p == e % p) ? 1.0 : 0.0;
}

// The r longest rows of G [p, p] in descending order (equal ones by index): their norms to sigma
// and sigma_out, the matching rows of V to Vsel [r, p].  One CTA, p <= 512.  Weights or tokens with NaN or
// infinity make norms that are NaN; those rank behind every number, so that the ranks are a permutation
// and every index read below has been written (the call then reports the failed factorisation).
__global__ void __launch_bounds__(512)
select_top_kernel(const double* __restrict__ G, const double* __restrict__ V, int p, int r, double* __restrict__ Vsel,
                  double* __restrict__ sigma, double* __restrict__ sigma_out) {
    __shared__ double norm[512];
    __shared__ int order[512];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = warp; i < p; i += 16) {
        double s = 0.0;
        for (int k = lane; k < p; k += 32) s = fma(G[(long long)i * p + k], G[(long long)i * p + k], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) norm[i] = s >= 0.0 ? s : -1.0;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < p; i += 512) {
        int rank = 0;
        for (int k = 0; k < p; ++k) rank += (norm[k] > norm[i] || (norm[k] == norm[i] && k < i)) ? 1 : 0;
        order[rank] = i;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < r; t += 512) {
        const double s = sqrt(norm[order[t]]);
        sigma[t] = s;
        if (sigma_out) sigma_out[t] = s;
    }
    for (int e = threadIdx.x; e < r * p; e += 512) Vsel[e] = V[(long long)order[e / p] * p + e % p];
}

// L_B[n, t] = fp16(sigma[t] * U[t, n])
__global__ void up_factor_kernel(const double* __restrict__ U, const double* __restrict__ sigma, int N, int r, __half* __restrict__ LB) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)N * r) return;
    const int n = (int)(e / r), t = (int)(e % r);
    LB[e] = __double2half(sigma[t] * U[(long long)t * N + n]);
}
// L_A[t, k] = fp16(src[t, k] / sigma[t] * *mul)
__global__ void down_factor_kernel(const double* __restrict__ src, const double* __restrict__ sigma, int K, int r,
                                   const double* __restrict__ mul, __half* __restrict__ LA) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < (long long)r * K) LA[e] = __double2half(src[e] / sigma[e / K] * (mul ? *mul : 1.0));
}

// Splits of k are chosen for a fixed SM count, so that the workspace size needs no device.
constexpr int kSplitSms = 148;

struct ConstructLayout {
    int p, tokens;                // tokens padded to 16 rows
    long long lda;                // columns of the wide error matrix, at most
    int pieces;                   // of the Gram matrix that is made beside the products of the next step (0: p is too large)
    bool sum_pieces;              // they are summed by a launch of their own, ahead of the factorisation
    size_t A, E, G, Xs, T[4], Y, part, C, L, V, Vsel, sigma, row_sq, scalars, fail, Wm, total;     // byte offsets
};

ConstructLayout construct_layout(int N, int K, int Tcal, int r, int n_split) {
    ConstructLayout L;
    int p = r + (r / 2 > 32 ? r / 2 : 32);
    p += p & 1;
    const int lim = (N < K ? N : K) & ~1;
    if (p > lim) p = lim;
    L.p = p;
    L.tokens = (Tcal + 15) / 16 * 16;
    const int wide = L.tokens <= K ? K + L.tokens : K;
    L.lda = wide;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off += (bytes + 255) / 256 * 256; return o; };
    // the wide error matrix, or (through the whitening factor) A, E and G: never both
    const size_t nk = (size_t)N * K * 8, apart = 2 * nk + (size_t)K * K * 8, joined = (size_t)N * wide * 8;
    L.A = take(joined > apart ? joined : apart);
    L.E = L.A + nk;
    L.G = L.E + nk;
    L.Xs = take((size_t)L.tokens * K * 8);
    for (int i = 0; i < 4; ++i) L.T[i] = take((size_t)p * N * 8);
    L.Y = take((size_t)p * wide * 8);
    // as many pieces as the product beside it has splits, of k = N both
    L.pieces = 0;
    for (int q = 4; p <= 96 && q <= 16 && L.pieces == 0; q *= 2)
        if (q == 16 || gemm64::split_count(p, wide, N, kSplitSms - q) <= q) L.pieces = q;
    // The factorisation in one CTA takes 4.9e-3 p^2 us, each piece that it sums itself 3.1e-4 p^2 more, the product beside it 2 p N
    // `wide` at 28 TFLOP/s; a launch that sums them first takes 3.6.  22 steps, ms, all in order / the CTA sums / summed first: 768 x 768,
    // r = 64 4.47 / 5.22 / 3.99; 1536 x 1536, r = 64 5.24 / 5.80 / 4.50; 2048 x 2048, r = 16 3.07 / 2.62 / 2.70, r = 64 5.99 / 5.46 / 5.01;
    // 4096 x 4096, r = 64 10.67 / 9.60 / 9.68.
    L.sum_pieces = 4.9e-3 * p * p + 3.1e-4 * (L.pieces - 1) * p * p > 2.0 * p * N * (double)wide / 28e6 + 3.6;
    size_t part = 0;
    auto need = [&](int m, int n, int k, int sms = kSplitSms) {
        const size_t b = gemm64::partial_bytes(m, n, k, sms);
        if (b > part) part = b;
    };
    need(N, L.tokens, K); need(N, K, K);
    for (int kc : {K, wide}) { need(p, kc, N); need(p, N, kc); need(p, p, kc); }
    need(p, p, N); need(p, N, p); need(r, N, p); need(r, K, N);
    for (int i0 = kMaxP; i0 < p; i0 += kMaxP) {
        const int nb = p - i0 < kMaxP ? p - i0 : kMaxP;
        need(p - i0, kMaxP, kMaxP); need(p - i0, p - i0, kMaxP); need(nb, i0, i0); need(nb, i0, nb);
    }
    for (int kc : {K, wide}) { need(p, kc, N, kSplitSms - L.pieces); need(p, N, kc, kSplitSms - 1); }
    L.part = take(part);
    L.C = take((size_t)p * p * 8 * (L.pieces > 1 ? L.pieces : 1));
    L.L = take((size_t)p * p * 8);
    L.V = take((size_t)p * p * 8);
    L.Vsel = take((size_t)(r > 0 ? r : 1) * p * 8);
    L.sigma = take((size_t)(r > 0 ? r : 1) * 8);
    L.row_sq = take((size_t)L.tokens * 8);
    L.scalars = take(64);
    L.fail = take(4);
    L.Wm = take(n_split > 0 ? (size_t)N * K * 2 : 0);
    L.total = off;
    return L;
}

inline int blocks_for(long long n, int threads) { return (int)((n + threads - 1) / threads); }

// What the steps share: stream, pieces of split products, failure flag.
struct Ctx {
    cudaStream_t st;
    double* part;
    int* fail;
};

// C[m, n] = a0 / *div * A B (+ a1 X1 + a2 X2)
int product(const Ctx& c, bool tb, int m, int n, int k, const double* A, long long lda, const double* B, long long ldb,
            double* C, long long ldc, double a0 = 1.0, const double* div = nullptr, const double* X1 = nullptr, double a1 = 0.0,
            const double* X2 = nullptr, double a2 = 0.0, int beside_ctas = 0) {
    gemm64::Args g = {};
    g.A = A; g.B = B; g.C = C; g.lda = lda; g.ldb = ldb; g.ldc = ldc; g.m = m; g.n = n; g.k = k;
    g.a0 = a0; g.a0_div = div; g.X1 = X1; g.a1 = a1; g.X2 = X2; g.a2 = a2;
    g.beside = beside_ctas > 0;                 // the launch before has this many SMs to itself
    return gemm64::run(g, tb, c.part, kSplitSms - beside_ctas, c.st);
}

#define ASER_STEP(call)                        \
    do {                                       \
        const int step_rc = (call);            \
        if (step_rc != ASER_OK) return step_rc; \
    } while (0)

int chol_inverse_block(const Ctx& c, const double* H, long long ldh, int p, double* Linv, long long ldl, double* G, long long ldg,
                       int pieces = 1) {
    switch ((p + 15) / 16) {
        case 1: chol_inverse_kernel<1><<<1, 256, 0, c.st>>>(H, ldh, p, pieces, Linv, ldl, G, ldg, c.fail); break;
        case 2: chol_inverse_kernel<2><<<1, 256, 0, c.st>>>(H, ldh, p, pieces, Linv, ldl, G, ldg, c.fail); break;
        case 3: chol_inverse_kernel<3><<<1, 256, 0, c.st>>>(H, ldh, p, pieces, Linv, ldl, G, ldg, c.fail); break;
        case 4: chol_inverse_kernel<4><<<1, 256, 0, c.st>>>(H, ldh, p, pieces, Linv, ldl, G, ldg, c.fail); break;
        case 5: chol_inverse_kernel<5><<<1, 256, 0, c.st>>>(H, ldh, p, pieces, Linv, ldl, G, ldg, c.fail); break;
        case 6: chol_inverse_kernel<6><<<1, 256, 0, c.st>>>(H, ldh, p, pieces, Linv, ldl, G, ldg, c.fail); break;
        default: chol_inverse_kernel<7><<<1, 256, 0, c.st>>>(H, ldh, p, pieces, Linv, ldl, G, ldg, c.fail); break;
    }
    return check_launch("chol_inverse_kernel");
}

// H [p, p] (overwritten where p > kMaxP) = L L^T: Linv = L^-1, G = L (both pitch p, zeros above the
// diagonal).  Larger matrices in blocks of kMaxP rows.
int chol_inverse(const Ctx& c, double* H, int p, double* Linv, double* G) {
    if (p <= kMaxP) return chol_inverse_block(c, H, p, p, Linv, p, G, p);
    cudaError_t e = cudaMemsetAsync(Linv, 0, (size_t)p * p * 8, c.st);
    if (e == cudaSuccess) e = cudaMemsetAsync(G, 0, (size_t)p * p * 8, c.st);
    if (e != cudaSuccess) return record_cuda_error(e, "construct: memset");
    for (int i0 = 0; i0 < p; i0 += kMaxP) {
        const int nb = p - i0 < kMaxP ? p - i0 : kMaxP, rest = p - i0 - nb;
        const long long d = (long long)i0 * p + i0, below = d + (long long)nb * p;
        ASER_STEP(chol_inverse_block(c, H + d, p, nb, Linv + d, p, G + d, p));
        if (rest > 0) {
            // rows below: L_ib = H_ib Linv_bb^T, then their Schur complement
            ASER_STEP(product(c, true, rest, nb, nb, H + below, p, Linv + d, p, G + below, p));
            ASER_STEP(product(c, true, rest, rest, nb, G + below, p, G + below, p, H + below + nb, p, -1.0, nullptr,
                              H + below + nb, 1.0));
        }
        if (i0 > 0) {       // row block of the inverse: -Linv_bb (L_b,0..i0 Linv_0..i0); H's rows are scratch by now
            ASER_STEP(product(c, false, nb, i0, i0, G + (long long)i0 * p, p, Linv, p, H + (long long)i0 * p, p));
            ASER_STEP(product(c, false, nb, i0, nb, Linv + d, p, H + (long long)i0 * p, p, Linv + (long long)i0 * p, p, -1.0));
        }
    }
    return ASER_OK;
}

}  // namespace

size_t construct_workspace_bytes(int N, int K, int Tcal, int r, int n_split) {
    return construct_layout(N, K, Tcal, r, n_split).total;
}

int launch_construct(const __half* W, const float* s, const __half* Xcal, int N, int K, int Tcal, int r,
                     double damping, int iters, uint8_t* Wq, float* w_scale, __half* LA, __half* LB,
                     double* sigma_out, double* S_out, const int* split_idx, int n_split, void* workspace,
                     cudaStream_t st) {
    const ConstructLayout L = construct_layout(N, K, Tcal, r, n_split);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    auto at = [&](size_t off) { return reinterpret_cast<double*>(ws + off); };
    double *A = at(L.A), *G = at(L.G), *Xs = at(L.Xs), *Y = at(L.Y), *C = at(L.C), *Li = at(L.L), *V = at(L.V);
    double *Vsel = at(L.Vsel), *sigma = at(L.sigma), *lambda = at(L.scalars), *bound = lambda + 3;
    int* fail = reinterpret_cast<int*>(ws + L.fail);
    const Ctx ctx{st, at(L.part), fail};
    const int p = L.p;

    const __half* Wquant = W;
    if (n_split > 0) {      // the quantizer sees W without the outlier columns; E below keeps them
        __half* Wm = reinterpret_cast<__half*>(ws + L.Wm);
        mask_columns_kernel<<<blocks_for((long long)N * K, 256), 256, 0, st>>>(W, N, K, split_idx, n_split, Wm);
        Wquant = Wm;
    }
    ASER_STEP(launch_pack_w4(Wquant, s, N, K, Wq, w_scale, st));
    if (r == 0) return ASER_OK;
    cudaError_t e = cudaMemsetAsync(fail, 0, sizeof(int), st);
    if (e != cudaSuccess) return record_cuda_error(e, "construct: memset");
    build_xs_kernel<<<L.tokens, 256, 0, st>>>(Xcal, s, Tcal, K, Xs, at(L.row_sq));
    lambda_kernel<<<1, 32, 0, st>>>(at(L.row_sq), L.tokens, K, damping, lambda, fail);

    // The matrix A [N, kc] to be decomposed, and the error matrix E (times *e_mul^-1) inside or beside it.
    // Above a damping of 1e-6 the smallest eigenvalue of the damped Gram matrix is far above the
    // rounding of its Cholesky factorisation at every supported K, so nothing is left to report.
    const bool factor = S_out != nullptr || damping < 1e-6 || L.tokens > K;
    const int kc = factor ? K : K + L.tokens;
    const double *E, *e_mul;
    long long lde;
    const int error_blocks = blocks_for((long long)N * (K / 8), 256);
    if (factor) {
        // G = X~^T X~ (the paper's X X^T), damped, its Cholesky factor in place, A = E S
        double* Ef = at(L.E);
        build_error_kernel<<<error_blocks, 256, 0, st>>>(W, s, Wq, w_scale, N, K, Ef, K, nullptr);
        ASER_STEP(dgemm(st, K, K, Tcal, 1.0, Xs, 1, K, Xs, K, 1, 0.0, G, K));
        damp_kernel<<<1, 256, 0, st>>>(G, K, damping);
        ASER_STEP(potrf_lower(st, G, K, K, fail));
        zero_upper_kernel<<<blocks_for((long long)K * K, 256), 256, 0, st>>>(G, K, K);
        if (S_out) {
            e = cudaMemcpyAsync(S_out, G, (size_t)K * K * 8, cudaMemcpyDeviceToDevice, st);
            if (e != cudaSuccess) return record_cuda_error(e, "construct: copy S");
        }
        ASER_STEP(product(ctx, false, N, K, K, Ef, K, G, K, A, K));
        E = Ef; lde = K; e_mul = nullptr;
    } else {
        // A = [ sqrt(lambda) E | E X~^T ]
        build_error_kernel<<<error_blocks, 256, 0, st>>>(W, s, Wq, w_scale, N, K, A, kc, lambda + 1);
        ASER_STEP(product(ctx, true, N, L.tokens, K, A, kc, Xs, K, A + K, kc, 1.0, lambda + 1));
        E = A; lde = kc; e_mul = lambda + 2;
    }

    // subspace iteration on A A^T with the basis as rows: t0 the current basis, t1 the term before it
    double *t0 = at(L.T[0]), *t1 = at(L.T[1]), *f0 = at(L.T[2]), *f1 = at(L.T[3]);
    auto swap = [](double*& x, double*& y) { double* t = x; x = y; y = t; };
    // normalize: t0 <- L^-1 t0 with L L^T = t0 t0^T; apply: with the factor there is; the same to t1 if it is still needed
    auto apply = [&](bool both) {
        gemm64::Args g = {};
        g.A = Li; g.lda = p; g.B = t0; g.ldb = N; g.C = f0; g.ldc = N; g.m = p; g.n = N; g.k = p; g.a0 = 1.0;
        if (both) { g.B2 = t1; g.C2 = f1; }
        if (both) { ASER_STEP(gemm64::run(g, false, ctx.part, kSplitSms, st)); swap(t1, f1); }
        else { ASER_STEP(product(ctx, false, p, N, p, Li, p, t0, N, f0, N)); }
        swap(t0, f0);
        return (int)ASER_OK;
    };
    auto normalize = [&](bool both) {
        ASER_STEP(product(ctx, true, p, p, N, t0, N, t0, N, C, p));
        ASER_STEP(chol_inverse(ctx, C, p, Li, V));
        return apply(both);
    };
    init_basis_kernel<<<blocks_for((long long)p * N, 256), 256, 0, st>>>(t0, (long long)p * N);
    ASER_STEP(normalize(false));
    ASER_STEP(normalize(false));
    int done = 0;
    for (; done < iters && done < 2; ++done) {
        ASER_STEP(product(ctx, false, p, kc, N, t0, N, A, kc, Y, kc));
        ASER_STEP(product(ctx, true, p, N, kc, Y, kc, A, kc, f0, N));
        swap(t0, f0);
        if (done == 0) {
            // The start vectors mix the whole spectrum, and the Gram matrix of Y A^T has its spread to the fourth power; with
            // the factor of Y Y^T taken out first it is the second.  Later bases come near the singular vectors in
            // descending order, whose Gram matrices are graded and factorise at any spread.
            ASER_STEP(product(ctx, true, p, p, kc, Y, kc, Y, kc, C, p));
            ASER_STEP(chol_inverse(ctx, C, p, Li, V));
            ASER_STEP(product(ctx, false, p, N, p, Li, p, t0, N, f0, N));
            swap(t0, f0);
        }
        ASER_STEP(normalize(false));
    }
    const int cycles = (iters - done + 11) / 12;
    for (int cycle = 0; cycle < cycles; ++cycle) {
        const int steps = (iters - done) / (cycles - cycle);
        for (int i = 0; i < steps; ++i, ++done) {
            if (i > 0 && L.pieces > 0) {
                // The basis of the step before is still as its product left it.  Its Gram matrix is made beside the first
                // product of this step, summed and factorised beside the second (40 us of one CTA), then the factor is applied to both
                // terms: the rows that the products see have the growth of one step, as their Gram matrix always had.
                gemm64::Args h = {};
                h.A = h.B = t0; h.lda = h.ldb = N; h.ldc = p; h.m = h.n = p; h.k = N; h.a0 = 1.0; h.side = true;
                ASER_STEP(gemm64::run_pieces(h, C, L.pieces, st));
                ASER_STEP(product(ctx, false, p, kc, N, t0, N, A, kc, Y, kc, 1.0, nullptr, nullptr, 0.0, nullptr, 0.0, L.pieces));
                if (L.sum_pieces) {
                    ASER_STEP(gemm64::sum_pieces(C, p, p, L.pieces, V, p, st));
                    ASER_STEP(chol_inverse_block(ctx, V, p, p, Li, p, nullptr, p));
                } else {
                    ASER_STEP(chol_inverse_block(ctx, C, p, p, Li, p, nullptr, p, L.pieces));
                }
                ASER_STEP(product(ctx, true, p, N, kc, Y, kc, A, kc, f0, N, 4.0, bound, t0, -2.0, t1, -1.0, 1));
                swap(t1, f0);
                swap(t0, t1);
                ASER_STEP(apply(i + 1 < steps));
                if (i + 1 == steps) ASER_STEP(normalize(false));
                continue;
            }
            ASER_STEP(product(ctx, false, p, kc, N, t0, N, A, kc, Y, kc));
            if (i == 0) {       // the basis is orthonormal here: Y Y^T holds its Ritz values
                ASER_STEP(product(ctx, true, p, p, kc, Y, kc, Y, kc, C, p));
                ASER_STEP(chol_inverse(ctx, C, p, Li, V));
                smallest_eigenvalue_kernel<<<1, 1024, 0, st>>>(Li, p, p, bound);
                ASER_STEP(product(ctx, true, p, N, kc, Y, kc, A, kc, f0, N, 2.0, bound, t0, -1.0));
            } else {
                ASER_STEP(product(ctx, true, p, N, kc, Y, kc, A, kc, f0, N, 4.0, bound, t0, -2.0, t1, -1.0));
            }
            swap(t1, f0);       // the new term to t1 ...
            swap(t0, t1);       // ... and into its place, the old basis behind it
            if (L.pieces == 0 || i + 1 == steps) ASER_STEP(normalize(i + 1 < steps));
        }
    }
    ASER_STEP(normalize(false));

    // Rayleigh-Ritz: rotate the rows of the Cholesky factor of (Ut A)(Ut A)^T until they are orthogonal
    ASER_STEP(product(ctx, false, p, kc, N, t0, N, A, kc, Y, kc));
    ASER_STEP(product(ctx, true, p, p, kc, Y, kc, Y, kc, C, p));
    ASER_STEP(chol_inverse(ctx, C, p, Li, V));
    double* Lrows = V;          // L, then the rotated rows
    double* Vrot = Li;          // the rotations (the inverse is not needed here)
    if (p <= kMaxP) {
        const int smem = 2 * p * p * 8;
        e = cudaFuncSetAttribute(jacobi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kMaxP * kMaxP * 8);
        if (e != cudaSuccess) return record_cuda_error(e, "jacobi smem attribute");
        jacobi_kernel<<<1, kJacobiThreads, smem, st>>>(Lrows, Vrot, p);
    } else {
        identity_kernel<<<blocks_for((long long)p * p, 256), 256, 0, st>>>(Vrot, p);
        for (int sweep = 0; sweep < 12; ++sweep)
            for (int round = 0; round < p - 1; ++round)
                jacobi_round_kernel<<<p / 2, 256, 0, st>>>(Lrows, p, Vrot, p, p, round);
    }
    select_top_kernel<<<1, 512, 0, st>>>(Lrows, Vrot, p, r, Vsel, sigma, sigma_out);
    // U_r^T = Vsel Ut;  L_B = U_r Sigma_r,  L_A = Sigma_r^-1 U_r^T E
    ASER_STEP(product(ctx, false, r, N, p, Vsel, p, t0, N, f0, N));
    up_factor_kernel<<<blocks_for((long long)N * r, 256), 256, 0, st>>>(f0, sigma, N, r, LB);
    ASER_STEP(product(ctx, false, r, K, N, f0, N, E, lde, Y, K));
    down_factor_kernel<<<blocks_for((long long)r * K, 256), 256, 0, st>>>(Y, sigma, K, r, e_mul, LA);
    ASER_STEP(check_launch("construct"));
    // an offline step: wait for it and report a failed factorisation
    int host_fail = 0;
    e = cudaMemcpyAsync(&host_fail, fail, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return record_cuda_error(e, "construct");
    if (host_fail) return record_error(ASER_ERR_SHAPE, "construct: the damped Gram matrix is not positive definite");
    return ASER_OK;
}

}  // namespace aser
