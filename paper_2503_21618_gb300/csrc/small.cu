// Small dense m x m kernels of the projection step (m = subspace size L):
// Cholesky factor and triangular inverse for Cholesky-QR2 B-orthonormalisation,
// and the symmetric eigensolver of the projected problem (Algorithm 1, "solve
// the eigenvalue problem A_hat s_i = theta_i B_hat s_i" once B_hat = I).
//
// FP64 arithmetic runs at a small fraction of the FP32 rate on this GPU, so
// the modes of the eigensolver are:
//  0. cyclic parallel Jacobi in FP64 (round-robin pair ordering, all m/2
//     rotations of a round applied at once) as ONE cooperative multi-block
//     kernel: each round is "rotations -> row phase -> grid barrier -> column
//     phase -> grid barrier", so the O(m^3) rotation work of a sweep is spread
//     over many SMs;
//  2. (default, m <= 448) the same Jacobi in FP32 in one block's shared memory
//     (m <= 160) or in double-float on a thread-block cluster first, the
//     vectors then refined by FP64 products (Ogita-Aishima) and groups of
//     close eigenvalues diagonalised in FP64;
//  1. (m <= 160) FP32 Jacobi, FP64 re-orthonormalisation (Cholesky of S0^T S0 ~
//     I), and the cooperative FP64 Jacobi polishes the nearly diagonal T =
//     S0^T A S0 in 2-3 sweeps (Jacobi converges quadratically; unlike
//     first-order refinement it is robust to clustered and graded spectra).
#include <cuda_runtime.h>
#include <cooperative_groups.h>
#include <float.h>

#include <algorithm>
#include <mutex>

#include "internal.h"

namespace slrf {

// ---------------------------------------------------------------------------
// column scaling of a Gram matrix: s_i = 1/sqrt(g_ii), G <- S G S
// ---------------------------------------------------------------------------
__global__ void k_colscale_diag(int m, const double *G, double *__restrict__ s) {
    chain_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const double g = G[(int64_t)i * m + i];
    s[i] = g > 0.0 ? 1.0 / sqrt(g) : 0.0;
}
__global__ void k_colscale(int m, double *__restrict__ G, const double *s) {
    chain_wait();
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e < (int64_t)m * m) G[e] *= s[e / m] * s[e % m];
}

void small_colscale(Ctx &ctx, int m, double *G, double *s) {
    const int64_t tot = (int64_t)m * m;
    ctx.before(KC_SMALL_DENSE, 16.0 * m, m);
    launch_chained(ctx, k_colscale_diag, (m + 63) / 64, 64, 0, m, G, s);
    ctx.after();
    ctx.before(KC_SMALL_DENSE, 16.0 * tot, tot);
    launch_chained(ctx, k_colscale, (unsigned)((tot + 255) / 256), 256, 0, m, G, s);
    ctx.after();
}

__global__ void k_scale_rows(int m, const double *s, double *__restrict__ T) {
    chain_wait();
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)m * m) return;
    T[e] *= s[e / m];
}
void small_scale_rows(Ctx &ctx, int m, const double *s, double *T) {
    const int64_t tot = (int64_t)m * m;
    ctx.before(KC_SMALL_DENSE, 16.0 * tot, tot);
    launch_chained(ctx, k_scale_rows, (unsigned)((tot + 255) / 256), 256, 0, m, s, T);
    ctx.after();
}

// ---------------------------------------------------------------------------
// Shifted refactorisation after a breakdown (*status > 0 on entry, else it
// returns): G + shift I = R^T R (R upper), one block, right-looking.  G is
// read and left untouched.  *status = -1 on success; an unrecoverable
// breakdown (a pivot not above 0) sets *status = k + 1, k the failing pivot.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_chol_shifted(int m, const double *G, double *__restrict__ Rg,
                                                        int32_t *__restrict__ status, int32_t *__restrict__ out_status,
                                                        int use_smem, double shift) {
    chain_wait();
    extern __shared__ double sm[];
    if (*(volatile int32_t *)status <= 0) return;
    double *A = use_smem ? sm : Rg;
    const int tid = threadIdx.x, bs = blockDim.x;
    __shared__ int bad;
    __shared__ double dinv;
    for (int e = tid; e < m * m; e += bs) A[e] = G[e] + ((e / m == e % m) ? shift : 0.0);
    if (tid == 0) bad = 0;
    __syncthreads();
    for (int k = 0; k < m; ++k) {
        if (tid == 0) {
            const double d = A[k * m + k];
            if (!(d > 0.0) || !isfinite(d)) {
                bad = k + 1;
            } else {
                const double r = sqrt(d);
                A[k * m + k] = r;
                dinv = 1.0 / r;
            }
        }
        __syncthreads();
        if (bad) break;
        for (int j = k + 1 + tid; j < m; j += bs) A[k * m + j] *= dinv;
        __syncthreads();
        const int r = m - k - 1;
        for (int e = tid; e < r * r; e += bs) {
            const int i = k + 1 + e / r, j = k + 1 + e % r;
            if (j >= i) A[i * m + j] -= A[k * m + i] * A[k * m + j];
        }
        __syncthreads();
    }
    if (!bad)
        for (int e = tid; e < m * m; e += bs) {
            const int i = e / m, j = e % m;
            if (j < i) A[e] = 0.0;
        }
    __syncthreads();
    if (use_smem)
        for (int e = tid; e < m * m; e += bs) Rg[e] = A[e];
    if (tid == 0) {
        const int32_t st = bad ? bad : -1;
        *status = st;
        if (out_status) *out_status = st;
    }
}

void raise_smem_limits();   // defined after the kernels it configures

// ---------------------------------------------------------------------------
// Blocked Cholesky factor and inverse: G = R^T R, X = R^{-1}, from the
// elimination of [G | I], whose right part ends as R^{-T}.  Right-looking in
// CHB x CHB blocks: the diagonal block on one CTA, the panel solves and the
// trailing updates of both parts spread over the GPU (FP64 issues at ~1.7
// FMAs per clock and SM here, so m^3/6 of them belong on many SMs; what is
// left is the chain of m pivots).  The right part costs no further steps: a
// separate triangular inverse by back substitution, one warp per column, was
// a chain of m dot products (m = 150: 136 us, m = 300: 321 us).  Factor and
// inverse at m = 150: 446 us on one CTA each, 181 us here.  The lower
// triangle of X holds the right part during the elimination; R is worked on
// in place (upper).  A breakdown at pivot k (a pivot at or below
// shift_on_fail) sets *status = k + 1 and stops the later steps; with
// shift_on_fail > 0 the one-block kernel then refactors G + shift I and
// k_triinv_upper inverts that factor.  `status` is a device word: the steps
// read it, and the last kernel copies it to `out_status` (a mapped host word
// costs each reader about a microsecond).
// ---------------------------------------------------------------------------
constexpr int CHB = 32;

__global__ void k_chol_init(int m, const double *G, double *__restrict__ A, double *__restrict__ X,
                            int32_t *__restrict__ status) {
    chain_wait();
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e == 0) *status = 0;
    if (e >= (int64_t)m * m) return;
    if (G != A) A[e] = G[e];
    X[e] = e / m == e % m ? 1.0 : 0.0;
}

// The kb x kb diagonal block on 8 warps: thread (i0, j) owns rows i0, i0 + 8,
// ... of column j in registers.  Per pivot the warp of row k scales the row
// by 1/sqrt(pivot) and publishes it, one barrier, everyone updates its rows
// below.  Bound by that chain (about 0.3 us per pivot; one warp with the
// block in shared memory took 62 us per 32 pivots).
__global__ void __launch_bounds__(256) k_chol_diag(int m, int k0, int kb, double *__restrict__ A,
                                                   int32_t *__restrict__ status, double pmin) {
    chain_wait();
    __shared__ double u[2][CHB];   // alternating by pivot: one barrier per pivot
    __shared__ int bad[2];
    if (*(volatile int32_t *)status != 0) return;   // uniform: the same word for every thread
    const int j = threadIdx.x & 31, i0 = threadIdx.x >> 5;
    double c[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = i0 + 8 * q;
        c[q] = (i < kb && j < kb && j >= i) ? A[(int64_t)(k0 + i) * m + k0 + j] : 0.0;
    }
    if (threadIdx.x < 2) bad[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int q0 = 0; q0 < 4; ++q0) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
            const int k = q0 * 8 + kk;
            if (k >= kb) break;
            if (i0 == kk) {
                const double d = __shfl_sync(0xffffffffu, c[q0], k);
                if (!(d > pmin) || !isfinite(d)) {
                    if (j == 0) bad[k & 1] = k0 + k + 1;
                } else {
                    c[q0] *= rsqrt(d);
                    u[k & 1][j] = c[q0];
                }
            }
            __syncthreads();
            if (bad[k & 1]) {   // uniform
                if (threadIdx.x == 0) *status = bad[k & 1];
                return;
            }
            const double uj = u[k & 1][j];
#pragma unroll
            for (int q = q0; q < 4; ++q) {
                const int i = i0 + 8 * q;
                if (i > k) c[q] = fma(-u[k & 1][i], uj, c[q]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = i0 + 8 * q;
        if (i < kb && j < kb) A[(int64_t)(k0 + i) * m + k0 + j] = j >= i ? c[q] : 0.0;
    }
}

// rows k0 .. k0+kb of the columns right of the block and of the right part's
// columns 0 .. k0+kb: x = R_kk^{-T} a, one warp per column (lane i = row i;
// the forward substitution with the unit-scaled factor broadcasts row p, so
// one FMA per step: FP64 FMAs of one warp issue ~70 clocks apart)
__global__ void __launch_bounds__(64) k_chol_panel(int m, int k0, int kb, double *__restrict__ A,
                                                   double *__restrict__ X, const int32_t *status) {
    chain_wait();
    __shared__ double Rk[CHB][CHB + 1], ri[CHB];
    if (*(volatile int32_t *)status != 0) return;
    if (threadIdx.x < kb) ri[threadIdx.x] = 1.0 / A[(int64_t)(k0 + threadIdx.x) * m + k0 + threadIdx.x];
    __syncthreads();
    for (int e = threadIdx.x; e < kb * kb; e += blockDim.x) {
        const int p = e / kb, i = e % kb;
        Rk[p][i] = A[(int64_t)(k0 + p) * m + k0 + i] * ri[p];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (c >= m) return;
    double *col = (c < k0 + kb ? X : A) + (int64_t)k0 * m + c;
    double v = lane < kb ? col[(int64_t)lane * m] : 0.0;
    for (int p = 0; p + 1 < kb; ++p) {
        const double vp = __shfl_sync(0xffffffffu, v, p);
        if (lane > p && lane < kb) v = fma(-Rk[p][lane], vp, v);
    }
    // entries above the right part's diagonal are zero and stay so
    if (lane < kb && (c >= k0 + kb || c <= k0 + lane)) col[(int64_t)lane * m] = v * ri[lane];
}

// Trailing rows i >= k0+kb: A[i][j] -= sum_p A[k0+p][i] A[k0+p][j] for j >= i
// and X[i][c] -= sum_p A[k0+p][i] X[k0+p][c] for the right part's columns
// c < k0+kb; 16 x 16 output tiles, the first `tl` tile columns the left part
__global__ void __launch_bounds__(256) k_chol_update(int m, int k0, int kb, int tl, double *__restrict__ A,
                                                     double *__restrict__ X, const int32_t *status) {
    chain_wait();
    __shared__ double Pi[CHB][17], Pj[CHB][17];
    if (*(volatile int32_t *)status != 0) return;
    const int r0 = k0 + kb;
    const bool left = (int)blockIdx.x < tl;
    if (left && blockIdx.x < blockIdx.y) return;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int i0 = r0 + blockIdx.y * 16, j0 = left ? r0 + blockIdx.x * 16 : (blockIdx.x - tl) * 16;
    const int jend = left ? m : r0;
    double *D = left ? A : X;
    for (int e = threadIdx.x; e < kb * 16; e += 256) {
        const int p = e / 16, q = e % 16;
        Pi[p][q] = (i0 + q < m) ? A[(int64_t)(k0 + p) * m + i0 + q] : 0.0;
        // above the right part's diagonal the matrix holds nothing yet
        Pj[p][q] = (j0 + q < jend && (left || j0 + q <= k0 + p)) ? D[(int64_t)(k0 + p) * m + j0 + q] : 0.0;
    }
    __syncthreads();
    const int i = i0 + ty, j = j0 + tx;
    if (i >= m || j >= jend || (left && j < i)) return;
    double s = 0.0;
#pragma unroll 8
    for (int p = 0; p < kb; ++p) s = fma(Pi[p][ty], Pj[p][tx], s);
    D[(int64_t)i * m + j] -= s;
}

// R's lower triangle to zero, X = (its lower triangle)^T
__global__ void k_chol_finish(int m, double *__restrict__ A, double *__restrict__ X,
                              const int32_t *status, int32_t *__restrict__ out_status) {
    chain_wait();
    const int32_t st = *(volatile int32_t *)status;
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e == 0 && out_status) *out_status = st;
    if (st != 0 || e >= (int64_t)m * m) return;
    const int i = (int)(e / m), j = (int)(e % m);
    if (j >= i) return;
    A[e] = 0.0;
    X[(int64_t)j * m + i] = X[e];
    X[e] = 0.0;
}

// X = R^{-1} of the shifted factor (runs only after a shifted refactorisation,
// *status < 0): one warp per column j, back substitution x_i = (delta_ij -
// sum_{k=i+1..j} R_ik x_k) / R_ii, the sum split over the lanes.
__global__ void __launch_bounds__(32) k_triinv_upper(int m, const double *R, double *__restrict__ X,
                                                     const int32_t *status) {
    chain_wait();
    extern __shared__ double xcol[];
    if (*(volatile int32_t *)status >= 0) return;
    double *rinv = xcol + m;
    const int j = blockIdx.x, lane = threadIdx.x;
    for (int i = lane; i <= j; i += 32) rinv[i] = 1.0 / R[(int64_t)i * m + i];
    for (int i = j + 1 + lane; i < m; i += 32) X[(int64_t)i * m + j] = 0.0;
    __syncwarp();
    for (int i = j; i >= 0; --i) {
        const double *Ri = R + (int64_t)i * m;
        double s = 0.0;
        for (int k = i + 1 + lane; k <= j; k += 32) s = fma(Ri[k], xcol[k], s);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane == 0) {
            const double x = ((i == j ? 1.0 : 0.0) - s) * rinv[i];
            xcol[i] = x;
            X[(int64_t)i * m + j] = x;
        }
        __syncwarp();
    }
}

void small_chol_inv(Ctx &ctx, int m, const double *G, double *R, double *Rinv, int32_t *status, int32_t *out_status,
                    double shift_on_fail) {
    const int64_t m2 = (int64_t)m * m;
    const unsigned eg = (unsigned)((m2 + 255) / 256);
    ctx.before(KC_SMALL_DENSE, 24.0 * m2, 0);
    launch_chained(ctx, k_chol_init, eg, 256, 0, m, G, R, Rinv, status);
    ctx.after();
    for (int k0 = 0; k0 < m; k0 += CHB) {
        const int kb = std::min(CHB, m - k0), rest = m - k0 - kb;
        ctx.before(KC_SMALL_DENSE, 16.0 * kb * kb, (double)kb * kb * kb / 3.0);
        launch_chained(ctx, k_chol_diag, 1, 256, 0, m, k0, kb, R, status, shift_on_fail);
        ctx.after();
        ctx.before(KC_SMALL_DENSE, 16.0 * kb * m, (double)kb * kb * m);
        launch_chained(ctx, k_chol_panel, (m + 1) / 2, 64, 0, m, k0, kb, R, Rinv, status);
        ctx.after();
        if (rest == 0) break;
        const int tl = (rest + 15) / 16, tr = (k0 + kb + 15) / 16;
        ctx.before(KC_SMALL_DENSE, 8.0 * rest * m, (double)rest * m * kb);
        launch_chained(ctx, k_chol_update, dim3(tl + tr, tl), 256, 0, m, k0, kb, tl, R, Rinv, status);
        ctx.after();
    }
    ctx.before(KC_SMALL_DENSE, 16.0 * m2, 0);
    launch_chained(ctx, k_chol_finish, eg, 256, 0, m, R, Rinv, status, out_status);
    ctx.after();
    if (shift_on_fail > 0.0 && G != R) {
        const size_t smem = (size_t)m * m * sizeof(double);
        const int use_smem = smem <= 200 * 1024;
        raise_smem_limits();
        ctx.before(KC_SMALL_DENSE, 16.0 * m2, 0);
        launch_chained(ctx, k_chol_shifted, 1, 1024, use_smem ? smem : 0, m, G, R, status, out_status, use_smem, shift_on_fail);
        ctx.after();
        ctx.before(KC_SMALL_DENSE, 16.0 * m2, 0);
        launch_chained(ctx, k_triinv_upper, m, 32, 2 * (size_t)m * sizeof(double), m, R, Rinv, status);
        ctx.after();
    }
}

// ---------------------------------------------------------------------------
// ||S||_F as FRO_PARTS partial sums of squares, one per block, summed by the
// readers (fro_norm, a whole warp)
constexpr int FRO_PARTS = 32, OA_PARTS = 64;   // OA_PARTS: blocks of k_oa_norms
__global__ void __launch_bounds__(256) k_fro(int m, const double *S, double *__restrict__ part) {
    chain_wait();
    __shared__ double red[8];
    double s = 0;
    for (int64_t e = blockIdx.x * 256 + threadIdx.x; e < (int64_t)m * m; e += FRO_PARTS * 256) s += S[e] * S[e];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int w = 0; w < 8; ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}
__device__ __forceinline__ double fro_norm(const double *part) {
    double s = part[threadIdx.x & 31];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    return sqrt(s);
}

// ---------------------------------------------------------------------------
// cyclic parallel Jacobi: round-robin pair ordering (circle method)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void rr_pair(int k, int r, int mp, int &a, int &b) {
    // circle method: position 0 fixed, positions 1..mp-1 rotate by r
    a = (k == 0) ? 0 : ((k - 1 + r) % (mp - 1)) + 1;
    b = ((mp - 2 - k + r) % (mp - 1)) + 1;
}

// ---------------------------------------------------------------------------
// FP32 cyclic Jacobi for m <= JMAX in one block: all m/2 rotations of a round
// applied at once, A in shared memory with an odd row pitch.  Bound by shared
// memory: the 2 x 2 block (k, l) of two pairs takes its row and its column
// rotation in one visit, so A is read and written once per round (rows, then
// columns, then the columns of V took three times that), and a thread's column
// pair and its rotation are fixed for the round: 1.52 -> 1.15 ms at m = 150.
// The vectors are not formed here: the rotations are logged and
// k_jacobi_vectors applies them, every row on its own SM.  Two block barriers
// per round: rotations, update.  A rotation is skipped below rel_tol of
// sqrt(|a_pp a_qq|); the sweeps stop once every rotation of a sweep was below
// sqrt(rel_tol) (quadratic convergence: the next sweep would find nothing), or
// when the log is full (max_sweeps: what is left then is the refinement's).
// Output: lam ascending (FP64), rank (the place of eigenvalue i in lam), the
// log and *nrounds.
// ---------------------------------------------------------------------------
constexpr int JMAX = 160;
constexpr int J32_SWEEPS = 40;   // at most; see log_sweeps

// x' = c x - s y, y' = s x + c y
__device__ __forceinline__ void rotate(float c, float s, float &x, float &y) {
    const float u = x, v = y;
    x = c * u - s * v;
    y = s * u + c * v;
}

// A rotation (1, 0: none) with its pair p < q
struct __align__(16) PairRotation {
    float c, s;
    int p, q;
};

// Padded order, row pitch and threads of the one-block Jacobi: in the update
// thread l + npair * kg takes the blocks (kg + i groups, l)
struct Jacobi32Shape {
    int mp, npair, ld, groups;
    __host__ __device__ explicit Jacobi32Shape(int m) {
        mp = m + (m & 1);
        npair = mp / 2;
        ld = mp + 1;
        groups = 1024 / npair < npair ? 1024 / npair : npair;
    }
    __host__ __device__ int threads() const { return (groups * npair + 31) / 32 * 32; }
    size_t bytes() const { return (size_t)mp * ld * sizeof(float); }
};

__global__ void __launch_bounds__(1024) k_jacobi32(int m, const double *S, double *__restrict__ lam,
                                                  int *__restrict__ rank, float2 *__restrict__ rlog,
                                                  int *__restrict__ nrounds, int max_sweeps, float rel_tol) {
    chain_wait();
    extern __shared__ float jsm[];
    const Jacobi32Shape sh(m);
    const int mp = sh.mp, npair = sh.npair, ld = sh.ld;
    float *A = jsm;   // mp x mp: an odd order's last row and column are zero
    const int tid = threadIdx.x, bs = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nwarp = bs >> 5;
    __shared__ PairRotation par[JMAX / 2];
    __shared__ int maxrel;             // largest relative pivot of the sweep (float bits)
    __shared__ double red[32];
    __shared__ float absmin;
    double fro = 0.0;
    for (int e = tid; e < mp * mp; e += bs) {
        const int i = e / mp, j = e - i * mp;
        const double v = i < m && j < m ? S[(int64_t)i * m + j] : 0.0;
        A[i * ld + j] = (float)v;
        fro += v * v;
    }
    for (int off = 16; off > 0; off >>= 1) fro += __shfl_xor_sync(0xffffffffu, fro, off);
    if (lane == 0) red[warp] = fro;
    __syncthreads();
    if (tid == 0) {
        double t = 0;
        for (int w = 0; w < nwarp; ++w) t += red[w];
        absmin = (float)(sqrt(t) * (double)rel_tol / sqrt((double)m));
        maxrel = 0;
    }
    __syncthreads();
    const int kg = tid / npair, l = tid - kg * npair;
    int64_t g = 0;   // rounds applied
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        for (int r = 0; r < mp - 1; ++r, ++g) {
            if (tid < npair) {
                int a, b;
                rr_pair(tid, r, mp, a, b);
                const int p = min(a, b), q = max(a, b);
                float c = 1.f, sv = 0.f;
                if (q < m) {
                    const float apq = A[p * ld + q];
                    const float app = A[p * ld + p], aqq = A[q * ld + q];
                    const float scale = sqrtf(fabsf(app * aqq));
                    if (fabsf(apq) > rel_tol * scale && fabsf(apq) > absmin) {
                        const float th = (aqq - app) / (2.f * apq);
                        const float t = (th >= 0.f ? 1.f : -1.f) / (fabsf(th) + sqrtf(1.f + th * th));
                        c = 1.f / sqrtf(1.f + t * t);
                        sv = t * c;
                        const float rel = fabsf(apq) / (scale > 0.f ? scale : 1.f);
                        atomicMax(&maxrel, __float_as_int(rel));
                    }
                }
                par[tid] = PairRotation{c, sv, p, q};
                rlog[g * npair + tid] = make_float2(a > b ? -c : c, sv);   // the sign: lower row first
            }
            __syncthreads();
            if (kg < sh.groups) {
                const PairRotation wl = par[l];
                for (int k = kg; k < npair; k += sh.groups) {
                    const PairRotation wk = par[k];
                    if (wk.s == 0.f && wl.s == 0.f) continue;
                    float *Ap = A + wk.p * ld, *Aq = A + wk.q * ld;
                    float xpp = Ap[wl.p], xpq = Ap[wl.q], xqp = Aq[wl.p], xqq = Aq[wl.q];
                    if (wk.s != 0.f) {
                        rotate(wk.c, wk.s, xpp, xqp);
                        rotate(wk.c, wk.s, xpq, xqq);
                    }
                    if (wl.s != 0.f) {
                        rotate(wl.c, wl.s, xpp, xpq);
                        rotate(wl.c, wl.s, xqp, xqq);
                    }
                    if (k == l) xpq = xqp = 0.f;
                    Ap[wl.p] = xpp;
                    Ap[wl.q] = xpq;
                    Aq[wl.p] = xqp;
                    Aq[wl.q] = xqq;
                }
            }
            __syncthreads();
        }
        const float top = __int_as_float(maxrel);   // 0: nothing rotated
        if (top < sqrtf(rel_tol)) break;
        __syncthreads();
        if (tid == 0) maxrel = 0;
        __syncthreads();
    }
    for (int i = tid; i < m; i += bs) {
        const float di = A[i * ld + i];
        int k = 0;
        for (int j = 0; j < m; ++j) {
            const float dj = A[j * ld + j];
            k += (dj < di) || (dj == di && j < i);
        }
        rank[i] = k;
        lam[k] = (double)di;
    }
    if (tid == 0) *nrounds = (int)g;
}

// ---------------------------------------------------------------------------
// Cyclic Jacobi for JMAX < m <= JDF_MAX on one thread-block cluster, in
// double-float arithmetic (hi + lo FP32 pairs, ~46 bits).
//
// The FP64 Jacobi over the whole GPU (k_jacobi_coop) is bound by its grid
// barriers and the FP64 pipe (32 ms at m = 300).  FP32 rotations would do for the
// accuracy, since the vectors are refined in FP64 afterwards, but the
// eigenvectors' signs come out of the rotation path: where two diagonal
// entries are close an FP32 rounding turns a rotation by 45 degrees the other
// way.  In double-float the path is the FP64 one (a decision differs only
// where the FP64 one is within ~1e-13), at ten FP32 instructions per
// operation on a pipe seventy times as fast.
//
// All m/2 rotations of a round (rr_pair) are applied at once, A in the shared
// memory of the C CTAs.  Position k of a round holds the pair (a_k, b_k).  A CTA
// owns a contiguous range of positions and the two full rows of each; from one
// round to the next the upper rows move down one position and the lower rows
// up one, so per round a CTA hands one row to each neighbour and the rest stay
// where they are.  Per round, between a block barrier (the inputs of the
// rotations are taken) and a cluster barrier:
//   update    (warps 1 ..) the 2 x 2 blocks (k, l) of the own positions k and
//             all l, rows and columns in one pass (A is kept in full, so the
//             columns of a block are two contiguous runs); the two rows that
//             move are written straight into the neighbours' free rows (DSMEM)
//   rotations (warp 0) of the next round, one lane per position, from the one
//             2 x 2 block each depends on and the diagonal, which every CTA
//             keeps in full (updated in closed form); they go to all CTAs
// The chain of double-float square roots and divisions (~1 us) thus hides behind
// the update: 8.3 ms at m = 300 on 16 CTAs, against 11.6 ms on 8 with it, and the
// rows' move, after the update; 8.0 with the divisions and the root of the skip
// test as hardware approximations (each first quotient is corrected by a second).
// The eigenvectors are not formed here: the rotations are logged (FP32) and
// k_jacobi_vectors applies them to the rows of I afterwards, every row on its
// own SM.  A rotation is skipped below rel_tol of sqrt(|a_pp a_qq|); the
// sweeps stop once every rotation of a sweep was below sqrt(rel_tol).
// Output: lam (FP64, unsorted), the log and *nrounds.
// ---------------------------------------------------------------------------
constexpr int JDF_MAX = 448;      // 7 positions per lane of k_jacobi_vectors
constexpr int JDF_CTAS = 16;      // with 8 a solve with 270 columns (n = 26 244) took 185 ms for 169
constexpr int JDF_SWEEPS = 20;    // at most; see log_sweeps
constexpr int JDF_THREADS = 544;  // 16 warps for the update, one for the rotations
static_assert(JDF_MAX <= 2 * 32 * JDF_CTAS, "one lane of warp 0 per position of a CTA");
constexpr int JVEC_ROUNDS = 8;    // rounds of the log per stage of k_jacobi_vectors
static_assert(JDF_MAX <= 2 * 32 * 7, "k_jacobi_vectors holds at most 7 positions per lane");

// double-float: the rounded operations are spelled out, so that no
// multiplication and addition of the error terms is contracted
struct df {
    float h, l;
};
__device__ __forceinline__ df df_renorm(float h, float l) {
    const float s = __fadd_rn(h, l);
    return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ df df_of(double x) {
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ df df_neg(df a) { return {-a.h, -a.l}; }
__device__ __forceinline__ df df_add(df a, df b) {
    const float s = __fadd_rn(a.h, b.h), v = __fsub_rn(s, a.h);
    float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, v)), __fsub_rn(b.h, v));
    e = __fadd_rn(e, __fadd_rn(a.l, b.l));
    return df_renorm(s, e);
}
__device__ __forceinline__ df df_mul(df a, df b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = fmaf(a.h, b.h, -p);
    e = fmaf(a.h, b.l, e);
    e = fmaf(a.l, b.h, e);
    return df_renorm(p, e);
}
// c x - s z
__device__ __forceinline__ df df_rot(df c, df x, df s, df z) {
    const float p = __fmul_rn(c.h, x.h), q = __fmul_rn(s.h, z.h);
    float pl = fmaf(c.h, x.h, -p), ql = fmaf(s.h, z.h, -q);
    pl = fmaf(c.h, x.l, pl);
    ql = fmaf(s.h, z.l, ql);
    pl = fmaf(c.l, x.h, pl);
    ql = fmaf(s.l, z.h, ql);
    const float d = __fsub_rn(p, q), v = __fsub_rn(d, p);
    float e = __fsub_rn(__fsub_rn(p, __fsub_rn(d, v)), __fadd_rn(q, v));
    e = __fadd_rn(e, __fsub_rn(pl, ql));
    return df_renorm(d, e);
}
__device__ __forceinline__ df df_div(df a, df b) {
    // both quotients to a few units in the last place: the second corrects the first
    const float q = __fdividef(a.h, b.h);
    const df r = df_add(a, df_neg(df_mul({q, 0.f}, b)));
    return df_renorm(q, __fdividef(r.h, b.h));
}
__device__ __forceinline__ df df_sqrt(df a) {
    const float y = rsqrtf(a.h), s = __fmul_rn(a.h, y);
    const df r = df_add(a, df_neg(df_mul({s, 0.f}, {s, 0.f})));
    return df_renorm(s, 0.5f * y * r.h);
}
__device__ __forceinline__ df df_rsqrt(df a) {
    const float y = rsqrtf(a.h);
    const df r = df_add({1.f, 0.f}, df_neg(df_mul(a, df_mul({y, 0.f}, {y, 0.f}))));
    return df_renorm(y, 0.5f * y * r.h);
}

// index of the upper (a) and lower (b) row of position k in round r
__device__ __forceinline__ int rr_top(int k, int r, int mp) {
    const int x = k - 1 + r;
    return k == 0 ? 0 : (x >= mp - 1 ? x - (mp - 1) : x) + 1;
}
__device__ __forceinline__ int rr_bot(int k, int r, int mp) {
    const int x = mp - 2 - k + r;
    return (x >= mp - 1 ? x - (mp - 1) : x) + 1;
}

struct JacobiShape {
    int mp, npair, ld, maxcnt;
    __host__ __device__ JacobiShape(int m, int C) {
        mp = m + (m & 1);
        npair = mp / 2;
        ld = mp;   // even: rows of 8-byte pairs start on 16 bytes
        maxcnt = (npair + C - 1) / C;
    }
    // rows (two free ones for arrivals), rotations and diagonal changes of two rounds, diagonal, row slots
    __host__ __device__ size_t bytes() const {
        return (size_t)(2 * maxcnt + 2) * ld * 8 + (size_t)npair * 48 + (size_t)ld * 8 + (size_t)maxcnt * 16;
    }
};

__global__ void __launch_bounds__(JDF_THREADS, 1)
k_jacobi_df(int m, const double *__restrict__ S, const double *__restrict__ fro_part, double *__restrict__ lam,
            float2 *__restrict__ rlog, int *__restrict__ nrounds, int max_sweeps, float rel_tol) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), c = (int)cl.block_rank();
    const JacobiShape sh(m, C);
    const int mp = sh.mp, npair = sh.npair, ld = sh.ld;
    extern __shared__ float4 jsm4[];
    float4 *par = jsm4;                                   // [2][npair]: c, s as (hi, lo)
    df *rows = reinterpret_cast<df *>(par + 2 * npair);
    df *pda = rows + (size_t)(2 * sh.maxcnt + 2) * ld;    // [2][npair]: change of a_aa
    df *diag = pda + 2 * npair;
    int *slots = reinterpret_cast<int *>(diag + ld);      // [2][upper, lower][maxcnt]
    __shared__ int nbfree[2][2];    // free slot of the lower / upper neighbour, by round parity
    __shared__ int myfree[2][2];    // own free slots for an upper / a lower row, by round parity
    __shared__ int mx[2];           // largest relative pivot of a sweep (float bits), by sweep parity
    __shared__ int allmx[JDF_CTAS]; // the CTAs' mx of the sweep that ends
    __shared__ float absmin;
    __shared__ int scale;           // ||S||_F < 2^scale; A holds S 2^-scale
    const int tid = threadIdx.x, bs = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nwarp = bs >> 5;
    const int k0 = c * npair / C, k1 = (c + 1) * npair / C, cnt = k1 - k0;
    const bool last = c == C - 1;
    auto slot_of = [&](int par_, int low) { return slots + (par_ * 2 + low) * sh.maxcnt; };
    cl.sync();   // every CTA runs before any writes to another's shared memory

    if (warp == 0) {
        const double f = fro_norm(fro_part);
        if (lane == 0) {
            scale = f > 0.0 && isfinite(f) ? ilogb(f) + 1 : 0;
            absmin = (float)(scalbn(f, -scale) * (double)rel_tol / sqrt((double)m));
            mx[0] = mx[1] = 0;
            myfree[0][0] = 2 * cnt;
            myfree[0][1] = 2 * cnt + 1;
            if (c > 0) cl.map_shared_rank(&nbfree[0][1], c - 1)[0] = 2 * cnt + 1;   // where c - 1 sends a lower row
            if (!last) cl.map_shared_rank(&nbfree[0][0], c + 1)[0] = 2 * cnt;       // where c + 1 sends an upper row
        }
    }
    __syncthreads();
    const double sc = scalbn(1.0, -scale);
    // the upper rows of the CTA's positions, then the lower ones
    for (int e = warp; e < 2 * cnt; e += nwarp) {
        const int low = e >= cnt, k = k0 + (low ? e - cnt : e);
        const int i = low ? rr_bot(k, 0, mp) : rr_top(k, 0, mp);
        for (int j = lane; j < ld; j += 32)
            rows[(size_t)e * ld + j] = i < m && j < m ? df_of(S[(int64_t)i * m + j] * sc) : df{0.f, 0.f};
        if (lane == 0) slot_of(0, low)[k - k0] = e;
    }
    for (int i = tid; i < ld; i += bs) diag[i] = i < m ? df_of(S[(int64_t)i * m + i] * sc) : df{0.f, 0.f};
    __syncthreads();

    // rotation of position k (a = upper, b = lower index) from its pivot; to every CTA and the log of round g
    auto rotation = [&](int k, int a, int b, df apq, int sweep, int64_t g, int pb) {
        df cc = {1.f, 0.f}, ss = {0.f, 0.f}, da = {0.f, 0.f};
        if (max(a, b) < m) {
            const df app = diag[min(a, b)], aqq = diag[max(a, b)];
            const float prod = fabsf(app.h * aqq.h), mag = prod > 0.f ? prod * rsqrtf(prod) : 0.f;
            if (fabsf(apq.h) > rel_tol * mag && fabsf(apq.h) > absmin) {
                // t = sign(th) / (|th| + sqrt(1 + th^2)), th = (a_qq - a_pp) / (2 a_pq)
                const df d = df_add(aqq, df_neg(app)), a2 = {2.f * apq.h, 2.f * apq.l};
                const df ad = d.h < 0.f ? df_neg(d) : d, aa = a2.h < 0.f ? df_neg(a2) : a2;
                const df h = df_sqrt(df_add(df_mul(ad, ad), df_mul(aa, aa)));
                df t = df_div(aa, df_add(ad, h));
                if (d.h != 0.f && (d.h > 0.f) != (apq.h > 0.f)) t = df_neg(t);
                cc = df_rsqrt(df_add({1.f, 0.f}, df_mul(t, t)));
                ss = df_mul(t, cc);
                da = df_neg(df_mul(t, apq));
                if (a > b) {
                    ss = df_neg(ss);
                    da = df_neg(da);
                }
                atomicMax(&mx[sweep & 1], __float_as_int(__fdividef(fabsf(apq.h), mag > 0.f ? mag : 1.f)));
            }
        }
        const float4 v = make_float4(cc.h, cc.l, ss.h, ss.l);
        for (int q = 0; q < C; ++q) {
            cl.map_shared_rank(par + pb * npair + k, q)[0] = v;
            cl.map_shared_rank(pda + pb * npair + k, q)[0] = da;
        }
        rlog[g * npair + k] = make_float2(cc.h, ss.h);
    };
    for (int j = tid; j < cnt; j += bs) {
        const int k = k0 + j, a = rr_top(k, 0, mp), b = rr_bot(k, 0, mp);
        rotation(k, a, b, rows[(size_t)slot_of(0, 0)[j] * ld + b], 0, 0, 0);
    }
    cl.sync();

    int64_t g = 0;   // rounds applied
    int cur = 0;
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        for (int r = 0; r < mp - 1; ++r) {
            const float4 *P = par + cur * npair;
            const int *sT = slot_of(cur, 0), *sB = slot_of(cur, 1);
            const int nxt = cur ^ 1, r1 = r + 1 == mp - 1 ? 0 : r + 1, s1 = r1 ? sweep : sweep + 1;
            // Warp 0 forms the rotations of the next round: each needs one
            // element as this round's update will leave it, so its block's
            // inputs are taken before the update starts.  Element (a', b') of
            // position k: rows and columns of the present positions kr and lc.
            const bool mine = warp == 0 && lane < cnt;
            df x00, x01, x10, x11;
            float4 pr, pc;
            bool row_low = false, col_low = true;
            if (mine) {
                const int k = k0 + lane;
                int kr = lane + 1, lc = k - 1;                       // (a_{k+1}, b_{k-1})
                if (k == 0) {                                        // (a_0, a_1)
                    kr = 0;
                    lc = 1;
                    col_low = false;
                } else if (lane + 1 == cnt) {
                    row_low = true;
                    if (last) {                                      // (b_k, b_{k-1})
                        kr = lane;
                    } else {                                         // (b_{k-1}, a_{k+1}): a_{k+1} is elsewhere
                        kr = lane - 1;
                        lc = k + 1;
                        col_low = false;
                    }
                }
                const df *ra = rows + (size_t)sT[kr] * ld, *rb = rows + (size_t)sB[kr] * ld;
                const int a = rr_top(lc, r, mp), b = rr_bot(lc, r, mp);
                x00 = ra[a];
                x01 = ra[b];
                x10 = rb[a];
                x11 = rb[b];
                pr = P[k0 + kr];
                pc = P[lc];
            }
            for (int l = tid; l < npair; l += bs) {
                const df da = pda[cur * npair + l];
                if (da.h != 0.f) {
                    const int a = rr_top(l, r, mp), b = rr_bot(l, r, mp);
                    diag[a] = df_add(diag[a], da);
                    diag[b] = df_add(diag[b], df_neg(da));
                }
            }
            __syncthreads();
            if (warp == 0) {
                if (mine) {
                    const int k = k0 + lane;
                    df apq;
                    if (pr.z != 0.f || pc.z != 0.f) {
                        const df ck = {pr.x, pr.y}, sk = {pr.z, pr.w}, cl_ = {pc.x, pc.y}, sl = {pc.z, pc.w};
                        const df u = row_low ? sk : ck, v = row_low ? df_neg(ck) : sk;
                        const df y0 = df_rot(u, x00, v, x10), y1 = df_rot(u, x01, v, x11);
                        apq = col_low ? df_rot(sl, y0, df_neg(cl_), y1) : df_rot(cl_, y0, sl, y1);
                    } else {
                        apq = row_low ? (col_low ? x11 : x10) : (col_low ? x01 : x00);
                    }
                    rotation(k, rr_top(k, r1, mp), rr_bot(k, r1, mp), apq, s1, g + 1, nxt);
                }
            } else {
                // The update: tasks (position j, 32 positions l), dealt to the
                // other warps.  The lowest upper row and the highest lower row
                // are written where the neighbours expect them, every element.
                df *const out_lo = c > 0 ? cl.map_shared_rank(rows, c - 1) + (size_t)nbfree[cur][0] * ld : nullptr;
                df *const out_hi = last ? nullptr : cl.map_shared_rank(rows, c + 1) + (size_t)nbfree[cur][1] * ld;
                int j = warp - 1, l0 = 0;
                while (j >= cnt) {
                    j -= cnt;
                    l0 += 32;
                }
                while (l0 < npair) {
                    const int k = k0 + j, l = l0 + lane;
                    if (l < npair) {
                        const float4 pk = P[k], pl = P[l];
                        const bool to_lo = j == 0 && c > 0, to_hi = j == cnt - 1 && !last;
                        if (pk.z != 0.f || pl.z != 0.f || to_lo || to_hi) {
                            df *ra = rows + (size_t)sT[j] * ld, *rb = rows + (size_t)sB[j] * ld;
                            df *wa = to_lo ? out_lo : ra, *wb = to_hi ? out_hi : rb;
                            const int a = rr_top(l, r, mp), b = rr_bot(l, r, mp);
                            if (l == k) {   // the pivot; the diagonal lives in diag
                                wa[b] = {0.f, 0.f};
                                wb[a] = {0.f, 0.f};
                            } else {
                                df xaa = ra[a], xab = ra[b], xba = rb[a], xbb = rb[b];
                                if (pk.z != 0.f || pl.z != 0.f) {
                                    const df ck = {pk.x, pk.y}, sk = {pk.z, pk.w}, cl_ = {pl.x, pl.y}, sl = {pl.z, pl.w};
                                    const df yaa = df_rot(ck, xaa, sk, xba), yab = df_rot(ck, xab, sk, xbb);
                                    const df yba = df_rot(sk, xaa, df_neg(ck), xba), ybb = df_rot(sk, xab, df_neg(ck), xbb);
                                    xaa = df_rot(cl_, yaa, sl, yab);
                                    xab = df_rot(sl, yaa, df_neg(cl_), yab);
                                    xba = df_rot(cl_, yba, sl, ybb);
                                    xbb = df_rot(sl, yba, df_neg(cl_), ybb);
                                }
                                wa[a] = xaa;
                                wa[b] = xab;
                                wb[a] = xba;
                                wb[b] = xbb;
                            }
                        }
                    }
                    j += nwarp - 1;
                    while (j >= cnt) {
                        j -= cnt;
                        l0 += 32;
                    }
                }
            }
            ++g;
            // the rows' new slots
            int *nT = slot_of(nxt, 0), *nB = slot_of(nxt, 1);
            for (int jj = bs - 1 - tid; jj < cnt; jj += bs) {
                nT[jj] = c == 0 && jj == 0 ? sT[0] : jj + 1 < cnt ? sT[jj + 1] : last ? sB[cnt - 1] : myfree[cur][0];
                nB[jj] = jj > 0 ? sB[jj - 1] : c == 0 ? sT[1] : myfree[cur][1];
            }
            if (warp == nwarp / 2 && lane == 0) {
                const int fT = c == 0 ? sB[cnt - 1] : sT[0], fB = last ? sT[0] : sB[cnt - 1];
                myfree[nxt][0] = fT;
                myfree[nxt][1] = fB;
                if (c > 0) cl.map_shared_rank(&nbfree[nxt][1], c - 1)[0] = fB;
                if (!last) cl.map_shared_rank(&nbfree[nxt][0], c + 1)[0] = fT;
            }
            if (tid == bs - 1) {
                if (r == 0) mx[(sweep + 1) & 1] = 0;
                if (r == mp - 2)
                    for (int q = 0; q < C; ++q) cl.map_shared_rank(&allmx[c], q)[0] = mx[sweep & 1];
            }
            cl.sync();
            cur = nxt;
        }
        float top = 0.f;
        for (int q = 0; q < C; ++q) top = fmaxf(top, __int_as_float(allmx[q]));
        if (top < sqrtf(rel_tol)) break;
    }
    if (c == 0) {
        for (int i = tid; i < m; i += bs) lam[i] = scalbn((double)diag[i].h + (double)diag[i].l, scale);
        if (tid == 0) *nrounds = (int)g;
    }
}

// Q = the product of the logged rotations, row by row of I, one warp per row.
// A serial chain over the rounds, so the row stays in registers in the order of
// the round's positions: a lane holds K consecutive ones (upper and lower
// index), and from round to round the upper ones move down one position and the
// lower ones up one (two shuffles).  The log streams through shared memory, G
// rounds ahead.  0.18 us a round; with the row in shared memory, gathered by index, 0.64
// (1.53 ms at m = 300, 0.42 now).
// A log entry (c, s) rotates (upper, lower), or (lower, upper) if c < 0; column
// i goes to column rank[i] of Q (rank = nullptr: i).
template <int K>
__global__ void __launch_bounds__(32) k_jacobi_vectors(int m, const float2 *rlog,
                                                       const int *nrounds, const int *rank,
                                                       double *__restrict__ Q) {
    chain_wait();
    constexpr int G = JVEC_ROUNDS;
    extern __shared__ float4 vsm4[];
    const int mp = m + (m & 1), npair = mp / 2;
    const int lane = threadIdx.x, row = blockIdx.x;
    const int n = *nrounds, nch = (n + G - 1) / G;
    const int stage = G * npair * (int)sizeof(float2);   // a multiple of 16
    char *buf = reinterpret_cast<char *>(vsm4);
    auto fetch = [&](int ch) {
        if (ch < nch) {
            // the last chunk's odd half of 16 bytes: the log has one more round
            const int bytes = (min(G, n - ch * G) * npair * (int)sizeof(float2) + 15) / 16 * 16;
            const char *src = reinterpret_cast<const char *>(rlog) + (int64_t)ch * stage;
            const unsigned dst = smem_addr(buf + (ch & 1) * stage);
            for (int o = lane * 16; o < bytes; o += 32 * 16)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + o), "l"(src + o) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float top[K], bot[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        const int k = lane * K + i;
        top[i] = k < npair && rr_top(k, 0, mp) == row ? 1.f : 0.f;
        bot[i] = k < npair && rr_bot(k, 0, mp) == row ? 1.f : 0.f;
    }
    fetch(0);
    fetch(1);
    for (int ch = 0; ch < nch; ++ch) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        const float2 *w = reinterpret_cast<const float2 *>(buf + (ch & 1) * stage) + lane * K;
        const int rounds = min(G, n - ch * G);
        for (int j = 0; j < rounds; ++j, w += npair) {
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const float2 v = lane * K + i < npair ? w[i] : make_float2(1.f, 0.f);
                const bool sw = v.x < 0.f;
                float x = sw ? bot[i] : top[i], y = sw ? top[i] : bot[i];
                rotate(fabsf(v.x), v.y, x, y);
                top[i] = sw ? y : x;
                bot[i] = sw ? x : y;
            }
            const float up = __shfl_down_sync(0xffffffffu, top[0], 1);      // next lane's first upper
            const float dn = __shfl_up_sync(0xffffffffu, bot[K - 1], 1);    // previous lane's last lower
            const float first = top[0], second = npair == 1 ? bot[0] : K > 1 ? top[K > 1 ? 1 : 0] : up;
            float t[K];
#pragma unroll
            for (int i = 0; i < K; ++i) {
                t[i] = i + 1 < K ? top[i + 1 < K ? i + 1 : 0] : up;
                if (lane * K + i == npair - 1) t[i] = bot[i];   // the last lower turns upper
            }
#pragma unroll
            for (int i = K - 1; i > 0; --i) bot[i] = bot[i - 1];
            bot[0] = dn;
#pragma unroll
            for (int i = 0; i < K; ++i) top[i] = t[i];
            if (lane == 0) {       // position 0: the upper stays, the next upper turns lower
                top[0] = first;
                bot[0] = second;
            }
        }
        __syncwarp();
        fetch(ch + 2);
    }
    const int r = n % (mp - 1);
#pragma unroll
    for (int i = 0; i < K; ++i) {
        const int k = lane * K + i;
        if (k >= npair) continue;
        const int a = rr_top(k, r, mp), b = rr_bot(k, r, mp);
        if (a < m) Q[(int64_t)row * m + (rank ? rank[a] : a)] = (double)top[i];
        if (b < m) Q[(int64_t)row * m + (rank ? rank[b] : b)] = (double)bot[i];
    }
}

void jacobi_vectors(Ctx &ctx, int m, const float2 *rlog, const int *nrounds, const int *rank, double *Q) {
    const int npair = (m + 1) / 2;
    const size_t smem = 2 * (size_t)JVEC_ROUNDS * npair * sizeof(float2);
    ctx.before(KC_SMALL_DENSE, 8.0 * m * m, 3.0 * (double)m * m * m * 8);
#define JV(K) case K: launch_chained(ctx, k_jacobi_vectors<K>, m, 32, smem, m, rlog, nrounds, rank, Q); break
    switch ((npair + 31) / 32) {
        JV(1); JV(2); JV(3); JV(4); JV(5); JV(6);
        default: launch_chained(ctx, k_jacobi_vectors<7>, m, 32, smem, m, rlog, nrounds, rank, Q); break;
    }
#undef JV
    ctx.after();
}

// ---------------------------------------------------------------------------
// cooperative FP64 Jacobi on a global m x m matrix A (overwritten; diag = lam)
// accumulating V <- V J.  Pairs whose |a_pq| is below eps abs_factor ||A||_F
// are left alone.  cnt[4] (device): rotation counters of the last two
// sweeps (0, 1) and their pre-check flags (2, 3).  All blocks
// compute the same rotations from the same data, so no broadcast is needed.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
k_jacobi_coop(int m, double *__restrict__ A, double *__restrict__ V, double *__restrict__ lam, int max_sweeps,
              const double *__restrict__ normA, double abs_factor, int *__restrict__ cnt,
              int32_t *__restrict__ info) {
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    const int mp = m + (m & 1);
    const int npair = mp / 2;
    __shared__ double cs[512], sn[512], dp[512], dq[512];
    __shared__ int pp[512], qq[512];
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gsz = (int64_t)gridDim.x * blockDim.x;
    const double eps = DBL_EPSILON;
    const double absmin = fro_norm(normA) * eps * abs_factor;
    // cnt[2 + (sweep & 1)]: set when some pair still passes the rotation test
    if (gtid == 0) cnt[2] = cnt[3] = 0;
    grid.sync();
    int sweep = 0;
    for (; sweep < max_sweeps; ++sweep) {
        if (blockIdx.x == 0 && threadIdx.x == 0) cnt[sweep & 1] = 0;
        // A sweep that would rotate nothing leaves A and V as they are: test
        // every pair against the rotation criterion first (one pass over A)
        // instead of running the sweep's 2 (mp - 1) grid barriers to find out.
        {
            int found = 0;
            for (int64_t e = gtid; e < (int64_t)m * m && !found; e += gsz) {
                const int p = (int)(e / m), q = (int)(e % m);
                if (q <= p) continue;
                const double apq = A[e];
                const double scale = sqrt(fabs(A[(int64_t)p * m + p] * A[(int64_t)q * m + q]));
                found = fabs(apq) > eps * scale && fabs(apq) > absmin;
            }
            if (found) atomicOr(&cnt[2 + (sweep & 1)], 1);
            grid.sync();
            const int any = *(volatile int *)&cnt[2 + (sweep & 1)];
            // the other flag was last read before this sweep's barriers: reset it for the next sweep
            if (gtid == 0) cnt[2 + ((sweep + 1) & 1)] = 0;
            if (!any) break;
        }
        __syncthreads();
        for (int r = 0; r < mp - 1; ++r) {
            // Every block derives all rotations of the round from the pair
            // blocks (p,p), (q,q), (p,q).  Those entries are not written by the
            // row phase (below), so a block still reading them here cannot race
            // with a block that has moved on to the row phase.
            for (int k = threadIdx.x; k < npair; k += blockDim.x) {
                int a, b;
                rr_pair(k, r, mp, a, b);
                const int p = min(a, b), q = max(a, b);
                double c = 1, s = 0, t = 0, app = 0, aqq = 0, apq = 0;
                if (q < m) {
                    apq = A[(int64_t)p * m + q];
                    app = A[(int64_t)p * m + p];
                    aqq = A[(int64_t)q * m + q];
                    const double scale = sqrt(fabs(app * aqq));
                    if (fabs(apq) > eps * scale && fabs(apq) > absmin) {
                        const double th = (aqq - app) / (2 * apq);
                        t = (th >= 0 ? 1.0 : -1.0) / (fabs(th) + sqrt(1.0 + th * th));
                        c = 1.0 / sqrt(1.0 + t * t);
                        s = t * c;
                        // every applied rotation counts: near-degenerate pairs
                        // converge only once they stop rotating
                        if (blockIdx.x == 0) atomicAdd(&cnt[sweep & 1], 1);
                    }
                }
                cs[k] = c;
                sn[k] = s;
                dp[k] = app - t * apq;   // rotated diagonal of the pair block
                dq[k] = aqq + t * apq;
                pp[k] = p;
                qq[k] = (q < m && s != 0.0) ? q : -1;
            }
            __syncthreads();
            // rows p, q <- J^T (rows p, q), except the pair block itself
            for (int64_t e = gtid; e < (int64_t)npair * m; e += gsz) {
                const int k = (int)(e / m), col = (int)(e % m);
                const int q = qq[k];
                if (q < 0) continue;
                const int p = pp[k];
                if (col == p || col == q) continue;
                const double c = cs[k], s = sn[k];
                const double apk = A[(int64_t)p * m + col], aqk = A[(int64_t)q * m + col];
                A[(int64_t)p * m + col] = c * apk - s * aqk;
                A[(int64_t)q * m + col] = s * apk + c * aqk;
            }
            grid.sync();
            // columns p, q <- (columns p, q) J; the pair block in closed form
            for (int64_t e = gtid; e < (int64_t)npair * m; e += gsz) {
                const int k = (int)(e / m), row = (int)(e % m);
                const int q = qq[k];
                if (q < 0) continue;
                const int p = pp[k];
                const double c = cs[k], s = sn[k];
                if (row == p) {
                    A[(int64_t)p * m + p] = dp[k];
                    A[(int64_t)p * m + q] = 0.0;
                } else if (row == q) {
                    A[(int64_t)q * m + q] = dq[k];
                    A[(int64_t)q * m + p] = 0.0;
                } else {
                    const double akp = A[(int64_t)row * m + p], akq = A[(int64_t)row * m + q];
                    A[(int64_t)row * m + p] = c * akp - s * akq;
                    A[(int64_t)row * m + q] = s * akp + c * akq;
                }
                const double vkp = V[(int64_t)row * m + p], vkq = V[(int64_t)row * m + q];
                V[(int64_t)row * m + p] = c * vkp - s * vkq;
                V[(int64_t)row * m + q] = s * vkp + c * vkq;
            }
            grid.sync();
        }
        const int n_rot = *(volatile int *)&cnt[sweep & 1];
        grid.sync();
        if (n_rot == 0) {
            ++sweep;
            break;
        }
    }
    for (int64_t i = gtid; i < m; i += gsz) lam[i] = A[i * m + i];
    if (gtid == 0 && info) *info = sweep;
}

__global__ void k_identity(int m, double *__restrict__ V) {
    chain_wait();
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e < (int64_t)m * m) V[e] = (e / m == e % m) ? 1.0 : 0.0;
}

// final ordering: lam ascending, Q columns permuted.  Every block ranks all
// eigenvalues (as integers of the same order: FP64 compares run on the slow
// FP64 pipe) and moves its rows, one warp per row.
__global__ void __launch_bounds__(256) k_sort_eig(int m, const double *lam_in, const double *S,
                                                  double *__restrict__ lam, double *__restrict__ Q) {
    chain_wait();
    __shared__ long long key[1024];
    __shared__ int rank[1024];
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        const long long b = __double_as_longlong(lam_in[i]);
        key[i] = b ^ ((b >> 63) & 0x7fffffffffffffffll);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        const long long ki = key[i];
        int r = 0;
#pragma unroll 4
        for (int j = 0; j < m; ++j) r += (key[j] < ki) || (key[j] == ki && j < i);
        rank[i] = r;
        if (blockIdx.x == 0) lam[r] = lam_in[i];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= m) return;
    for (int j = lane; j < m; j += 32) Q[(int64_t)row * m + rank[j]] = S[(int64_t)row * m + j];
}

// Matrices of the eigensolver's workspace in front of its vectors and counters:
// the group blocks (2 mp^2 doubles) and S0, S1, G, Y, T, V (6 m^2)
static size_t syev_matrix_bytes(int m) {
    const size_t mp = (size_t)(m + (m & 1)), m2 = (size_t)m * m;
    return (2 * mp * mp + 6 * m2) * sizeof(double);
}
size_t small_syev_work_bytes(int m) {
    // + lam0, partial norms, counters, component labels and sizes (2 m ints)
    return syev_matrix_bytes(m) + (2 * (size_t)m + 2) * sizeof(double) + 2 * (size_t)m * sizeof(int) + 4096;
}
// The rotation log of the Jacobi that precedes the refinement (one entry per
// pair and round, one round more) takes the matrices' place behind S0, which are
// written after the vectors are formed.  It holds 13 sweeps, a few less below
// m = 10; 6 to 9 are the rule.
static int log_sweeps(int m, int most) {
    const size_t mp = (size_t)(m + (m & 1));
    const size_t room = syev_matrix_bytes(m) - (size_t)m * m * sizeof(double) - 16;   // the log starts on 16 bytes
    const size_t rounds = room / (mp / 2 * sizeof(float2)) - 1;
    return (int)std::min<size_t>(most, rounds / (mp - 1));
}

// ---------------------------------------------------------------------------
// Iterative refinement of an approximate eigendecomposition (Ogita and
// Aishima, "Iterative refinement for symmetric eigenvalue decomposition",
// Japan J. Indust. Appl. Math. 35, 2018).  With Xh the current eigenvector
// matrix, G = Xh^T Xh, T = Xh^T S Xh and R = I - G, the exact eigenvectors
// are X = Xh (I + E) with, to first order in the error,
//   E + E^T = R                         (orthonormality)
//   T + E^T D + D E = D                 (diagonalisation, D = eigenvalues)
// so lam_i = t_ii / g_ii, e_ii = r_ii / 2 and, for i != j,
//   e_ij = (t_ij + lam_j r_ij) / (lam_j - lam_i).
// A pair is refined this way only while the step is small: its eigenvalues
// more than delta = 2 ||T - D||_F apart and |e_ij| <= 1/8; other pairs get
// e_ij = r_ij / 2 (orthonormality only) and are left to k_oa_components.
// (The paper's delta also carries ||S|| ||R||; here every step is preceded
// by a Newton-Schulz orthonormalisation X <- X (3 I - X^T X) / 2, which
// keeps R at rounding level, so that term is dropped: with the FP32
// Jacobi's ||R|| ~ 1e-4 it would group most of a graded spectrum.)  The
// products are FP64 GEMMs; three steps reach FP64 accuracy from the FP32
// Jacobi's vectors wherever the pairs are separated.
// ---------------------------------------------------------------------------
// lam_t = t_ii / g_ii, and per block the partial sum of ||T - D||_F^2 over its
// rows (fixed order; one block for the whole matrix took 33 us at m = 150,
// all of it FP64 issue; this takes 5)
__global__ void __launch_bounds__(256) k_oa_norms(int m, const double *G, const double *T,
                                                  double *__restrict__ lam_t, double *__restrict__ part) {
    chain_wait();
    __shared__ double red[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double off = 0.0;
    for (int i = blockIdx.x * 8 + warp; i < m; i += OA_PARTS * 8) {
        const double *Ti = T + (int64_t)i * m;
        const double ti = Ti[i], li = ti / G[(int64_t)i * m + i];
        if (lane == 0) lam_t[i] = li;
        for (int j = lane; j < m; j += 32) {
            const double d = i == j ? ti - li : Ti[j];
            off = fma(d, d, off);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) off += __shfl_xor_sync(0xffffffffu, off, o);
    if (lane == 0) red[warp] = off;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int w = 0; w < 8; ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

// Ep = I + E (row-major), one thread per entry over many blocks (the FP64
// divisions spread over the GPU); the pair threshold is delta = 2 ||T - D||_F
__global__ void __launch_bounds__(256) k_oa_step(int m, const double *G, const double *T,
                                                 const double *lam_t, const double *part,
                                                 double *__restrict__ Ep) {
    chain_wait();
    __shared__ double delta;
    if (threadIdx.x < 32) {
        double s = part[threadIdx.x] + part[threadIdx.x + 32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) delta = 2.0 * sqrt(s);
    }
    __syncthreads();
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)m * m) return;
    const int i = (int)(e / m), j = (int)(e % m);
    const double r = (i == j ? 1.0 : 0.0) - G[e];
    double v;
    if (i == j) {
        v = 1.0 + 0.5 * r;
    } else {
        const double li = lam_t[i], lj = lam_t[j], num = T[e] + lj * r;
        const bool sep = fabs(li - lj) > delta && 8.0 * fabs(num) <= fabs(lj - li);
        v = sep ? num / (lj - li) : 0.5 * r;
    }
    Ep[e] = v;
}

// After the refinement T = Q^T S Q is diagonal up to rounding except inside
// groups of (nearly) equal eigenvalues.  Indices joined by an off-diagonal
// entry above tau = 4 m u ||S||_F (about ten times the rounding of the FP64
// products) form components (label propagation); each
// component of two or more is diagonalised by cyclic FP64 Jacobi and its
// columns of Q rotated; lam receives the diagonal (unsorted).  Workspace:
// label, size (m ints each), blk, W (m^2 doubles each), Qc (m^2 doubles).
__global__ void __launch_bounds__(1024) k_oa_components(int m, const double *T,
                                                       const double *normS, double *__restrict__ Q,
                                                       double *__restrict__ lam, int *__restrict__ label,
                                                       int *__restrict__ size, double *__restrict__ blk,
                                                       double *__restrict__ Wm, double *__restrict__ Qc) {
    chain_wait();
    const int tid = threadIdx.x, bs = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nwarp = bs >> 5;
    __shared__ int changed, k, nrot;
    __shared__ int members[1024];
    __shared__ double cs[512], sn[512];
    __shared__ int pp[512], qq[512];
    const double tau = 4.0 * m * 1.1102230246251565e-16 * fro_norm(normS);
    // T is symmetric (its product is mirrored); |t| > tau compared as integers
    const long long tau_bits = __double_as_longlong(tau);
    auto joined = [&](int i, int j) {
        return (__double_as_longlong(T[(int64_t)i * m + j]) & 0x7fffffffffffffffll) > tau_bits;
    };
    for (int i = tid; i < m; i += bs) {
        label[i] = i;
        size[i] = 0;
    }
    __syncthreads();
    // labels only decrease and label[i] <= i, so the jumps end; a chain of
    // m indices needs at most m passes
    for (int pass = 0; pass <= m; ++pass) {
        if (tid == 0) changed = 0;
        __syncthreads();
        for (int e = tid; e < m * m; e += bs) {
            const int i = e / m, j = e % m;
            if (j <= i || !joined(i, j)) continue;
            const int li = label[i], lj = label[j];
            if (li != lj) {
                const int l = min(li, lj);
                atomicMin(&label[i], l);
                atomicMin(&label[j], l);
                changed = 1;
            }
        }
        __syncthreads();
        for (int i = tid; i < m; i += bs) {
            int l = label[i];
            while (label[l] != l) l = label[l];
            atomicMin(&label[i], l);
        }
        __syncthreads();
        const int c = changed;
        __syncthreads();
        if (!c) break;
    }
    for (int i = tid; i < m; i += bs) atomicAdd(&size[label[i]], 1);
    __syncthreads();
    for (int i = tid; i < m; i += bs)
        if (size[label[i]] == 1) lam[i] = T[(int64_t)i * m + i];
    for (int r = 0; r < m; ++r) {
        if (size[r] < 2) continue;   // uniform: every thread reads the same entry
        if (tid == 0) {
            int c = 0;
            for (int i = r; i < m && c < 1024; ++i)
                if (label[i] == r) members[c++] = i;
            k = c;
        }
        __syncthreads();
        const int kk = k;
        for (int e = tid; e < kk * kk; e += bs) {
            const int a = e / kk, b = e % kk;
            const int ia = members[a], ib = members[b];
            blk[e] = 0.5 * (T[(int64_t)ia * m + ib] + T[(int64_t)ib * m + ia]);
            Wm[e] = a == b ? 1.0 : 0.0;
        }
        __syncthreads();
        const int kp = kk + (kk & 1), npair = kp / 2;
        for (int sweep = 0; sweep < 40; ++sweep) {
            if (tid == 0) nrot = 0;
            __syncthreads();
            for (int rd = 0; rd < kp - 1; ++rd) {
                for (int t = tid; t < npair; t += bs) {
                    int a, b;
                    rr_pair(t, rd, kp, a, b);
                    const int p = min(a, b), q = max(a, b);
                    double c = 1.0, s = 0.0;
                    if (q < kk) {
                        const double apq = blk[p * kk + q];
                        if (fabs(apq) > tau) {
                            const double app = blk[p * kk + p], aqq = blk[q * kk + q];
                            const double th = (aqq - app) / (2.0 * apq);
                            const double tt = (th >= 0 ? 1.0 : -1.0) / (fabs(th) + sqrt(1.0 + th * th));
                            c = 1.0 / sqrt(1.0 + tt * tt);
                            s = tt * c;
                            atomicAdd(&nrot, 1);
                        }
                    }
                    cs[t] = c;
                    sn[t] = s;
                    pp[t] = p;
                    qq[t] = (q < kk && s != 0.0) ? q : -1;
                }
                __syncthreads();
                for (int t = warp; t < npair; t += nwarp) {
                    const int q = qq[t];
                    if (q < 0) continue;
                    const int p = pp[t];
                    const double c = cs[t], s = sn[t];
                    for (int col = lane; col < kk; col += 32) {
                        const double apk = blk[p * kk + col], aqk = blk[q * kk + col];
                        blk[p * kk + col] = c * apk - s * aqk;
                        blk[q * kk + col] = s * apk + c * aqk;
                    }
                }
                __syncthreads();
                for (int t = warp; t < npair; t += nwarp) {
                    const int q = qq[t];
                    if (q < 0) continue;
                    const int p = pp[t];
                    const double c = cs[t], s = sn[t];
                    for (int row = lane; row < kk; row += 32) {
                        const double akp = blk[row * kk + p], akq = blk[row * kk + q];
                        blk[row * kk + p] = c * akp - s * akq;
                        blk[row * kk + q] = s * akp + c * akq;
                        const double wkp = Wm[row * kk + p], wkq = Wm[row * kk + q];
                        Wm[row * kk + p] = c * wkp - s * wkq;
                        Wm[row * kk + q] = s * wkp + c * wkq;
                    }
                }
                __syncthreads();
                for (int t = tid; t < npair; t += bs) {
                    const int q = qq[t];
                    if (q < 0) continue;
                    const int p = pp[t];
                    blk[p * kk + q] = 0.0;
                    blk[q * kk + p] = 0.0;
                }
                __syncthreads();
            }
            const int nr = nrot;
            __syncthreads();
            if (nr == 0) break;
        }
        for (int a = tid; a < kk; a += bs) lam[members[a]] = blk[a * kk + a];
        for (int e = tid; e < m * kk; e += bs) {
            const int row = e / kk, b = e % kk;
            Qc[e] = Q[(int64_t)row * m + members[b]];
        }
        __syncthreads();
        for (int e = tid; e < m * kk; e += bs) {
            const int row = e / kk, a = e % kk;
            double v = 0.0;
            for (int b = 0; b < kk; ++b) v = fma(Qc[row * kk + b], Wm[b * kk + a], v);
            Q[(int64_t)row * m + members[a]] = v;
        }
        __syncthreads();
    }
}

// At most one cooperative (grid-barrier) kernel of this process is in flight
// on the device at any time: concurrent handles on other streams take turns,
// so two partially resident cooperative grids can never wait on each other.
static std::mutex g_coop_mutex;

// Returns the launch's or the wait's error: a refused cooperative launch (too
// few co-resident blocks, say) must not leave the caller polishing an
// unrotated matrix.
static cudaError_t coop_jacobi(Ctx &ctx, int m, double *A, double *V, double *lam, int max_sweeps,
                               const double *normA, double abs_factor, int *cnt) {
    static const int per_sm = [] {
        int b = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_jacobi_coop, 256, 0);
        return b;
    }();
    const int64_t work = (int64_t)((m + 1) / 2) * m;
    int blocks = (int)std::min<int64_t>((work + 255) / 256, std::min(per_sm * ctx.sm_count, ctx.sm_count));
    if (blocks < 1) blocks = 1;
    int32_t *info = nullptr;
    void *args[] = {&m, &A, &V, &lam, &max_sweeps, (void *)&normA, &abs_factor, &cnt, &info};
    thread_local cudaEvent_t done = nullptr;
    if (!done) {
        const cudaError_t e = cudaEventCreateWithFlags(&done, cudaEventDisableTiming);
        if (e != cudaSuccess) {
            done = nullptr;
            return e;
        }
    }
    std::lock_guard<std::mutex> lock(g_coop_mutex);
    ctx.before(KC_SMALL_DENSE, 24.0 * m * m, 9.0 * (double)m * m * m * 3);
    cudaError_t e = cudaLaunchCooperativeKernel((const void *)k_jacobi_coop, dim3(blocks), dim3(256), args, 0,
                                                ctx.stream);
    ctx.after();
    if (e != cudaSuccess) return e;
    e = cudaEventRecord(done, ctx.stream);
    if (e != cudaSuccess) return e;
    return cudaEventSynchronize(done);
}

// Whether the current device places the double-float Jacobi's cluster (its size is
// not a portable one)
static bool jacobi_df_fits() {
    constexpr int kMaxDevices = 64;
    static std::once_flag once[kMaxDevices];
    static bool fits[kMaxDevices];
    int dev = 0;
    cudaGetDevice(&dev);
    const int i = dev < 0 || dev >= kMaxDevices ? 0 : dev;
    std::call_once(once[i], [i] {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = JDF_CTAS;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.gridDim = dim3(JDF_CTAS);
        cfg.blockDim = dim3(JDF_THREADS);
        cfg.dynamicSmemBytes = JacobiShape(JDF_MAX, JDF_CTAS).bytes();
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int n = 0;
        raise_smem_limits();
        fits[i] =
            cudaFuncSetAttribute(k_jacobi_df, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&n, k_jacobi_df, &cfg) == cudaSuccess && n > 0;
        if (!fits[i]) cudaGetLastError();
    });
    return fits[i];
}

cudaError_t small_syev(Ctx &ctx, int m, const double *S, double *lam, double *Q, double *work, int mode) {
    const size_t m2 = (size_t)m * m;
    const size_t mp = (size_t)(m + (m & 1));
    double *S0 = work;
    void *Ag = S0 + m2;
    void *Vg = S0 + m2 + mp * mp;
    double *S1 = S0 + m2 + 2 * mp * mp;
    double *G = S1 + m2;
    double *Ym = G + m2;
    double *Tm = Ym + m2;
    double *Vm = Tm + m2;
    double *lam0 = Vm + m2;
    double *normA = lam0 + m;             // FRO_PARTS partial sums of ||S||_F^2
    double *oa_part = normA + FRO_PARTS;  // OA_PARTS partial sums of the refinement's ||T - D||_F^2
    int *cnt = reinterpret_cast<int *>(oa_part + OA_PARTS);
    int32_t *cst = cnt + 4;   // cnt[6]: rounds of the Jacobi
    int *label = cst + 4, *csize = label + m;   // label: the FP32 Jacobi's ranks first
    // 16-byte aligned (work is a multiple of 8 bytes) for the vectors' 16-byte loads
    float2 *rlog = reinterpret_cast<float2 *>((reinterpret_cast<uintptr_t>(Ag) + 15) / 16 * 16);

    ctx.before(KC_SMALL_DENSE, 8.0 * m2, 2.0 * m2);
    launch_chained(ctx, k_fro, FRO_PARTS, 256, 0, m, S, normA);
    ctx.after();
    auto identity = [&](double *V) {
        ctx.before(KC_SMALL_DENSE, 8.0 * m2, 0);
        launch_chained(ctx, k_identity, (unsigned)((m2 + 255) / 256), 256, 0, m, V);
        ctx.after();
    };
    // The one-block FP32 stage takes m <= JMAX (A in its shared memory), the
    // double-float cluster m <= JDF_MAX; beyond that, without the refinement, and
    // on a device that does not place the cluster, the cooperative FP64 Jacobi.
    if (mode == 0 || m > JDF_MAX || (m > JMAX && (mode == 1 || !jacobi_df_fits()))) {
        identity(Vm);
        cudaMemcpyAsync(Tm, S, m2 * sizeof(double), cudaMemcpyDeviceToDevice, ctx.stream);
        const cudaError_t e = coop_jacobi(ctx, m, Tm, Vm, lam0, 60, normA, 0.5 / m, cnt);
        if (e != cudaSuccess) return e;
        ctx.before(KC_SMALL_DENSE, 16.0 * m2, 0);
        launch_chained(ctx, k_sort_eig, (m + 7) / 8, 256, 0, m, lam0, Vm, lam, Q);
        ctx.after();
        return cudaGetLastError();
    }
    // stage 1: eigenvectors to single precision
    raise_smem_limits();
    if (m <= JMAX) {
        const Jacobi32Shape sh(m);
        ctx.before(KC_SMALL_DENSE, 8.0 * m2, 6.0 * (double)m * m2 * 8);
        launch_chained(ctx, k_jacobi32, 1, sh.threads(), sh.bytes(), m, S, lam0, label, rlog, cnt + 6,
                       log_sweeps(m, J32_SWEEPS), 1e-6f);
        ctx.after();
        jacobi_vectors(ctx, m, rlog, cnt + 6, label, S0);
    } else {
        ctx.before(KC_SMALL_DENSE, 12.0 * m2, 9.0 * (double)m * m2 * 8);
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = JDF_CTAS;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.gridDim = dim3(JDF_CTAS);
        cfg.blockDim = dim3(JDF_THREADS);
        cfg.dynamicSmemBytes = JacobiShape(m, JDF_CTAS).bytes();
        cfg.stream = ctx.stream;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        const cudaError_t je =
            cudaLaunchKernelEx(&cfg, k_jacobi_df, m, S, (const double *)normA, lam0, rlog, cnt + 6,
                               log_sweeps(m, JDF_SWEEPS), 1e-10f);
        ctx.after();
        if (je != cudaSuccess) return je;
        jacobi_vectors(ctx, m, rlog, cnt + 6, nullptr, S0);
    }
    if (mode == 2) {
        // stage 2: three rounds of an orthonormalisation step and a
        // refinement step X <- X (I + E) from the FP64 products G = X^T X and
        // T = X^T (S X); then the groups of nearly equal eigenvalues are
        // diagonalised and the pairs sorted
        double *X0 = S0, *X1 = S1;
        const unsigned eg = (unsigned)((m2 + 255) / 256);
        for (int it = 0; it < 3; ++it) {
            small_ns_factor(ctx, m, X0, Vm);
            dgemm(ctx, 0, 0, m, m, m, X0, m, Vm, m, 0.0, X1, m, 1, nullptr, KC_SMALL_DENSE);
            std::swap(X0, X1);
            dgemm(ctx, 1, 0, m, m, m, X0, m, X0, m, 0.0, G, m, 1, nullptr, KC_SMALL_DENSE, true);
            dgemm(ctx, 0, 0, m, m, m, S, m, X0, m, 0.0, Ym, m, 1, nullptr, KC_SMALL_DENSE);
            dgemm(ctx, 1, 0, m, m, m, X0, m, Ym, m, 0.0, Tm, m, 1, nullptr, KC_SMALL_DENSE, true);
            ctx.before(KC_SMALL_DENSE, 16.0 * m2, 4.0 * m2);
            launch_chained(ctx, k_oa_norms, OA_PARTS, 256, 0, m, G, Tm, lam0, oa_part);
            ctx.after();
            ctx.before(KC_SMALL_DENSE, 24.0 * m2, 8.0 * m2);
            launch_chained(ctx, k_oa_step, eg, 256, 0, m, G, Tm, lam0, oa_part, Vm);
            ctx.after();
            dgemm(ctx, 0, 0, m, m, m, X0, m, Vm, m, 0.0, X1, m, 1, nullptr, KC_SMALL_DENSE);
            std::swap(X0, X1);
        }
        // the last refinement step leaves R at the square of its largest
        // accepted steps: three orthonormalisation steps bring it back to
        // rounding level before the groups are rotated
        for (int it = 0; it < 3; ++it) {
            small_ns_factor(ctx, m, X0, Vm);
            dgemm(ctx, 0, 0, m, m, m, X0, m, Vm, m, 0.0, X1, m, 1, nullptr, KC_SMALL_DENSE);
            std::swap(X0, X1);
        }
        dgemm(ctx, 0, 0, m, m, m, S, m, X0, m, 0.0, Ym, m, 1, nullptr, KC_SMALL_DENSE);
        dgemm(ctx, 1, 0, m, m, m, X0, m, Ym, m, 0.0, Tm, m, 1, nullptr, KC_SMALL_DENSE, true);
        if (m > JMAX) {
            // a large group of close eigenvalues is too much for one block:
            // the cooperative Jacobi rotates whatever the refinement left
            // above rounding level (it returns after one look if nothing is).
            // That level is 1/2 eps ||S||_F: the entries of T = X^T S X between
            // separated pairs are rounding of at most 0.28 eps ||S||_F (m = 161
            // .. 448, spectra over up to six decades), so these cost no sweep,
            // and a pair that the refinement took for too close to separate is
            // rotated to it.
            identity(Vm);
            const cudaError_t e = coop_jacobi(ctx, m, Tm, Vm, lam0, 60, normA, 0.5, cnt);
            if (e != cudaSuccess) return e;
            dgemm(ctx, 0, 0, m, m, m, X0, m, Vm, m, 0.0, X1, m, 1, nullptr, KC_SMALL_DENSE);
            ctx.before(KC_SMALL_DENSE, 16.0 * m2, 0);
            launch_chained(ctx, k_sort_eig, (m + 7) / 8, 256, 0, m, lam0, X1, lam, Q);
            ctx.after();
            return cudaGetLastError();
        }
        ctx.before(KC_SMALL_DENSE, 24.0 * m2, 4.0 * m2);
        launch_chained(ctx, k_oa_components, 1, 1024, 0, m, Tm, normA, X0, lam0, label, csize, (double *)Ag,
                                                     (double *)Vg, X1);
        ctx.after();
        ctx.before(KC_SMALL_DENSE, 16.0 * m2, 0);
        launch_chained(ctx, k_sort_eig, (m + 7) / 8, 256, 0, m, lam0, X0, lam, Q);
        ctx.after();
        return cudaGetLastError();
    }
    // stage 2: FP64 re-orthonormalisation S1 = S0 R^{-1}, G = S0^T S0 = R^T R
    dgemm(ctx, 1, 0, m, m, m, S0, m, S0, m, 0.0, G, m, 1, nullptr, KC_SMALL_DENSE, true);
    small_chol_inv(ctx, m, G, G, Ym, cst, nullptr, 0.0);
    dgemm(ctx, 0, 0, m, m, m, S0, m, Ym, m, 0.0, S1, m, 1, nullptr, KC_SMALL_DENSE);
    // T = S1^T A S1, then polish T by FP64 Jacobi, S = S1 V
    dgemm(ctx, 0, 0, m, m, m, S, m, S1, m, 0.0, Ym, m, 1, nullptr, KC_SMALL_DENSE);
    dgemm(ctx, 1, 0, m, m, m, S1, m, Ym, m, 0.0, Tm, m, 1, nullptr, KC_SMALL_DENSE);
    identity(Vm);
    const cudaError_t e = coop_jacobi(ctx, m, Tm, Vm, lam0, 20, normA, 0.5 / m, cnt);
    if (e != cudaSuccess) return e;
    dgemm(ctx, 0, 0, m, m, m, S1, m, Vm, m, 0.0, S0, m, 1, nullptr, KC_SMALL_DENSE);
    ctx.before(KC_SMALL_DENSE, 16.0 * m2, 0);
    launch_chained(ctx, k_sort_eig, (m + 7) / 8, 256, 0, m, lam0, S0, lam, Q);
    ctx.after();
    return cudaGetLastError();
}

// Kernel attributes are process-wide: a handle lowering a kernel's dynamic
// shared-memory limit to its own size while another thread is about to launch
// with more would fail that launch ("invalid argument").  So the limits are
// raised once, to the most any launch here uses (200 KB), and never changed.
void raise_smem_limits() {
    constexpr int kMaxDevices = 64;
    static std::once_flag once[kMaxDevices];
    int dev = 0;
    cudaGetDevice(&dev);
    std::call_once(once[dev < 0 || dev >= kMaxDevices ? 0 : dev], [] {   // per device, with it current
        const int lim = 200 * 1024;
        cudaFuncSetAttribute(k_chol_shifted, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_triinv_upper, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        cudaFuncSetAttribute(k_jacobi32, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
        cudaFuncSetAttribute(k_jacobi_df, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    });
}

}  // namespace slrf
