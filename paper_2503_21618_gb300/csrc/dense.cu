// FP64 kernels of the projection step of Algorithm 1: real SpMM (A U, B U,
// A X, B X), tall-skinny GEMMs (Grams U^T B U, U^T A U and the basis changes
// X = U S), residuals rho_i, and the filter combination of the
// residual-corrected form.  Everything here is FP64: these quantities set the
// accuracy of the Ritz values (relative error 1e-10) and residuals (1e-8).
#include <cuda_runtime.h>

#include "internal.h"

namespace slrf {

// ---------------------------------------------------------------------------
// Y = A X, Z = B X (either may be null); thread per (row, column).  Bound by
// the FP64 pipe (one FMA per entry, column and output at ~0.5 TFMA/s: 0.25 ms
// for A X on the 2D pencil of n = 89 401 with 150 columns).  NB: a node-block
// pencil, whose rows hold whole neighbour nodes (three consecutive columns)
// and whose mass couples equal dofs only: row r of a node takes every third
// mass entry (its zeros cost as much as the others otherwise).
// ---------------------------------------------------------------------------
template <bool DO_A, bool DO_B, bool NB>
__global__ void __launch_bounds__(256)
k_spmm_real(int n, int m, const int32_t *__restrict__ rowptr, const int32_t *__restrict__ col,
            const double2 *__restrict__ ab, const double *__restrict__ X, int64_t ldx, double *__restrict__ Y,
            int64_t ldy, double *__restrict__ Z, int64_t ldz) {
    const int c = blockIdx.x * 32 + threadIdx.x;
    if (c >= m) return;
    for (int row = blockIdx.y * 8 + threadIdx.y; row < n; row += gridDim.y * 8) {
        const int k0 = __ldg(rowptr + row), k1 = __ldg(rowptr + row + 1);
        double ya = 0.0, zb = 0.0;
        if (NB) {
            const int r = row % 3;   // the same for the warp
            if (DO_A)
                for (int k = k0; k < k1; k += 3) {
                    double2 w[3];
                    double x[3];
#pragma unroll
                    for (int t = 0; t < 3; ++t) {
                        x[t] = X[(int64_t)__ldg(col + k + t) * ldx + c];
                        w[t] = __ldg(ab + k + t);
                    }
#pragma unroll
                    for (int t = 0; t < 3; ++t) ya = fma(w[t].x, x[t], ya);
                    if (DO_B) {
                        const double xb = r == 0 ? x[0] : r == 1 ? x[1] : x[2];
                        const double wb = r == 0 ? w[0].y : r == 1 ? w[1].y : w[2].y;
                        zb = fma(wb, xb, zb);
                    }
                }
            else
                for (int k = k0 + r; k < k1; k += 3)
                    zb = fma(__ldg(&ab[k].y), X[(int64_t)__ldg(col + k) * ldx + c], zb);
        } else {
            for (int k = k0; k < k1; ++k) {
                const double x = X[(int64_t)__ldg(col + k) * ldx + c];
                const double2 w = __ldg(ab + k);
                if (DO_A) ya = fma(w.x, x, ya);
                if (DO_B) zb = fma(w.y, x, zb);
            }
        }
        if (DO_A) Y[(int64_t)row * ldy + c] = ya;
        if (DO_B) Z[(int64_t)row * ldz + c] = zb;
    }
}

void spmm_real(Ctx &ctx, const DevPencil &A, int m, const double *X, int64_t ldx, double *Y, int64_t ldy,
               double *Z, int64_t ldz) {
    if (!Y && !Z) return;
    const int gx = (m + 31) / 32;
    int gy = ctx.sm_count * 8 / gx;
    if (gy > (A.n + 7) / 8) gy = (A.n + 7) / 8;
    if (gy < 1) gy = 1;
    dim3 grid(gx, gy), block(32, 8);
    const int nout = (Y ? 1 : 0) + (Z ? 1 : 0);
    const bool nb = A.nb_coef != nullptr;
    const double bytes = 4.0 * (A.n + 1) + 20.0 * A.nnz + 8.0 * A.n * m * (1 + nout);
    ctx.before(KC_SPMM_REAL, bytes, 2.0 * ((Y ? 1.0 : 0.0) + (Z ? (nb ? 1.0 / 3 : 1.0) : 0.0)) * A.nnz * m);
#define SR(a, b, c) k_spmm_real<a, b, c><<<grid, block, 0, ctx.stream>>>(A.n, m, A.rowptr, A.col, A.ab64, X, ldx, Y, ldy, Z, ldz)
    if (Y && Z) {
        if (nb) SR(true, true, true);
        else SR(true, true, false);
    } else if (Y) {
        SR(true, false, false);
    } else {
        if (nb) SR(false, true, true);
        else SR(false, true, false);
    }
#undef SR
    ctx.after();
}

// ---------------------------------------------------------------------------
// DGEMM, row-major, C = op(A) op(B) (+ beta C), 64x64x16 tiles, 4x4 per thread.
// On GB300 the FP64 tensor-core path (mma.sync m8n8k4 f64) measured slower
// than this CUDA-core kernel on the Gram shapes (0.62 vs 0.70 TFLOP/s at
// 89 401 x 150, 0.79 vs 0.90 at 187 200 x 300), so FP64 products stay here.
// ---------------------------------------------------------------------------
constexpr int BM = 64, BN = 64, BK = 16;

template <int OPA, int OPB>
__global__ void __launch_bounds__(256)
k_dgemm(int M, int N, int K, int Kc, const double *__restrict__ A, int64_t lda, const double *__restrict__ B,
        int64_t ldb, double beta, double *__restrict__ C, int64_t ldc, double *__restrict__ work) {
    __shared__ double As[BK][BM + 1];
    __shared__ double Bs[BK][BN + 1];
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int i0 = blockIdx.y * BM, j0 = blockIdx.x * BN;
    const int kbeg = blockIdx.z * Kc;
    const int kend = min(K, kbeg + Kc);
    double acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;

    for (int k0 = kbeg; k0 < kend; k0 += BK) {
        // load op(A) tile [BM x BK] into As[kk][ii]
#pragma unroll
        for (int t = 0; t < (BM * BK) / 256; ++t) {
            const int e = tid + t * 256;
            int ii, kk;
            if (OPA == 1) { ii = e % BM; kk = e / BM; }   // A is K x M: coalesce along i
            else { kk = e % BK; ii = e / BK; }             // A is M x K: coalesce along k
            const int gi = i0 + ii, gk = k0 + kk;
            double v = 0.0;
            if (gi < M && gk < kend) v = OPA ? A[(int64_t)gk * lda + gi] : A[(int64_t)gi * lda + gk];
            As[kk][ii] = v;
        }
#pragma unroll
        for (int t = 0; t < (BN * BK) / 256; ++t) {
            const int e = tid + t * 256;
            int jj, kk;
            if (OPB == 0) { jj = e % BN; kk = e / BN; }   // B is K x N
            else { kk = e % BK; jj = e / BK; }             // B is N x K
            const int gj = j0 + jj, gk = k0 + kk;
            double v = 0.0;
            if (gj < N && gk < kend) v = OPB ? B[(int64_t)gj * ldb + gk] : B[(int64_t)gk * ldb + gj];
            Bs[kk][jj] = v;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            double a[4], b[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                a[q] = As[kk][ty + 16 * q];
                b[q] = Bs[kk][tx + 16 * q];
            }
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[p][q] = fma(a[p], b[q], acc[p][q]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const int gi = i0 + ty + 16 * p;
        if (gi >= M) continue;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int gj = j0 + tx + 16 * q;
            if (gj >= N) continue;
            if (work) {
                work[((int64_t)blockIdx.z * M + gi) * N + gj] = acc[p][q];
            } else {
                double *o = C + (int64_t)gi * ldc + gj;
                *o = (beta != 0.0 ? beta * *o : 0.0) + acc[p][q];
            }
        }
    }
}

__global__ void k_split_reduce(int M, int N, int split, const double *__restrict__ work, double beta,
                               double *__restrict__ C, int64_t ldc) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= (int64_t)M * N) return;
    double s = 0.0;
    for (int z = 0; z < split; ++z) s += work[(int64_t)z * M * N + e];
    const int i = (int)(e / N), j = (int)(e % N);
    double *o = C + (int64_t)i * ldc + j;
    *o = (beta != 0.0 ? beta * *o : 0.0) + s;
}

// Small products (the m x m x m GEMMs of the projection) on 8 x 8 output
// tiles: 64 outputs times a four-way split of each K chunk per CTA, the next
// chunk's loads in flight during the FMAs, the four sums added in a fixed
// order.  Bound by the FP64 pipe (~1.7 FMAs per clock and SM), so the tiles
// are small enough that the most loaded SM has little more than the average:
// m = 150 on 100 CTAs of 16 x 16 took 17 us, on 361 of 8 x 8 about 10 us.
// symmetric: the result is known to be symmetric (X^T X, X^T S X): only the
// tiles on and above the diagonal are computed, and mirrored.
template <int OPA, int OPB>
__global__ void __launch_bounds__(256)
k_dgemm_small(int M, int N, int K, const double *A, int64_t lda, const double *B,
              int64_t ldb, double beta, double *__restrict__ C, int64_t ldc, int symmetric,
              int ns) {
    chain_wait();
    constexpr int T = 8, KC = 32;
    __shared__ double As[KC][T + 1], Bs[KC][T + 1], red[3][T * T];
    if (symmetric && blockIdx.x < blockIdx.y) return;
    const int tid = threadIdx.x;
    const int i0 = blockIdx.y * T, j0 = blockIdx.x * T;
    // this thread's element of each staged chunk (lanes along the contiguous index)
    const int ai = OPA ? tid & 7 : tid >> 5, ak = OPA ? tid >> 3 : tid & 31;
    const int bj = OPB ? tid >> 5 : tid & 7, bk = OPB ? tid & 31 : tid >> 3;
    auto load_a = [&](int k0) {
        const int i = i0 + ai, k = k0 + ak;
        return i < M && k < K ? (OPA ? A[(int64_t)k * lda + i] : A[(int64_t)i * lda + k]) : 0.0;
    };
    auto load_b = [&](int k0) {
        const int j = j0 + bj, k = k0 + bk;
        return j < N && k < K ? (OPB ? B[(int64_t)j * ldb + k] : B[(int64_t)k * ldb + j]) : 0.0;
    };
    const int o = tid & 63, kq = tid >> 6, i = o >> 3, j = o & 7;
    double s = 0.0, av = load_a(0), bv = load_b(0);
    for (int k0 = 0; k0 < K; k0 += KC) {
        As[ak][ai] = av;
        Bs[bk][bj] = bv;
        __syncthreads();
        if (k0 + KC < K) {
            av = load_a(k0 + KC);
            bv = load_b(k0 + KC);
        }
#pragma unroll
        for (int kk = 0; kk < KC / 4; ++kk) s = fma(As[kq * (KC / 4) + kk][i], Bs[kq * (KC / 4) + kk][j], s);
        __syncthreads();
    }
    if (kq) red[kq - 1][o] = s;
    __syncthreads();
    const int gi = i0 + i, gj = j0 + j;
    if (kq || gi >= M || gj >= N || (symmetric && gi > gj)) return;
    s = ((s + red[0][o]) + red[1][o]) + red[2][o];
    double *c = C + (int64_t)gi * ldc + gj;
    if (ns) s = (gi == gj ? 1.5 : 0.0) - 0.5 * s;
    *c = (beta != 0.0 ? beta * *c : 0.0) + s;
    if (symmetric && gi != gj) C[(int64_t)gj * ldc + gi] = s;
}

int gram_split(const Ctx &ctx, int m, int64_t n) {
    const int tiles = ((m + BM - 1) / BM) * ((m + BN - 1) / BN);
    int split = (ctx.sm_count * 4 + tiles - 1) / tiles;
    const int64_t maxs = (n + 255) / 256;    // keep at least 256 rows per slice
    if (split > maxs) split = (int)maxs;
    if (split < 1) split = 1;
    return split;
}

void small_ns_factor(Ctx &ctx, int m, const double *X, double *E) {
    const dim3 grid((m + 7) / 8, (m + 7) / 8);
    ctx.before(KC_SMALL_DENSE, 16.0 * m * m, (double)m * m * m);
    launch_chained(ctx, k_dgemm_small<1, 0>, grid, 256, 0, m, m, m, X, (int64_t)m, X, (int64_t)m, 0.0, E, (int64_t)m,
                   1, 1);
    ctx.after();
}

void dgemm(Ctx &ctx, int opA, int opB, int M, int N, int K, const double *A, int64_t lda, const double *B,
           int64_t ldb, double beta, double *C, int64_t ldc, int split, double *work, int kc, bool symmetric) {
    if (M <= 0 || N <= 0) return;
    if (split < 1 || !work) split = 1;
    if (split == 1 && M <= 1024 && N <= 1024 && K <= 4096) {
        const dim3 grid((N + 7) / 8, (M + 7) / 8);
        const int sym = symmetric && beta == 0.0 && M == N ? 1 : 0;
        ctx.before(kc, 8.0 * ((double)M * K + (double)K * N + (double)M * N), 2.0 * M * N * (double)K);
#define LS(a, b) launch_chained(ctx, k_dgemm_small<a, b>, grid, 256, 0, M, N, K, A, lda, B, ldb, beta, C, ldc, sym, 0)
        if (opA == 0 && opB == 0) LS(0, 0);
        else if (opA == 1 && opB == 0) LS(1, 0);
        else if (opA == 0 && opB == 1) LS(0, 1);
        else LS(1, 1);
#undef LS
        ctx.after();
        return;
    }
    int Kc = (K + split - 1) / split;
    Kc = (Kc + BK - 1) / BK * BK;
    split = (K + Kc - 1) / Kc;
    if (split < 1) split = 1;
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, split);
    double *w = split > 1 ? work : nullptr;
    ctx.before(kc, 8.0 * ((double)M * K + (double)K * N + (double)M * N), 2.0 * M * N * (double)K);
#define L(a, b) k_dgemm<a, b><<<grid, 256, 0, ctx.stream>>>(M, N, K, Kc, A, lda, B, ldb, beta, C, ldc, w)
    if (opA == 0 && opB == 0) L(0, 0);
    else if (opA == 1 && opB == 0) L(1, 0);
    else if (opA == 0 && opB == 1) L(0, 1);
    else L(1, 1);
#undef L
    ctx.after();
    if (split > 1) {
        const int64_t tot = (int64_t)M * N;
        ctx.before(kc, 8.0 * tot * (split + 1), 0);
        k_split_reduce<<<(unsigned)((tot + 255) / 256), 256, 0, ctx.stream>>>(M, N, split, work, beta, C, ldc);
        ctx.after();
    }
}

// ---------------------------------------------------------------------------
// residuals: R = BX diag(theta) - AX, per-column ||R||^2, ||BX||^2, ||AX||^2
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
k_residual(int n, int m, const double *__restrict__ AX, const double *__restrict__ BX, int64_t ld,
           const double *__restrict__ theta, double *__restrict__ R, int64_t ldr, double *__restrict__ part) {
    const int c = blockIdx.x * 32 + threadIdx.x;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    if (c < m) {
        const double th = theta[c];
        for (int row = blockIdx.y * 8 + threadIdx.y; row < n; row += gridDim.y * 8) {
            const double ax = AX[(int64_t)row * ld + c];
            const double bx = BX[(int64_t)row * ld + c];
            const double r = fma(bx, th, -ax);
            if (R) R[(int64_t)row * ldr + c] = r;
            s0 = fma(r, r, s0);
            s1 = fma(bx, bx, s1);
            s2 = fma(ax, ax, s2);
        }
    }
    __shared__ double red[8][32][3];
    red[threadIdx.y][threadIdx.x][0] = s0;
    red[threadIdx.y][threadIdx.x][1] = s1;
    red[threadIdx.y][threadIdx.x][2] = s2;
    __syncthreads();
    if (threadIdx.y == 0 && c < m) {
        double a = 0, b = 0, d = 0;
        for (int y = 0; y < 8; ++y) {
            a += red[y][threadIdx.x][0];
            b += red[y][threadIdx.x][1];
            d += red[y][threadIdx.x][2];
        }
        double *o = part + ((int64_t)blockIdx.y * m + c) * 3;
        o[0] = a;
        o[1] = b;
        o[2] = d;
    }
}

__global__ void k_residual_reduce(int m, int gy, const double *__restrict__ part, const double *__restrict__ theta,
                                  double *__restrict__ rho, double *__restrict__ rho_ax) {
    const int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (c >= m) return;
    double a = 0, b = 0, d = 0;
    for (int g = lane; g < gy; g += 32) {
        const double *o = part + ((int64_t)g * m + c) * 3;
        a += o[0];
        b += o[1];
        d += o[2];
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, off);
        b += __shfl_xor_sync(0xffffffffu, b, off);
        d += __shfl_xor_sync(0xffffffffu, d, off);
    }
    if (lane == 0) {
        const double nr = sqrt(a);
        rho[c] = nr / (fabs(theta[c]) * sqrt(b));
        if (rho_ax) rho_ax[c] = nr / sqrt(d);
    }
}

void residual(Ctx &ctx, int n, int m, const double *AX, const double *BX, int64_t ld, const double *theta,
              double *Rout, int64_t ldr, double *rho, double *rho_ax, double *work) {
    const int gx = (m + 31) / 32;
    int gy = ctx.sm_count * 4 / gx;
    if (gy > (n + 7) / 8) gy = (n + 7) / 8;
    if (gy > 1024) gy = 1024;
    if (gy < 1) gy = 1;
    ctx.before(KC_RESIDUAL, 8.0 * n * m * (Rout ? 3 : 2), 8.0 * n * m);
    k_residual<<<dim3(gx, gy), dim3(32, 8), 0, ctx.stream>>>(n, m, AX, BX, ld, theta, Rout, ldr, work);
    ctx.after();
    ctx.before(KC_RESIDUAL, 24.0 * gy * m, 0);
    k_residual_reduce<<<(m * 32 + 255) / 256, 256, 0, ctx.stream>>>(m, gy, work, theta, rho, rho_ax);
    ctx.after();
}

// ---------------------------------------------------------------------------
// U = X diag(phi) + Ucorr
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_filter_combine(int n, int m, const double *__restrict__ X, int64_t ldx,
                                 const double *__restrict__ phi, const T *__restrict__ Uc, int ldc,
                                 double *__restrict__ U, int64_t ldu) {
    const int c = blockIdx.x * 32 + threadIdx.x;
    if (c >= m) return;
    const double ph = phi ? phi[c] : 0.0;
    for (int row = blockIdx.y * 8 + threadIdx.y; row < n; row += gridDim.y * 8) {
        const double x = X ? X[(int64_t)row * ldx + c] * ph : 0.0;
        U[(int64_t)row * ldu + c] = x + (double)Uc[(int64_t)row * ldc + c];
    }
}

template <typename T>
void filter_combine(Ctx &ctx, int n, int m, const double *X, int64_t ldx, const double *phi, const T *Ucorr,
                    int ldc, double *U, int64_t ldu) {
    const int gx = (m + 31) / 32;
    int gy = ctx.sm_count * 8 / gx;
    if (gy > (n + 7) / 8) gy = (n + 7) / 8;
    if (gy < 1) gy = 1;
    ctx.before(KC_FILTER_COMBINE, (double)n * m * (8 * (X ? 2 : 1) + sizeof(T)), 2.0 * n * m);
    k_filter_combine<T><<<dim3(gx, gy), dim3(32, 8), 0, ctx.stream>>>(n, m, X, ldx, phi, Ucorr, ldc, U, ldu);
    ctx.after();
}
template void filter_combine<float>(Ctx &, int, int, const double *, int64_t, const double *, const float *, int,
                                    double *, int64_t);
template void filter_combine<double>(Ctx &, int, int, const double *, int64_t, const double *, const double *,
                                     int, double *, int64_t);

void fill_zero(Ctx &ctx, void *p, size_t bytes) { cudaMemsetAsync(p, 0, bytes, ctx.stream); }

void copy_block(Ctx &ctx, int n, int m, const double *src, int64_t lds, double *dst, int64_t ldd) {
    cudaMemcpy2DAsync(dst, (size_t)ldd * 8, src, (size_t)lds * 8, (size_t)m * 8, (size_t)n,
                      cudaMemcpyDeviceToDevice, ctx.stream);
}

}  // namespace slrf
