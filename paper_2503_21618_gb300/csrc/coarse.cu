// Exact solve of one multigrid level by dense shifted inverses.
//
// The cycle's coarse-grid correction is only as good as the level it stops
// at.  Stopping at a level of ~10^3 unknowns with an exact solve there
// (instead of smoothing it and recursing once more) cuts the COCG
// iterations per pole on the 2D bench pencil from ~15 to ~10.  A level of
// that size is solved exactly by its shifted inverses: per solve, with the
// poles known, every matrix M_j = A_l - sigma_j B_l (complex symmetric,
// Im M_j = -Im(sigma_j) B_l definite, so every leading block is nonsingular
// and no pivoting is needed) is formed densely and inverted; the cycle then
// applies Z_j = M_j^{-1} R_j, one batched product per visit.  The inverse is
// symmetric to the last bit, so the cycle stays a complex symmetric operator,
// as COCG requires.
//
// The elimination is the symmetric sweep in blocks of CB rows K (the rest R),
// which keeps M complex symmetric, so only its block upper triangle is held
// and half the arithmetic of Gauss-Jordan is done:
//   P = M_KK^{-1},  T = P M_KR,  M_RR -= M_KR^T T,  M_KR = T,  M_KK = -P;
// after the last block M holds -M^{-1}.  It runs in the inverses' own storage
// (a copy padded to whole blocks would double the memory of the level); the
// last block's padding, the identity, is put in where its tiles are loaded.
// Two launches per block: the panel (T, every block column its own
// CTA), and the update, one CTA per 64 x 64 tile, whose first CTA takes the
// next diagonal block and sweeps it in registers while the others work, so
// most of the chain of 64 pivots (~15 us) hides behind the update.  Bound by FP32
// arithmetic: 4 N n^3 flops (n = 1283, N = 4: 34 GF, 0.45 ms at 75 TFLOP/s);
// cuBLAS complex GEMMs on the whole matrix, with the diagonal blocks and
// block copies in launches of their own, took 3.9 ms there, this 1.15 ms.
// Error of the cycle against FP64 inverses (100 poles of 25 1D pencils, levels of 334
// to 1 500 unknowns): geometric mean 2.6e-5, RMS 5.2e-5 (by Gauss-Jordan with
// cuBLAS 2.5e-5 and 5.0e-5; a conditioned level, 2D, 2e-6 to 6e-6 both ways).
// (The chain in a launch of its own beside the update was slower: it is as long
// as the update.)
#include <cublas_v2.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "internal.h"
#include "sweep_rule.h"

namespace slrf {

namespace {

constexpr int CB = 64;   // block size of the sweep

// M_j = A - sigma_j B on the level's CSR pattern of (a, b) pairs, dense, rows
// of ld = coarse_inverse_ld(n) entries (the one beyond n, if any, is zero and
// stays so)
__global__ void k_dense_shift(int n, int ld, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
                              const float2 *__restrict__ ab, PoleSet<float> ps, float2 *__restrict__ M) {
    const int row = blockIdx.x;
    const int j = blockIdx.y;
    float2 *Mr = M + ((int64_t)j * n + row) * ld;
    for (int c = threadIdx.x; c < ld; c += blockDim.x) Mr[c] = make_float2(0.f, 0.f);
    __syncthreads();
    const float sr = ps.re[j], si = ps.im[j];
    for (int k = ptr[row] + threadIdx.x; k < ptr[row + 1]; k += blockDim.x) {
        const float2 w = ab[k];
        Mr[col[k]] = make_float2(w.x - sr * w.y, -si * w.y);
    }
}

// Thread (ty, tx) of 16 x 16 holds of a CB x CB tile the rows 4 ty .. 4 ty+3
// and the columns 2 tx, 2 tx + 1, 2 tx + 32, 2 tx + 33: a row's operands are
// one broadcast and the columns' two conflict-free 16-byte shared loads.
__device__ __forceinline__ int tile_col(int tx, int q) { return 2 * tx + 32 * (q >> 1) + (q & 1); }

// 16-byte asynchronous copies to shared memory; the second form writes zeros
// (and reads nothing) unless `in`
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool in) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(in ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// acc -= A^T B over KR rows of two staged panels of CB columns
template <int KR>
__device__ __forceinline__ void tile_product(const float2 (*A)[CB], const float2 (*B)[CB], int ty, int tx,
                                             float2 (&acc)[4][4]) {
#pragma unroll 4
    for (int k = 0; k < KR; ++k) {
        const float4 a01 = *reinterpret_cast<const float4 *>(&A[k][4 * ty]);
        const float4 a23 = *reinterpret_cast<const float4 *>(&A[k][4 * ty + 2]);
        const float4 b01 = *reinterpret_cast<const float4 *>(&B[k][2 * tx]);
        const float4 b23 = *reinterpret_cast<const float4 *>(&B[k][2 * tx + 32]);
        const float2 a[4] = {make_float2(a01.x, a01.y), make_float2(a01.z, a01.w), make_float2(a23.x, a23.y),
                             make_float2(a23.z, a23.w)};
        const float2 b[4] = {make_float2(b01.x, b01.y), make_float2(b01.z, b01.w), make_float2(b23.x, b23.y),
                             make_float2(b23.z, b23.w)};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][q] = cfma(make_float2(-a[i].x, -a[i].y), b[q], acc[i][q]);
    }
}

// 1 / p of a pivot, in the middle of the chain of pivots: the hardware reciprocal of
// |p|^2, then one Newton step q + q (1 - p q) in fused operations, 0.48 units of
// rounding (RMS) where correctly rounded quotients by |p|^2 leave 0.64.  That counts:
// the pivots of banded levels (1D) follow from one another, and their errors are
// what the inverse's error grows from.
__device__ __forceinline__ float2 rcp_newton(float2 p) {
    float d;
    asm("rcp.approx.f32 %0, %1;" : "=f"(d) : "f"(p.x * p.x + p.y * p.y));
    const float2 q = make_float2(p.x * d, -p.y * d);
    const float2 e = make_float2(fmaf(p.y, q.y, fmaf(-p.x, q.x, 1.f)), fmaf(-p.y, q.x, -p.x * q.y));
    return make_float2(fmaf(q.x, e.x, fmaf(-q.y, e.y, q.x)), fmaf(q.x, e.y, fmaf(q.y, e.x, q.y)));
}
// Where |p|^2 is near the ends of FP32's range (pencils scaled to 1e-15 and below or
// 1e15 and above) p is brought to the middle by a power of two first; the same
// branch for the whole block.
__device__ __forceinline__ float2 pivot_rcp(float2 p) {
    const float d = p.x * p.x + p.y * p.y;
    if (d >= 1e-30f && d <= 1e30f) return rcp_newton(p);
    const int e = ilogbf(fmaxf(fabsf(p.x), fabsf(p.y)));
    const float2 q = rcp_newton(make_float2(scalbnf(p.x, -e), scalbnf(p.y, -e)));
    return make_float2(scalbnf(q.x, -e), scalbnf(q.y, -e));
}

// Pivot k (column k: registers S[.][qk] of lane tx = kx; row k: S[ki][.] of ty =
// k4) with w = row k / pivot, r = column k, applied to the register rows i
// (mask), the pivot's own row and column included.
template <int KI, int QK>
__device__ __forceinline__ void pivot_rows(float2 (&S)[4][4], const float2 (&w)[4], const float2 (&r)[4], float2 pinv,
                                           bool own_row, bool own_col, int mask) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (!(mask >> i & 1)) continue;
#pragma unroll
        for (int q = 0; q < 4; ++q) S[i][q] = cfma(make_float2(-r[i].x, -r[i].y), w[q], S[i][q]);
        if (own_col) S[i][QK] = cmul(pinv, r[i]);
        if (i == KI && own_row) {
#pragma unroll
            for (int q = 0; q < 4; ++q) S[i][q] = w[q];
            if (own_col) S[i][QK] = make_float2(-pinv.x, -pinv.y);
        }
    }
}

__device__ __forceinline__ void publish_row(float2 *row, const float2 (&v)[4], int tx) {
    *reinterpret_cast<float4 *>(row + 2 * tx) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    *reinterpret_cast<float4 *>(row + 2 * tx + 32) = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
}

// The symmetric sweep of all CB pivots of a tile in registers: S -> -S^{-1}.
// Per pivot the owners publish its row (= its column), one barrier, everyone
// updates.  A chain of 64 such steps, so a step is cut into what the next one
// needs and the rest: pivot k is applied to the register row that holds row k+1
// first, which is published; the other three rows follow after the barrier,
// beside the loads and the reciprocal of pivot k+1: 17 us for the first block
// against 21.
struct Pivot {
    float2 w[4], r[4], pinv;
};
template <int HALF, int KI>
__device__ __forceinline__ void sweep_step(float2 (&S)[4][4], float2 (*row)[CB], int ty, int tx, int k8, Pivot &v) {
    constexpr int QK = 2 * HALF + (KI & 1), KP = (KI + 3) & 3, NEXT = (KI + 1) & 3;
    const int k4 = 8 * HALF + k8, k = 4 * k4 + KI;
    const float2 *rk = row[KI & 1];
    __syncthreads();
    const float2 p = rk[k];
    const float4 c01 = *reinterpret_cast<const float4 *>(rk + 2 * tx);
    const float4 c23 = *reinterpret_cast<const float4 *>(rk + 2 * tx + 32);
    const float4 r01 = *reinterpret_cast<const float4 *>(rk + 4 * ty);
    const float4 r23 = *reinterpret_cast<const float4 *>(rk + 4 * ty + 2);
    // the rest of pivot k - 1: the register rows other than KI
    const bool prow = ty == (k - 1) >> 2, pcol = tx == ((k - 1) & 31) >> 1;
    constexpr int REST = 15 & ~(1 << KI);
    if constexpr (KI > 0) {
        pivot_rows<KP, 2 * HALF + (KP & 1)>(S, v.w, v.r, v.pinv, prow, pcol, REST);
    } else {
        if (k8 > 0) pivot_rows<3, 2 * HALF + 1>(S, v.w, v.r, v.pinv, prow, pcol, REST);
        else if (HALF == 1) pivot_rows<3, 1>(S, v.w, v.r, v.pinv, prow, pcol, REST);
    }
    v.pinv = pivot_rcp(p);
    v.w[0] = cmul(v.pinv, make_float2(c01.x, c01.y));
    v.w[1] = cmul(v.pinv, make_float2(c01.z, c01.w));
    v.w[2] = cmul(v.pinv, make_float2(c23.x, c23.y));
    v.w[3] = cmul(v.pinv, make_float2(c23.z, c23.w));
    v.r[0] = make_float2(r01.x, r01.y);
    v.r[1] = make_float2(r01.z, r01.w);
    v.r[2] = make_float2(r23.x, r23.y);
    v.r[3] = make_float2(r23.z, r23.w);
    pivot_rows<KI, QK>(S, v.w, v.r, v.pinv, ty == k4, tx == (k & 31) >> 1, 1 << NEXT);
    if (k + 1 < CB && ty == (k + 1) >> 2) publish_row(row[(KI + 1) & 1], S[NEXT], tx);
}
__device__ __forceinline__ void tile_sweep(float2 (&S)[4][4], float2 (*row)[CB], int ty, int tx) {
    if (ty == 0) publish_row(row[0], S[0], tx);
    Pivot v;
    for (int k8 = 0; k8 < CB / 8; ++k8) {
        sweep_step<0, 0>(S, row, ty, tx, k8, v);
        sweep_step<0, 1>(S, row, ty, tx, k8, v);
        sweep_step<0, 2>(S, row, ty, tx, k8, v);
        sweep_step<0, 3>(S, row, ty, tx, k8, v);
    }
    for (int k8 = 0; k8 < CB / 8; ++k8) {
        sweep_step<1, 0>(S, row, ty, tx, k8, v);
        sweep_step<1, 1>(S, row, ty, tx, k8, v);
        sweep_step<1, 2>(S, row, ty, tx, k8, v);
        sweep_step<1, 3>(S, row, ty, tx, k8, v);
    }
    pivot_rows<3, 3>(S, v.w, v.r, v.pinv, ty == CB / 4 - 1, tx == 15, 14);
}

// Sweep of the diagonal block at k0: M_KK = -P
__device__ __forceinline__ void sweep_store(float2 (&S)[4][4], float2 (*row)[CB], int n, int ld, int k0,
                                            float2 *__restrict__ M, int ty, int tx) {
    tile_sweep(S, row, ty, tx);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = 4 * ty + i, c = tile_col(tx, q);
            if (max(r, c) < n - k0) M[(int64_t)(k0 + r) * ld + k0 + c] = S[i][q];
        }
}

__global__ void __launch_bounds__(256) k_first_block(int n, int ld, float2 *__restrict__ M) {
    chain_wait();
    __shared__ __align__(16) float2 row[2][CB];
    float2 *Mj = M + (int64_t)blockIdx.x * n * ld;
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    float2 S[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = 4 * ty + i, c = tile_col(tx, q);
            S[i][q] = r < n && c < n ? Mj[(int64_t)r * ld + c] : make_float2(r == c ? 1.f : 0.f, 0.f);
        }
    sweep_store(S, row, n, ld, 0, Mj, ty, tx);
}

// Panel of block K: the old rows M_K* (from the upper triangle: M_KJ for J >
// K, M_JK^T for J < K) to Cp, T = P M_K* to Tp and in place of the old block;
// one CTA per matrix and 32 columns.  Cp and Tp have the columns of the other
// blocks only (pitch lq).
constexpr int PC = 32, PLD = PC + 2;   // columns of a panel CTA, their pitch
__global__ void __launch_bounds__(256) k_sweep_panel(int n, int ld, int lq, int K, float2 *__restrict__ M,
                                                     float2 *__restrict__ Cp, float2 *__restrict__ Tp) {
    chain_wait();
    extern __shared__ __align__(16) float2 sm[];
    float2(*sP)[CB] = reinterpret_cast<float2(*)[CB]>(sm);
    float2(*sC)[PLD] = reinterpret_cast<float2(*)[PLD]>(sm + CB * CB);
    const int j = blockIdx.x, Jh = blockIdx.y >> 1, J = Jh + (Jh >= K ? 1 : 0);
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    float2 *Mj = M + (int64_t)j * n * ld;
    float2 *C = Cp + (int64_t)j * CB * lq, *T = Tp + (int64_t)j * CB * lq;
    const int k0 = K * CB, c0 = J * CB + (blockIdx.y & 1) * PC, q0 = Jh * CB + (blockIdx.y & 1) * PC;
#pragma unroll
    for (int q = 0; q < CB * CB / 2 / 256; ++q) {   // -P, symmetric
        const int e = tid + 256 * q, r = k0 + e / (CB / 2), c = k0 + e % (CB / 2) * 2;
        const bool in = r < n && c < n;
        cp_async16(&sP[0][0] + 2 * e, in ? Mj + (int64_t)r * ld + c : Mj, in);
    }
    if (J > K)   // block K is not the last: all its rows are there
#pragma unroll
        for (int q = 0; q < CB * PC / 2 / 256; ++q) {
            const int e = tid + 256 * q, r = e / (PC / 2), c = e % (PC / 2) * 2;
            const bool in = c0 + c < n;
            cp_async16(&sC[r][c], in ? Mj + (int64_t)(k0 + r) * ld + c0 + c : Mj, in);
        }
    else         // all columns of block J are there
#pragma unroll
        for (int e = tid; e < CB * PC; e += 256)
            sC[e % CB][e / CB] = k0 + e % CB < n ? Mj[(int64_t)(c0 + e / CB) * ld + k0 + e % CB] : make_float2(0.f, 0.f);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
#pragma unroll
    for (int e = tid; e < CB * PC; e += 256) C[(int64_t)(e / PC) * lq + q0 + e % PC] = sC[e / PC][e % PC];
    float2 acc[4][2] = {};
#pragma unroll 4
    for (int k = 0; k < CB; ++k) {   // P^T = P
        const float4 a01 = *reinterpret_cast<const float4 *>(&sP[k][4 * ty]);
        const float4 a23 = *reinterpret_cast<const float4 *>(&sP[k][4 * ty + 2]);
        const float4 b01 = *reinterpret_cast<const float4 *>(&sC[k][2 * tx]);
        const float2 a[4] = {make_float2(-a01.x, -a01.y), make_float2(-a01.z, -a01.w), make_float2(-a23.x, -a23.y),
                             make_float2(-a23.z, -a23.w)};
        const float2 b[2] = {make_float2(b01.x, b01.y), make_float2(b01.z, b01.w)};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < 2; ++q) acc[i][q] = cfma(a[i], b[q], acc[i][q]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = 4 * ty + i;
        const float4 v = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
        *reinterpret_cast<float4 *>(T + (int64_t)r * lq + q0 + 2 * tx) = v;
        if (J > K && c0 + 2 * tx < n) *reinterpret_cast<float4 *>(Mj + (int64_t)(k0 + r) * ld + c0 + 2 * tx) = v;
    }
    if (J < K) {   // transposed, through shared memory
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < 2; ++q) sC[4 * ty + i][2 * tx + q] = acc[i][q];
        __syncthreads();
#pragma unroll
        for (int e = tid; e < CB * PC; e += 256)
            if (k0 + e % CB < n) Mj[(int64_t)(c0 + e / CB) * ld + k0 + e % CB] = sC[e % CB][e / CB];
    }
}

// M_IJ -= Cp_I^T T_J for the tiles I <= J off block K; the first CTA of each
// matrix takes the next diagonal block and sweeps it.  The product is summed from
// zero and subtracted once: 64 roundings at the size of M's entries instead of one
// cost accuracy, though the tile's loads
// would then hide behind the product (cycle call with 1 156 unknowns and 4 poles 945
// us for 979).
__global__ void __launch_bounds__(256, 3) k_sweep_update(int n, int ld, int lq, int nb, int K, float2 *__restrict__ M,
                                                         const float2 *Cp, const float2 *Tp) {
    chain_wait();
    extern __shared__ __align__(16) float2 sm[];
    float2(*sA)[CB] = reinterpret_cast<float2(*)[CB]>(sm);
    float2(*sB)[CB] = sA + CB;
    const int j = blockIdx.x;   // the matrices fastest: every first CTA starts at once
    // tile t of the upper triangle of the nb - 1 blocks other than K
    const bool next = K + 1 < nb;
    int Ih, Jh;
    {
        int t = blockIdx.y;
        const int q = nb - 1;
        // the next diagonal block (position K among the others) comes first
        const int td = next ? K * q - K * (K - 1) / 2 : -1;
        if (next) t = t == 0 ? td : (t <= td ? t - 1 : t);
        int i = 0, rem = t;
        while (rem >= q - i) {
            rem -= q - i;
            ++i;
        }
        Ih = i;
        Jh = i + rem;
    }
    const int I = Ih + (Ih >= K ? 1 : 0), J = Jh + (Jh >= K ? 1 : 0);
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    float2 *Mj = M + (int64_t)j * n * ld;
    const float2 *C = Cp + (int64_t)j * CB * lq + Ih * CB, *T = Tp + (int64_t)j * CB * lq + Jh * CB;
    float2 *D = Mj + (int64_t)I * CB * ld + J * CB;
    // whether the thread's rows i (bit i) and column pairs h (bit 4 + h) are inside
    const int nr = n - I * CB - 4 * ty, nc = n - J * CB - 2 * tx;
    const unsigned in = (nr >= 4 ? 15u : nr > 0 ? (1u << nr) - 1 : 0u) | (nc > 0 ? 16u : 0u) | (nc > 32 ? 32u : 0u);
    auto inside = [&](int i, int h) { return (in >> i & 1) && (in >> (4 + h) & 1); };
    // both panels by asynchronous copies, in two halves of K: all of a thread's
    // 16 loads are in flight at once and the product starts on the first half
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int q = 0; q < CB * CB / 4 / 256; ++q) {
            const int e = tid + 256 * q, r = h * (CB / 2) + e / (CB / 2), c = e % (CB / 2) * 2;
            cp_async16(&sA[r][c], C + (int64_t)r * lq + c);
            cp_async16(&sB[r][c], T + (int64_t)r * lq + c);
        }
        cp_async_commit();
    }
    float2 m[4][4] = {};
    cp_async_wait<1>();
    __syncthreads();
    tile_product<CB / 2>(sA, sB, ty, tx, m);
    cp_async_wait<0>();
    __syncthreads();
    tile_product<CB / 2>(sA + CB / 2, sB + CB / 2, ty, tx, m);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            // outside: the identity, which only the last diagonal block's sweep uses
            const int r = 4 * ty + i, c = 2 * tx + 32 * h;
            float4 v = make_float4(r == c ? 1.f : 0.f, 0.f, r == c + 1 ? 1.f : 0.f, 0.f);
            if (inside(i, h)) v = *reinterpret_cast<const float4 *>(D + (int64_t)r * ld + c);
            m[i][2 * h] = cadd(m[i][2 * h], make_float2(v.x, v.y));
            m[i][2 * h + 1] = cadd(m[i][2 * h + 1], make_float2(v.z, v.w));
        }
    if (next && blockIdx.y == 0) {
        __syncthreads();   // the panels' shared memory holds the pivot rows from here
        sweep_store(m, sA, n, ld, (K + 1) * CB, Mj, ty, tx);
        return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (inside(i, h))
                *reinterpret_cast<float4 *>(D + (int64_t)(4 * ty + i) * ld + 2 * tx + 32 * h) =
                    make_float4(m[i][2 * h].x, m[i][2 * h].y, m[i][2 * h + 1].x, m[i][2 * h + 1].y);
}

// M = -M, the lower triangle from the upper one, in place, 32 x 32 tiles
__global__ void __launch_bounds__(256) k_sweep_finish(int n, int ld, float2 *M) {
    chain_wait();
    __shared__ float2 s[32][33];
    if (blockIdx.x < blockIdx.y) return;
    float2 *Mj = M + (int64_t)blockIdx.z * n * ld;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
#pragma unroll
    for (int i = ty; i < 32; i += 8) {
        const int r = r0 + i, c = c0 + tx;
        // inside a diagonal block both halves are swept; its upper one counts
        const float2 v = r >= n || c >= n ? make_float2(0.f, 0.f)
                                          : (r <= c ? Mj[(int64_t)r * ld + c] : Mj[(int64_t)c * ld + r]);
        s[i][tx] = make_float2(-v.x, -v.y);
    }
    __syncthreads();
#pragma unroll
    for (int i = ty; i < 32; i += 8) {
        if (r0 + i < n && c0 + tx < n) Mj[(int64_t)(r0 + i) * ld + c0 + tx] = s[i][tx];
        if (r0 != c0 && c0 + i < n && r0 + tx < n) Mj[(int64_t)(c0 + i) * ld + r0 + tx] = s[tx][i];
    }
}

constexpr size_t SWEEP_SMEM = 2 * CB * CB * sizeof(float2);   // three CTAs of the update per SM
constexpr size_t SWEEP_SMEM_TWO = 100 * 1024;                 // two
constexpr size_t PANEL_SMEM = (CB * CB + CB * PLD) * sizeof(float2);

// The kernels' shared-memory limit, raised once per device
void raise_sweep_smem() {
    static std::once_flag once[64];
    int dev = 0;
    cudaGetDevice(&dev);
    std::call_once(once[dev < 0 || dev >= 64 ? 0 : dev], [] {
        cudaFuncSetAttribute(k_sweep_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PANEL_SMEM);
        cudaFuncSetAttribute(k_sweep_update, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SWEEP_SMEM_TWO);
    });
}

}  // namespace

size_t coarse_inverse_work_bytes(int n, int N) {
    const size_t nb = (n + CB - 1) / CB;
    return 2 * (size_t)N * (nb - 1) * CB * CB * sizeof(float2);
}

void coarse_inverse(Ctx &ctx, int n, const PoleSet<float> &ps, const int32_t *ptr, const int32_t *col,
                    const float2 *ab, float2 *M, void *work) {
    const int N = ps.N, nb = (n + CB - 1) / CB, ld = coarse_inverse_ld(n), lq = (nb - 1) * CB;
    float2 *Cp = reinterpret_cast<float2 *>(work);            // N x (CB x lq)
    float2 *Tp = Cp + (size_t)N * lq * CB;                    // N x (CB x lq)
    raise_sweep_smem();
    const size_t update_smem =
        sweep_three_per_sm(ctx.sm_count, (int64_t)N * (nb - 1) * nb / 2) ? SWEEP_SMEM : SWEEP_SMEM_TWO;
    ctx.before(KC_MG_COARSE, 8.0 * N * n * n, 0);
    k_dense_shift<<<dim3(n, N), 128, 0, ctx.stream>>>(n, ld, ptr, col, ab, ps, M);
    ctx.after();
    ctx.before(KC_MG_COARSE, 16.0 * N * CB * CB, 8.0 * N * CB * CB * CB);
    launch_chained(ctx, k_first_block, N, 256, 0, n, ld, M);
    ctx.after();
    if (nb > 1)
        for (int K = 0; K < nb; ++K) {
            ctx.before(KC_MG_COARSE, 24.0 * N * CB * n, 8.0 * N * CB * CB * (double)n);
            launch_chained(ctx, k_sweep_panel, dim3(N, 2 * (nb - 1)), 256, PANEL_SMEM, n, ld, lq, K, M, Cp, Tp);
            ctx.after();
            ctx.before(KC_MG_COARSE, 8.0 * N * n * (double)n, 4.0 * N * CB * (double)n * n);
            launch_chained(ctx, k_sweep_update, dim3(N, (nb - 1) * nb / 2), 256, update_smem, n, ld, lq, nb, K, M, Cp, Tp);
            ctx.after();
        }
    ctx.before(KC_MG_COARSE, 12.0 * N * n * (double)n, 0);
    const unsigned g = (unsigned)((n + 31) / 32);
    launch_chained(ctx, k_sweep_finish, dim3(g, g, N), 256, 0, n, ld, M);
    ctx.after();
}

int coarse_inverse_apply(Ctx &ctx, void *cublas, const KrylovDims &d, int n, const float2 *Minv, const float2 *R,
                         float2 *Z) {
    cublasHandle_t hb = reinterpret_cast<cublasHandle_t>(cublas);
    cublasStatus_t st = cublasSetStream(hb, ctx.stream);
    if (st != CUBLAS_STATUS_SUCCESS) return (int)st;
    const int W = d.W();
    const cuComplex one = make_cuComplex(1.f, 0.f), zero = make_cuComplex(0.f, 0.f);
    // column-major: Z_j^T (Lp x n, ld W) = R_j^T (Lp x n, ld W) * Minv_j (symmetric)
    ctx.before(KC_MG_COARSE, (double)d.N * n * n * 8 + 2.0 * n * W * 8 * d.frac,
               8.0 * d.N * (double)n * n * d.Lp * d.frac);
    st = cublasCgemmStridedBatched(hb, CUBLAS_OP_N, CUBLAS_OP_N, d.Lp, n, n, &one, R, W, d.Lp, Minv,
                                   coarse_inverse_ld(n), (int64_t)n * coarse_inverse_ld(n), &zero, Z, W, d.Lp, d.N);
    ctx.after();
    return (int)st;
}

}  // namespace slrf
