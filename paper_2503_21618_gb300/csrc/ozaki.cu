// FP64-accurate Gram G = X^T Y on the integer tensor cores (Ozaki scheme).
//
// FP64 arithmetic on this GPU runs at ~1 TFLOP/s (CUDA cores and the FP64
// tensor path alike, measured), while int8 mma.sync runs at ~150 TOP/s.  The
// Gram of two tall n x m blocks is therefore computed from exact integer
// pieces (error-free splitting, Ozaki et al., Numer. Algorithms 59, 2012):
//
//  * every column a of X is scaled by 2^-e_a, e_a = exponent of max_i |X_ia|
//    plus one, so |X_ia 2^-e_a| < 1/2;
//  * the scaled value is rounded to a fixed-point integer F with 7S fraction
//    bits and cut into S balanced base-128 digits D_s in [-64, 64] (int8):
//    X_ia = 2^e_a sum_s D_s,ia 2^(-7(s+1)) + (rounding below 2^(e_a - 7S - 1));
//  * products of digits are exact in int32 (|D E| <= 2^12; a K-slice of at
//    most 2^19/(d+1) rows keeps every partial sum below 2^31), and all digit
//    pairs with the same s + t = d share one scale, so
//        G_ab = 2^(e_a + f_b) sum_{d < S} 2^(-7(d+2)) sum_{s+t=d} D_s^T E_t;
//  * the int32 sums are converted to FP64 once per (CTA, d) and the K-slices
//    are reduced in a fixed order.
// With S = 7 the truncation error is ~2^-50 relative to max|X_a| max|Y_b| n.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <climits>

#include "internal.h"

namespace slrf {

constexpr int OZ_S = 7;          // digits per value
constexpr int OZ_TM = 64;        // CTA output tile (rows a) = (cols b)

// ---------------------------------------------------------------------------
// column exponents: e[a] = ilogb(max_i |X_ia|) + 2 (so |X 2^-e| < 1/2)
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ int oz_exponent(unsigned long long maxbits) {
    return maxbits ? ilogb(__longlong_as_double((long long)maxbits)) + 2 : 0;
}

// max |X_ia| (blockIdx.z = 0) and max |Y_ia| (1) per column, as bit patterns,
// which order like the values; row i of X counts times f[i] if f != nullptr.
// Bound by HBM: four loads in flight per thread and integer compares (FP64
// ones issue on the slow FP64 pipe; one load at a time took 34 us for 107 MB).
__global__ void __launch_bounds__(256) k_oz_colmax(int64_t n, int m, const double *__restrict__ X, int64_t ldx,
                                                   const double *__restrict__ Y, int64_t ldy,
                                                   const double *__restrict__ f, unsigned long long *__restrict__ maxbits) {
    __shared__ unsigned long long red[8][32];
    const int a = blockIdx.x * 32 + threadIdx.x;
    const double *Z = blockIdx.z ? Y : X;
    const int64_t ld = blockIdx.z ? ldy : ldx;
    const int64_t step = (int64_t)gridDim.y * 8;
    unsigned long long mx = 0;
    if (a < m)
        for (int64_t i0 = blockIdx.y * 8 + threadIdx.y; i0 < n; i0 += 4 * step) {
            unsigned long long v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t i = i0 + u * step;
                v[u] = 0;
                if (i < n) v[u] = abs_bits(f ? Z[i * ld + a] * f[i] : Z[i * ld + a]);
                if (v[u] > 0x7ff0000000000000ull) v[u] = 0;   // a NaN does not count
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) mx = max(mx, v[u]);
        }
    red[threadIdx.y][threadIdx.x] = mx;
    __syncthreads();
    if (threadIdx.y || a >= m) return;
#pragma unroll
    for (int y = 1; y < 8; ++y) mx = max(mx, red[y][threadIdx.x]);
    atomicMax(maxbits + (size_t)blockIdx.z * m + a, mx);
}
static dim3 colmax_grid(const Ctx &ctx, int64_t n, int m, int operands) {
    const int gx = (m + 31) / 32;
    const int64_t gy = std::min<int64_t>((n + 31) / 32, (ctx.sm_count * 8 + gx * operands - 1) / (gx * operands));
    return dim3(gx, (unsigned)std::max<int64_t>(gy, 1), operands);
}

__global__ void k_oz_exponent(int m, const unsigned long long *__restrict__ maxbits, int *__restrict__ e) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a < m) e[a] = oz_exponent(maxbits[a]);
}

// ---------------------------------------------------------------------------
// digits: slices[s][a][i] (transposed, row pitch npad bytes), integer-exact
// ---------------------------------------------------------------------------
__device__ __forceinline__ void oz_digits(double x, int e, int8_t d[OZ_S]) {
    // F = round(x 2^(7S - e)) exactly, from the integer significand
    long long F = 0;
    if (x != 0.0) {
        const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
        const int ex = (int)((bits >> 52) & 0x7ff);
        unsigned long long mant = bits & ((1ull << 52) - 1);
        int E;
        if (ex == 0) {
            E = -1074;                 // subnormal
        } else {
            mant |= 1ull << 52;
            E = ex - 1075;
        }
        const int sh = E - e + 7 * OZ_S;   // x 2^(7S-e) = mant 2^sh
        unsigned long long mag;
        if (sh >= 0)
            mag = mant << sh;              // |x 2^-e| < 1/2 keeps this below 2^(7S-1)
        else if (sh > -64)
            mag = (mant + (1ull << (-sh - 1))) >> (-sh);
        else
            mag = 0;
        F = (bits >> 63) ? -(long long)mag : (long long)mag;
    }
#pragma unroll
    for (int s = 0; s < OZ_S; ++s) {
        const int k = 7 * (OZ_S - 1 - s);
        long long D;
        if (k > 0)
            D = (F + (1ll << (k - 1))) >> k;   // balanced digit (round half up)
        else
            D = F;
        F -= D << k;
        d[s] = (int8_t)D;
    }
}

__global__ void __launch_bounds__(256)
k_oz_split(int64_t n, int m, int64_t npad, const double *__restrict__ X, int64_t ldx, const int *__restrict__ e,
           int8_t *__restrict__ slices, int mpad) {
    // 32 x 32 tile: read along a (coalesced), write along i (coalesced)
    __shared__ int8_t tile[OZ_S][32][33];
    const int a0 = blockIdx.x * 32, i0base = blockIdx.y * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;   // 32 x 8
    for (int64_t i0 = i0base; i0 < npad; i0 += (int64_t)gridDim.y * 32) {
        for (int r = ty; r < 32; r += 8) {
            const int64_t i = i0 + r;
            const int a = a0 + tx;
            int8_t d[OZ_S];
            const double x = (i < n && a < m) ? X[i * ldx + a] : 0.0;
            oz_digits(x, a < m ? e[a] : 0, d);
#pragma unroll
            for (int s = 0; s < OZ_S; ++s) tile[s][r][tx] = d[s];
        }
        __syncthreads();
        for (int c = ty; c < 32; c += 8) {
            const int a = a0 + c;
            if (a < mpad) {
                const int64_t i = i0 + tx;
#pragma unroll
                for (int s = 0; s < OZ_S; ++s) slices[((int64_t)s * mpad + a) * npad + i] = tile[s][tx][c];
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// IMMA Gram of digit slices: work[z][a][b] = sum_d 2^(-7(d+2)) sum_{s+t=d} D_s^T E_t
// over the K-slice z.  CTA = 4 warps, 64 x 64 tile, warp 32 x 32 (2 x 4 mma).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void imma16832(int c[4], const unsigned a[4], const unsigned b[2]) {
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};\n"
                 : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__global__ void __launch_bounds__(128)
k_oz_gram(int m, int mpad, int64_t npad, int64_t kslice, const int8_t *__restrict__ SX,
          const int8_t *__restrict__ SY, double *__restrict__ work, int symmetric) {
    // a symmetric Gram needs the tiles on and above the diagonal only
    if (symmetric && blockIdx.y > blockIdx.x) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, q = lane & 3;
    const int a_base = blockIdx.y * OZ_TM + (warp >> 1) * 32;
    const int b_base = blockIdx.x * OZ_TM + (warp & 1) * 32;
    const int64_t k_begin = blockIdx.z * kslice;
    const int64_t k_end = min(npad, k_begin + kslice);
    const int64_t plane = (int64_t)mpad * npad;
    double acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 4; ++h) acc[i][j][h] = 0.0;

    for (int d = 0; d < OZ_S; ++d) {
        int c[2][4][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int h = 0; h < 4; ++h) c[i][j][h] = 0;
        for (int s = 0; s <= d; ++s) {
            const int8_t *Xs = SX + s * plane;
            const int8_t *Yt = SY + (d - s) * plane;
            for (int64_t k = k_begin; k < k_end; k += 32) {
                unsigned af[2][4], bf[4][2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int8_t *r0 = Xs + (int64_t)(a_base + i * 16 + g) * npad + k + 4 * q;
                    const int8_t *r1 = r0 + 8 * npad;
                    af[i][0] = __ldg(reinterpret_cast<const unsigned *>(r0));
                    af[i][1] = __ldg(reinterpret_cast<const unsigned *>(r1));
                    af[i][2] = __ldg(reinterpret_cast<const unsigned *>(r0 + 16));
                    af[i][3] = __ldg(reinterpret_cast<const unsigned *>(r1 + 16));
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int8_t *r = Yt + (int64_t)(b_base + j * 8 + g) * npad + k + 4 * q;
                    bf[j][0] = __ldg(reinterpret_cast<const unsigned *>(r));
                    bf[j][1] = __ldg(reinterpret_cast<const unsigned *>(r + 16));
                }
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) imma16832(c[i][j], af[i], bf[j]);
            }
        }
        const double scale = ldexp(1.0, -7 * (d + 2));
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int h = 0; h < 4; ++h) acc[i][j][h] = fma((double)c[i][j][h], scale, acc[i][j][h]);
    }
    // C fragment: c0, c1 at (row g, cols 2q, 2q+1); c2, c3 at (row g+8, ...)
    double *W = work + (int64_t)blockIdx.z * m * m;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int a = a_base + i * 16 + g + (h >= 2 ? 8 : 0);
                const int b = b_base + j * 8 + 2 * q + (h & 1);
                if (a < m && b < m) W[(int64_t)a * m + b] = acc[i][j][h];
            }
}

// Sum of the K-slices in a fixed order: 32 outputs and 8 groups of slices per
// block (one thread per output walked up to 390 slices, a load latency each:
// 40 us at 175 slices of 150 x 150)
__global__ void __launch_bounds__(256) k_oz_reduce(int m, int split, const double *__restrict__ work,
                                                   const unsigned long long *__restrict__ maxbits,
                                                   double *__restrict__ G, int64_t ldg, int symmetric) {
    __shared__ double red[8][32];
    const int64_t idx = blockIdx.x * (int64_t)32 + threadIdx.x;
    const bool live = idx < (int64_t)m * m;
    int a = live ? (int)(idx / m) : 0, b = live ? (int)(idx % m) : 0;
    const int ga = a, gb = b;
    if (symmetric && a > b) {   // mirror the upper triangle (computed tiles only)
        a = gb;
        b = ga;
    }
    const double *w = work + (int64_t)a * m + b;
    double s = 0.0;
    for (int z0 = threadIdx.y; z0 < split; z0 += 32) {
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = z0 + 8 * u < split ? w[(int64_t)(z0 + 8 * u) * m * m] : 0.0;
#pragma unroll
        for (int u = 0; u < 4; ++u) s += v[u];
    }
    red[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y || !live) return;
#pragma unroll
    for (int y = 1; y < 8; ++y) s += red[y][threadIdx.x];
    G[(int64_t)ga * ldg + gb] = ldexp(s, oz_exponent(maxbits[a]) + oz_exponent(maxbits[m + b]));
}

// ---------------------------------------------------------------------------
// Tensor-core (tcgen05) form of the same Gram.
//
// The digits are the seven balanced base-128 digits above, stored as bf16
// (|D| <= 64 is exact in bf16) and multiplied by tcgen05.mma (kind::f16, bf16
// operands, FP32 accumulation in tensor memory).  A digit product is at most
// 2^12 and a diagonal d sums at most 7 of them per row of K, so with K-slices
// of at most 512 rows every partial sum stays below 2^24 and the FP32
// accumulation is exact; the seven diagonals live in seven TMEM accumulators
// and are combined in FP64 once per K-slice, then the K-slices are reduced in
// a fixed order (k_oz_reduce).
//
// Operand "panel" layout (UMMA canonical K-major, no swizzle): an operand
// with R rows (the M or N side) and depth K is stored per digit s, K-step of
// 32, and 64-row panel as 8 x 4 core matrices of 8 rows x 8 K-elements
// (128 contiguous bytes, row r at 16 r):
//   [s][ks][panel][row%64 / 8][k%32 / 8][row%8][k%8]
// so one (digit, K-step) block of consecutive panels is contiguous, the
// 8-row groups of consecutive panels are 512 bytes apart (the descriptor's
// stride offset) and K-adjacent cores 128 bytes apart (its leading offset).
// ---------------------------------------------------------------------------
constexpr int TC_KSTEP = 32;        // K rows per pipeline stage
constexpr int TC_MAXSTEPS = 15;     // K steps per slice: 480 rows (sums below 2^24; the combined integer below 2^63)
constexpr int TC_KMAX = 512;        // K of a tall product in one slice (beyond 480 rows combined in FP64)
constexpr int TC_TM = 128, TC_TN = 64;
constexpr unsigned TC_PANEL = 4096u;   // one digit of a 64-row panel per K step, bytes
constexpr unsigned TC_STAGE_A = OZ_S * 2 * TC_PANEL, TC_STAGE_B = OZ_S * TC_PANEL;
constexpr int TC_NS = 2;
constexpr int TC_EPI = 8;              // epilogue warps
constexpr int TC_THREADS = 32 * (2 + TC_EPI);
constexpr int TC_EPI_LD = 17;          // staging pitch of an epilogue warp's 32 x 16 block
constexpr size_t TC_SMEM = 1024 + TC_NS * (size_t)(TC_STAGE_A + TC_STAGE_B) + (size_t)TC_EPI * 32 * TC_EPI_LD * 8;

// Digits of two K-adjacent values of an operand row as packed bf16 pairs.  v
// holds round(x 2^(7S - e)) plus the bias sum_{k<6} 64 128^k of the six lower
// digits, so that digit s > 0 is seven bits of v less 64: shift, permute the
// two values' low halves together, then (bits | 0x4300) is the bf16 128 +
// digit + 64 and one packed subtraction of 192 leaves the digit.  The top
// digit, at most 128 in magnitude, is what lies above them: added to the bits
// of 1.5 2^23 it is a float of at most eight significant bits, whose upper
// half is its bf16.  About 2.5 instructions per digit.
__device__ __forceinline__ uint32_t oz_digit_pair(long long v0, long long v1, int s) {
    const int k = 7 * (OZ_S - 1 - s);
    if (s == 0) {
        const float f0 = __int_as_float(0x4b400000 + (int)(v0 >> k)) - 12582912.f;
        const float f1 = __int_as_float(0x4b400000 + (int)(v1 >> k)) - 12582912.f;
        return __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
    }
    uint32_t x0, x1;
    if (k <= 21) {
        x0 = (uint32_t)v0 >> k;
        x1 = (uint32_t)v1 >> k;
    } else {
        x0 = (uint32_t)(v0 >> k);
        x1 = (uint32_t)(v1 >> k);
    }
    uint32_t w = (__byte_perm(x0, x1, 0x5410) & 0x007f007fu) | 0x43004300u;
    __nv_bfloat162 d = *reinterpret_cast<__nv_bfloat162 *>(&w);
    const __nv_bfloat16 c192 = __ushort_as_bfloat16(0x4340);
    d = __hsub2(d, __nv_bfloat162(c192, c192));
    return *reinterpret_cast<uint32_t *>(&d);
}

// round(x 2^(7S - e)) + bias from the integer significand; |x 2^-e| < 1
__device__ __forceinline__ long long oz_biased(double x, int e) {
    constexpr long long BIAS = 64ll * ((1ll << 42) - 1) / 127;
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7ff);
    const unsigned long long mant = (bits & ((1ull << 52) - 1)) | ((unsigned long long)(ex != 0) << 52);
    const int r = e - (max(ex, 1) - 1075) - 7 * OZ_S;   // x 2^(7S - e) = mant 2^-r
    unsigned long long mag;
    if (r > 0)
        mag = ((mant >> (min(r, 64) - 1)) + 1) >> 1;
    else
        mag = mant << -r;   // subnormal columns only
    return ((bits >> 63) ? -(long long)mag : (long long)mag) + BIAS;
}

// the seven digits' 16-byte groups of eight K-adjacent values
__device__ __forceinline__ void oz_store_digits(const long long v[8], __nv_bfloat16 *__restrict__ out,
                                                int64_t digit_stride) {
#pragma unroll
    for (int s = 0; s < OZ_S; ++s) {
        uint4 q;
        q.x = oz_digit_pair(v[0], v[1], s);
        q.y = oz_digit_pair(v[2], v[3], s);
        q.z = oz_digit_pair(v[4], v[5], s);
        q.w = oz_digit_pair(v[6], v[7], s);
        *reinterpret_cast<uint4 *>(out + s * digit_stride) = q;
    }
}

// Digits of X (rows i < n, columns a < m) into the panel layout with K = rows
// of X and the panel rows = columns a, zero in the K padding (panel rows from
// m on stay unwritten: they only reach output rows or columns that nothing
// reads).  One block per (K step, 64-column panel, operand): thread (a, 8
// consecutive i), reads and writes coalesced.  Row i counts times f[i].
// Bound by HBM (8 bytes read, 14 written per value): 53 us for 89 401 x 150
// against 102 us with 64-bit digit arithmetic and scattered 16-byte writes.
__global__ void __launch_bounds__(256) k_oz_split_panel(int64_t n, int m, int64_t nks, int np,
                                                        const double *__restrict__ X, int64_t ldx,
                                                        const double *__restrict__ Y, int64_t ldy,
                                                        const double *__restrict__ f,
                                                        const unsigned long long *__restrict__ maxbits,
                                                        __nv_bfloat16 *__restrict__ PX, __nv_bfloat16 *__restrict__ PY) {
    const int panel = blockIdx.x % np;
    const int64_t ks = blockIdx.x / np;
    const int a = panel * 64 + (threadIdx.x & 63), kc = threadIdx.x >> 6;
    if (a >= m) return;
    const double *Z = blockIdx.y ? Y : X;
    const int64_t ld = blockIdx.y ? ldy : ldx;
    const int e = oz_exponent(maxbits[(size_t)blockIdx.y * m + a]);
    const int64_t i0 = ks * TC_KSTEP + kc * 8;
    double x[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) x[t] = i0 + t < n ? Z[(i0 + t) * ld + a] : 0.0;
    if (f)
#pragma unroll
        for (int t = 0; t < 8; ++t)
            if (i0 + t < n) x[t] *= f[i0 + t];
    long long v[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = oz_biased(x[t], e);
    const int r = threadIdx.x & 63;
    __nv_bfloat16 *out = (blockIdx.y ? PY : PX) + (ks * np + panel) * 2048 + ((r >> 3) * 4 + kc) * 64 + (r & 7) * 8;
    oz_store_digits(v, out, nks * np * 2048);
}

// V 2^e for an int64 V, rounded to nearest even, in integer arithmetic: FP64
// conversions and FMAs issue at ~1.7 per clock and SM, and four of them per
// output were half of the tall product's time.
__device__ __forceinline__ double oz_int_to_double(long long V, int e) {
    if (V == 0) return 0.0;
    const bool neg = V < 0;
    unsigned long long u = neg ? 0ull - (unsigned long long)V : (unsigned long long)V;
    const int lz = __clzll((long long)u);
    u <<= lz;
    unsigned long long mant = u >> 11;                       // 53 bits
    const unsigned rem = (unsigned)u & 0x7ffu;
    mant += rem > 0x400u || (rem == 0x400u && (mant & 1));   // a carry to 2^53 raises the exponent below
    const int ex = 63 - lz + e;                              // of the leading bit
    if (ex < -1022 || ex > 1022) {
        const double d = ldexp((double)mant, ex - 52);
        return neg ? -d : d;
    }
    const unsigned long long b = mant + ((unsigned long long)(ex + 1022) << 52);
    return __longlong_as_double((long long)(b | ((unsigned long long)neg << 63)));
}

// sum_d v_d 2^(7(6-d) + e) of the seven FP32 accumulators (exact integers
// below 2^24), for slices of at most 480 rows.  The sum has up to 65 bits (a
// tall product's rows carry one more bit): a large one is halved with the bit
// that is lost kept as a sticky one, so it is rounded once.
__device__ __forceinline__ double oz_combine(const float v[OZ_S], int e) {
    const long long h = (long long)__float2int_rn(v[0]) * 128 + __float2int_rn(v[1]);
    long long l = __float2int_rn(v[OZ_S - 1]);
#pragma unroll
    for (int d = 2; d < OZ_S - 1; ++d) l += (long long)__float2int_rn(v[d]) * (1 << (7 * (OZ_S - 1 - d)));
    const bool big = (unsigned long long)(h + (1ll << 26)) >> 27 != 0;   // |h| above 2^26
    return oz_int_to_double(big ? ((h << 34) + (l >> 1)) | (l & 1) : (h << 35) + l, e + big);
}
// the same times 2^-56 in FP64, for longer slices
__device__ __forceinline__ double oz_combine_f64(const float v[OZ_S]) {
    long long t = 0;
#pragma unroll
    for (int d = 1; d < OZ_S; ++d) t += (long long)__float2int_rn(v[d]) * (1ll << (7 * (OZ_S - 1 - d)));
    return fma((double)t, 0x1p-56, (double)__float2int_rn(v[0]) * 0x1p-14);
}

// Persistent CTAs over output blocks a in [128 ta, +128), b in [64 tb, +64).
// Gram (TALL = false): item = (K-slice z of `steps` K steps, block), the
// blocks below the diagonal left out if symmetric; work[z][a][b] (m x m per
// slice) receives sum_d 2^(-7(d+2)) sum_{s+t=d} D_s^T E_t for a, b < m.  Tall
// product (TALL = true): item = (row block, column block), one slice; C[a][b]
// receives that sum times 2^(ea[a] + eb[b]) for a < nrows, b < m.
// Warp 0: TMEM allocation and the bulk copies of the digit panels (two
// stages; it runs ahead into the next item during an epilogue).  Warp 1 lane
// 0: the MMAs.  Warps 2..9: epilogue (a warp reads the TMEM lanes of its
// quarter: rows; the two warps of a quarter take 32 columns each), integer
// combination, rows staged in shared memory for coalesced stores.
// Bound by the MMAs: 28 digit pairs.  One by one, at N = 64, they are bound by
// shared memory (6 KB in 48 clocks each); the digits of B that share a digit of
// A are one MMA of up to N = 256 (12 KB in 128 clocks): 175 -> 129 us per Gram,
// 249 -> 231 us per tall product at 89 401 x 150 (the latter's epilogue shows).
// Before that the fill, the allocation and the epilogue of a CTA per block were
// exposed (186 and 319 us).
struct OzItem {
    int ta, tb;
    int64_t ks0;
    int nsteps, z;
};
template <bool TALL>
__device__ __forceinline__ OzItem oz_item(int64_t w, int nta, int ntb, int live, int symmetric, int steps, int64_t nks) {
    OzItem it;
    if (TALL) {
        it.ta = (int)(w / ntb);
        it.tb = (int)(w % ntb);
        it.ks0 = 0;
        it.nsteps = (int)nks;
        it.z = 0;
        return it;
    }
    it.z = (int)(w / live);
    int q = (int)(w % live);
    it.ta = 0;
    if (symmetric) {
        while (q >= ntb - 2 * it.ta) {
            q -= ntb - 2 * it.ta;
            ++it.ta;
        }
        it.tb = q + 2 * it.ta;
    } else {
        it.ta = q / ntb;
        it.tb = q % ntb;
    }
    it.ks0 = (int64_t)it.z * steps;
    it.nsteps = (int)min((int64_t)steps, nks - it.ks0);
    return it;
}

template <bool TALL>
__global__ void __launch_bounds__(TC_THREADS, 1)
k_oz_gram_tc(int m, int nta, int ntb, int live, int64_t items, int64_t nks, int steps, int npx, int npy,
             const __nv_bfloat16 *__restrict__ PX, const __nv_bfloat16 *__restrict__ PY, double *__restrict__ work,
             int symmetric, int32_t *__restrict__ err, int64_t nrows, double *__restrict__ C, int64_t ldc,
             const int *__restrict__ ea, const unsigned long long *__restrict__ eb_bits) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr unsigned long long LIMIT_NS = 1000000000ull;
    unsigned long long *full = reinterpret_cast<unsigned long long *>(smem), *empty = full + TC_NS;
    unsigned long long *tfull = empty + TC_NS, *tfree = tfull + 1;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + 128);
    unsigned char *stA = smem + 1024;
    unsigned char *stB = stA + TC_NS * TC_STAGE_A;
    double *stage = reinterpret_cast<double *>(stB + TC_NS * TC_STAGE_B);
    if (threadIdx.x == 0) {
        for (int i = 0; i < TC_NS; ++i) {
            mbar_init(full + i, 1);
            mbar_init(empty + i, 1);
        }
        mbar_init(tfull, 1);
        mbar_init(tfree, TC_EPI);
        mbar_fence_init();
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_addr(tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(tmem_slot);

    if (warp == 0) {   // ---- producer: 7 A blocks (4 or 8 KB) and 7 B blocks (4 KB) per stage
        int fill = 0, ok = 1;
        for (int64_t w = blockIdx.x; w < items && ok; w += gridDim.x) {
            const OzItem it = oz_item<TALL>(w, nta, ntb, live, symmetric, steps, nks);
            const unsigned abytes = min(2, npx - 2 * it.ta) * TC_PANEL;
            for (int k = 0; k < it.nsteps; ++k, ++fill) {
                const int st = fill % TC_NS, u = fill / TC_NS;
                if (u > 0 && lane == 0) ok = mbar_wait_bounded(empty + st, (u - 1) & 1, LIMIT_NS);
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) {
                    if (lane == 0) atomicExch(err, 3);
                    break;
                }
                if (lane == 0) mbar_expect_tx(full + st, OZ_S * (abytes + TC_PANEL));
                __syncwarp();
                const int64_t ks = it.ks0 + k;
                if (lane < OZ_S)
                    bulk_g2s(stA + st * TC_STAGE_A + lane * 2 * TC_PANEL,
                             PX + (((int64_t)lane * nks + ks) * npx + 2 * it.ta) * 2048, abytes, full + st);
                else if (lane < 2 * OZ_S)
                    bulk_g2s(stB + st * TC_STAGE_B + (lane - OZ_S) * TC_PANEL,
                             PY + (((int64_t)(lane - OZ_S) * nks + ks) * npy + it.tb) * 2048, TC_PANEL, full + st);
            }
        }
        // every copy has landed before the CTA gives its shared memory back
        if (lane == 0)
            for (int f = max(0, fill - TC_NS); f < fill; ++f)
                mbar_wait_bounded(full + f % TC_NS, (f / TC_NS) & 1, LIMIT_NS);
        __syncwarp();
    } else if (warp == 1) {   // ---- MMA issuer
        if (lane == 0) {
            int use = 0, n = 0;
            bool ok = true;
            for (int64_t w = blockIdx.x; w < items && ok; w += gridDim.x, ++n) {
                const OzItem it = oz_item<TALL>(w, nta, ntb, live, symmetric, steps, nks);
                if (n > 0 && !mbar_wait_bounded(tfree, (n - 1) & 1, LIMIT_NS)) {   // accumulators read out
                    atomicExch(err, 6);
                    break;
                }
                for (int k = 0; k < it.nsteps; ++k, ++use) {
                    const int st = use % TC_NS;
                    ok = mbar_wait_bounded(full + st, (use / TC_NS) & 1, LIMIT_NS);
                    if (!ok) {
                        atomicExch(err, 4);
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t a0 = umma_desc(smem_addr(stA + st * TC_STAGE_A));
                    const uint64_t b0 = umma_desc(smem_addr(stB + st * TC_STAGE_B));
                    // digit s of A times the digits t0 .. of B: their panels follow one another in the
                    // stage, as the sums d = s + t do in TMEM, so up to four of them are one MMA
#pragma unroll
                    for (int k16 = 0; k16 < 2; ++k16)
#pragma unroll
                        for (int sd = 0; sd < OZ_S; ++sd)
#pragma unroll
                            for (int t0 = 0; t0 < OZ_S - sd; t0 += 4)
                                umma_bf16(tmem + (uint32_t)((sd + t0) * TC_TN),
                                          umma_desc_at(a0, sd * 2 * TC_PANEL + k16 * 256u),
                                          umma_desc_at(b0, t0 * TC_PANEL + k16 * 256u),
                                          umma_idesc_bf16(TC_TM, (OZ_S - sd - t0 < 4 ? OZ_S - sd - t0 : 4) * TC_TN),
                                          sd == 0 && k16 == 0 ? (k > 0) : 1u);
                    umma_commit(empty + st);   // stage free once these MMAs have read it
                }
                umma_commit(tfull);            // accumulators final once every MMA above completes
            }
        }
        __syncwarp();
    } else {   // ---- epilogue: lane = TMEM lane 32 (warp % 4) + lane = row a, columns 32 h .. 32 h + 31
        const int quarter = warp & 3, h = (warp - 2) >> 2;
        double *sw = stage + (size_t)(warp - 2) * 32 * TC_EPI_LD;
        const bool wide = nks > TC_MAXSTEPS && TALL;
        int n = 0;
        for (int64_t w = blockIdx.x; w < items; w += gridDim.x, ++n) {
            const OzItem it = oz_item<TALL>(w, nta, ntb, live, symmetric, steps, nks);
            const bool ok = mbar_wait_bounded(tfull, n & 1, LIMIT_NS);
            if (__any_sync(0xffffffffu, !ok)) {
                if (lane == 0) atomicExch(err, 5);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int64_t a0 = (int64_t)it.ta * TC_TM + quarter * 32, rows = TALL ? nrows : m;
            double *O = TALL ? C : work + (int64_t)it.z * m * m;
            const int64_t ldo = TALL ? ldc : m;
            const int e_a = TALL && a0 + lane < nrows ? ea[a0 + lane] : 0;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int b0 = it.tb * TC_TN + h * 32 + c * 16;
                float v[OZ_S][16];
#pragma unroll
                for (int d = 0; d < OZ_S; ++d)
                    tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(d * TC_TN + h * 32 + c * 16), v[d]);
                if (c == 1) {   // this warp's accumulators are in registers
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tfree);
                }
                if (a0 < rows && b0 < m) {   // uniform over the warp
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        float u[OZ_S];
#pragma unroll
                        for (int d = 0; d < OZ_S; ++d) u[d] = v[d][j];
                        const int eb = TALL && b0 + j < m ? oz_exponent(eb_bits[b0 + j]) : 0;
                        sw[lane * TC_EPI_LD + j] =
                            wide ? ldexp(oz_combine_f64(u), e_a + eb) : oz_combine(u, e_a + eb - 56);
                    }
                    __syncwarp();
                    const int j = lane & 15, b = b0 + j;
                    for (int r = lane >> 4; r < 32; r += 2)
                        if (a0 + r < rows && b < m) O[(a0 + r) * ldo + b] = sw[r * TC_EPI_LD + j];
                    __syncwarp();
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// The kernels' shared-memory limit, raised once per device (attributes are
// process-wide and every launch uses the same size).
static void raise_tc_smem() {
    static bool raised[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !raised[dev]) {
        cudaFuncSetAttribute(k_oz_gram_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM);
        cudaFuncSetAttribute(k_oz_gram_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM);
        raised[dev] = true;
    }
}

// blocks of the Gram's output with work
static int gram_live(int m, bool symmetric) {
    const int nta = (m + TC_TM - 1) / TC_TM, ntb = (m + TC_TN - 1) / TC_TN;
    if (!symmetric) return nta * ntb;
    int c = 0;
    for (int a = 0; a < nta; ++a) c += ntb - 2 * a;
    return c;
}
// K steps per slice: the one whose rounds of items over the SMs take the
// fewest K steps, an item costing about two steps beyond its own
static int gram_steps(int64_t nks, int live, int sm_count) {
    int best = TC_MAXSTEPS;
    int64_t cost = INT64_MAX;
    for (int s = TC_MAXSTEPS; s >= 2; --s) {
        const int64_t items = (nks + s - 1) / s * live, c = (items + sm_count - 1) / sm_count * (s + 2);
        if (c < cost) {
            cost = c;
            best = s;
        }
    }
    return best;
}

static void ozaki_gram_tc(Ctx &ctx, int64_t n, int m, const double *X, int64_t ldx, const double *Y, int64_t ldy,
                          double *G, void *work, bool symmetric, int32_t *err, bool same_x) {
    const int64_t nks = (n + TC_KSTEP - 1) / TC_KSTEP;
    const int nta = (m + TC_TM - 1) / TC_TM, ntb = (m + TC_TN - 1) / TC_TN, np = ntb;
    const int live = gram_live(m, symmetric), steps = gram_steps(nks, live, ctx.sm_count);
    const int nz = (int)((nks + steps - 1) / steps);
    char *w = reinterpret_cast<char *>(work);
    __nv_bfloat16 *PX = reinterpret_cast<__nv_bfloat16 *>(w);
    __nv_bfloat16 *PY = PX + (size_t)OZ_S * nks * np * 2048;
    unsigned long long *mb = reinterpret_cast<unsigned long long *>(PY + (size_t)OZ_S * nks * np * 2048);
    double *part = reinterpret_cast<double *>(mb + 2 * m);
    raise_tc_smem();
    // same_x: the panels and maxima of X are those of the last call on this work block
    const int first = same_x ? 1 : 0, ops = 2 - first;
    cudaMemsetAsync(mb + (size_t)first * m, 0, ops * (size_t)m * sizeof(unsigned long long), ctx.stream);
    const double *X0 = same_x ? Y : X;
    const int64_t ld0 = same_x ? ldy : ldx;
    unsigned long long *mb0 = mb + (size_t)first * m;
    ctx.before(KC_GRAM, 8.0 * (double)n * m * ops, 0);
    k_oz_colmax<<<colmax_grid(ctx, n, m, ops), dim3(32, 8), 0, ctx.stream>>>(n, m, X0, ld0, Y, ldy, nullptr, mb0);
    ctx.after();
    ctx.before(KC_GRAM, (8.0 + 2.0 * OZ_S) * (double)n * m * ops, 0);
    k_oz_split_panel<<<dim3((unsigned)(nks * np), ops), 256, 0, ctx.stream>>>(n, m, nks, np, X0, ld0, Y, ldy, nullptr, mb0,
                                                                             same_x ? PY : PX, PY);
    ctx.after();
    const int64_t items = (int64_t)nz * live;
    const double pairs = OZ_S * (OZ_S + 1) / 2.0;
    ctx.before(KC_GRAM, 2.0 * OZ_S * (double)nks * TC_KSTEP * 64.0 * 3.0 * live + 8.0 * nz * m * m,
               2.0 * pairs * (double)live * TC_TM * TC_TN * nks * TC_KSTEP);
    k_oz_gram_tc<false><<<(unsigned)std::min<int64_t>(items, ctx.sm_count), TC_THREADS, TC_SMEM, ctx.stream>>>(
        m, nta, ntb, live, items, nks, steps, np, np, PX, PY, part, symmetric ? 1 : 0, err, 0, nullptr, 0, nullptr, nullptr);
    ctx.after();
    ctx.before(KC_GRAM, 8.0 * (double)nz * m * m, 0);
    k_oz_reduce<<<(unsigned)(((int64_t)m * m + 31) / 32), dim3(32, 8), 0, ctx.stream>>>(m, nz, part, mb, G, m,
                                                                                        symmetric ? 1 : 0);
    ctx.after();
}

// ---------------------------------------------------------------------------
size_t ozaki_gram_work_bytes(int64_t n, int m, int sm_count, bool tensor_core) {
    const int64_t npad = (n + 63) / 64 * 64;
    const int mpad = (m + OZ_TM - 1) / OZ_TM * OZ_TM;
    const size_t slices = 2 * (size_t)OZ_S * mpad * npad;
    const size_t split = (size_t)sm_count * 4;
    const size_t mma_sync = slices + split * m * m * sizeof(double) + 2 * (size_t)m * (sizeof(int) + 8) + 1024;
    if (!tensor_core) return mma_sync;
    // tensor-core form: bf16 digit panels of both operands and one m x m partial per K-slice
    const int64_t nks = (n + TC_KSTEP - 1) / TC_KSTEP;
    const int np = (m + TC_TN - 1) / TC_TN;
    const int steps = std::min(gram_steps(nks, gram_live(m, false), sm_count), gram_steps(nks, gram_live(m, true), sm_count));
    const int64_t nz = (nks + steps - 1) / steps;
    const size_t tc = (size_t)OZ_S * nks * 2 * np * 2048 * sizeof(__nv_bfloat16) + (size_t)nz * m * m * sizeof(double) +
                      2 * (size_t)m * 8 + 1024;
    return std::max(mma_sync, tc);
}

void ozaki_gram(Ctx &ctx, int64_t n, int m, const double *X, int64_t ldx, const double *Y, int64_t ldy, double *G,
                void *work, bool symmetric, int32_t *tc_err, bool same_x) {
    if (tc_err) {   // tensor-core form (tcgen05)
        ozaki_gram_tc(ctx, n, m, X, ldx, Y, ldy, G, work, symmetric, tc_err, same_x);
        return;
    }
    const int64_t npad = (n + 63) / 64 * 64;
    const int mpad = (m + OZ_TM - 1) / OZ_TM * OZ_TM;
    char *w = reinterpret_cast<char *>(work);
    int8_t *SX = reinterpret_cast<int8_t *>(w);
    int8_t *SY = SX + (size_t)OZ_S * mpad * npad;
    unsigned long long *mb = reinterpret_cast<unsigned long long *>(SY + (size_t)OZ_S * mpad * npad);
    int *ex = reinterpret_cast<int *>(mb + 2 * m);
    int *ey = ex + m;
    double *part = reinterpret_cast<double *>(reinterpret_cast<char *>(ey + m) + 16 - ((uintptr_t)(ey + m) & 15));
    const int tiles = mpad / OZ_TM;
    const int live = symmetric ? tiles * (tiles + 1) / 2 : tiles * tiles;   // tiles with work
    // K-slices: enough CTAs to fill the GPU, each at most 2^16 rows (int32 bound)
    int split = (ctx.sm_count * 4 + live - 1) / live;
    int64_t kslice = (npad + split - 1) / split;
    kslice = (kslice + 31) / 32 * 32;
    if (kslice > 65536) kslice = 65536;
    split = (int)((npad + kslice - 1) / kslice);

    cudaMemsetAsync(mb, 0, 2 * (size_t)m * sizeof(unsigned long long), ctx.stream);
    ctx.before(KC_GRAM, 8.0 * (double)n * m * 2, 0);
    k_oz_colmax<<<colmax_grid(ctx, n, m, 2), dim3(32, 8), 0, ctx.stream>>>(n, m, X, ldx, Y, ldy, nullptr, mb);
    k_oz_exponent<<<(2 * m + 127) / 128, 128, 0, ctx.stream>>>(2 * m, mb, ex);
    ctx.after();
    // digits (rows beyond n and columns beyond m become zeros)
    const dim3 sgrid(mpad / 32, (unsigned)std::min<int64_t>(npad / 32, 4096)), sblock(32, 8);
    ctx.before(KC_GRAM, 8.0 * (double)n * m * 2 + 2.0 * OZ_S * mpad * npad, 0);
    k_oz_split<<<sgrid, sblock, 0, ctx.stream>>>(n, m, npad, X, ldx, ex, SX, mpad);
    k_oz_split<<<sgrid, sblock, 0, ctx.stream>>>(n, m, npad, Y, ldy, ey, SY, mpad);
    ctx.after();
    const dim3 ggrid(tiles, tiles, split);
    const double pairs = OZ_S * (OZ_S + 1) / 2.0;
    ctx.before(KC_GRAM, 2.0 * OZ_S * mpad * npad,
               2.0 * pairs * (double)live * OZ_TM * OZ_TM * npad);
    k_oz_gram<<<ggrid, 128, 0, ctx.stream>>>(m, mpad, npad, kslice, SX, SY, part, symmetric ? 1 : 0);
    ctx.after();
    ctx.before(KC_GRAM, 8.0 * (double)split * m * m, 0);
    k_oz_reduce<<<(unsigned)(((int64_t)m * m + 31) / 32), dim3(32, 8), 0, ctx.stream>>>(m, split, part, mb, G, m,
                                                                                        symmetric ? 1 : 0);
    ctx.after();
}

// ---------------------------------------------------------------------------
// Tall product C = (A diag(cs)) B on the same digits: A is n x k (row-major,
// n large, k small), B is k x m, C is n x m.  Rows of A take their own
// exponent (max over the row of |A_ai cs_i|), columns of B theirs, so the
// error is ~2^-50 of max_i |A_ai cs_i| * sum_i |B_ib|; the optional column
// scaling cs (nullptr = 1) lets a caller whose columns differ widely in size
// split the well-scaled A diag(cs) instead of A.
// ---------------------------------------------------------------------------
constexpr int OZ_TA = 128;       // tall product: CTA tile rows (4 warps x 32)
constexpr int OZ_TB = 32;        // tall product: CTA tile columns

// One warp per row: exponent e[a] and the digits of A_a diag(cs), written to
// slices[s][a][i] (row pitch kpad, zero beyond k and beyond n).
__global__ void __launch_bounds__(256)
k_oz_rowsplit(int64_t n, int k, int kpad, int64_t npad, const double *__restrict__ A, int64_t lda,
              const double *__restrict__ cs, int *__restrict__ e, int8_t *__restrict__ slices) {
    const int lane = threadIdx.x & 31;
    const int64_t a = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (a >= npad) return;
    const bool live = a < n;
    double mx = 0.0;
    if (live)
        for (int i = lane; i < k; i += 32) mx = fmax(mx, fabs(A[a * lda + i] * (cs ? cs[i] : 1.0)));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    const int ea = mx > 0.0 ? ilogb(mx) + 2 : 0;
    if (lane == 0 && live) e[a] = ea;
    for (int i = lane; i < kpad; i += 32) {
        const double x = (live && i < k) ? A[a * lda + i] * (cs ? cs[i] : 1.0) : 0.0;
        int8_t d[OZ_S];
        oz_digits(x, ea, d);
#pragma unroll
        for (int s = 0; s < OZ_S; ++s) slices[((int64_t)s * npad + a) * kpad + i] = d[s];
    }
}

// C tile 128 x 32 per CTA, warp 32 x 32 (2 x 4 mma), all of K per CTA (k is
// small: kpad <= 2^16 keeps each diagonal's int32 sum exact).
__global__ void __launch_bounds__(128)
k_oz_tall(int64_t n, int m, int kpad, int64_t npad, int mpad, const int8_t *__restrict__ SA,
          const int8_t *__restrict__ SB, const int *__restrict__ ea, const int *__restrict__ eb, double *__restrict__ C,
          int64_t ldc) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, q = lane & 3;
    const int64_t a_base = blockIdx.y * (int64_t)OZ_TA + warp * 32;
    const int b_base = blockIdx.x * OZ_TB;
    const int64_t planeA = npad * kpad, planeB = (int64_t)mpad * kpad;
    double acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 4; ++h) acc[i][j][h] = 0.0;
    for (int d = 0; d < OZ_S; ++d) {
        int c[2][4][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int h = 0; h < 4; ++h) c[i][j][h] = 0;
        for (int s = 0; s <= d; ++s) {
            const int8_t *As = SA + s * planeA;
            const int8_t *Bt = SB + (d - s) * planeB;
            for (int kk = 0; kk < kpad; kk += 32) {
                unsigned af[2][4], bf[4][2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int8_t *r0 = As + (a_base + i * 16 + g) * kpad + kk + 4 * q;
                    const int8_t *r1 = r0 + 8 * (int64_t)kpad;
                    af[i][0] = __ldg(reinterpret_cast<const unsigned *>(r0));
                    af[i][1] = __ldg(reinterpret_cast<const unsigned *>(r1));
                    af[i][2] = __ldg(reinterpret_cast<const unsigned *>(r0 + 16));
                    af[i][3] = __ldg(reinterpret_cast<const unsigned *>(r1 + 16));
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int8_t *r = Bt + (int64_t)(b_base + j * 8 + g) * kpad + kk + 4 * q;
                    bf[j][0] = __ldg(reinterpret_cast<const unsigned *>(r));
                    bf[j][1] = __ldg(reinterpret_cast<const unsigned *>(r + 16));
                }
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) imma16832(c[i][j], af[i], bf[j]);
            }
        }
        const double scale = ldexp(1.0, -7 * (d + 2));
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int h = 0; h < 4; ++h) acc[i][j][h] = fma((double)c[i][j][h], scale, acc[i][j][h]);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int64_t a = a_base + i * 16 + g + (h >= 2 ? 8 : 0);
                const int b = b_base + j * 8 + 2 * q + (h & 1);
                if (a < n && b < m) C[a * ldc + b] = ldexp(acc[i][j][h], ea[a] + eb[b]);
            }
}

// Tall product on tcgen05: row exponents and digits of A diag(2^es) into the
// K-major panel layout of k_oz_gram_tc's A operand (panel rows = rows a of A,
// K = its columns i, zero beyond k).  One block per 64-row panel: thread
// (row, 8 consecutive columns of each K step), the row's maximum over its
// four threads first (the second read hits L1), all in integer arithmetic:
// the column scaling is a power of two added to the exponents.
// Bound by HBM (8 bytes read, 14 written per value).
__global__ void __launch_bounds__(256) k_oz_rowsplit_panel(int64_t n, int k, const double *__restrict__ A, int64_t lda,
                                                           const int *__restrict__ es, int64_t nks, int np,
                                                           int *__restrict__ e, __nv_bfloat16 *__restrict__ out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = warp * 8 + (lane >> 2), kc = lane & 3;
    const int64_t a = (int64_t)blockIdx.x * 64 + row;
    const bool live = a < n;
    const double *Ar = A + a * lda;
    // largest exponent of the row's scaled entries (+2), from the bits
    int emax = INT_MIN;
    if (live)
        for (int64_t ks = 0; ks < nks; ++ks) {
            const int i0 = (int)ks * TC_KSTEP + kc * 8;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int i = i0 + t;
                if (i >= k) continue;
                const unsigned long long b = abs_bits(Ar[i]);
                int ex = (int)(b >> 52);
                if (b == 0 || b > 0x7ff0000000000000ull) continue;   // a NaN does not count
                if (ex == 0) ex = 12 - __clzll((long long)b);   // subnormal: the leading bit's exponent
                emax = max(emax, ex - 1023 + (es ? es[i] : 0));
            }
        }
    emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 1));
    emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 2));
    // |x 2^-ea| < 1: the rows take one bit more than the columns of a Gram, for
    // what the power-of-two scaling loses against an exact one (with K <= 512
    // the digit sums stay below 2^24)
    const int ea = emax == INT_MIN ? 0 : emax + 1;
    if (!live) return;
    if (kc == 0) e[a] = ea;
    for (int64_t ks = 0; ks < nks; ++ks) {
        const int i0 = (int)ks * TC_KSTEP + kc * 8;
        long long v[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int i = i0 + t;
            v[t] = oz_biased(i < k ? Ar[i] : 0.0, i < k && es ? ea - es[i] : ea);
        }
        oz_store_digits(v, out + (ks * np + blockIdx.x) * 2048 + ((row >> 3) * 4 + kc) * 64 + (row & 7) * 8,
                        nks * np * 2048);
    }
}

// cs = f 2^es with f in [3/4, 3/2) (0 for 0): the power of two scales the tall
// operand exactly, f the rows of the small one
__global__ void k_oz_scale_split(int k, const double *__restrict__ cs, int *__restrict__ es, double *__restrict__ f) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= k) return;
    const double c = cs[i];
    int x = c != 0.0 && isfinite(c) ? ilogb(c) : 0;
    if (fabs(scalbn(c, -x)) >= 1.5) ++x;
    es[i] = x;
    f[i] = scalbn(c, -x);
}

// C = (A diag(cs)) B with A n x k, B k x m, k <= 512 (one K-slice: the FP32
// tensor-memory sums of digit products stay exact), on tcgen05.  *err (a
// mapped host word) records a bounded wait that gave up.
static void ozaki_tall_tc(Ctx &ctx, int64_t n, int k, int m, const double *A, int64_t lda, const double *cs,
                          const double *B, int64_t ldb, double *C, int64_t ldc, void *work, int kc, int32_t *err) {
    const int64_t nks = (k + TC_KSTEP - 1) / TC_KSTEP;
    const int nta = (int)((n + TC_TM - 1) / TC_TM), ntb = (m + TC_TN - 1) / TC_TN;
    const int npa = (int)((n + 63) / 64), npb = ntb;
    char *w = reinterpret_cast<char *>(work);
    __nv_bfloat16 *PA = reinterpret_cast<__nv_bfloat16 *>(w);
    __nv_bfloat16 *PB = PA + (size_t)OZ_S * nks * npa * 2048;
    unsigned long long *mb = reinterpret_cast<unsigned long long *>(PB + (size_t)OZ_S * nks * npb * 2048);
    double *f = reinterpret_cast<double *>(mb + m);
    int *es = reinterpret_cast<int *>(f + k);
    int *ea = es + k;
    raise_tc_smem();
    if (cs) {
        ctx.before(kc, 20.0 * k, 0);
        k_oz_scale_split<<<(k + 127) / 128, 128, 0, ctx.stream>>>(k, cs, es, f);
        ctx.after();
    }
    // B: column maxima and digit panels (panel rows = columns b, K = rows of B)
    cudaMemsetAsync(mb, 0, (size_t)m * sizeof(unsigned long long), ctx.stream);
    ctx.before(kc, 8.0 * (double)k * m * 2 + 2.0 * OZ_S * nks * TC_KSTEP * 64.0 * npb, 0);
    k_oz_colmax<<<colmax_grid(ctx, k, m, 1), dim3(32, 8), 0, ctx.stream>>>(k, m, B, ldb, nullptr, 0, cs ? f : nullptr, mb);
    k_oz_split_panel<<<dim3((unsigned)(nks * npb), 1), 256, 0, ctx.stream>>>(k, m, nks, npb, B, ldb, nullptr, 0,
                                                                            cs ? f : nullptr, mb, PB, nullptr);
    ctx.after();
    // A: row exponents and digit panels
    ctx.before(kc, 8.0 * (double)n * k + 2.0 * OZ_S * nks * TC_KSTEP * 64.0 * npa, 0);
    k_oz_rowsplit_panel<<<(unsigned)npa, 256, 0, ctx.stream>>>(n, k, A, lda, cs ? es : nullptr, nks, npa, ea, PA);
    ctx.after();
    const double pairs = OZ_S * (OZ_S + 1) / 2.0;
    const int64_t items = (int64_t)nta * ntb;
    ctx.before(kc, 2.0 * OZ_S * (double)nks * TC_KSTEP * 64.0 * (2.0 * nta * ntb + (double)nta * ntb) +
                       8.0 * (double)n * m,
               2.0 * pairs * (double)nta * ntb * TC_TM * TC_TN * nks * TC_KSTEP);
    k_oz_gram_tc<true><<<(unsigned)std::min<int64_t>(items, ctx.sm_count), TC_THREADS, TC_SMEM, ctx.stream>>>(
        m, nta, ntb, 0, items, nks, (int)nks, npa, npb, PA, PB, nullptr, 0, err, n, C, ldc, ea, mb);
    ctx.after();
}

size_t ozaki_tall_work_bytes(int64_t n, int k, int m, bool tensor_core) {
    const int64_t npad = (n + OZ_TA - 1) / OZ_TA * OZ_TA;
    const int kpad = (k + 31) / 32 * 32, mpad = (m + OZ_TB - 1) / OZ_TB * OZ_TB;
    const size_t mma_sync = (size_t)OZ_S * npad * kpad + (size_t)OZ_S * mpad * kpad + 256 +
                            (size_t)npad * sizeof(int) + (size_t)m * (sizeof(int) + 8) + 1024;
    if (!tensor_core) return mma_sync;
    // tensor-core form: bf16 digit panels of A (rows) and B (columns), maxima, scalings, exponents
    const int64_t nks = (k + TC_KSTEP - 1) / TC_KSTEP;
    const int64_t npa = (n + 63) / 64, npb = (m + TC_TN - 1) / TC_TN;
    const size_t tc = (size_t)OZ_S * nks * (npa + npb) * 2048 * sizeof(__nv_bfloat16) + (size_t)m * 8 + (size_t)k * 12 +
                      (size_t)n * sizeof(int) + 1024;
    return std::max(mma_sync, tc);
}

bool ozaki_tall_fits(int k) { return (k + 31) / 32 * 32 <= 65536; }

void ozaki_tall(Ctx &ctx, int64_t n, int k, int m, const double *A, int64_t lda, const double *cs, const double *B,
                int64_t ldb, double *C, int64_t ldc, void *work, int kc, int32_t *tc_err) {
    if (tc_err && k <= TC_KMAX) {
        ozaki_tall_tc(ctx, n, k, m, A, lda, cs, B, ldb, C, ldc, work, kc, tc_err);
        return;
    }
    const int64_t npad = (n + OZ_TA - 1) / OZ_TA * OZ_TA;
    const int kpad = (k + 31) / 32 * 32, mpad = (m + OZ_TB - 1) / OZ_TB * OZ_TB;
    char *w = reinterpret_cast<char *>(work);
    int8_t *SA = reinterpret_cast<int8_t *>(w);
    int8_t *SB = SA + (size_t)OZ_S * npad * kpad;
    char *tail = reinterpret_cast<char *>(SB + (size_t)OZ_S * mpad * kpad);
    tail += (256 - ((uintptr_t)tail & 255)) & 255;
    unsigned long long *mb = reinterpret_cast<unsigned long long *>(tail);
    int *eb = reinterpret_cast<int *>(mb + m);
    int *ea = eb + m;
    // B: column exponents and transposed digits (rows = K, columns = m)
    cudaMemsetAsync(mb, 0, (size_t)m * sizeof(unsigned long long), ctx.stream);
    ctx.before(kc, 8.0 * (double)k * m * 2 + 1.0 * OZ_S * mpad * kpad, 0);
    k_oz_colmax<<<colmax_grid(ctx, k, m, 1), dim3(32, 8), 0, ctx.stream>>>(k, m, B, ldb, nullptr, 0, nullptr, mb);
    k_oz_exponent<<<(m + 127) / 128, 128, 0, ctx.stream>>>(m, mb, eb);
    const dim3 sgrid(mpad / 32, (unsigned)std::min<int64_t>(kpad / 32, 4096)), sblock(32, 8);
    k_oz_split<<<sgrid, sblock, 0, ctx.stream>>>(k, m, kpad, B, ldb, eb, SB, mpad);
    ctx.after();
    // A: row exponents and digits
    ctx.before(kc, 8.0 * (double)n * k + 1.0 * OZ_S * npad * kpad, 0);
    k_oz_rowsplit<<<(unsigned)(npad / 8), 256, 0, ctx.stream>>>(n, k, kpad, npad, A, lda, cs, ea, SA);
    ctx.after();
    const dim3 grid(mpad / OZ_TB, (unsigned)(npad / OZ_TA));
    const double pairs = OZ_S * (OZ_S + 1) / 2.0;
    ctx.before(kc, (double)OZ_S * (npad * kpad * (double)(mpad / OZ_TB) + (double)mpad * kpad) + 8.0 * (double)n * m,
               2.0 * pairs * (double)npad * mpad * kpad);
    k_oz_tall<<<grid, 128, 0, ctx.stream>>>(n, m, kpad, npad, mpad, SA, SB, ea, eb, C, ldc);
    ctx.after();
}

}  // namespace slrf
