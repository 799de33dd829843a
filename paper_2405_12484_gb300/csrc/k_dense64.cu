// FP64 dense kernels of the prefactorisation (Sec. 7.2: Eq. cms_boundary
// and the reduced system of Eq. global_subspace / Eq. dd, computed on the
// device): the batched inverse of SPD matrices and a batched GEMM, row-major
// storage.  Matrices handed to the inverse are padded to a multiple of the
// 64-wide block with identity rows/columns.
//
// This chip issues two FP64 FMAs per clock and SM (1.2 TFLOP/s in all): one
// 64 x 64 x 64 product on one SM took 82 us.  So the products run on the
// BF16 tensor cores without giving up FP64: the error-free splitting of
// Ozaki, Ogita, Oishi and Rump ("Error-free transformations of matrix
// multiplication", 2012) in fixed point.  Per row of 64 values, a common
// power of two makes every value a 62-bit integer, cut into eight balanced
// base-256 digits (-128 .. 127, exact in BF16).  A product of two digits has
// at most 14 bits, so the FP32 accumulators hold the sums over 64 values of
// all pairs (i, j) of one order i + j = d exactly (at most 8 x 64 x 2^14 =
// 2^23).  The orders 0 .. 7 (36 pairs) are combined in 64-bit integers and
// rounded once; the dropped orders are below 2^-60 of the row maxima's
// product (FP64's own rounding is 2^-53).  Rows with an infinity or a NaN
// give NaN.
#include <algorithm>

#include "pd_internal.h"

namespace pdg {

namespace {

constexpr int NB = 64;        // block of the inverse, tile of the GEMM
constexpr int kDig = 8;       // digits of a value
constexpr int kThr = 512;     // threads of the digit kernels: 16 warps, one 16 x 16 part of a 64 x 64 tile each
// digits of one 64 x 64 block: [16-column group 4][16-row group 4][digit 8]
// fragments of 32 lanes x 16 bytes, in the register order of the A operand
// of mma.m16n8k16 (which, for the transposed operand, is also the order of
// two neighbouring B operands); 16 KB per 16-column group
constexpr int kGrpVec = 4 * kDig * 32;
constexpr int kBlkVec = 4 * kGrpVec;
constexpr int kNanExp = 1 << 28;   // exponent of a row that holds an infinity or a NaN
constexpr int kSmemDig = 2 * 16 * kBlkVec;   // dynamic shared memory: the digits of two blocks (128 KB)

// Exponent field -> E with |x| < 2^E for every x of that or a smaller field.
__device__ __forceinline__ int row_exponent(int field) {
    return field == 2047 ? kNanExp : (field == 0 ? 0 : field - 1022);
}

__device__ __forceinline__ int exponent_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// round(x 2^(62 - E)) plus the bias that makes bytes 0..6 balanced digits (|x| < 2^E; subnormals count as 0)
__device__ __forceinline__ long long biased_fixed(double x, int E) {
    constexpr long long kBias = 0x80808080808080ll;
    const long long bits = __double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7ff);
    if (ex == 0 || E == kNanExp) return kBias;
    const long long m = (bits & 0xfffffffffffffll) | (1ll << 52);
    const int sh = ex - 1013 - E;   // <= 9
    const long long v = sh >= 0 ? m << sh : (sh > -54 ? (m + (1ll << (-sh - 1))) >> -sh : 0);
    return (bits < 0 ? -v : v) + kBias;
}

// digit d (0 = most significant) of a biased value, as the bits of a float
__device__ __forceinline__ uint32_t digit_bits(long long u, int d) {
    if (d == 0) return __float_as_uint((float)(int)(u >> 56));
    const uint32_t byte = (uint32_t)(u >> (8 * (7 - d))) & 0xffu;
    return __float_as_uint(__uint_as_float(0x4b000000u | byte) - 8388736.0f);
}

// x 2^n (by the exponent field where the result is a normal number)
__device__ __forceinline__ double scale2(double x, int n) {
    const int f = exponent_field(x);
    if (f == 0 || f + n <= 0 || f + n >= 2047) return f == 0 ? 0.0 : ldexp(x, n);
    return __hiloint2double(__double2hiint(x) + (n << 20), __double2loint(x));
}

// Digits of the 16 x 16 block (mb, k16) of sm, whose rows have exponents es: one fragment per digit.
__device__ __forceinline__ void digits_block(const double (*sm)[NB + 1], const int* es, int mb, int k16, int lane,
                                             uint4* dst) {
    const int r = 16 * mb + (lane >> 2), c = 16 * k16 + 2 * (lane & 3);
    const int e0 = es[r], e1 = es[r + 8];
    const long long u0 = biased_fixed(sm[r][c], e0), u1 = biased_fixed(sm[r][c + 1], e0);
    const long long u2 = biased_fixed(sm[r + 8][c], e1), u3 = biased_fixed(sm[r + 8][c + 1], e1);
    const long long u4 = biased_fixed(sm[r][c + 8], e0), u5 = biased_fixed(sm[r][c + 9], e0);
    const long long u6 = biased_fixed(sm[r + 8][c + 8], e1), u7 = biased_fixed(sm[r + 8][c + 9], e1);
#pragma unroll
    for (int d = 0; d < kDig; ++d)   // two exact BF16 values: the upper halves of two floats
        dst[d * 32 + lane] = make_uint4(__byte_perm(digit_bits(u0, d), digit_bits(u1, d), 0x7632),
                                        __byte_perm(digit_bits(u2, d), digit_bits(u3, d), 0x7632),
                                        __byte_perm(digit_bits(u4, d), digit_bits(u5, d), 0x7632),
                                        __byte_perm(digit_bits(u6, d), digit_bits(u7, d), 0x7632));
}

// Row exponents (es: 64 ints of shared memory) and digits of the 64 x 64 block in sm.  Synchronises once; the
// digits are complete after the caller's next barrier.
__device__ __noinline__ void split_block(const double (*sm)[NB + 1], int* es, uint4* dig) {
    const int r = threadIdx.x >> 3;
    int f = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) f = max(f, exponent_field(sm[r][(threadIdx.x & 7) + 8 * k]));
    f = max(f, __shfl_xor_sync(0xffffffffu, f, 1));
    f = max(f, __shfl_xor_sync(0xffffffffu, f, 2));
    f = max(f, __shfl_xor_sync(0xffffffffu, f, 4));
    if ((threadIdx.x & 7) == 0) es[r] = row_exponent(f);
    __syncthreads();
    const int warp = threadIdx.x >> 5, mb = warp >> 2, k16 = warp & 3;
    digits_block(sm, es, mb, k16, threadIdx.x & 31, dig + (k16 * 4 + mb) * kDig * 32);
}

// A block's digits from shared to global memory (after a barrier).
__device__ __forceinline__ void store_digits(uint4* dst, const uint4* src, int* ex, const int* es) {
    for (int l = threadIdx.x; l < kBlkVec; l += kThr) dst[l] = src[l];
    if (threadIdx.x < NB) ex[threadIdx.x] = es[threadIdx.x];
}

// The digits of two blocks from global to shared memory, one group of asynchronous copies per 16 columns.
__device__ __forceinline__ void load_digits(uint4* sA, const uint4* A, uint4* sB, const uint4* B) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
#pragma unroll
        for (int l = 0; l < kGrpVec / kThr; ++l) {
            const int o = g * kGrpVec + l * kThr + threadIdx.x;
            const uint32_t da = (uint32_t)__cvta_generic_to_shared(sA + o), db = (uint32_t)__cvta_generic_to_shared(sB + o);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(da), "l"(A + o) : "memory");
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(db), "l"(B + o) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
}

__device__ __forceinline__ void mma_digits(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// The warp's 16 x 16 part of A B^T over one block of 64 columns, by order: acc[d] = sum_{i + j = d} A_i B_j^T, digits in
// shared memory.  Sixteen warps cover 64 x 64: 16-row group warp / 4, 16-column group warp & 3.  ASYNC: the
// digits are on their way (load_digits); else the caller has synchronised.  Rolled: unrolled
// copies would not fit the instruction cache.
template <bool ASYNC>
__device__ __forceinline__ void mma_block(const uint4* A, const uint4* B, float (&acc)[kDig][2][4]) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, mb = warp >> 2, nb = warp & 3;
#pragma unroll
    for (int d = 0; d < kDig; ++d)
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[d][q][k] = 0.f;
#pragma unroll 1
    for (int g = 0; g < 4; ++g) {
        if (ASYNC) {
            if (g == 0) asm volatile("cp.async.wait_group 3;" ::: "memory");
            if (g == 1) asm volatile("cp.async.wait_group 2;" ::: "memory");
            if (g == 2) asm volatile("cp.async.wait_group 1;" ::: "memory");
            if (g == 3) asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
        }
        uint4 a[kDig];
#pragma unroll
        for (int i = 0; i < kDig; ++i) a[i] = A[((g * 4 + mb) * kDig + i) * 32 + lane];
#pragma unroll
        for (int j = 0; j < kDig; ++j) {
            const uint4 b = B[((g * 4 + nb) * kDig + j) * 32 + lane];
#pragma unroll
            for (int i = 0; i < kDig - j; ++i) {
                mma_digits(acc[i + j][0], a[i], b.x, b.z);
                mma_digits(acc[i + j][1], a[i], b.y, b.w);
            }
        }
    }
}

// Row and column of element k (0..3) of 8-column group q (0, 1) of the calling thread's part of the tile.
__device__ __forceinline__ int tile_row(int k) {
    return 16 * (threadIdx.x >> 7) + ((threadIdx.x & 31) >> 2) + 8 * (k >> 1);
}
__device__ __forceinline__ int tile_col(int q, int k) {
    return 16 * ((threadIdx.x >> 5) & 3) + 8 * q + 2 * (threadIdx.x & 3) + (k & 1);
}

__device__ __forceinline__ int small_int(float x) {   // |x| <= 2^22: by the magic constant 1.5 2^23
    return (int)__float_as_uint(x + 12582912.0f) - 0x4b400000;
}

// The eight exact sums of one output -> FP64 (e: sum of the two rows' exponents), rounded once, in integer
// arithmetic only (on the FP64 pipe this would cost more than the products).
__device__ __forceinline__ double combine(const float (&acc)[kDig][2][4], int q, int k, int e) {
    const float a0 = acc[0][q][k], a1 = acc[1][q][k], a2 = acc[2][q][k], a3 = acc[3][q][k];
    const float a4 = acc[4][q][k], a5 = acc[5][q][k], a6 = acc[6][q][k], a7 = acc[7][q][k];
    // value = (H 2^32 + L) 2^(56 - 124 + e)
    const long long H = ((long long)small_int(a0) << 24) + ((long long)small_int(a1) << 16) +
                        ((long long)small_int(a2) << 8) + small_int(a3);
    const long long L = ((long long)__float2int_rn(a4) << 24) + ((long long)__float2int_rn(a5) << 16) +
                        ((long long)__float2int_rn(a6) << 8) + __float2int_rn(a7);
    const int s = min(32, __clzll(H < 0 ? -H : H) - 2);
    const long long t = (H << s) + (L >> (32 - s));   // |t| < 2^62, value = t 2^(e - 36 - s)
    if (e >= kNanExp / 2) return __longlong_as_double(0x7ff8000000000000ll);
    if (t == 0) return 0.0;
    const unsigned long long a = t < 0 ? (unsigned long long)-t : (unsigned long long)t;
    const int lz = __clzll((long long)a);
    const unsigned long long n = a << lz, m = (n >> 11) + ((n >> 10) & 1);   // 53 bits (2^53 carries into the exponent)
    const int field = 1023 + 63 - lz + e - 36 - s;
    unsigned long long bits = ((unsigned long long)(field - 1) << 52) + m;
    if (field <= 0) bits = 0;
    if (field >= 2047) bits = 0x7ff0000000000000ull;
    return __longlong_as_double((long long)(bits | ((unsigned long long)t & 0x8000000000000000ull)));
}
// Digits of op(X) by blocks of 64 x 64 (zero beyond rows x cols): block (row block blockIdx.x, column chunk
// blockIdx.y) of batch item blockIdx.z.  trans: element (r, k) is X[k ld + r], else X[r ld + k].
__global__ void __launch_bounds__(kThr) k_split64(const double* __restrict__ X, int ld, int64_t sX, int rows, int cols,
                                                 int trans, uint4* __restrict__ dig, int* __restrict__ ex) {
    __shared__ double sm[NB][NB + 1];
    __shared__ int es[NB];
    X += (int64_t)blockIdx.z * sX;
    const int r0 = blockIdx.x * NB, k0 = blockIdx.y * NB;
    for (int l = threadIdx.x; l < NB * NB; l += kThr) {
        const int hi = l / NB, lo = l % NB, r = trans ? lo : hi, k = trans ? hi : lo;
        double v = 0.0;
        if (r0 + r < rows && k0 + k < cols)
            v = trans ? X[(int64_t)(k0 + k) * ld + r0 + r] : X[(int64_t)(r0 + r) * ld + k0 + k];
        sm[r][k] = v;
    }
    __syncthreads();
    const int64_t blk = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    split_block(sm, es, dig + blk * kBlkVec);
    if (threadIdx.x < NB) ex[blk * NB + threadIdx.x] = es[threadIdx.x];
}

// C = alpha A B^T + beta C from the digits of A (MB row blocks) and of B (gridDim.x row blocks), KC chunks of 64.
__global__ void __launch_bounds__(kThr) k_gemm64(int M, int N, int KC, double alpha, const uint4* __restrict__ dA,
                                                const int* __restrict__ eA, const uint4* __restrict__ dB,
                                                const int* __restrict__ eB, double beta, double* __restrict__ C, int ldc,
                                                int64_t sC) {
    extern __shared__ uint4 dsm[];
    const int64_t za = (int64_t)blockIdx.z * KC * gridDim.y, zb = (int64_t)blockIdx.z * KC * gridDim.x;
    C += (int64_t)blockIdx.z * sC;
    double sum[2][4];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) sum[q][k] = 0.0;
    for (int kc = 0; kc < KC; ++kc) {
        const int64_t ba = za + (int64_t)kc * gridDim.y + blockIdx.y, bb = zb + (int64_t)kc * gridDim.x + blockIdx.x;
        float acc[kDig][2][4];
        if (kc > 0) __syncthreads();   // the previous chunk's digits are read
        load_digits(dsm, dA + ba * kBlkVec, dsm + kBlkVec, dB + bb * kBlkVec);
        mma_block<true>(dsm, dsm + kBlkVec, acc);
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int k = 0; k < 4; ++k)
                sum[q][k] += combine(acc, q, k, eA[ba * NB + tile_row(k)] + eB[bb * NB + tile_col(q, k)]);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int r = blockIdx.y * NB + tile_row(k), c = blockIdx.x * NB + tile_col(q, k);
            if (r >= M || c >= N) continue;
            double* p = C + (int64_t)r * ldc + c;
            *p = (beta == 0.0) ? alpha * sum[q][k] : fma(alpha, sum[q][k], beta * *p);
        }
}

// ---- inverse of an SPD matrix: symmetric block sweeps
//
// Sweeping block k of the symmetric B (pivot D = B_kk, P = D^-1, C_i = B_ik):
// B_ij -= C_i P C_j^T, B_ik = C_i P, B_kk = -P; after every block has been
// swept B = -A^-1.  The pivots are the Schur complements of a block
// Cholesky factorisation, so a non-positive one shows that A is not positive
// definite.  Half the operations of factor + triangular inversion, and two
// launches per 64 columns: k_sweep_panel forms W = C P (and the digits of C
// and W), k_sweep_update forms B - W C^T on the lower tiles; its first block
// per matrix also inverts the next pivot while the others update.
// W = C P with P rounded to FP64 is not as good as a triangular solve where C P C^T cancels; there the panel refines
// it (see cancels and refine_panel).  Errors max |X - X*| / max |X*| against extended precision, blocked Cholesky on the
// FP64 pipe / plain sweeps / these: lattices of 400 vertices moved by up to 45 % of an edge, two decades of stiffness,
// dt = 1 s 1.6e-8 / 1.3e-7 / 1.2e-9; I + v v^T with a condition of 2^20 over two pivots 2.0e-11 / 1.1e-6 / 7.1e-12; regular
// lattices, two decades, dt = 1/150 s 1.7e-15 / 2.3e-15 / 2.3e-15 (not refined).
// What bounds it: one matrix is a chain of n / 64 steps, each the pivot's inversion on one SM (about 60 us), its
// tile and the panel (25 us); the tiles of a batch are bound by the tensor cores (36 products per FP64
// product, mma.sync).  Measured against the blocked Cholesky factorisation and substitution on the FP64 pipe
// that it replaces (GB300, events): n = 512 x 25 matrices 9.9 -> 1.06 ms, 512 x 200 50.0 -> 6.4 ms, 1472 x 8
// 50.6 -> 4.7 ms, 1984 x 1 30.3 -> 3.1 ms, 2880 x 1 60.8 -> 4.6 ms (the choice of refinement is 1 % of these);
// dense_gemm's error against exact sums 4e-16 of sum |a||b| on rows of ordinary range (2e-15 on the FP64 pipe), 2^-60 of
// the row maxima's product for entries far below the maximum of their row of 64.

// Double-float arithmetic (pairs of floats, about 48 bits) for the pivot blocks: an FP64 instruction of a warp
// occupies its quarter of the SM for about 60 clocks, these 15 FP32 ones for 15.  The intrinsics keep the
// compiler from contracting the error terms away.
struct DF {
    float h, l;
};
__device__ __forceinline__ DF df_norm(float h, float l) {   // |l| <= |h|
    const float s = __fadd_rn(h, l);
    return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ DF df_mul(DF a, DF b) {
    const float h = __fmul_rn(a.h, b.h);
    return df_norm(h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -h))));
}
__device__ __forceinline__ DF df_recip(DF d) {   // one Newton step with the exact residual
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d.h));
    return df_norm(r, __fmul_rn(r, __fmaf_rn(-d.l, r, __fmaf_rn(-d.h, r, 1.0f))));
}
// c - a b; the sum is left unnormalised (its low part a few roundings of the high one), df_norm before the next product
__device__ __forceinline__ DF df_fnma(DF a, DF b, DF c) {
    const float h = __fmul_rn(a.h, b.h);
    const float l = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -h)));
    const float s = __fsub_rn(c.h, h), t = __fsub_rn(s, c.h);
    const float e = __fsub_rn(__fsub_rn(c.h, __fsub_rn(s, t)), __fadd_rn(h, t));
    return {s, __fadd_rn(e, __fsub_rn(c.l, l))};
}

// (a __grid_constant__ parameter: its address goes to the routines out of line without a copy on the stack)
struct SweepArgs {
    double* A;             // the matrix (lower tiles), swept in place
    int lda, nblk;         // row stride, n / 64
    int64_t sA;
    double* P;             // per matrix: 64 x 64 inverse of the pivot, then its digits
    uint4* dP;
    int* eP;
    uint4* dD;             // per matrix: digits of the scaled pivot D' = S D S, S = 2^-ex; eD: their exponents + ex
    int *eD, *ex;
    float *sx, *nu;        // per matrix: square roots of the diagonal of X = D'^-1, its largest -X_kj / (sx_k sx_j)
    uint4 *dC, *dW;        // per matrix: digits of the panel C and of W, nblk blocks each
    int *eC, *eW;
    int* err;
};

struct PivotSmem {
    int es[NB], es2[NB], ex[NB];
    DF col[2][NB];
    float sx[NB];
    unsigned nu;
    int bad;
};

// Inverse of the pivot block in sm (its lower part is read) -> P and its digits; sets the error
// flag when a pivot is not positive.  dsm: digits of two blocks.
//   D' = S D S with powers of two S that bring its diagonal into [1, 4)
//   X  = D'^-1 by symmetric sweeps in double-float (registers, element (ty + 32 a, tx + 16 b), the 16-column groups
//        that reach the lower part; one barrier per column), relative error about 2^-46 cond(D')
//   X += (I - X D') X, both products exact to FP64 by digits: squares that error
//   P  = S X S
__device__ __noinline__ void finish_pivot(const SweepArgs& S, int z, double (*sm)[NB + 1], uint4* dsm, PivotSmem& T) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    if (threadIdx.x == 0) {
        T.bad = 0;
        T.nu = 0;
    }
    __syncthreads();
    if (threadIdx.x < NB) {
        const double d = sm[threadIdx.x][threadIdx.x];
        const int f = exponent_field(d);
        const bool ok = d > 0.0 && f != 2047 && f != 0;
        if (!ok) T.bad = 1;
        T.ex[threadIdx.x] = ok ? (f - 1023) >> 1 : 0;
    }
    __syncthreads();
    // groups b of a row group a: 2 a + 2 of 16 columns (b >> 1 <= a)
    DF m[2][4];
    {
        double v[2][4];
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2 * a + 2; ++b) {
                const int r = ty + 32 * a, c = tx + 16 * b;
                v[a][b] = scale2(r >= c ? sm[r][c] : sm[c][r], -(T.ex[r] + T.ex[c]));
                m[a][b].h = (float)v[a][b];
                m[a][b].l = (float)(v[a][b] - (double)m[a][b].h);
            }
        __syncthreads();
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2 * a + 2; ++b) {
                const int r = ty + 32 * a, c = tx + 16 * b;
                sm[r][c] = v[a][b];
                sm[c][r] = v[a][b];
            }
    }
    __syncthreads();
    split_block(sm, T.es, dsm);             // digits of D'
#pragma unroll
    for (int kb = 0; kb < 4; ++kb)
#pragma unroll 1
        for (int kt = 0; kt < 16; ++kt) {
            const int k = 16 * kb + kt, ka = kb >> 1, kr = k & 31;   // row k: ty = kr of row group ka
            DF* col = T.col[kt & 1];        // the other one may still be read
            if (tx == kt) {                 // column k, row groups from ka on
#pragma unroll
                for (int a = ka; a < 2; ++a) col[ty + 32 * a] = df_norm(m[a][kb].h, m[a][kb].l);
            }
            if (ty == kr) {                 // the rest of it is row k
#pragma unroll
                for (int b = 0; b < 2 * ka; ++b) col[tx + 16 * b] = df_norm(m[ka][b].h, m[ka][b].l);
            }
            __syncthreads();
            DF d = col[k];
            if (!(d.h > 0.f) || !(d.h < 3e38f)) {
                if (threadIdx.x == 0) T.bad = 1;
                d = {1.f, 0.f};
            }
            const DF p = df_recip(d);
            DF wi[2];
#pragma unroll
            for (int a = 0; a < 2; ++a) wi[a] = df_mul(col[ty + 32 * a], p);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const DF cj = col[tx + 16 * b];
#pragma unroll
                for (int a = b >> 1; a < 2; ++a) {
                    DF v = df_fnma(wi[a], cj, m[a][b]);
                    if (a == ka && ty == kr) v = df_mul(cj, p);
                    if (b == kb && tx == kt) v = (a == ka && ty == kr) ? DF{-p.h, -p.l} : wi[a];
                    m[a][b] = v;
                }
            }
        }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2 * a + 2; ++b) {      // X = -(swept matrix)
            const int r = ty + 32 * a, c = tx + 16 * b;
            const double v = -((double)m[a][b].h + (double)m[a][b].l);
            if (r >= c) {
                sm[r][c] = v;
                sm[c][r] = v;
            }
            if (r == c) T.sx[r] = sqrtf(fmaxf(-m[a][b].h, 0.f));
        }
    __syncthreads();
    uint4 *dD = dsm, *dX = dsm + kBlkVec;
    // for the panel's choice and its refinement (see k_sweep_panel)
    float nu = 0.f;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2 * a + 2; ++b)
            if (ty + 32 * a > tx + 16 * b) nu = fmaxf(nu, __fdividef(m[a][b].h, T.sx[ty + 32 * a] * T.sx[tx + 16 * b]));
    const unsigned wnu = __reduce_max_sync(0xffffffffu, __float_as_uint(nu));
    if ((threadIdx.x & 31) == 0) atomicMax(&T.nu, wnu);
    for (int l = threadIdx.x; l < kBlkVec; l += kThr) S.dD[(int64_t)z * kBlkVec + l] = dD[l];
    if (threadIdx.x < NB) {
        S.eD[z * NB + threadIdx.x] = T.es[threadIdx.x] + T.ex[threadIdx.x];
        S.ex[z * NB + threadIdx.x] = T.ex[threadIdx.x];
        S.sx[z * NB + threadIdx.x] = T.sx[threadIdx.x];
    }
    split_block(sm, T.es2, dX);
    double x[2][4];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) x[q][e] = sm[tile_row(e)][tile_col(q, e)];
    __syncthreads();
    float acc[kDig][2][4];
    mma_block<false>(dX, dD, acc);
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) {       // R = I - X D'
            const int r = tile_row(e), c = tile_col(q, e);
            double v = -combine(acc, q, e, T.es2[r] + T.es[c]);
            if (r == c) v += 1.0;
            sm[r][c] = v;
        }
    __syncthreads();
    split_block(sm, T.es, dD);              // (its barrier: every read of D' digits is past)
    __syncthreads();
    mma_block<false>(dD, dX, acc);
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) {       // X + R X, unscaled
            const int r = tile_row(e), c = tile_col(q, e);
            sm[r][c] = scale2(x[q][e] + combine(acc, q, e, T.es[r] + T.es2[c]), -(T.ex[r] + T.ex[c]));
        }
    __syncthreads();
    split_block(sm, T.es, dD);
    __syncthreads();
    store_digits(S.dP + (int64_t)z * kBlkVec, dD, S.eP + z * NB, T.es);
    double* P = S.P + (int64_t)z * NB * NB;
    for (int l = threadIdx.x; l < NB * NB; l += kThr) P[l] = sm[l / NB][l % NB];
    if (threadIdx.x == 0) {
        S.nu[z] = __uint_as_float(T.nu);
        if (T.bad) atomicOr(S.err, ERR_NOT_SPD);
    }
}

__global__ void __launch_bounds__(kThr) k_sweep_first(const __grid_constant__ SweepArgs S) {
    extern __shared__ uint4 dsm[];
    __shared__ double sm[NB][NB + 1];
    __shared__ PivotSmem T;
    const double* A = S.A + (int64_t)blockIdx.x * S.sA;
    for (int l = threadIdx.x; l < NB * NB; l += kThr) sm[l / NB][l % NB] = A[(int64_t)(l / NB) * S.lda + l % NB];
    finish_pivot(S, blockIdx.x, sm, dsm, T);
}

// x 2^-e to 20 bits (zero below 2^-100, infinite above 2^100)
__device__ __forceinline__ float coarse(double x, int e) {
    const int hi = __double2hiint(x), f = ((hi >> 20) & 0x7ff) - 1023 - e;
    const unsigned sign = (unsigned)hi & 0x80000000u;
    if (f < -100) return 0.f;
    if (f > 100) return __uint_as_float(sign | 0x7f800000u);
    return __uint_as_float(sign | (unsigned)(f + 127) << 23 | ((unsigned)hi & 0xfffffu) << 3);
}

// Whether W = C P of the row block in sm needs the refinement: P is rounded to FP64, so W C^T is off by up to
// u |C| P |C|^T, where a Cholesky factorisation is off by u times the diagonal of B.  The first is C P C^T (at most
// that diagonal) where nothing cancels, as in the M-matrices of well-shaped elements (C <= 0 <= P); in general it is
// at most C P C^T + 4 t+ t- + 2 nu t^2 with t+- = sum_k (C_ik)+- P_kk^1/2, t their sum, and nu the most negative entry of
// P relative to its diagonal.  Refine where the added terms exceed twice the diagonal: never on the lattices of the
// slabs and shells (largest measured 0.7), on about half of the row blocks of lattices with vertices moved by up to 30 or 45 %.
__device__ __forceinline__ bool cancels(const SweepArgs& S, int z, int i, const double (*sm)[NB + 1]) {
    const int r = threadIdx.x >> 3;
    const double* A = S.A + (int64_t)z * S.sA;
    const double d = A[(int64_t)(i * NB + r) * (S.lda + 1)];
    const int e = (exponent_field(d) - 1023) >> 1;
    float tp = 0.f, tm = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int c = (threadIdx.x & 7) + 8 * k;
        const float v = coarse(sm[r][c], S.ex[z * NB + c] + e) * S.sx[z * NB + c];
        tp += fmaxf(v, 0.f);
        tm += fmaxf(-v, 0.f);
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        tp += __shfl_xor_sync(0xffffffffu, tp, o);
        tm += __shfl_xor_sync(0xffffffffu, tm, o);
    }
    const float t = tp + tm;
    return !(4.f * tp * tm + 2.f * S.nu[z] * t * t <= 2.f * fabsf(coarse(d, 2 * e)));
}

// W += (C - W D) P with exact products: W D is C to rounding then, as with a triangular solve.  T: the tile of C
// (transposed if flip); sC, sP: digits, sP those of P on entry and exit.
__device__ __noinline__ void refine_panel(const SweepArgs& S, int z, const double* T, bool flip, double (*sm)[NB + 1],
                                          int* es, uint4* sC, uint4* sP, double (&w)[2][4]) {
    float acc[kDig][2][4];
    const uint4 *dP = S.dP + (int64_t)z * kBlkVec, *dD = S.dD + (int64_t)z * kBlkVec;
    __syncthreads();           // es and the digits in sC and sP are read
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) sm[tile_row(e)][tile_col(q, e)] = scale2(w[q][e], S.ex[z * NB + tile_col(q, e)]);
    for (int l = threadIdx.x; l < kBlkVec; l += kThr) sP[l] = dD[l];
    __syncthreads();
    split_block(sm, es, sC);   // W S^-1, so that W D = (W S^-1) D' S^-1
    __syncthreads();
    mma_block<false>(sC, sP, acc);
    double res[2][4];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int r = tile_row(e), c = tile_col(q, e);
            res[q][e] = T[flip ? (int64_t)c * S.lda + r : (int64_t)r * S.lda + c] -
                        combine(acc, q, e, es[r] + S.eD[z * NB + c]);
        }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) sm[tile_row(e)][tile_col(q, e)] = res[q][e];
    for (int l = threadIdx.x; l < kBlkVec; l += kThr) sP[l] = dP[l];
    __syncthreads();
    split_block(sm, es, sC);
    __syncthreads();
    mma_block<false>(sC, sP, acc);
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) w[q][e] += combine(acc, q, e, es[tile_row(e)] + S.eP[z * NB + tile_col(q, e)]);
}

// Row block blockIdx.y of matrix blockIdx.x: C_i, W_i = C_i P into the matrix, the digits of both.
__global__ void __launch_bounds__(kThr) k_sweep_panel(const __grid_constant__ SweepArgs S, int k) {
    extern __shared__ uint4 dsm[];
    __shared__ double sm[NB][NB + 1];
    __shared__ int es[NB];
    const int z = blockIdx.x, i = blockIdx.y;
    double* A = S.A + (int64_t)z * S.sA;
    double* T = A + (int64_t)(i >= k ? i : k) * NB * S.lda + (i >= k ? k : i) * NB;   // lower tile of (i, k)
    if (i == k) {
        const double* P = S.P + (int64_t)z * NB * NB;
        for (int l = threadIdx.x; l < NB * NB; l += kThr) T[(int64_t)(l / NB) * S.lda + l % NB] = -P[l];
        return;
    }
    const bool flip = i < k;   // stored as its transpose
    for (int l = threadIdx.x; l < NB * NB; l += kThr) {
        const double v = T[(int64_t)(l / NB) * S.lda + l % NB];
        if (flip) sm[l % NB][l / NB] = v;
        else sm[l / NB][l % NB] = v;
    }
    __syncthreads();
    const int64_t blk = (int64_t)z * S.nblk + i;
    uint4 *sC = dsm, *sP = dsm + kBlkVec;
    const uint4* dP = S.dP + (int64_t)z * kBlkVec;
    for (int l = threadIdx.x; l < kBlkVec; l += kThr) sP[l] = dP[l];
    const bool own = cancels(S, z, i, sm);
    split_block(sm, es, sC);
    const bool refine = __syncthreads_or(own) != 0;
    store_digits(S.dC + blk * kBlkVec, sC, S.eC + blk * NB, es);
    float acc[kDig][2][4];
    mma_block<false>(sC, sP, acc);
    double w[2][4];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e)
            w[q][e] = combine(acc, q, e, es[tile_row(e)] + S.eP[z * NB + tile_col(q, e)]);
    if (refine) {
        double v[2][4];        // (w stays in registers)
        memcpy(v, w, sizeof(v));
        refine_panel(S, z, T, flip, sm, es, sC, sP, v);
        memcpy(w, v, sizeof(v));
    }
    __syncthreads();           // es and the digits of C are rewritten below
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) sm[tile_row(e)][tile_col(q, e)] = w[q][e];
    __syncthreads();
    for (int l = threadIdx.x; l < NB * NB; l += kThr)
        T[(int64_t)(l / NB) * S.lda + l % NB] = flip ? sm[l % NB][l / NB] : sm[l / NB][l % NB];
    split_block(sm, es, sC);
    __syncthreads();
    store_digits(S.dW + blk * kBlkVec, sC, S.eW + blk * NB, es);
}

// Lower tile (i, j), i, j != k, of one matrix: B_ij -= W_i C_j^T.  Tile 0 is the next pivot (k + 1, k + 1), which its
// block then inverts (all matrices' first, so that the long blocks start first); the others follow row by row.
__global__ void __launch_bounds__(kThr) k_sweep_update(const __grid_constant__ SweepArgs S, int k, int batch) {
    extern __shared__ uint4 dsm[];
    __shared__ double sm[NB][NB + 1];
    __shared__ PivotSmem ps;
    const int z = blockIdx.x % batch, tile = blockIdx.x / batch, m = S.nblk - 1;
    const int next = k + 1 < S.nblk ? k : -1;          // index of block k + 1 among the blocks other than k
    int i, j;
    const bool pivot = next >= 0 && tile == 0;
    if (pivot) {
        i = j = next;
    } else {
        // tile number t of the lower triangle (row by row), the next pivot's tile moved to the front
        int t = tile;
        if (next >= 0) {
            const int tn = next * (next + 1) / 2 + next;
            t = t <= tn ? t - 1 : t;
        }
        i = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
        while (i * (i + 1) / 2 > t) --i;
        while ((i + 1) * (i + 2) / 2 <= t) ++i;
        j = t - i * (i + 1) / 2;
        if (i >= m) return;   // (not reached: the grid has m (m + 1) / 2 tiles)
    }
    i += i >= k;
    j += j >= k;
    const int64_t bi = (int64_t)z * S.nblk + i, bj = (int64_t)z * S.nblk + j;
    float acc[kDig][2][4];
    load_digits(dsm, S.dW + bi * kBlkVec, dsm + kBlkVec, S.dC + bj * kBlkVec);
    mma_block<true>(dsm, dsm + kBlkVec, acc);
    double* T = S.A + (int64_t)z * S.sA + (int64_t)i * NB * S.lda + j * NB;
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = tile_row(2 * h), c = tile_col(q, 0), ew = S.eW[bi * NB + r];
            double2* p = reinterpret_cast<double2*>(T + (int64_t)r * S.lda + c);
            double2 v = *p;
            v.x -= combine(acc, q, 2 * h, ew + S.eC[bj * NB + c]);
            v.y -= combine(acc, q, 2 * h + 1, ew + S.eC[bj * NB + c + 1]);
            *p = v;
            if (pivot) {
                sm[r][c] = v.x;
                sm[r][c + 1] = v.y;
            }
        }
    if (!pivot) return;
    __syncthreads();
    finish_pivot(S, z, sm, dsm, ps);
}

// X = -B, both triangles, from the lower tiles
__global__ void __launch_bounds__(kThr) k_sweep_store(const double* __restrict__ A, int lda, int64_t sA,
                                                     double* __restrict__ X, int ldx, int64_t sX) {
    if (blockIdx.x > blockIdx.y) return;
    __shared__ double sm[NB][NB + 1];
    A += (int64_t)blockIdx.z * sA;
    X += (int64_t)blockIdx.z * sX;
    const int i = blockIdx.y, j = blockIdx.x;
    for (int l = threadIdx.x; l < NB * NB; l += kThr) {
        const int r = l / NB, c = l % NB;
        const double v = -A[(int64_t)(i * NB + r) * lda + j * NB + c];
        sm[r][c] = v;
        X[(int64_t)(i * NB + r) * ldx + j * NB + c] = v;
    }
    if (i == j) return;
    __syncthreads();
    for (int l = threadIdx.x; l < NB * NB; l += kThr) {
        const int r = l / NB, c = l % NB;
        X[(int64_t)(j * NB + r) * ldx + i * NB + c] = sm[c][r];
    }
}

__global__ void k_set_identity(double* __restrict__ A, int n, int lda, int64_t sA) {
    A += (int64_t)blockIdx.y * sA;
    const int64_t tot = (int64_t)n * n;
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < tot; l += (int64_t)gridDim.x * blockDim.x) {
        int r = (int)(l / n), c = (int)(l % n);
        A[(int64_t)r * lda + c] = (r == c) ? 1.0 : 0.0;
    }
}

inline int grid_for(int64_t n) {
    int64_t b = (n + 255) / 256;
    return (int)(b < 65535 ? (b > 0 ? b : 1) : 65535);
}

// Temporary device memory of one call, stream-ordered.
struct Scratch {
    void* p = nullptr;
    cudaStream_t s;
    explicit Scratch(size_t bytes, cudaStream_t st) : s(st) { PDG_CUDA(cudaMallocAsync(&p, bytes, s)); }
    ~Scratch() { cudaFreeAsync(p, s); }
    Scratch(const Scratch&) = delete;
    Scratch& operator=(const Scratch&) = delete;
};

// the digit kernels' dynamic shared memory exceeds the default limit
void allow_digit_smem() {
    static PerDevice known;
    if (max_dynamic_smem(known, k_gemm64, k_sweep_first, k_sweep_panel, k_sweep_update) < kSmemDig) throw Fail{PD_ERR_UNSUPPORTED};
}

constexpr int64_t kSplitBytes = 16 * (int64_t)kBlkVec + 4 * NB;   // digits and exponents of one 64 x 64 block
constexpr int64_t kScratchMax = int64_t(64) << 20;               // digits held at once (larger calls go in slices)

}  // namespace

void dense_gemm(bool ta, bool tb, int M, int N, int K, double alpha, const double* A, int lda, int64_t sA,
                const double* B, int ldb, int64_t sB, double beta, double* C, int ldc, int64_t sC, int batch,
                cudaStream_t s) {
    if (M <= 0 || N <= 0 || batch <= 0) return;
    allow_digit_smem();
    const int KC = (K + NB - 1) / NB, nbN = (N + NB - 1) / NB, nbM = (M + NB - 1) / NB;
    // slices of the batch, or of the rows of one item, whose digits fit in kScratchMax (and the grid's limits)
    const int64_t cap = std::max<int64_t>(1, kScratchMax / (kSplitBytes * std::max(KC, 1)));
    const int mb = (int)std::max<int64_t>(1, std::min<int64_t>(std::min(nbM, 65535), cap - nbN));
    const int zb = mb < nbM ? 1 : (int)std::max<int64_t>(1, std::min<int64_t>(std::min(batch, 65535), cap / (mb + nbN)));
    const int64_t nA = (int64_t)zb * std::max(KC, 1) * mb, nBl = (int64_t)zb * std::max(KC, 1) * nbN;
    Scratch w((size_t)(kSplitBytes * (nA + nBl)), s);
    uint4* dA = static_cast<uint4*>(w.p);
    uint4* dB = dA + nA * kBlkVec;
    int* eA = reinterpret_cast<int*>(dB + nBl * kBlkVec);
    int* eB = eA + nA * NB;
    for (int z0 = 0; z0 < batch; z0 += zb) {
        const int nz = std::min(zb, batch - z0);
        // op(B)^T: its rows are the columns of op(B)
        if (KC > 0) {
            k_split64<<<dim3(nbN, KC, nz), kThr, 0, s>>>(B + z0 * sB, ldb, sB, N, K, tb ? 0 : 1, dB, eB);
            PDG_CHECK_LAUNCH();
        }
        for (int m0 = 0; m0 < nbM; m0 += mb) {
            const int rows = std::min(M - m0 * NB, mb * NB), nm = (rows + NB - 1) / NB;
            const double* Am = A + z0 * sA + (int64_t)m0 * NB * (ta ? 1 : lda);
            if (KC > 0) {
                k_split64<<<dim3(nm, KC, nz), kThr, 0, s>>>(Am, lda, sA, rows, K, ta ? 1 : 0, dA, eA);
                PDG_CHECK_LAUNCH();
            }
            k_gemm64<<<dim3(nbN, nm, nz), kThr, kSmemDig, s>>>(rows, N, KC, alpha, dA, eA, dB, eB, beta,
                                                       C + z0 * sC + (int64_t)m0 * NB * ldc, ldc, sC);
            PDG_CHECK_LAUNCH();
        }
    }
}

void dense_set_identity(double* A, int n, int lda, int64_t strideA, int batch, cudaStream_t s) {
    dim3 g(grid_for((int64_t)n * n), batch);
    k_set_identity<<<g, 256, 0, s>>>(A, n, lda, strideA);
    PDG_CHECK_LAUNCH();
}

// X = A^-1 (batched SPD matrices, n a multiple of 64, even row stride); A is overwritten.  A pivot that is not
// positive sets ERR_NOT_SPD in d_err.
void dense_spd_inverse(double* A, int n, int lda, int64_t sA, double* X, int ldx, int64_t sX, int batch, int* d_err,
                       cudaStream_t s) {
    if (n <= 0 || batch <= 0) return;
    allow_digit_smem();
    const int nblk = n / NB;
    const int zb = (int)std::max<int64_t>(1, std::min<int64_t>(batch, kScratchMax / (kSplitBytes * (2 * nblk + 2))));
    const int64_t nP = zb, nC = (int64_t)zb * nblk;
    constexpr int64_t kPivotBytes = sizeof(double) * NB * NB + 4 * (2 * NB + 1);   // P, ex, sx and nu
    Scratch w((size_t)(kSplitBytes * (2 * nP + 2 * nC) + kPivotBytes * nP), s);
    SweepArgs S{};
    S.lda = lda;
    S.nblk = nblk;
    S.sA = sA;
    S.err = d_err;
    S.dP = static_cast<uint4*>(w.p);
    S.dD = S.dP + nP * kBlkVec;
    S.dC = S.dD + nP * kBlkVec;
    S.dW = S.dC + nC * kBlkVec;
    S.P = reinterpret_cast<double*>(S.dW + nC * kBlkVec);
    S.eP = reinterpret_cast<int*>(S.P + nP * NB * NB);
    S.eD = S.eP + nP * NB;
    S.ex = S.eD + nP * NB;
    S.eC = S.ex + nP * NB;
    S.eW = S.eC + nC * NB;
    S.sx = reinterpret_cast<float*>(S.eW + nC * NB);
    S.nu = S.sx + nP * NB;
    for (int z0 = 0; z0 < batch; z0 += zb) {
        const int nz = std::min(zb, batch - z0);
        S.A = A + z0 * sA;
        k_sweep_first<<<nz, kThr, kSmemDig, s>>>(S);
        PDG_CHECK_LAUNCH();
        for (int k = 0; k < nblk; ++k) {
            k_sweep_panel<<<dim3(nz, nblk), kThr, kSmemDig, s>>>(S, k);
            PDG_CHECK_LAUNCH();
            if (nblk > 1) {
                k_sweep_update<<<nz * (nblk * (nblk - 1) / 2), kThr, kSmemDig, s>>>(S, k, nz);
                PDG_CHECK_LAUNCH();
            }
        }
        k_sweep_store<<<dim3(nblk, nblk, nz), kThr, 0, s>>>(S.A, lda, sA, X + z0 * sX, ldx, sX);
        PDG_CHECK_LAUNCH();
    }
}

int64_t dense_scratch_bytes(int n, int batch) {
    const int64_t nblk = (n + NB - 1) / NB;
    const int64_t inv = kSplitBytes * (2 * nblk + 2), prod = 2 * kSplitBytes * nblk * nblk;
    return std::max(inv, std::min<int64_t>(kScratchMax, std::max(inv, prod) * std::max(batch, 1)));
}

int dense_block() { return NB; }

}  // namespace pdg

// ---------------------------------------------------------------- prefactor helpers
namespace pdg {

namespace {

// K by rows (Sec. 7.1) in FP64.  Per element the ten products V_e (gamma_s + gamma_v) g_a . g_b of its corners'
// gradients, from the rest positions; then one thread per free vertex adds its elements' entries in increasing
// (element, corner) order: a fixed order without atomics.  On the host the same sums took 5.4 ms for 50K elements.
__global__ void __launch_bounds__(128) k_tet_stiffness(int n_t, const int4* __restrict__ tets,
                                                       const double* __restrict__ rest, const float* __restrict__ gs,
                                                       const float* __restrict__ gv, double* __restrict__ out) {
    const int t = blockIdx.x * 128 + threadIdx.x;
    if (t >= n_t) return;
    const int4 q = tets[t];
    const double* p[4] = {rest + 3 * (int64_t)q.x, rest + 3 * (int64_t)q.y, rest + 3 * (int64_t)q.z,
                          rest + 3 * (int64_t)q.w};
    double D[3][3];   // columns = edges
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int k = 0; k < 3; ++k) D[c][k] = p[k + 1][c] - p[0][c];
    double g[4][3];   // rows of D^-1 times det
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;   // row k of the adjugate: cross product of the other two edges
        g[k + 1][0] = D[1][k1] * D[2][k2] - D[2][k1] * D[1][k2];
        g[k + 1][1] = D[2][k1] * D[0][k2] - D[0][k1] * D[2][k2];
        g[k + 1][2] = D[0][k1] * D[1][k2] - D[1][k1] * D[0][k2];
    }
    const double det = D[0][0] * g[1][0] + D[1][0] * g[1][1] + D[2][0] * g[1][2];
#pragma unroll
    for (int c = 0; c < 3; ++c) g[0][c] = -(g[1][c] + g[2][c] + g[3][c]);
    // V w / det^2 = w / (6 det)
    const double w = ((double)gs[t] + (double)gv[t]) / (6.0 * det);
    double* o = out + 10 * (int64_t)t;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = a; b < 4; ++b)
            o[a * (7 - a) / 2 + b] = w * (g[a][0] * g[b][0] + g[a][1] * g[b][1] + g[a][2] * g[b][2]);
}

__global__ void __launch_bounds__(128) k_assemble_rows(int n_free, const int* __restrict__ inc_ptr,
                                                       const int* __restrict__ inc, const int4* __restrict__ tets,
                                                       const double* __restrict__ ke, const double* __restrict__ mass,
                                                       double inv_h2, const int* __restrict__ ptr,
                                                       const int* __restrict__ col, double* __restrict__ val,
                                                       const int* __restrict__ fptr, const int* __restrict__ fcol,
                                                       double* __restrict__ fval, float* __restrict__ fval32,
                                                       float* __restrict__ mh2, int* __restrict__ err) {
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i >= n_free) return;
    const int lo = ptr[i], hi = ptr[i + 1], flo = fptr[i], fhi = fptr[i + 1];
    for (int k = lo; k < hi; ++k) val[k] = 0.0;
    for (int k = flo; k < fhi; ++k) fval[k] = 0.0;
    bool lost = false;
    for (int n = inc_ptr[i]; n < inc_ptr[i + 1]; ++n) {
        const int t = inc[n] >> 2, a = inc[n] & 3;
        const int4 q4 = tets[t];
        const int q[4] = {q4.x, q4.y, q4.z, q4.w};
        const double* e = ke + 10 * (int64_t)t;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int x = min(a, b), y = max(a, b);
            const double v = e[x * (7 - x) / 2 + y];
            if (q[b] < n_free) {
                const int k = find_col(col, lo, hi, q[b]);
                if (k >= 0) val[k] += v;
                else lost = true;
            } else {
                const int k = find_col(fcol, flo, fhi, q[b] - n_free);
                if (k >= 0) fval[k] += v;
                else lost = true;
            }
        }
    }
    const int d = find_col(col, lo, hi, i);
    const double m = mass[i] * inv_h2;
    if (d >= 0) val[d] += m;
    else lost = true;
    if (lost) atomicOr(err, ERR_NO_PLACE);
    mh2[i] = (float)m;
    for (int k = flo; k < fhi; ++k) fval32[k] = (float)fval[k];
}

// Dense K_ii (identity beyond the domain's rows) and K_ib of every domain from the rows of K (both zeroed before):
// dom = (first internal vertex, count, offset and count of the boundary list) of a domain.  An entry without a place
// sets ERR_NO_PLACE.
__global__ void __launch_bounds__(128) k_domain_blocks(const int4* __restrict__ dom, const int* __restrict__ bnd,
                                                       int n_int, const int* __restrict__ ptr,
                                                       const int* __restrict__ col, const double* __restrict__ val,
                                                       double* __restrict__ Kii, int NI, double* __restrict__ Kib,
                                                       int NBp, int* __restrict__ err) {
    const int r = blockIdx.x * 128 + threadIdx.x;
    if (r >= NI) return;
    const int4 D = dom[blockIdx.y];
    double* ii = Kii + ((int64_t)blockIdx.y * NI + r) * NI;
    if (r >= D.y) {
        ii[r] = 1.0;
        return;
    }
    double* ib = Kib + ((int64_t)blockIdx.y * NI + r) * NBp;
    for (int k = ptr[D.x + r]; k < ptr[D.x + r + 1]; ++k) {
        const int p = domain_place(col[k], D.x, D.y, bnd, D.z, D.w, n_int);
        if (p < 0) atomicOr(err, ERR_NO_PLACE);
        else if (p < D.y) ii[p] = val[k];
        else ib[p - D.y] = val[k];
    }
}

// S[j, c] = K entries between interface vertices
__global__ void __launch_bounds__(128) k_interface_rows(int n_int, int n_B, const int* __restrict__ ptr,
                                                        const int* __restrict__ col, const double* __restrict__ val,
                                                        double* __restrict__ S, int ld) {
    const int j = blockIdx.x * 128 + threadIdx.x;
    if (j >= n_B) return;
    for (int k = ptr[n_int + j]; k < ptr[n_int + j + 1]; ++k)
        if (col[k] >= n_int) S[(int64_t)j * ld + col[k] - n_int] = val[k];
}

// S[bidx[a], bidx[b]] += Sd[a, b]; one launch per domain keeps the sum order fixed
__global__ void k_add_block(double* __restrict__ S, int ldS, const double* __restrict__ Sd, int ldSd,
                            const int* __restrict__ bidx, int nb) {
    const int64_t n = (int64_t)nb * nb;
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n; l += (int64_t)gridDim.x * blockDim.x) {
        int a = (int)(l / nb), b = (int)(l % nb);
        S[(int64_t)bidx[a] * ldS + bidx[b]] += Sd[(int64_t)a * ldSd + b];
    }
}

__device__ __forceinline__ float round_tf32(float x) {
    uint32_t y;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(y) : "f"(x));
    return __uint_as_float(y);
}

// dst[r, c] = src[r, c] (or src[c, r] when transposed), converted to the storage precision
__global__ void k_cast_block(const double* __restrict__ src, int lds, int rows, int cols, int transpose, int prec,
                             float* __restrict__ d32, __nv_bfloat16* __restrict__ d16, int64_t off, int ldd) {
    const int64_t n = (int64_t)rows * cols;
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n; l += (int64_t)gridDim.x * blockDim.x) {
        int r = (int)(l / cols), c = (int)(l % cols);
        double v = transpose ? src[(int64_t)c * lds + r] : src[(int64_t)r * lds + c];
        int64_t o = off + (int64_t)r * ldd + c;
        if (prec == PD_PREC_BF16) d16[o] = __double2bfloat16(v);
        else if (prec == PD_PREC_TF32) d32[o] = round_tf32((float)v);
        else d32[o] = (float)v;
    }
}

// the same cast into the tiled axpy layout (ax_tile_width), chunks of CW outputs
__global__ void k_cast_tiled(const double* __restrict__ src, int lds, int rows, int cols, int transpose, int prec,
                             float* __restrict__ d32, __nv_bfloat16* __restrict__ d16, int64_t off, int CW, int VN) {
    const int64_t n = (int64_t)rows * cols;
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n; l += (int64_t)gridDim.x * blockDim.x) {
        int r = (int)(l / cols), c = (int)(l % cols);
        double v = transpose ? src[(int64_t)c * lds + r] : src[(int64_t)r * lds + c];
        const int o0 = c / CW * CW;
        const int64_t o = off + (int64_t)o0 * rows + (int64_t)r * ax_tile_width(cols, o0, CW, VN) + (c - o0);
        if (prec == PD_PREC_BF16) d16[o] = __double2bfloat16(v);
        else if (prec == PD_PREC_TF32) d32[o] = round_tf32((float)v);
        else d32[o] = (float)v;
    }
}

// BF16 tile in the tensor-core fragment order (rows padded to 16; see k_axpy_mma):
// element (r, c) of chunk o0 = c - c % CW lands in its 16 x 8 block at the
// lane and register the mma B operand reads it from.
__global__ void k_cast_frag16(const double* __restrict__ src, int lds, int rows, int cols, int transpose,
                              __nv_bfloat16* __restrict__ d16, int64_t off, int CW) {
    const int64_t n = (int64_t)rows * cols;
    const int kp = (rows + 15) & ~15;
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n; l += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(l / cols), c = (int)(l % cols);
        const double v = transpose ? src[(int64_t)c * lds + r] : src[(int64_t)r * lds + c];
        const int o0 = c / CW * CW;
        const int w = ax_tile_width(cols, o0, CW, 8);
        const int kb = r >> 4, kk = r & 15, cc = c - o0, nb = cc >> 3, nn = cc & 7;
        const int q = (kk & 7) >> 1, j = (kk & 1) + ((kk >> 3) << 1);
        d16[off + (int64_t)o0 * kp + ((int64_t)kb * (w >> 3) + nb) * 128 + (4 * nn + q) * 4 + j] =
            __double2bfloat16(v);
    }
}

// TF32 tile (rows padded to 8) in the register order of the B operand of
// mma.m16n8k8 (tf32): 8 x 8 blocks, lane 4 n + (k mod 4) holding rows k mod 4
// and k mod 4 + 4 of output n; values rounded to TF32.
__global__ void k_cast_frag32(const double* __restrict__ src, int lds, int rows, int cols, int transpose,
                              float* __restrict__ d32, int64_t off, int CW) {
    const int64_t n = (int64_t)rows * cols;
    const int kp = (rows + 7) & ~7;
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n; l += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(l / cols), c = (int)(l % cols);
        const double v = transpose ? src[(int64_t)c * lds + r] : src[(int64_t)r * lds + c];
        const int o0 = c / CW * CW;
        const int w = ax_tile_width(cols, o0, CW, 8);
        const int kb = r >> 3, kk = r & 7, cc = c - o0, nb = cc >> 3, nn = cc & 7;
        d32[off + (int64_t)o0 * kp + ((int64_t)kb * (w >> 3) + nb) * 64 + (4 * nn + (kk & 3)) * 2 + (kk >> 2)] =
            round_tf32((float)v);
    }
}

// BF16 row-form block in the tensor-core fragment order (rows and columns
// padded to 16, see k_rowdot_mma): element (r, c) lands in 16 x 16 block
// (r / 16, c / 16) at the lane and register of the mma A operand.
__global__ void k_cast_rowfrag16(const double* __restrict__ src, int lds, int rows, int cols, int transpose,
                                 __nv_bfloat16* __restrict__ d16, int64_t off, int Kp) {
    const int64_t n = (int64_t)rows * cols;
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n; l += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(l / cols), c = (int)(l % cols);
        const double v = transpose ? src[(int64_t)c * lds + r] : src[(int64_t)r * lds + c];
        const int rb = r >> 4, kb = c >> 4, rr = r & 15, kk = c & 15;
        const int g = rr & 7, rhi = rr >> 3, q = (kk & 7) >> 1, j = kk & 1, khi = kk >> 3;
        d16[off + ((int64_t)rb * (Kp >> 4) + kb) * 256 + (4 * g + q) * 8 + (rhi + 2 * khi) * 2 + j] =
            __double2bfloat16(v);
    }
}

// dst[i][k] = S[r0 + i][cols ? c0 + cols[k] : c0 + k]
__global__ void k_copy_block_idx(const double* __restrict__ S, int ldS, int r0, int nr, const int* __restrict__ cols,
                                 int c0, int nc, double* __restrict__ dst, int ldd) {
    const int64_t n = (int64_t)nr * nc;
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n; l += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(l / nc), k = (int)(l % nc);
        const int c = c0 + (cols ? cols[k] : k);
        dst[(int64_t)i * ldd + k] = S[(int64_t)(r0 + i) * ldS + c];
    }
}

inline int grid_of(int64_t n) {
    int64_t b = (n + 255) / 256;
    return (int)(b < 65535 ? (b > 0 ? b : 1) : 65535);
}

}  // namespace

// K (and K_fp, m / dt^2) of the mesh's materials for time step dt, on the device.
void launch_assemble_K(pd_mesh* m, double inv_h2, cudaStream_t s) {
    if (m->n_free <= 0) return;
    DBuf<double> ke, fval;
    ke.alloc(10 * (size_t)m->n_t);
    fval.alloc(m->Kfp_col.size());
    k_tet_stiffness<<<(m->n_t + 127) / 128, 128, 0, s>>>(m->n_t, m->d_tets.p, m->d_rest64.p, m->d_gamma.p,
                                                        m->d_gamma.p + m->n_t, ke.p);
    PDG_CHECK_LAUNCH();
    k_assemble_rows<<<(m->n_free + 127) / 128, 128, 0, s>>>(
        m->n_free, m->d_inc_ptr.p, m->d_inc.p, m->d_tets.p, ke.p, m->d_mass64.p, inv_h2, m->d_K_ptr.p, m->d_K_col.p,
        m->d_K_val.p, m->d_kfp_ptr.p, m->d_kfp_col.p, fval.p, m->d_kfp_val.p, m->d_mh2.p, m->d_err.p);
    PDG_CHECK_LAUNCH();   // (the temporaries' release is stream-ordered, or waits for the device)
}

void launch_domain_blocks(const pd_mesh* m, const int4* dom, const int* bnd, double* Kii, int NI, double* Kib, int NBp,
                          cudaStream_t s) {
    if (m->n_dom <= 0) return;
    k_domain_blocks<<<dim3((NI + 127) / 128, m->n_dom), 128, 0, s>>>(dom, bnd, m->n_int, m->d_K_ptr.p, m->d_K_col.p,
                                                                    m->d_K_val.p, Kii, NI, Kib, NBp, m->d_err.p);
    PDG_CHECK_LAUNCH();
}

void launch_interface_rows(const pd_mesh* m, double* S, int ld, cudaStream_t s) {
    if (m->n_B <= 0) return;
    k_interface_rows<<<(m->n_B + 127) / 128, 128, 0, s>>>(m->n_int, m->n_B, m->d_K_ptr.p, m->d_K_col.p, m->d_K_val.p, S,
                                                        ld);
    PDG_CHECK_LAUNCH();
}

void launch_prefactor_add_block(double* S, int ldS, const double* Sd, int ldSd, const int* bidx, int nb,
                                cudaStream_t s) {
    if (nb <= 0) return;
    k_add_block<<<grid_of((int64_t)nb * nb), 256, 0, s>>>(S, ldS, Sd, ldSd, bidx, nb);
    PDG_CHECK_LAUNCH();
}

void launch_copy_block_idx(const double* S, int ldS, int r0, int nr, const int* cols, int c0, int nc, double* dst,
                           int ldd, cudaStream_t s) {
    if (nr <= 0 || nc <= 0) return;
    k_copy_block_idx<<<grid_of((int64_t)nr * nc), 256, 0, s>>>(S, ldS, r0, nr, cols, c0, nc, dst, ldd);
    PDG_CHECK_LAUNCH();
}

void launch_cast_block(const double* src, int lds, int rows, int cols, int transpose, int prec, float* dst32,
                       __nv_bfloat16* dst16, int64_t dst_off, int ldd, cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return;
    k_cast_block<<<grid_of((int64_t)rows * cols), 256, 0, s>>>(src, lds, rows, cols, transpose, prec, dst32, dst16,
                                                                dst_off, ldd);
    PDG_CHECK_LAUNCH();
}

void launch_cast_frag32(const double* src, int lds, int rows, int cols, int transpose, float* dst32,
                        int64_t dst_off, int CW, cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return;
    k_cast_frag32<<<grid_of((int64_t)rows * cols), 256, 0, s>>>(src, lds, rows, cols, transpose, dst32, dst_off, CW);
    PDG_CHECK_LAUNCH();
}

void launch_cast_rowfrag16(const double* src, int lds, int rows, int cols, int transpose, __nv_bfloat16* dst16,
                           int64_t dst_off, int Kp, cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return;
    k_cast_rowfrag16<<<grid_of((int64_t)rows * cols), 256, 0, s>>>(src, lds, rows, cols, transpose, dst16, dst_off,
                                                                    Kp);
    PDG_CHECK_LAUNCH();
}

void launch_cast_frag16(const double* src, int lds, int rows, int cols, int transpose, __nv_bfloat16* dst16,
                        int64_t dst_off, int CW, cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return;
    k_cast_frag16<<<grid_of((int64_t)rows * cols), 256, 0, s>>>(src, lds, rows, cols, transpose, dst16, dst_off, CW);
    PDG_CHECK_LAUNCH();
}

void launch_cast_tiled(const double* src, int lds, int rows, int cols, int transpose, int prec, float* dst32,
                       __nv_bfloat16* dst16, int64_t dst_off, int CW, int VN, cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return;
    k_cast_tiled<<<grid_of((int64_t)rows * cols), 256, 0, s>>>(src, lds, rows, cols, transpose, prec, dst32, dst16,
                                                                dst_off, CW, VN);
    PDG_CHECK_LAUNCH();
}

}  // namespace pdg
