// Stage (b), split precision: the contraction of Eq. chi_mat as an Ozaki-style
// error-free slice expansion on the BF16 tensor cores (tcgen05, accumulators in TMEM).
//
// With A[p][G] = s_p M[p][G], s_p = sqrt(-Delta_p) (Delta < 0), chi = -A^H A.  In real
// form Z = [Re A | Im A] interleaved by column (j = 2G + {0: Re, 1: Im}) and
// chi_GG' = -(C[2G][2G'] + C[2G+1][2G'+1]) - i (C[2G][2G'+1] - C[2G+1][2G']),  C = Z^T Z.
//
// Splitting (per chunk of pairs and per complex column G, exponent E_G with
// max_p |Z[p][2G+c]| < 2^(E_G - 1)):
//     Z[p][j] = 2^(E_G + 1) sum_{i=1..s} 2^(-9 i) z_i[p][j],   z_i integers,
// |z_1| <= 128 and |z_i| <= 256 otherwise, so the slices are exact in BF16.  Products of slices
// are exact, and so is the FP32 sum of a slice group
//     C_t = sum_{i+k=t} z_i^T z_k     (t = 2 .. s+1, triangular truncation)
// while it stays below 2^24.  The groups are therefore summed in K-segments (oz_segment): 512 pairs
// for t = 2 (|z_1 z_1| <= 2^14, so a segment's sum is at most 2^23 and the sum of two of them that
// makes an entry of chi is exact too), 256 for t = 3 (2 products, 2^24) and for t = 4 (2^25 if
// every digit took its largest value with one sign; the rounding then lies 2^-36 below the leading
// group), longer ones for t >= 5, whose rounding lies below 2^-27 2^-24 of the result.  The
// epilogue adds the segments, times 2^(-9 (t - 2)), in two-float arithmetic in registers and adds
//     chi += -2^(E_G + E_G' - 16) (hi + lo)
// once per tile in FP64, with atomic adds so that the chunks (pair segments) of one chi block may
// run concurrently in one launch (one chunk's sums are the same bits in every run).  FP64 is kept for
// Delta, the scaling, the accumulation across chunks and the symmetrisation.
//
// The FP64 contraction of computed pair elements takes the same route with seven slices (62 bits of
// each column's largest entry, where a double keeps 53 of each entry) and without any FP32 sum beyond
// a segment: the segments' sums, whole numbers, are added as 64-bit integers over a K block of 1024
// pairs, and the blocks in FP64 (OzProd::F64 below).
#include "internal.h"
#include "ptx.cuh"
#include "fft_tf.cuh"
#include "oz_digits.cuh"
#include <cuda_bf16.h>
#include <algorithm>

namespace gw {

// Slices for a requested accuracy of 6 nslices bits (the ABI's nslices, 3..8): the fewest 9-bit
// slices whose dropped products (i + k > s + 1) lie no higher.  With six-bit digits the dropped
// products come to 2^(-6 nslices - 3.6) sqrt(nslices - 1) of the operands' scales, with these to
// 2^(-9 s - 1.6) sqrt(s - 1): 3, 3, 4, 5, 5, 6 slices for nslices = 3 .. 8.
int oz_slices(int nslices) { return nslices <= 4 ? 3 : nslices == 5 ? 4 : nslices <= 7 ? 5 : 6; }

constexpr int kOzBM = 128, kOzBK = 64; // rows of A (and of B) per CTA of a pair; K entries per ring stage
constexpr int kOzThreads = 384;        // a warpgroup with the TMA and MMA warps, two of epilogue warps
constexpr int kOzNoColumn = -400;      // exponent of an all-zero column
constexpr int kOzMaxExpo = 390;        // exponents that the FP64 contraction's scaling takes, +-
constexpr int kOzF64Slices = 7;

// K runs in blocks of kOzKBlock K-steps (of 64 entries), every slice group over one block before
// the next, so that a slice comes from DRAM once per block and from L2 for its other products.
// (On 48^3 and 72^3 chunks, on N_G = 6000 self-energy products and on 2000 x 2000 products, 8, 16 and
// 32 K-steps run within 3 % of one another.)
constexpr int kOzKBlock = 16;
// K-steps that slice group t sums in FP32 before the epilogue takes the sum (bounds at the top of
// this file)
// (F64: every sum whose rounding would show is exact whatever the digits.  A pair adds at most 2^14 to t = 2,
// 2^16 to t = 3, 2^17 to t = 4, 3 2^16 to t = 5 and 2^18 to t = 6, so 512, 256, 128, 64 and 64 pairs stay
// within 2^24.  t = 7 (5 2^16) over 128 pairs and t = 8 (6 2^16) over 1024 may be rounded by up to 4 and 32 in
// each of their 48 and 448 MMA steps: 2^-51 and 2^-54 of a pair's largest product 2^14 at most, and only where
// the digits of those slices have one sign throughout.)
template <bool F64>
__device__ __forceinline__ int oz_segment(int t)
{
    if (F64) return t == 2 ? 8 : t == 3 ? 4 : t == 4 || t == 7 ? 2 : t == 8 ? kOzKBlock : 1;
    return t == 2 ? 8 : t <= 4 ? 4 : kOzKBlock;
}

// ------------------------------------------------------------------ split, step 1: column exponents
// E[g] = max_p ilogb(max(|Re A|, |Im A|)) + 2 over the chunk, A = s_p M[p][g].
__global__ void oz_sqrt_kernel(const double *__restrict__ delta, int64_t n, double *__restrict__ sp)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) sp[i] = sqrt(-delta[i]);
}

// GUARD: sets *guard where an entry is not finite or a column's scale is out of range (FP64
// contraction: the DMMA kernel then takes the chunk).
// SCALE = false: of M itself (the column operand of a general product).
template <bool GUARD, bool SCALE>
__global__ void oz_colexp_kernel(const double2 *__restrict__ M, int64_t P, int ng, const double *__restrict__ sp,
                                 int *__restrict__ E, int *guard)
{
    __shared__ int red[8][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int g = blockIdx.x * 32 + lane;
    int e = kOzNoColumn;
    if (g < ng) {
        for (int64_t p = (int64_t)blockIdx.y * 8 + wid; p < P; p += (int64_t)gridDim.y * 8) {
            const double2 m = M[p * ng + g];
            const double b = oz_bits_d(oz_absmax_bits(m.x, m.y)), a = SCALE ? b * sp[p] : b;
            e = max(e, oz_expo_pos(a, kOzNoColumn));
            if constexpr (GUARD)
                if ((oz_dbits(a) & 0x7fffffffffffffffull) >= 0x7ff0000000000000ull || e > kOzMaxExpo) *guard = 1;
        }
    }
    red[wid][lane] = e;
    __syncthreads();
    if (wid == 0 && g < ng) {
        for (int w = 1; w < 8; ++w) e = max(e, red[w][lane]);
        atomicMax(E + g, e);
    }
}

__global__ void oz_fill_kernel(int *E, int n, int v)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) E[i] = v;
}

// ------------------------------------------------------------------ split, step 2: slices
// A block forms the slices of a 64-pair x 32-column tile of M and stores them straight into
// Z[i][j][p] (j = 2 g + {Re, Im}, K-major rows of kpad pairs).  Thread roles: warp w takes tile
// rows 32 (w & 1) .. + 31 (lane = row: column g = row / 2, component row & 1) and pairs
// 16 (w >> 1) .. + 15, so a warp reads 32 consecutive doubles of M per pair, and each thread
// writes each slice's 16 digits of its row as one aligned 32-byte segment (two 16-byte stores).
struct OzTileThread {
    int row, gl, c, pl0;
};
__device__ __forceinline__ OzTileThread oz_tile_thread()
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    OzTileThread t;
    t.row = 32 * (w & 1) + lane;
    t.gl = t.row >> 1;
    t.c = t.row & 1;
    t.pl0 = 16 * (w >> 1);
    return t;
}

// the s slices of the 16 biased integers nb[t] = N_t + bias (consecutive pairs of one row) into
// out + i plane + [0, 16)
__device__ __forceinline__ void oz_store_row_digits(const long long nb[16], int s, __nv_bfloat16 *out, int64_t plane)
{
    for (int i = 0; i < s; ++i) {
        uint32_t w[8];
#pragma unroll
        for (int t = 0; t < 16; t += 2) {
            uint16_t d[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const long long v = nb[t + u];
                d[u] = i == 0 ? oz_small_bf16((int)(v >> (kOzBeta * (s - 1))))
                              : oz_small_bf16((int)((v >> (kOzBeta * (s - 1 - i))) & 511) - 256);
            }
            w[t >> 1] = (uint32_t)d[0] | ((uint32_t)d[1] << 16);
        }
        uint4 *o = (uint4 *)(out + i * plane);
        o[0] = make_uint4(w[0], w[1], w[2], w[3]);
        o[1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
}

// Z[i][j][p] (bf16, K-major rows of length kpad) for a 64-pair x 32-column block.
// Five blocks per SM (48 registers, a 24-byte spill) keep more of the 16 loads per thread in flight
// than the four the unconstrained build allows: the split preparation of a 48^3 q-point (16 chunks)
// takes 5.04 against 5.32 ms (six blocks, 40 registers and a 60-byte spill: 5.17 ms).
// GUARD: as in oz_colexp_kernel, for a column that is not zero but below the exponent range.
template <bool GUARD, bool SCALE>
__global__ void __launch_bounds__(256, 5) oz_slice_kernel(const double2 *__restrict__ M, int64_t P, int ng,
                                                       const double *__restrict__ spv, const int *__restrict__ E,
                                                       int s, int64_t kpad, __nv_bfloat16 *__restrict__ Z, int *guard)
{
    const int64_t p0 = (int64_t)blockIdx.y * 64;
    const OzTileThread tt = oz_tile_thread();
    const int g = blockIdx.x * 32 + tt.gl;
    if (g >= ng) return;
    // N = round(a 2^(9 s - 1 - E)) and its balanced base-512 digits, in integer arithmetic
    const int sh = oz_frac_bits(s) - E[g];
    const double *Md = (const double *)M;
    const long long bias = oz_digit_bias<kOzBeta>(s);
    long long nb[16];
#pragma unroll
    for (int t = 0; t < 16; ++t) {
        const int64_t p = p0 + tt.pl0 + t;
        const double b = p < P ? Md[2 * (p * ng + g) + tt.c] : 0.0, a = SCALE ? (p < P ? b * spv[p] : 0.0) : b;
        if constexpr (GUARD)
            if (E[g] < -kOzMaxExpo && a != 0.0) *guard = 1;
        nb[t] = oz_round_scaled(a, sh) + bias;
    }
    const int64_t j = 2 * (int64_t)g + tt.c;
    oz_store_row_digits(nb, s, Z + j * kpad + p0 + tt.pl0, 2 * (int64_t)ng * kpad);
}

// ------------------------------------------------------------------ split for several frequencies
// The scale s_p(w) = sqrt(-Delta_p(w)) is the only thing that changes with the frequency, so a
// group of up to kOzGroupW frequencies shares one read of M: exponents E[w][g] in one pass,
// slices Z_w in another (each frequency's slices at Z + w zstride), the digits as in
// oz_slice_kernel.
constexpr int kOzGroupW = 8;

__global__ void __launch_bounds__(256) oz_colexp_multi_kernel(const double2 *__restrict__ M, int64_t P, int ng,
                                                              const double *__restrict__ sp, int64_t dstride,
                                                              int nw, int *__restrict__ E)
{
    __shared__ int red[8][32][kOzGroupW];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int g = blockIdx.x * 32 + lane;
    int e[kOzGroupW];
#pragma unroll
    for (int w = 0; w < kOzGroupW; ++w) e[w] = kOzNoColumn;
    if (g < ng) {
        for (int64_t p = (int64_t)blockIdx.y * 8 + wid; p < P; p += (int64_t)gridDim.y * 8) {
            const double2 m = M[p * ng + g];
            const double a0 = oz_bits_d(oz_absmax_bits(m.x, m.y));
#pragma unroll
            for (int w = 0; w < kOzGroupW; ++w)
                if (w < nw) {
                    const double a = a0 * sp[(int64_t)w * dstride + p];
                    e[w] = max(e[w], oz_expo_pos(a, kOzNoColumn));
                }
        }
    }
#pragma unroll
    for (int w = 0; w < kOzGroupW; ++w) red[wid][lane][w] = e[w];
    __syncthreads();
    if (wid == 0 && g < ng) {
#pragma unroll
        for (int w = 0; w < kOzGroupW; ++w)
            if (w < nw) {
                int v = red[0][lane][w];
                for (int k = 1; k < 8; ++k) v = max(v, red[k][lane][w]);
                atomicMax(E + (int64_t)w * ng + g, v);
            }
    }
}

__global__ void __launch_bounds__(256) oz_slice_multi_kernel(const double2 *__restrict__ M, int64_t P, int ng,
                                                             const double *__restrict__ spv, int64_t dstride, int nw,
                                                             const int *__restrict__ E, int s, int64_t kpad,
                                                             int64_t zstride, __nv_bfloat16 *__restrict__ Z)
{
    const int64_t p0 = (int64_t)blockIdx.y * 64;
    const OzTileThread tt = oz_tile_thread();
    const int g = blockIdx.x * 32 + tt.gl;
    if (g >= ng) return;
    const long long bias = oz_digit_bias<kOzBeta>(s);
    // the thread's 16 entries of the block's tile of M, read once for every frequency
    const double *Md = (const double *)M;
    double m[16];
#pragma unroll
    for (int t = 0; t < 16; ++t) {
        const int64_t p = p0 + tt.pl0 + t;
        m[t] = p < P ? Md[2 * (p * ng + g) + tt.c] : 0.0;
    }
    const int64_t j = 2 * (int64_t)g + tt.c;
    for (int w = 0; w < nw; ++w) {
        const int sh = oz_frac_bits(s) - E[(int64_t)w * ng + g];
        long long nb[16];
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            const int64_t p = p0 + tt.pl0 + t;
            const double a = p < P ? m[t] * spv[(int64_t)w * dstride + p] : 0.0;
            nb[t] = oz_round_scaled(a, sh) + bias;
        }
        oz_store_row_digits(nb, s, Z + w * zstride + j * kpad + p0 + tt.pl0, 2 * (int64_t)ng * kpad);
    }
}

// ------------------------------------------------------------------ general product: slices
// Y = A B with A split by rows and B by columns: x = 2^(E+1) sum_{i=1..s} 2^(-9 i) z_i, the same
// balanced base-512 digits as oz_slice_kernel, in the same layout (real and imaginary parts in
// rows of their own, K the complex inner index), so that with C the real product of the 2 rows
// slice rows by the 2 nout slice columns
//     Re Y[r][c] = C[2r][2c] - C[2r+1][2c+1],   Im Y[r][c] = C[2r][2c+1] + C[2r+1][2c],
// and E = max(ilogb) + 2 over a row of A or a
// column of B (both parts of a complex entry).
// exponent of a complex entry: ilogb(max(|Re|, |Im|)) + 2
__device__ __forceinline__ int oz_expo(double2 x)
{
    return oz_expo_bits(oz_absmax_bits(x.x, x.y), kOzNoColumn);
}

__device__ __forceinline__ int oz_block_max(int e, int *red)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    if (lane == 0) red[wid] = e;
    __syncthreads();
    if (threadIdx.x < 32) {
        e = threadIdx.x < (int)(blockDim.x >> 5) ? red[threadIdx.x] : kOzNoColumn;
        for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
        if (threadIdx.x == 0) red[0] = e;
    }
    __syncthreads();
    return red[0];
}

// digits of two consecutive entries x0, x1 of a row: 32-bit stores at out + i plane32
__device__ __forceinline__ void oz_store_pair(double x0, double x1, int sh, int s, long long bias, uint32_t *out,
                                              int64_t plane32)
{
    const long long n0 = oz_round_scaled(x0, sh) + bias, n1 = oz_round_scaled(x1, sh) + bias;
    for (int k = 0; k < s - 1; ++k)
        out[(int64_t)(s - 1 - k) * plane32] =
            (uint32_t)oz_small_bf16((int)((n0 >> (kOzBeta * k)) & 511) - 256) |
            (uint32_t)oz_small_bf16((int)((n1 >> (kOzBeta * k)) & 511) - 256) << 16;
    out[0] = (uint32_t)oz_small_bf16((int)(n0 >> (kOzBeta * (s - 1)))) |
             (uint32_t)oz_small_bf16((int)(n1 >> (kOzBeta * (s - 1)))) << 16;
}

// One block per complex row p of A: E[p], then the slice rows Z[i][2 p + c][g] (c = 0 the real,
// c = 1 the imaginary parts), zero for g >= ka.  A[p][g] is read at A[p sr + g sk] (sr = ka, sk = 1
// for row-major A [rows][ka]; sr = 1, sk = nout for the columns of a row-major B [ka][nout]).
// CONJ: of conj(A).
template <bool CONJ>
__global__ void __launch_bounds__(256) oz_split_kernel(const double2 *__restrict__ A, int64_t rows, int ka,
                                                       int64_t sr, int64_t sk, int s, int64_t kpad,
                                                       uint16_t *__restrict__ Z, int *__restrict__ E)
{
    __shared__ int red[8];
    const int64_t p = blockIdx.x;
    const double2 *a = A + p * sr;
    int e = kOzNoColumn;
    for (int g = threadIdx.x; g < ka; g += blockDim.x) e = max(e, oz_expo(a[g * sk]));
    e = oz_block_max(e, red);
    if (threadIdx.x == 0) E[p] = e;
    const int sh = oz_frac_bits(s) - e;
    const long long bias = oz_digit_bias<kOzBeta>(s);
    const int64_t plane32 = rows * kpad; // 2 rows kpad entries of 16 bits
    uint32_t *z0 = (uint32_t *)(Z + 2 * p * kpad), *z1 = (uint32_t *)(Z + (2 * p + 1) * kpad);
    for (int64_t k = threadIdx.x; 2 * k < kpad; k += blockDim.x) {
        const int64_t g = 2 * k;
        const double2 zero = make_double2(0.0, 0.0);
        const double2 x = g < ka ? a[g * sk] : zero, y = g + 1 < ka ? a[(g + 1) * sk] : zero;
        oz_store_pair(x.x, y.x, sh, s, bias, z0 + k, plane32);
        oz_store_pair(CONJ ? -x.y : x.y, CONJ ? -y.y : y.y, sh, s, bias, z1 + k, plane32);
    }
}

// ------------------------------------------------------------------ plasmon-pole prep. step, split
// The A operand of X^T = P^T conj(M_n)^T straight from the pole parameters, P never stored:
// P[g][c] = A[g][c] / (d - sgn wt[g][c]) with A = v Omega^2 / (2 wt) (gpp_setup_tf_kernel),
// d = E - E_n, sgn = -1 for an occupied band n and +1 for an empty one.  At / Wt hold A and wt
// transposed ([c][g]) in two-float form, so that row c of P^T is one contiguous row and the
// pole runs on the FP32 pipes.  One block per row c and up to kGppMaxE energies per launch,
// sharing each read of the row:
//  * pass 1, the row exponent per energy, from P in FP32 after the exact two-float subtraction
//    x = d - sgn wt (relative error ~2^-22 however close the pole), padded by 2^-10 so that the
//    exponent is never below the one of the exact maximum;
//  * pass 2, P = A conj(x) / |x|^2 in two-float arithmetic (the reciprocal by one Newton step,
//    relative error near 2^-46, below the 2^-43 five slices keep), then the balanced base-512
//    digits of N = round(P 2^sh) in the layout of oz_split_kernel.  N is formed without 64-bit steps: v = hi 2^sh splits in FP32 into t 2^S + r, both
//    exact (|r| <= 2^(S-1), S two digits, three for six slices), and the low part
//    L = rint(r) + rint(lo 2^sh) (below 2^20, 2^29 for six slices) gives the S / 9 lowest digits
//    and a carry into t, which holds the others, in 32-bit integers.  N differs from
//    round((hi + lo) 2^sh) by one unit of the last digit at most.
__device__ __forceinline__ tf tf_recip(tf d)
{
    const float r0 = __frcp_rn(d.hi);
    const tf p = tf_mul(d, tf{r0, 0.0f});
    const tf e = tf_sub(tf{1.0f, 0.0f}, p); // 1 - d r0, of order 2^-23
    return tf_fast2sum(r0, __fmul_rn(r0, e.hi));
}

__device__ __forceinline__ tcx gpp_pole_tf(float4 a4, float4 w4, tf d, float sgn)
{
    const tcx a{{a4.x, a4.y}, {a4.z, a4.w}};
    // x = d - sgn wt (sgn = +-1: exact negation)
    const tcx x{tf_sub(d, tf{sgn * w4.x, sgn * w4.y}), tf{-sgn * w4.z, -sgn * w4.w}};
    const tf den = tf_add(tf_mul(x.re, x.re), tf_mul(x.im, x.im));
    return tc_rmul(tc_mulc(x, a), tf_recip(den)); // conj(x) a / |x|^2
}

// max(|Re P|, |Im P|) in FP32 from the exact two-float x
__device__ __forceinline__ float gpp_pole_mag(float4 a4, float4 w4, tf d, float sgn)
{
    const float xr = tf_sub(d, tf{sgn * w4.x, sgn * w4.y}).hi, xi = -sgn * w4.z;
    const float r = __frcp_rn(__fmaf_rn(xr, xr, __fmul_rn(xi, xi)));
    const float pr = __fmaf_rn(a4.x, xr, __fmul_rn(a4.z, xi)), pi = __fmaf_rn(a4.z, xr, -__fmul_rn(a4.x, xi));
    return fmaxf(fabsf(pr), fabsf(pi)) * r;
}

__device__ __forceinline__ int tf_expo(float a)
{
    if (!(a > 0.0f)) return kOzNoColumn;
    const int be = (int)((__float_as_uint(a) >> 23) & 0xff);
    return (be == 0 ? -127 : be - 127) + 2;
}

__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi)
{
    return (__float_as_uint(lo) >> 16) | (__float_as_uint(hi) & 0xffff0000u);
}

// N = round(v 2^sh) as L + T 2^(9 low), 2^sh = s1 s2
__device__ __forceinline__ void tf_fixed(tf v, float s1, float s2, int low, int &L, int &T)
{
    const float vh = __fmul_rn(__fmul_rn(v.hi, s1), s2);
    const float t = rintf(__fmul_rn(vh, low == 2 ? 0x1p-18f : 0x1p-27f));
    const float r = __fmaf_rn(low == 2 ? -0x1p18f : -0x1p27f, t, vh);
    L = __float2int_rn(r) + __float2int_rn(__fmul_rn(__fmul_rn(v.lo, s1), s2));
    T = __float2int_rn(t);
}

__device__ __forceinline__ uint32_t oz_digit_pair(int a, int b)
{
    return bf16_pair(__int_as_float(0x4B400000 + a) - 12582912.0f, __int_as_float(0x4B400000 + b) - 12582912.0f);
}

// Digits of round(v 2^sh) of two consecutive entries of a row (2^sh = s1 s2), stored as they come:
// slice i at zr + i plane32.
__device__ __forceinline__ void tf_digits_store(tf v0, tf v1, float s1, float s2, int s, uint32_t *zr, int64_t plane32)
{
    const int low = s <= 5 ? 2 : 3;
    int L0, T0, L1, T1;
    tf_fixed(v0, s1, s2, low, L0, T0);
    tf_fixed(v1, s1, s2, low, L1, T1);
    for (int i = s - 1; i >= 1; --i) {
        const int d0 = ((L0 + 256) & 511) - 256, d1 = ((L1 + 256) & 511) - 256;
        zr[i * plane32] = oz_digit_pair(d0, d1);
        L0 = (L0 - d0) >> kOzBeta;
        L1 = (L1 - d1) >> kOzBeta;
        if (i == s - low) { // the low parts are used up: carry into the high ones
            L0 += T0;
            L1 += T1;
        }
    }
    zr[0] = oz_digit_pair(L0, L1);
}

template <int NE>
__global__ void __launch_bounds__(256, NE > 4 ? 3 : 4) gpp_prep_split_kernel(const float4 *__restrict__ At,
                                                                const float4 *__restrict__ Wt, int ng, GppEnergies en,
                                                                int cnt, float sgn, int s, int64_t kpad,
                                                                int64_t zstride, uint16_t *__restrict__ Z,
                                                                int *__restrict__ E)
{
    __shared__ int red[8][NE];
    __shared__ float2 dsm[NE];
    __shared__ float2 ssm[NE];
    const int c = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x < NE) {
        const tf t = tf_from(threadIdx.x < cnt ? en.d[threadIdx.x] : 0.0);
        dsm[threadIdx.x] = make_float2(t.hi, t.lo);
    }
    __syncthreads();
    const float4 *a = At + (int64_t)c * ng, *w = Wt + (int64_t)c * ng;
    float mx[NE];
#pragma unroll
    for (int j = 0; j < NE; ++j) mx[j] = 0.0f;
    for (int g = threadIdx.x; g < ng; g += blockDim.x) {
        const float4 a4 = a[g], w4 = w[g];
#pragma unroll
        for (int j = 0; j < NE; ++j)
            if (j < cnt) mx[j] = fmaxf(mx[j], gpp_pole_mag(a4, w4, tf{dsm[j].x, dsm[j].y}, sgn));
    }
#pragma unroll
    for (int j = 0; j < NE; ++j) {
        float v = mx[j];
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (lane == 0) red[wid][j] = __float_as_int(v);
    }
    __syncthreads();
    if (threadIdx.x < cnt) {
        float v = 0.0f;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) v = fmaxf(v, __int_as_float(red[k][threadIdx.x]));
        const int e = tf_expo(v * (1.0f + 0x1p-10f));
        E[(int64_t)threadIdx.x * ng + c] = e;
        // 2^sh in two factors, each inside the FP32 exponent range
        const int sh = max(-250, min(250, oz_frac_bits(s) - e));
        ssm[threadIdx.x] = make_float2(__int_as_float((127 + sh / 2) << 23), __int_as_float((127 + sh - sh / 2) << 23));
    }
    __syncthreads();
    const int64_t plane32 = (int64_t)ng * kpad;
    for (int64_t k = threadIdx.x; 2 * k < kpad; k += blockDim.x) {
        // entries 2 k and 2 k + 1 of the row; padding entries have a = 0, so P = 0 there
        float4 a4[2], w4[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const bool in = 2 * k + u < ng;
            a4[u] = in ? a[2 * k + u] : make_float4(0.f, 0.f, 0.f, 0.f);
            w4[u] = in ? w[2 * k + u] : make_float4(1.f, 0.f, 0.f, 0.f);
        }
        for (int j = 0; j < cnt; ++j) {
            const tf d{dsm[j].x, dsm[j].y};
            const tcx p0 = gpp_pole_tf(a4[0], w4[0], d, sgn), p1 = gpp_pole_tf(a4[1], w4[1], d, sgn);
            const float2 sc = ssm[j];
            uint32_t *z = (uint32_t *)(Z + j * zstride + (int64_t)2 * c * kpad) + k;
            tf_digits_store(p0.re, p1.re, sc.x, sc.y, s, z, plane32);
            tf_digits_store(p0.im, p1.im, sc.x, sc.y, s, z + kpad / 2, plane32);
        }
    }
}

// ------------------------------------------------------------------ tcgen05 GEMM
// Persistent and batched: a launch takes a table of jobs (one job = one chunk's slices for one chi
// block, or one general product, each with its own sizes, tensor maps and exponents) and a list of
// items (job, tile, K range).  A pair of CTAs (a cluster of two, cta_group::2) takes items c,
// c + clusters, ... in the same order in every role, so the TMA warps, the MMA warp and the
// epilogue warps need no exchange beyond the mbarriers.
//
// What bounds it: the tensor pipe, fed from L2.  A pair works on 256 x 256 real entries; each CTA
// loads 128 rows of A and 128 of B per K-step, 32 KB, so the ring holds six stages (one CTA on a
// 128 x 256 tile loads 48 KB per K-step for half the work and holds four).  A 256 x 128 tile is no
// alternative: an MMA of a pair takes as long with 128 columns as with 256 (33.5 against 19.0 ms
// for the 16 chunks of a 48^3 q-point).  The sums of a tile stay in registers as two-float pairs
// over all its slice groups and K-segments (64 per epilogue thread: Re or Im parts, two of the real
// products each), so a segment costs TMEM loads and FP32 adds, and FP64 work and atomics come once
// per item.  Two accumulators in TMEM alternate between segments, so a segment's epilogue overlaps
// the next one's MMAs.  The issuing warp runs converged (umma_f16_run): issued by a lone thread the 16
// launches of a 48^3 q-point take 19.2 ms instead of 17.5.
//
// Measured (split contraction of one 8192-pair chunk, N_G = 2000, 7-slice accuracy): 1.09 ms, 15
// products of nine-bit slices, 1.80 PFLOP/s on them; one CTA per tile with 28 products of six-bit
// slices and an FP64 atomic epilogue per slice group took 2.44 ms (1.50 PFLOP/s).  General product of the
// self-energy (N_G = 6000, 384 bands): 19.1 against 54.3 ms.
struct OzCfg {
    static constexpr unsigned Bytes = kOzBM * kOzBK * 2;     // of A, and of B, per stage and CTA
    static constexpr int Stages = 6;                         // TMA ring depth
    static constexpr int Cols = 256, Bufs = 2;               // accumulators in TMEM
    // idesc: D = F32, A = B = BF16, both K-major, N = 256, M = 256 over the pair
    static constexpr uint32_t Idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(Cols >> 3) << 17) |
                                      ((uint32_t)(2 * kOzBM >> 4) << 24);
    static constexpr size_t Smem = 1024 + Stages * 2 * (size_t)Bytes + (2 * Stages + 2 * Bufs + 1) * 8 + 16;
};

// The segments of an item of nk K-steps with s slices, in the order every role walks them: K block
// by K block, from the least significant group up, the group's segments of the block.
template <bool F64>
struct OzSegments {
    int nk, s, kc, t, k0, len;
    __device__ __forceinline__ OzSegments(int nk_, int s_) : nk(nk_), s(s_), kc(0), t(s_ + 1), k0(0) { cut(); }
    __device__ __forceinline__ void cut() { len = min(min(nk, kc + kOzKBlock) - k0, oz_segment<F64>(t)); }
    // of a K block: first segment of its group, last segment of all
    __device__ __forceinline__ bool opens() const { return k0 == kc; }
    __device__ __forceinline__ bool closes() const { return t == 2 && k0 + len >= min(nk, kc + kOzKBlock); }
    __device__ __forceinline__ bool more() const { return kc < nk; }
    __device__ __forceinline__ void next()
    {
        k0 += len;
        if (k0 >= min(nk, kc + kOzKBlock)) {
            if (--t < 2) {
                t = s + 1;
                kc += kOzKBlock;
            }
            k0 = kc;
        }
        cut();
    }
};

// A pair's waits end within a millisecond unless something failed; the bound keeps the time until
// every warp of both CTAs has given up short.
__device__ __forceinline__ bool pair_wait(uint64_t *b, unsigned parity) { return bar_wait(b, parity, 1LL << 22); }

// hi + lo += x with the rounding error of hi + x kept in lo
__device__ __forceinline__ void oz_add(float &hi, float &lo, float x)
{
    const float s = __fadd_rn(hi, x), b = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
    hi = s;
}

// x 2^ex as a double, from the bits (no conversion on the FP64 pipe); 0 below 2^-1022
__device__ __forceinline__ double oz_scaled_double(float x, int ex)
{
    const uint32_t u = __float_as_uint(x);
    const int e = (int)((u >> 23) & 0xff) + 896 + ex;
    if ((u & 0x7f800000u) == 0 || e <= 0) return 0.0;
    return __hiloint2double((int)((u & 0x80000000u) | ((uint32_t)min(e, 2046) << 20) | ((u >> 3) & 0xfffffu)),
                            (int)(u << 29));
}

// where an epilogue thread's sums belong: complex row g of nr, columns g0 .. of nc
struct OzPlace {
    int g, g0, nr, nc, eg;
    const int *ecol;
    double *row, *part;
};

// Split: the Hermitian contraction above (upper tiles, chi epilogue), two-float sums.  General: the
// product out += A B (all tiles, each owned by one pair of CTAs, plain FP64 adds).  F64: the Hermitian
// contraction with seven slices, sums exact up to the last unit of a 64-bit integer per K block of 1024
// pairs: segments whose FP32 sums are exact whatever the digits (oz_segment), groups t = 8..5 in units of
// 2^-54 (|sum| < 2^57), rounded to units of 2^-37 before t = 4..2 (|sum| <= 2 1024 2^14 2^37 = 2^62), 2^-51 of
// a pair's largest product.  A block's sum goes to chi (or to the part's place in scratch) in FP64, so a
// chunk of 8192 pairs is rounded eight times where a chain of DMMAs is rounded 2048 times.  Measured on a
// chunk of 8192 pairs, N_G = 2000: 3.12 ms (28 products, 1.18 PFLOP/s, the epilogue of the 55 segments of
// a K block its bound; segments of 256 pairs throughout, 26 of them, take 2.45 but leave 1e-11 where the digits of
// many pairs have one sign) and 0.33 ms for the slices where the DMMA kernel, at 0.86 of its pipe's rate, takes
// 138; error of chi against 64 bits 1.1e-15 where it leaves 1.9e-15.  One code path for t = 2 and another for
// the rest spills 872 bytes instead of 232: 4.58 ms.
enum class OzProd { Split, General, F64 };
template <OzProd MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kOzThreads, 1)
    oz_gemm_kernel(const OzJob *__restrict__ jobs, const OzItem *__restrict__ items, int nitems, OzScratch scr,
                   int *status, const int *guard)
{
    using C = OzCfg;
    constexpr int ST = C::Stages, NB = C::Bufs;
    constexpr bool GEN = MODE == OzProd::General, F64 = MODE == OzProd::F64;
    if (F64 && *guard) return; // the DMMA kernel takes the chunk
    extern __shared__ __align__(1024) unsigned char smraw[];
    unsigned char *sm = (unsigned char *)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = sm;                 // [stages][Bytes]
    unsigned char *sB = sA + ST * C::Bytes; // [stages][Bytes]
    uint64_t *full = (uint64_t *)(sB + ST * C::Bytes); // used in CTA 0: both CTAs' loads count there
    uint64_t *empty = full + ST;            // each CTA its own, by the pair's commit
    uint64_t *tfull = empty + ST;           // likewise
    uint64_t *tempty = tfull + NB;          // used in CTA 0: 16 epilogue warps arrive
    uint64_t *fin = tempty + NB;
    uint32_t *tslot = (uint32_t *)(fin + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int cl0 = blockIdx.x >> 1, ncl = gridDim.x >> 1;
    if (threadIdx.x == 0) {
        for (int i = 0; i < ST; ++i) {
            bar_init(&full[i], 1);
            bar_init(&empty[i], 1);
        }
        for (int i = 0; i < NB; ++i) {
            bar_init(&tfull[i], 1);
            bar_init(&tempty[i], 16);
        }
        bar_init(fin, 1);
        bar_fence_init();
    }
    if (warp == 1) tmem_alloc_pair(tslot, NB * C::Cols);
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    const uint32_t tbase = *tslot;
    bool ok = true;

    // registers: 384 x 168 at launch; the epilogue warps hold a tile's sums (128 of them) and take
    // 224 a thread, the warpgroup of the TMA and MMA warps keeps 56 (2 x 224 + 56 = 3 x 168)
    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        if (warp == 0 && lane == 0) {
            uint32_t it = 0;
            const uint32_t full0 = cluster_map(full, 0);
            for (int item = cl0; item < nitems && ok; item += ncl) {
                const OzItem w = items[item];
                const OzJob &jb = jobs[w.job];
                const int ra = (2 * w.I + (int)rank) * kOzBM, rb = (2 * w.J + (int)rank) * kOzBM;
                for (OzSegments<F64> g(w.nk, jb.s); g.more() && ok; g.next())
                    for (int i = 1; i < g.t && ok; ++i)
                        for (int kb = 0; kb < g.len; ++kb, ++it) {
                            const uint32_t st = it % ST;
                            if (!pair_wait(&empty[st], ((it / ST) & 1) ^ 1)) { ok = false; break; }
                            if (rank == 0) bar_expect(&full[st], 4 * C::Bytes);
                            const int k = (w.kb0 + g.k0 + kb) * kOzBK;
                            tma3_pair(sA + st * C::Bytes, &jb.tmA, full0 + 8 * st, k, ra, i - 1);
                            tma3_pair(sB + st * C::Bytes, &jb.tmB, full0 + 8 * st, k, rb, g.t - i - 1);
                        }
            }
            // copies in flight land before the pair tears down (they count at CTA 0's barriers)
            if (!ok && rank == 0)
                for (uint32_t j = it > ST ? it - ST : 0; j < it; ++j) pair_wait(&full[j % ST], (j / ST) & 1);
            if (!ok) atomicOr(status, kStatusTimeout);
        }
        if (warp == 1 && rank == 0) { // the warp converged (umma_f16_run)
            const uint32_t lead = elect_lane(), tb = __shfl_sync(0xffffffffu, tbase, 0);
            const uint32_t ad = sdesc_sw128_low(su32(sA)), bd = sdesc_sw128_low(su32(sB));
            auto wait = [&](uint64_t *b, uint32_t parity) {
                if (!__all_sync(0xffffffffu, pair_wait(b, parity))) ok = false;
            };
            uint32_t st = 0, ph = 0, seg = 0;
            for (int item = cl0; item < nitems && ok; item += ncl) {
                const OzItem w = items[item];
                for (OzSegments<F64> g(w.nk, jobs[w.job].s); g.more() && ok; g.next(), ++seg) {
                    const uint32_t b = seg % NB;
                    wait(&tempty[b], ((seg / NB) & 1) ^ 1);
                    tc_fence_after();
                    const int n = (g.t - 1) * g.len; // ring stages of the segment
                    for (int j = 0; j < n && ok; ++j) {
                        wait(&full[st], ph);
                        tc_fence_after();
                        const uint32_t o = st * (C::Bytes >> 4);
#pragma unroll
                        for (int kk = 0; kk < kOzBK / 16; ++kk)
                            umma_f16_pair(lead, tb + b * C::Cols, ad + o + kk * 2, bd + o + kk * 2, kSdescSw128High,
                                          C::Idesc, (j == 0 && kk == 0) ? 0u : 1u);
                        umma_commit_pair(lead, &empty[st]);
                        if (++st == ST) {
                            st = 0;
                            ph ^= 1;
                        }
                    }
                    umma_commit_pair(lead, &tfull[b]);
                }
            }
            // every issued MMA has completed before the pair tears down
            umma_commit_pair(lead, fin);
            wait(fin, 0);
            if (!ok && lead) atomicOr(status, kStatusTimeout);
        } else if (warp == 1 && lane == 0) {
            pair_wait(fin, 0); // the pair's last commit has reached this CTA too
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        // epilogue: warps 4..11 -> TMEM lane quadrant (warp % 4) and half of the columns, one tile
        // row per thread
        constexpr int COLS = C::Cols / 2;             // columns per thread
        constexpr int NO = COLS / 2;                  // sums per thread: Re or Im parts of a complex row
        const int q = warp & 3, half = (warp - 4) >> 2;
        const int r = q * 32 + lane;                  // row of this CTA's half of the tile
        const int odd = r & 1;                        // 0 Re part, 1 Im part
        // chi: Re = C[2G][2G'] + C[2G+1][2G'+1], Im = C[2G][2G'+1] - C[2G+1][2G']; general product: Re =
        // C[2r][2c] - C[2r+1][2c+1], Im = C[2r][2c+1] + C[2r+1][2c].  The other row's term comes
        // from the neighbouring lane.
        const uint32_t flip = !GEN && odd ? 0x80000000u : 0u, rflip = GEN && !odd ? 0x80000000u : 0u;
        const uint32_t tempty0 = cluster_map(tempty, 0);
        constexpr int64_t kPart = 2 * 8 * 32 * NO; // doubles of one part
        auto place = [&](const OzItem &w, const OzJob &jb) {
            OzPlace p;
            p.g = (2 * w.I + (int)rank) * (kOzBM / 2) + (r >> 1);
            p.g0 = w.J * kOzBM + half * NO;
            p.nr = GEN ? jb.rows_a : jb.ng;
            p.nc = GEN ? jb.cols_b : jb.ng;
            p.ecol = GEN ? jb.E2 : jb.E;
            p.eg = p.g < p.nr ? __ldg(jb.E + p.g) - 16 : 0;
            p.row = (GEN ? jb.out + (int64_t)p.g * jb.ldo : jb.chi + 2 * (int64_t)p.g * jb.ng) + 2 * p.g0 + odd;
            // a part of a split tile: this warp's sums go to its place in scratch, lane by lane
            p.part = !GEN && w.parts > 1 ? scr.sums + ((int64_t)w.slot * w.parts + w.part) * kPart +
                                               ((int)rank * 8 + warp - 4) * (32 * NO) + lane
                                         : nullptr;
            return p;
        };
        float hi[F64 ? 1 : NO], lo[F64 ? 1 : NO];
        long long acc[F64 ? NO : 1];
        uint32_t seg = 0;
        for (int item = cl0; item < nitems && ok; item += ncl) {
            const OzItem w = items[item];
            const OzJob &jb = jobs[w.job];
            if constexpr (!F64) {
#pragma unroll
                for (int j = 0; j < NO; ++j) hi[j] = lo[j] = 0.0f;
            }
            for (OzSegments<F64> sg(w.nk, jb.s); sg.more(); sg.next(), ++seg) {
                const uint32_t b = seg % NB;
                const bool got = pair_wait(&tfull[b], (seg / NB) & 1);
                if (!__all_sync(0xffffffffu, got)) { ok = false; break; } // warp-uniform exit
                tc_fence_after();
                const float wt = __int_as_float((127 - kOzBeta * (sg.t - 2)) << 23); // the group's weight
                if constexpr (F64) {
                    if (sg.opens() && sg.t == jb.s + 1) {
#pragma unroll
                        for (int j = 0; j < NO; ++j) acc[j] = 0;
                    } else if (sg.opens() && sg.t == 4) {
#pragma unroll
                        for (int j = 0; j < NO; ++j) acc[j] = (acc[j] + (1 << 16)) >> 17;
                    }
                }
                const uint32_t ta = tbase + ((uint32_t)(q * 32) << 16) + b * C::Cols + half * COLS;
                // F64: the group's unit is 2^ush of the sum's (t = 2: 2^37, into the high word)
                const int ush = sg.t >= 5 ? kOzBeta * (8 - sg.t) : 37 - kOzBeta * (sg.t - 2);
                const int umul = sg.t == 2 ? 0 : 1 << ush, hmul = sg.t == 2 ? 1 << (ush - 32) : 0;
#pragma unroll
                for (int c0 = 0; c0 < COLS; c0 += 32) {
                    uint32_t v[32];
                    GW_TMEM_LD32(ta + c0, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int cc = 0; cc < 16; ++cc) {
                        const uint32_t rv = __shfl_xor_sync(0xffffffffu, v[2 * cc + 1], 1) ^ rflip;
                        const float x0 = __uint_as_float(v[2 * cc] ^ flip), x1 = __uint_as_float(rv);
                        if constexpr (F64) { // added as integers: two sums of 2^24 may not fit FP32
                            const int xi = __float2int_rn(x0) + __float2int_rn(x1);
                            acc[(c0 >> 1) + cc] += (long long)xi * umul + ((long long)(xi * hmul) << 32);
                        } else {
                            oz_add(hi[(c0 >> 1) + cc], lo[(c0 >> 1) + cc], __fmul_rn(wt, __fadd_rn(x0, x1)));
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) bar_arrive_cluster(tempty0 + 8 * b);
                if constexpr (F64) {
                    if (sg.closes()) { // the K block's sums, |E| <= 400: the scale is a normal number
                        const OzPlace p = place(w, jb);
#pragma unroll
                        for (int j = 0; j < NO; ++j)
                            if (p.g < p.nr && p.g0 + j < p.nc && p.g <= p.g0 + j) {
                                const int ex = p.eg + __ldg(p.ecol + p.g0 + j) - 37;
                                const double y = (double)acc[j] * __hiloint2double((1023 + ex) << 20, 0);
                                if (p.part) __stcg(p.part + 32 * j, sg.kc == 0 ? y : __ldcg(p.part + 32 * j) + y);
                                else if (y != 0.0) atomicAdd(p.row + 2 * j, -y);
                            }
                    }
                }
            }
            if (!ok) break;
            const OzPlace p = place(w, jb);
            const int g = p.g, g0 = p.g0, nr = p.nr, nc = p.nc, eg = p.eg;
            const int *ecol = p.ecol;
            double *row = p.row, *part = p.part;
#pragma unroll
            for (int j = 0; j < NO; ++j)
                if (!F64 && g < nr && g0 + j < nc && (GEN || g <= g0 + j)) {
                    const int ex = eg + __ldg(ecol + g0 + j);
                    const int q = F64 ? 0 : j;
                    const double y = oz_scaled_double(hi[q], ex) + oz_scaled_double(lo[q], ex);
                    if constexpr (GEN) row[2 * j] = jb.add ? row[2 * j] + y : y; // the pair of CTAs owns the tile
                    else if (part) __stcg(part + 32 * j, y);
                    else if (y != 0.0) atomicAdd(row + 2 * j, -y); // other pair segments may add here too
                }
            if (!GEN && part) {
                // the warp that finishes a split tile's rows last adds all parts, in their order
                __threadfence();
                __syncwarp();
                int *flag = scr.flags + w.slot * 16 + (int)rank * 8 + warp - 4;
                int last = 0;
                if (lane == 0) last = atomicAdd(flag, 1) == w.parts - 1;
                if (__shfl_sync(0xffffffffu, last, 0)) {
                    __threadfence();
                    const double *p0 = part - (int64_t)w.part * kPart;
                    for (int j0 = 0; j0 < NO; j0 += 16) { // 16 loads in flight
                        double y[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j) y[j] = 0.0;
                        for (int i = 0; i < w.parts; ++i) {
                            double v[16];
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                const int c = g0 + j0 + j;
                                v[j] = g < nr && c < nc && g <= c ? __ldcg(p0 + i * kPart + 32 * (j0 + j)) : 0.0;
                            }
#pragma unroll
                            for (int j = 0; j < 16; ++j) y[j] += v[j];
                        }
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (y[j] != 0.0) atomicAdd(row + 2 * (j0 + j), -y[j]);
                    }
                    if (lane == 0) *flag = 0;
                }
            }
        }
        if (!ok && lane == 0) atomicOr(status, kStatusTimeout);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    if (warp == 1) tmem_dealloc_pair(tbase, NB * C::Cols);
}

// ------------------------------------------------------------------ host launchers
cudaError_t launch_oz_sqrt(const double *delta, int64_t n, double *sp, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    oz_sqrt_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(delta, n, sp);
    return cudaGetLastError();
}

cudaError_t launch_oz_colexp(const double2 *M, int64_t P, int ng, const double *sp, int *E, int *guard,
                             cudaStream_t st)
{
    oz_fill_kernel<<<(ng + 255) / 256, 256, 0, st>>>(E, ng, kOzNoColumn);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || P == 0) return e;
    int gy = (int)std::min<int64_t>((P + 63) / 64, 256);
    const dim3 grid((ng + 31) / 32, gy);
    if (!sp) oz_colexp_kernel<false, false><<<grid, 256, 0, st>>>(M, P, ng, sp, E, guard);
    else if (guard) oz_colexp_kernel<true, true><<<grid, 256, 0, st>>>(M, P, ng, sp, E, guard);
    else oz_colexp_kernel<false, true><<<grid, 256, 0, st>>>(M, P, ng, sp, E, guard);
    return cudaGetLastError();
}

int oz_group_w() { return kOzGroupW; }

cudaError_t launch_oz_split_multi(const double2 *M, int64_t P, int ng, const double *sp, int64_t dstride, int nw,
                                  int *E, int s, int64_t kpad, void *Z, int64_t zstride, cudaStream_t st)
{
    if (nw < 1 || nw > kOzGroupW) return cudaErrorInvalidValue;
    oz_fill_kernel<<<(unsigned)(((int64_t)nw * ng + 255) / 256), 256, 0, st>>>(E, nw * ng, kOzNoColumn);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (P > 0) {
        const int gy = (int)std::min<int64_t>((P + 63) / 64, 256);
        oz_colexp_multi_kernel<<<dim3((ng + 31) / 32, gy), 256, 0, st>>>(M, P, ng, sp, dstride, nw, E);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    oz_slice_multi_kernel<<<dim3((ng + 31) / 32, (unsigned)(kpad / 64)), 256, 0, st>>>(
        M, P, ng, sp, dstride, nw, E, s, kpad, zstride, (__nv_bfloat16 *)Z);
    return cudaGetLastError();
}

cudaError_t launch_oz_slice(const double2 *M, int64_t P, int ng, const double *sp, const int *E, int s,
                            int64_t kpad, void *Z, int *guard, cudaStream_t st)
{
    const dim3 grid((ng + 31) / 32, (unsigned)(kpad / 64));
    __nv_bfloat16 *z = (__nv_bfloat16 *)Z;
    if (!sp) oz_slice_kernel<false, false><<<grid, 256, 0, st>>>(M, P, ng, sp, E, s, kpad, z, guard);
    else if (guard) oz_slice_kernel<true, true><<<grid, 256, 0, st>>>(M, P, ng, sp, E, s, kpad, z, guard);
    else oz_slice_kernel<false, true><<<grid, 256, 0, st>>>(M, P, ng, sp, E, s, kpad, z, guard);
    return cudaGetLastError();
}

template <OzProd MODE>
static cudaError_t launch_gemm(const OzJob *jobs, const OzItem *items, int nitems, int clusters, OzScratch scr,
                               int *status, const int *guard, cudaStream_t st)
{
    if (nitems == 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(oz_gemm_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)OzCfg::Smem);
    if (e != cudaSuccess) return e;
    oz_gemm_kernel<MODE><<<2 * clusters, kOzThreads, OzCfg::Smem, st>>>(jobs, items, nitems, scr, status, guard);
    return cudaGetLastError();
}

int oz_f64_slices() { return kOzF64Slices; }

size_t oz_part_bytes() { return sizeof(double) * 2 * 8 * 32 * (OzCfg::Cols / 4); }
int oz_slot_flags() { return 16; }

cudaError_t launch_oz_gemm_jobs(const OzJob *jobs, const OzItem *items, int nitems, int clusters, OzScratch scr,
                                int *status, const int *guard, cudaStream_t st)
{
    return guard ? launch_gemm<OzProd::F64>(jobs, items, nitems, clusters, scr, status, guard, st)
                 : launch_gemm<OzProd::Split>(jobs, items, nitems, clusters, scr, status, guard, st);
}

cudaError_t launch_oz_gemm_general(const OzJob *jobs, const OzItem *items, int nitems, int clusters, int *status,
                                   cudaStream_t st)
{
    return launch_gemm<OzProd::General>(jobs, items, nitems, clusters, OzScratch{}, status, nullptr, st);
}

cudaError_t launch_oz_split(const double2 *A, int64_t rows, int ka, int64_t sr, int64_t sk, bool conj, int s,
                            int64_t kpad, void *Z, int *E, cudaStream_t st)
{
    if (rows == 0) return cudaSuccess;
    if (conj) oz_split_kernel<true><<<(unsigned)rows, 256, 0, st>>>(A, rows, ka, sr, sk, s, kpad, (uint16_t *)Z, E);
    else oz_split_kernel<false><<<(unsigned)rows, 256, 0, st>>>(A, rows, ka, sr, sk, s, kpad, (uint16_t *)Z, E);
    return cudaGetLastError();
}

cudaError_t launch_gpp_prep_split(const float4 *At, const float4 *Wt, int ng, const double *d, int cnt, float sgn,
                                  int s, int64_t kpad, int64_t zstride, void *Z, int *E, cudaStream_t st)
{
    if (ng == 0 || cnt == 0) return cudaSuccess;
    if (cnt > kGppMaxE) return cudaErrorInvalidValue;
    GppEnergies en{};
    for (int j = 0; j < cnt; ++j) en.d[j] = d[j];
    if (cnt <= 4)
        gpp_prep_split_kernel<4><<<(unsigned)ng, 256, 0, st>>>(At, Wt, ng, en, cnt, sgn, s, kpad, zstride,
                                                               (uint16_t *)Z, E);
    else
        gpp_prep_split_kernel<kGppMaxE><<<(unsigned)ng, 256, 0, st>>>(At, Wt, ng, en, cnt, sgn, s, kpad, zstride,
                                                                      (uint16_t *)Z, E);
    return cudaGetLastError();
}

int oz_box_rows() { return kOzBM; }
int oz_box_k() { return kOzBK; }

} // namespace gw
