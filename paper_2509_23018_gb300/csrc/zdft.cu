// Stage (a), last-axis transform of the pair products on the BF16 tensor cores.
//
// For a line l = (i0, i1) of the grid and a pair (v, c), the pruned transform of the pair
// product along the last axis at the kept frequencies kz[q] is
//     F[v][c][l][q] = sum_{i2} conj(psi_v[l][i2]) W_q[i2] psi_c[l][i2],   W_q[i2] = e^{+2 pi i kz[q] i2 / N},
// the first stage of the forward transform of the product (the definition after Eq. ff-ch).
// Over the pairs of a block it is, line by line, a complex matrix product whose operands
// belong to one band each: rows psi_c[l] (conduction), columns W_q conj(psi_v[l]) (valence).
// Written in real form (K = 2 N: Re and Im of each point interleaved), it runs as an
// Ozaki-style split product (the scheme of stage (b)):
//   * each operand row / column is scaled by its own power of two 2^E (|x| < 2^E) and cut into
//     six balanced base-256 digits, x = 2^E sum_{i<6} d_i 2^(-7-8i), |d_i| <= 128; a digit
//     times its scale is exact in BF16 (eight significant bits), so the slices carry their
//     scales and the tensor cores accumulate true values;
//   * the slice products i + j <= 5 are kept (the rest lies below 2^-48 of the operands'
//     scales); the products with i + j = 0, 1, 2 go to three FP32 accumulators of their own:
//     each of their terms is a multiple of one unit of that group with |sum| <= 3 * 144 * 2^14
//     < 2^24, so those sums are exact; i + j = 3..5 share a fourth accumulator (its rounding
//     lies 2^-48 below the leading group);
//   * the four accumulators are summed in two-float arithmetic (two-sums for the exact groups)
//     into F, which the pair kernel's remaining stages (middle and first axis) take from there.
// The row slices of a block of conduction bands are formed once (zd_rows_kernel), as the images
// of the shared-memory tiles that the product copies; the valence columns are formed on the chip,
// from psi_v and the twiddles, by producer warps, once for all the row tiles of a line.
#include "internal.h"
#include "ptx.cuh"
#include "fft_tf.cuh"
#include "zd_tiles.cuh"

#include <algorithm>

namespace gw {

// ------------------------------------------------------------------ digits
// Balanced base-256 digits of y = (h + l) 2^(7 - E), |y| < 128 (two-float value, exponent E):
// N = round(y 2^40) = T 2^24 + U with T, U exact FP32 integers, digits taken from the low end,
// each digit times its weight 2^(E - 7 - 8i) returned as the BF16 bits of slice i.
__device__ __forceinline__ void zd_digits(float h, float l, int E, uint16_t out[kZdSlices])
{
    // 2^(47 - E) in two factors so that each stays a normal FP32 for any E in [-100, 100]
    const int sh = 47 - E;
    const float s1 = __int_as_float((127 + sh / 2) << 23), s2 = __int_as_float((127 + sh - sh / 2) << 23);
    const float Y = __fmul_rn(__fmul_rn(h, s1), s2), L = __fmul_rn(__fmul_rn(l, s1), s2);
    const float T = rintf(__fmul_rn(Y, 0x1p-24f));
    float U = __fadd_rn(rintf(__fmaf_rn(-0x1p24f, T, Y)), rintf(L)); // |U| <= 2^24
    float d[kZdSlices];
#pragma unroll
    for (int i = kZdSlices - 1; i >= 3; --i) {
        const float q = rintf(__fmul_rn(U, 0.00390625f));
        d[i] = __fmaf_rn(-256.0f, q, U);
        U = q;
    }
    float V = __fadd_rn(T, U); // |V| < 2^23 + 2
#pragma unroll
    for (int i = 2; i >= 1; --i) {
        const float q = rintf(__fmul_rn(V, 0.00390625f));
        d[i] = __fmaf_rn(-256.0f, q, V);
        V = q;
    }
    d[0] = V;
    // weights: slice i holds d_i 2^(E - 7 - 8 i)
#pragma unroll
    for (int i = 0; i < kZdSlices; ++i) {
        const int e = E - 7 - 8 * i;
        const float w = __int_as_float((127 + max(-126, e)) << 23);
        out[i] = (uint16_t)(__float_as_uint(__fmul_rn(d[i], w)) >> 16);
    }
}

// The same digits where the line's scale 2^(47 - E) and every weight are normal FP32 numbers
// (-70 <= E <= 120).
__device__ __forceinline__ void zd_digits_n(float h, float l, int E, uint16_t out[kZdSlices])
{
    const float sc = __int_as_float((127 + 47 - E) << 23);
    const float Y = __fmul_rn(h, sc);
    const float T = rintf(__fmul_rn(Y, 0x1p-24f));
    float U = __fadd_rn(rintf(__fmaf_rn(-0x1p24f, T, Y)), rintf(__fmul_rn(l, sc)));
    float d[kZdSlices];
#pragma unroll
    for (int i = kZdSlices - 1; i >= 3; --i) {
        const float q = rintf(__fmul_rn(U, 0.00390625f));
        d[i] = __fmaf_rn(-256.0f, q, U);
        U = q;
    }
    float V = __fadd_rn(T, U);
#pragma unroll
    for (int i = 2; i >= 1; --i) {
        const float q = rintf(__fmul_rn(V, 0.00390625f));
        d[i] = __fmaf_rn(-256.0f, q, V);
        V = q;
    }
    d[0] = V;
    const int w0 = (127 + E - 7) << 23;
#pragma unroll
    for (int i = 0; i < kZdSlices; ++i)
        out[i] = (uint16_t)(__float_as_uint(__fmul_rn(d[i], __int_as_float(w0 - i * (8 << 23)))) >> 16);
}

// exponent E with |x| < 2^E for a line's largest component magnitude m (E = -126 for m = 0)
__device__ __forceinline__ int zd_expo(float m)
{
    if (!(m > 0.0f)) return -126;
    const int be = (int)((__float_as_uint(m) >> 23) & 0xff);
    return (be == 0 ? -126 : be - 127) + 1;
}

// ------------------------------------------------------------------ operand tiles in shared memory
constexpr int kZdMaxStages = 9;                        // stages per tile: lines of up to 72 points
constexpr unsigned kZdSlice = kZdM * kZdKB * 2;        // one row slice of one stage: 4 KB
constexpr unsigned kZdStage = kZdSlices * kZdSlice;    // 24 KB

// ------------------------------------------------------------------ row slices
// A[l][mt][ks][slice] (4 KB images of the swizzled tile of 128 rows x 16 real entries, so that one
// bulk copy of 24 KB brings a stage) of the rows psi[r][l][.], r < nr, zero above and past the line's
// n points: one warp per row of a line, 8 warps per block.
__global__ void __launch_bounds__(256) zd_rows_kernel(const float4 *__restrict__ psi, int nr, int n, int nlines,
                                                      int nmt, unsigned char *__restrict__ A)
{
    const int lane = threadIdx.x & 31, l = blockIdx.y, r = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int nst = zd_stages(n);
    unsigned char *dst = A + ((int64_t)l * nmt + r / kZdM) * nst * kZdStage;
    const int rt = r % kZdM;
    const float4 *row = psi + ((int64_t)min(r, nr - 1) * nlines + l) * n;
    float m = 0.0f;
    float4 x[3];
#pragma unroll
    for (int u = 0; u < 3; ++u) {
        const int i = lane + 32 * u;
        x[u] = i < n && r < nr ? row[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        m = fmaxf(m, fmaxf(fabsf(x[u].x), fabsf(x[u].z)) * (1.0f + 0x1p-20f));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    const int E = zd_expo(m);
#pragma unroll
    for (int u = 0; u < 3; ++u) {
        const int i = lane + 32 * u;
        if (i >= 8 * nst) break;
        uint16_t dr[kZdSlices], di[kZdSlices];
        zd_digits(x[u].x, x[u].y, E, dr);
        zd_digits(x[u].z, x[u].w, E, di);
        unsigned char *p = dst + (i >> 3) * kZdStage + sw32_off(rt, 2 * (i & 7));
#pragma unroll
        for (int s = 0; s < kZdSlices; ++s) *(uint32_t *)(p + s * kZdSlice) = (uint32_t)dr[s] | ((uint32_t)di[s] << 16);
    }
}

// E[band][l]: exponent of a line's columns W_q conj(psi): |W_q psi| <= |Re psi| + |Im psi|
// (-70 <= E, so that the digits' scale and every weight stay normal FP32 numbers)
__global__ void __launch_bounds__(256) zd_colexp_kernel(const float4 *__restrict__ psi, int nb, int n, int nlines,
                                                        int *__restrict__ E)
{
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= (int64_t)nb * nlines) return;
    float m = 0.0f;
    for (int i = lane; i < n; i += 32) {
        const float4 x = psi[w * n + i];
        m = fmaxf(m, (fabsf(x.x) + fabsf(x.z)) * (1.0f + 0x1p-20f));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) E[w] = min(120, max(-70, zd_expo(m)));
}

size_t zd_row_bytes(int nr, int n, int lines)
{
    return (size_t)lines * ((nr + kZdM - 1) / kZdM) * zd_stages(n) * kZdStage;
}

cudaError_t launch_zd_rows(const void *psi, int nr, int n, int lines, void *A, cudaStream_t st)
{
    const int nmt = (nr + kZdM - 1) / kZdM;
    zd_rows_kernel<<<dim3(nmt * (kZdM / 8), lines), 256, 0, st>>>((const float4 *)psi, nr, n, lines, nmt,
                                                                  (unsigned char *)A);
    return cudaGetLastError();
}

cudaError_t launch_zd_colexp(const void *psi, int nb, int n, int lines, int *E, cudaStream_t st)
{
    const int64_t warps = (int64_t)nb * lines;
    zd_colexp_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>((const float4 *)psi, nb, n, lines, E);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ the product
// One block per SM, persistent over units u = (line l, valence tile of CT bands); per unit the
// producer warps form the tile's column slices (CT bands, 2 K2P real columns each, K2 rounded up to
// even; the others of 128 are zero), all stages of 16 real entries resident (points past the line's
// end are zero), and the block runs over the row tiles of 128 conduction bands, whose slices the TMA
// warp copies stage by stage into a ring.  Lines whose column stages leave no room for the ring (57 to
// 72 points) take tiles of 96 columns.  One thread issues the tcgen05 products into four accumulators
// of 128 TMEM columns each, and the
// epilogue warps sum the accumulators into F.  A 128 x N x 16 product costs about the same time at
// N = 64 as at N = 128 (feeding the 128 x 16 A operand sets the pace, whether A is read from shared
// memory or from TMEM), so the tile is 128 columns wide; its four accumulators then fill the 512 TMEM
// columns and are not double-buffered.  Each is handed back on its own as soon as its TMEM
// loads have landed, least significant first, and a tile's first two stages issue their products in
// that order: 15 of the 21 belong to the first accumulator handed back.
// A stage's columns are released by the last row tile's products, so the producers refill them while
// that tile finishes; the line tiles of the next unit are loaded a unit ahead.
//
// What bounds it: the tensor pipe and, behind it, F's stores.  A 128 x 128 x 16 product reads 8 KB of
// operands in its 64 clocks, all that shared memory delivers, so whatever else passes through it (the row
// stages' copies, the producers' stores) adds to the products' time.  1.80 ms for a 48^3 block of 8192
// pairs (16 x 512 bands, K2 = 15), 1.13 ms of it with nothing but the products; 1.45 without F's stores,
// 4.9 GB.  Issued by a lone thread, which moves every descriptor from its own registers to uniform ones, a
// product took 95 clocks whatever its size, 1.97 ms in all.  With the valence bands in the rows
// (resident) and each tile of conduction columns formed for one row tile it took 2.30 ms; F stored entry
// by entry, 32 half sectors an instruction, 2.9 ms; exchanged in quads by shuffles 2.25 ms; row stages in
// a ring of two instead of three 2.4 ms.
//  warps 0..3: TMA, MMA (and TMEM), two producers; warps 4..11: epilogue (TMEM lane quadrant
//  warp % 4, half of the columns each); warps 12..15: producers.
constexpr int kZdThreads = 512;
constexpr int kZdProducers = 6; // producer warps
constexpr int kZdPsiSlots = 2;  // ring of valence-band line tiles
constexpr int kZdMaxRing = 4;   // ring of row stages (2 to 4, what shared memory holds)
constexpr int kZdRounds = 3;    // (band, frequency) pairs per producer lane: 64 pairs, 6 warps x 4

// two-sum with the sum's rounding error
__device__ __forceinline__ float zd_2sum(float a, float b, float &e)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

struct ZdArgs {
    CUtensorMap tmV;        // valence grids as FP32 [nv][lines][4N], box {4N, 1, CT} (zd_line_split)
    const unsigned char *A; // row slices (zd_rows_kernel) of the block's cb conduction bands
    const int *E;           // [nv][lines] column exponents
    const int *kz;          // [K2] kept last-axis frequencies
    float4 *F;              // [lines][vb cb][K2P] two-float, row vl cb + cl
    int *status;
    int n, lines, lsplit, nv, v0, vb, cb, K2, K2P, CT, nvt, nmt, nunits, ast; // ast: stages of the row ring
};

template <int NT>
__global__ void __launch_bounds__(kZdThreads, 1) zd_gemm_kernel(const __grid_constant__ ZdArgs a,
                                                                const float4 *__restrict__ twf)
{
    constexpr unsigned kBSlice = NT * kZdKB * 2, kBStage = kZdSlices * kBSlice;
    // idesc: D = F32, A = B = BF16, both K-major, N = NT, M = 128
    constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NT >> 3) << 17) |
                                ((uint32_t)(kZdM >> 4) << 24);
    extern __shared__ __align__(1024) unsigned char smraw[];
    unsigned char *sm = (unsigned char *)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
    const int nst = zd_stages(a.n), ncol = 2 * a.K2P;     // stages; real columns per valence band
    const uint32_t ast = a.ast;
    unsigned char *sA = sm;                               // ast x 24 KB
    unsigned char *sB = sA + ast * kZdStage;              // nst x 24 KB (18 KB at 96 columns)
    float4 *ring = (float4 *)(sB + nst * kBStage);        // [slots][CT][N] valence line tiles
    const int rst = zd_ring_stride(a.CT, a.n);
    float4 *wt = ring + kZdPsiSlots * rst;                // [N] twiddles W^t
    int2 *ctab = (int2 *)(wt + a.n);                      // [64] column pair -> (band, F offset)
    uint64_t *bar = (uint64_t *)(ctab + 64);
    uint64_t *aFull = bar, *aEmpty = aFull + kZdMaxRing, *bFull = aEmpty + kZdMaxRing, *bEmpty = bFull + kZdMaxStages,
             *tFull = bEmpty + kZdMaxStages, *tEmpty = tFull + 1, *pFull = tEmpty + 4, *pEmpty = pFull + kZdPsiSlots,
             *fin = pEmpty + kZdPsiSlots;
    uint32_t *tslot = (uint32_t *)(fin + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < a.n; i += blockDim.x) wt[i] = twf[i];
    // the epilogue's column pairs (Re, Im of entry q of band vl of the tile): vl and the offset
    // vl cb K2P + q of its F entry from the row's first (padding pairs: vl >= CT)
    for (int pi = threadIdx.x; pi < 64; pi += blockDim.x) {
        const int vl = pi / a.K2P, q = pi - vl * a.K2P;
        ctab[pi] = make_int2(vl, vl * a.cb * a.K2P + q);
    }
    // columns that no frequency fills stay zero in every stage
    for (int i = threadIdx.x; i < nst * (int)kBStage / 16; i += blockDim.x)
        ((uint4 *)sB)[i] = make_uint4(0u, 0u, 0u, 0u);
    fence_async_shared();
    if (threadIdx.x == 0) {
        for (int i = 0; i < kZdMaxRing; ++i) {
            bar_init(&aFull[i], 1);
            bar_init(&aEmpty[i], 1);
        }
        for (int i = 0; i < kZdMaxStages; ++i) {
            bar_init(&bFull[i], kZdProducers);
            bar_init(&bEmpty[i], 1);
        }
        bar_init(tFull, 1);
        for (int i = 0; i < 4; ++i) bar_init(&tEmpty[i], 8);
        for (int i = 0; i < kZdPsiSlots; ++i) {
            bar_init(&pFull[i], 1);
            bar_init(&pEmpty[i], kZdProducers);
        }
        bar_init(fin, 1);
        bar_fence_init();
    }
    if (warp == 1) tmem_alloc(tslot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = *tslot;
    bool ok = true;

    // registers: 512 x 128 at launch; the epilogue warps hold 64 columns of two accumulators and
    // take 176 a thread, the other two warpgroups keep 80
    if (warp >= 4 && warp < 12) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 176;");
        // ---- epilogue: a quadrant's 32 rows (conduction bands) x 64 of the 128 columns per warp.  The
        // 16 x 256-bit load shape gives the four lanes of a quad four consecutive entries (Re, Im) of
        // one row, so that a store instruction writes 64 contiguous bytes (whole sectors) of 8 rows.
        const int q4 = warp & 3, half = (warp - 4) >> 2;
        const uint32_t ta = tbase + ((uint32_t)(q4 * 32) << 16) + half * 64;
        uint32_t tile = 0;
        for (int u = blockIdx.x; u < a.nunits && ok; u += gridDim.x) {
            const int l = u / a.nvt, vt = u - l * a.nvt;
            const int vmax = min(a.CT, a.vb - vt * a.CT);
            for (int mt = 0; mt < a.nmt; ++mt, ++tile) {
                const bool got = bar_wait(tFull, tile & 1);
                if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                tc_fence_after();
                auto release = [&](int g) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) bar_arrive(&tEmpty[g]);
                };
                // s + e: the sum of the groups so far and its error, from the least significant up.
                // Registers 32 h + 4 j + 2 i + {0, 1}: row 16 h + 8 i + lane / 4, entry 4 j + lane % 4
                uint32_t s[64], e[64];
                GW_TMEM_LD_16X256_X8(ta + 3 * kZdAcc, e);
                GW_TMEM_LD_16X256_X8(ta + 3 * kZdAcc + (16u << 16), e + 32);
                tmem_wait_ld();
                release(3);
                GW_TMEM_LD_16X256_X8(ta + 2 * kZdAcc, s);
                GW_TMEM_LD_16X256_X8(ta + 2 * kZdAcc + (16u << 16), s + 32);
                tmem_wait_ld();
                release(2);
#pragma unroll
                for (int c = 0; c < 64; ++c) {
                    float er;
                    s[c] = __float_as_uint(zd_2sum(__uint_as_float(s[c]), __uint_as_float(e[c]), er));
                    e[c] = __float_as_uint(er);
                }
#pragma unroll
                for (int c0 = 0; c0 < 64; c0 += 16) {
                    const uint32_t tc = ta + ((uint32_t)(c0 >> 5) << 20) + (c0 & 16) * 2;
                    uint32_t v[32];
                    GW_TMEM_LD_16X256_X4(tc + kZdAcc, v);
                    GW_TMEM_LD_16X256_X4(tc, v + 16);
                    tmem_wait_ld();
                    if (c0 == 48) {
                        release(1);
                        if (lane == 0) bar_arrive(&tEmpty[0]);
                    }
#pragma unroll
                    for (int g = 0; g < 2; ++g)
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            float er;
                            s[c0 + c] =
                                __float_as_uint(zd_2sum(__uint_as_float(v[16 * g + c]), __uint_as_float(s[c0 + c]), er));
                            e[c0 + c] = __float_as_uint(__fadd_rn(__uint_as_float(e[c0 + c]), er));
                        }
                }
                const int64_t unit0 = ((int64_t)l * a.vb + (int64_t)vt * a.CT) * a.cb;
                const int r0 = mt * kZdM + q4 * 32 + (lane >> 2);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int2 cp = ctab[half * 32 + 4 * j + (lane & 3)];
#pragma unroll
                    for (int i = 0; i < 4; ++i) { // rows r0 + 8 i
                        const int c = 32 * (i >> 1) + 4 * j + 2 * (i & 1), cl = r0 + 8 * i;
                        float h[2], y[2];
#pragma unroll
                        for (int m = 0; m < 2; ++m) {
                            const float t = __uint_as_float(e[c + m]), b = __uint_as_float(s[c + m]);
                            h[m] = __fadd_rn(b, t);
                            y[m] = __fsub_rn(t, __fsub_rn(h[m], b));
                        }
                        if (cp.x < vmax && cl < a.cb) {
                            const int64_t fi = (unit0 + cl) * a.K2P + cp.y;
                            if (!GW_IN(fi, (int64_t)a.lines * a.cb * a.vb * a.K2P, a.status)) continue;
                            a.F[fi] = make_float4(h[0], y[0], h[1], y[1]);
                        }
                    }
                }
            }
        }
        if (!ok && lane == 0) atomicOr(a.status, kStatusTimeout);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        if (warp == 0) {
            // ---- TMA: line tiles one unit ahead, row slices stage by stage
            if (lane == 0) {
                uint32_t it = 0, nu = 0, np = 0;
                const unsigned pbytes = (unsigned)a.CT * a.n * 16; // CT lines of N two-float points
                auto lines = [&](int u) {
                    if (u >= a.nunits) return;
                    const uint32_t ps = np % kZdPsiSlots;
                    if (!bar_wait(&pEmpty[ps], ((np / kZdPsiSlots) & 1) ^ 1)) {
                        ok = false;
                        return;
                    }
                    const int l = u / a.nvt, vt = u - l * a.nvt;
                    bar_expect(&pFull[ps], pbytes);
                    tma3(ring + ps * rst, &a.tmV, &pFull[ps], 0, l * a.lsplit, a.v0 + vt * a.CT);
                    ++np;
                };
                lines(blockIdx.x);
                for (int u = blockIdx.x; u < a.nunits && ok; u += gridDim.x, ++nu) {
                    lines(u + gridDim.x);
                    const unsigned char *src = a.A + (int64_t)(u / a.nvt) * a.nmt * nst * kZdStage;
                    for (int j = 0; j < a.nmt * nst && ok; ++j, ++it) {
                        const uint32_t as = it % ast;
                        if (!bar_wait(&aEmpty[as], ((it / ast) & 1) ^ 1)) { ok = false; break; }
                        bar_expect(&aFull[as], kZdStage);
                        bulk_copy(sA + as * kZdStage, src + (int64_t)j * kZdStage, kZdStage, &aFull[as]);
                    }
                }
                // every copy has landed before the block may leave
                for (uint32_t j = it > ast ? it - ast : 0; j < it; ++j) bar_wait(&aFull[j % ast], (j / ast) & 1);
                for (uint32_t j = np > kZdPsiSlots ? np - kZdPsiSlots : 0; j < np; ++j)
                    bar_wait(&pFull[j % kZdPsiSlots], (j / kZdPsiSlots) & 1);
                if (!ok) atomicOr(a.status, kStatusTimeout);
            }
        } else if (warp == 1) {
            // ---- MMA issue, the warp converged (umma_f16_run)
            {
                const uint32_t lead = elect_lane(), tb = __shfl_sync(0xffffffffu, tbase, 0);
                auto wait = [&](uint64_t *b, uint32_t parity) {
                    if (!__all_sync(0xffffffffu, bar_wait(b, parity))) ok = false;
                };
                // The pipe holds few products, so what this warp does between two stages shows: a
                // stage's barriers are awaited between the products of the stage before.
                // descriptor address fields count 16-byte units: offsets below 256 KB add in place
                const uint32_t ad0 = sdesc_sw32_low(su32(sA)), bd0 = sdesc_sw32_low(su32(sB));
                uint32_t as = 0, ph = 0, tph = 1, nu = 0;
                if (blockIdx.x < a.nunits) {
                    wait(&bFull[0], 0);
                    wait(&aFull[0], 0);
                }
                tc_fence_after();
                for (int u = blockIdx.x; u < a.nunits && ok; u += gridDim.x, ++nu) {
                    const bool more = u + (int)gridDim.x < a.nunits;
                    for (int mt = 0; mt < a.nmt && ok; ++mt, tph ^= 1) {
                        const bool last = mt == a.nmt - 1;
                        // The 21 products of a stage, unrolled, descriptors advanced by constant offsets.
                        // A tile's first two stages go together, accumulator by accumulator as the
                        // epilogue hands them back (the least significant, with 15 products, first);
                        // a group's first product of the tile starts its accumulator.
                        // products of A slice i with the B slices j0 .. j1, one after the other: A is read once
                        auto run = [&](int i, int j0, int j1, uint32_t ad, uint32_t bd, uint32_t acc0) {
#pragma unroll
                            for (int j = 0; j < kZdSlices; ++j)
                                if (j >= j0 && j <= j1) {
                                    const int g = i + j < 3 ? i + j : 3;
                                    umma_f16_run(lead, tb + g * kZdAcc, ad + (uint32_t)((i * kZdSlice) >> 4),
                                                 bd + (uint32_t)((j * kBSlice) >> 4), kSdescSw32High, kIdesc,
                                                 i == 0 && j == g ? acc0 : 1u, j - j0, j1 - j0 + 1);
                                }
                        };
                        auto issue = [&](int g, uint32_t ad, uint32_t bd, uint32_t acc0) {
#pragma unroll
                            for (int i = 0; i < kZdSlices; ++i)
                                if (g == 3) run(i, i < 3 ? 3 - i : 0, kZdSlices - 1 - i, ad, bd, acc0);
                                else if (i <= g) run(i, g - i, g - i, ad, bd, acc0);
                        };
                        auto advance = [&] {
                            if (++as == ast) {
                                as = 0;
                                ph ^= 1;
                            }
                        };
                        auto await = [&](bool newb, int ks, uint32_t unit) { // stage ks of this unit or the next
                            if (newb) wait(&bFull[ks], unit & 1);
                            wait(&aFull[as], ph);
                            tc_fence_after();
                        };
                        {
                            const uint32_t s0 = as;
                            const uint32_t a0 = ad0 + (uint32_t)((s0 * kZdStage) >> 4);
                            advance();
                            const uint32_t s1 = as;
                            const uint32_t a1 = ad0 + (uint32_t)((s1 * kZdStage) >> 4), b1 = bd0 + (kBStage >> 4);
                            wait(&tEmpty[3], tph);
                            tc_fence_after();
                            issue(3, a0, bd0, 0u);
                            await(mt == 0, 1, nu);
                            wait(&tEmpty[2], tph);
                            tc_fence_after();
                            issue(2, a0, bd0, 0u);
                            issue(3, a1, b1, 1u);
                            issue(2, a1, b1, 1u);
                            wait(&tEmpty[1], tph);
                            wait(&tEmpty[0], tph);
                            tc_fence_after();
                            issue(1, a0, bd0, 0u);
                            issue(0, a0, bd0, 0u);
                            umma_commit_lead(lead, &aEmpty[s0]);
                            if (last) umma_commit_lead(lead, &bEmpty[0]);
                            issue(1, a1, b1, 1u);
                            advance();
                            await(mt == 0, 2, nu);
                            issue(0, a1, b1, 1u);
                            umma_commit_lead(lead, &aEmpty[s1]);
                            if (last) umma_commit_lead(lead, &bEmpty[1]);
                        }
                        for (int ks = 2; ks < nst && ok; ++ks) {
                            const uint32_t ad = ad0 + (uint32_t)((as * kZdStage) >> 4);
                            const uint32_t bd = bd0 + (uint32_t)((ks * kBStage) >> 4);
                            const uint32_t cur = as;
                            advance();
                            run(0, 0, 5, ad, bd, 1u);
                            run(1, 0, 4, ad, bd, 1u);
                            // the next stage: of this tile, of the next tile or of the next unit
                            if (ks + 1 < nst) await(mt == 0, ks + 1, nu);
                            else if (!last || more) await(last, 0, nu + 1);
                            run(2, 0, 3, ad, bd, 1u);
                            run(3, 0, 2, ad, bd, 1u);
                            run(4, 0, 1, ad, bd, 1u);
                            run(5, 0, 0, ad, bd, 1u);
                            umma_commit_lead(lead, &aEmpty[cur]);
                            if (last) umma_commit_lead(lead, &bEmpty[ks]);
                        }
                        umma_commit_lead(lead, tFull);
                    }
                }
                umma_commit_lead(lead, fin);
                wait(fin, 0);
                if (!ok && lead) atomicOr(a.status, kStatusTimeout);
            }
        } else {
            // ---- producers: column slices of the valence tile, stage by stage.  A lane owns point
            // i2 = 8 ks + k2 (k2 = lane % 8) of up to three (band, frequency) pairs, the same in every
            // stage and unit.
            const int pw = warp < 4 ? warp - 2 : warp - 10, k2 = lane & 7, npair = a.CT * a.K2;
            int vl[kZdRounds], col[kZdRounds], w0[kZdRounds], dw[kZdRounds]; // twiddle index, its step per stage
#pragma unroll
            for (int j = 0; j < kZdRounds; ++j) {
                const int p = (j * kZdProducers + pw) * 4 + (lane >> 3);
                vl[j] = p < npair ? p / a.K2 : -1;
                const int q = p < npair ? p - vl[j] * a.K2 : 0, kz = a.kz[q];
                col[j] = vl[j] * ncol + 2 * q;
                w0[j] = (kz * k2) % a.n;
                dw[j] = (kz * 8) % a.n;
            }
            uint32_t nu = 0;
            for (int u = blockIdx.x; u < a.nunits && ok; u += gridDim.x, ++nu) {
                const int l = u / a.nvt, vt = u - l * a.nvt;
                const uint32_t ps = nu % kZdPsiSlots;
                const bool pgot = bar_wait(&pFull[ps], (nu / kZdPsiSlots) & 1);
                if (!__all_sync(0xffffffffu, pgot)) { ok = false; break; }
                const float4 *pl = ring + ps * rst;
                int E[kZdRounds], w[kZdRounds];
#pragma unroll
                for (int j = 0; j < kZdRounds; ++j) {
                    const int v = vt * a.CT + vl[j];
                    w[j] = w0[j];
                    E[j] = vl[j] >= 0 && v < a.vb ? __ldg(a.E + (int64_t)(a.v0 + v) * a.lines + l) : -70;
                }
                for (int ks = 0; ks < nst; ++ks) {
                    const bool got = bar_wait(&bEmpty[ks], (nu & 1) ^ 1);
                    if (!__all_sync(0xffffffffu, got)) { ok = false; break; } // warp-uniform exit
                    unsigned char *B = sB + ks * kBStage;
#pragma unroll
                    for (int j = 0; j < kZdRounds; ++j) {
                        if (vl[j] < 0) continue;
                        const int i2 = ks * 8 + k2;
                        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (i2 < a.n && vt * a.CT + vl[j] < a.vb) x = pl[vl[j] * a.n + i2];
                        const tcx b = tc_mulc(tcx{{x.x, x.y}, {x.z, x.w}}, tc_load(wt + w[j])); // conj(x) W
                        w[j] += dw[j];
                        if (w[j] >= a.n) w[j] -= a.n;
                        uint16_t dr[kZdSlices], di[kZdSlices];
                        zd_digits_n(b.re.hi, b.re.lo, E[j], dr);
                        zd_digits_n(b.im.hi, b.im.lo, E[j], di);
                        const int colr = col[j];
                        if (!GW_IN(colr + 1, NT, a.status)) continue;
                        // rows (Re c, Im c): Re column (Re b, -Im b); Im column (Im b, Re b).  The lanes of
                        // pairs 2 and 3 store their Im column first: the four pairs' columns, 64 bytes
                        // apart, would share banks two by two
                        const bool im = (lane & 16) != 0;
                        unsigned char *p0 = B + sw32_off(colr + im, 2 * k2), *p1 = B + sw32_off(colr + !im, 2 * k2);
#pragma unroll
                        for (int sl = 0; sl < kZdSlices; ++sl) {
                            const uint32_t vr = (uint32_t)dr[sl] | ((uint32_t)(di[sl] ^ 0x8000u) << 16);
                            const uint32_t vi = (uint32_t)di[sl] | ((uint32_t)dr[sl] << 16);
                            *(uint32_t *)(p0 + sl * kBSlice) = im ? vi : vr;
                            *(uint32_t *)(p1 + sl * kBSlice) = im ? vr : vi;
                        }
                    }
                    fence_async_shared();
                    __syncwarp();
                    if (lane == 0) bar_arrive(&bFull[ks]);
                }
                if (lane == 0) bar_arrive(&pEmpty[ps]);
            }
            if (!ok && lane == 0) atomicOr(a.status, kStatusTimeout);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tbase, 512);
}

// Entries of F per (row, line): the kept frequencies, padded to whole 32-byte sectors.
int zd_row_entries(int K2) { return (K2 + 1) / 2 * 2; }

static int zd_bands(int nt, int K2) { return std::max(1, std::min(6, nt / (2 * zd_row_entries(K2)))); }

static size_t zd_smem(int n, int K2, int nt, int ast)
{
    return 1024 + ast * (size_t)kZdStage + zd_stages(n) * (size_t)(kZdSlices * nt * kZdKB * 2) +
           16 * (size_t)kZdPsiSlots * zd_ring_stride(zd_bands(nt, K2), n) + 16 * (size_t)n + 8 * 64 + 8 * 48 + 64;
}

// The tile's columns (128, or 96 for long lines) and the stages of the row ring: what shared memory
// holds (48-point lines: 128 columns, three stages; 72: 96 columns, two).  False: neither fits.
static bool zd_shape(int n, int K2, int &nt, int &ast)
{
    const size_t room = (size_t)227 * 1024;
    for (nt = 128; nt >= 96; nt -= 32)
        if (2 * zd_row_entries(K2) <= nt && zd_smem(n, K2, nt, 2) <= room) {
            for (ast = kZdMaxRing; zd_smem(n, K2, nt, ast) > room; --ast) {}
            return true;
        }
    return false;
}

// The route's shapes: lines of 24 to 72 points (at least three stages; 3 * 144 * 2^14 < 2^24), at most
// 32 kept frequencies.
bool zd_supported(int n, int K2)
{
    int nt, ast;
    return n >= 24 && n <= 8 * kZdMaxStages && n % zd_line_split(n) == 0 && K2 >= 1 && K2 <= 32 &&
           zd_shape(n, K2, nt, ast);
}

// A tensor map's box takes 256 entries: longer lines (4 n FP32) are mapped as two.
int zd_line_split(int n) { return n > 64 ? 2 : 1; }

int zd_valence_per_tile(int n, int K2)
{
    int nt = 128, ast = 2;
    zd_shape(n, K2, nt, ast);
    return zd_bands(nt, K2);
}

cudaError_t launch_zd_gemm(const CUtensorMap &tmV, const void *A, const int *E, const int *kz, const float4 *twf, int n,
                           int lines, int nv, int v0, int vb, int cb, int K2, float4 *F, int *status, cudaStream_t st)
{
    ZdArgs a;
    int nt;
    if (!zd_shape(n, K2, nt, a.ast)) return cudaErrorInvalidValue;
    a.tmV = tmV;
    a.A = (const unsigned char *)A;
    a.E = E;
    a.kz = kz;
    a.F = F;
    a.status = status;
    a.n = n;
    a.lines = lines;
    a.lsplit = zd_line_split(n);
    a.nv = nv;
    a.v0 = v0;
    a.vb = vb;
    a.cb = cb;
    a.K2 = K2;
    a.K2P = zd_row_entries(K2);
    a.CT = zd_bands(nt, K2);
    a.nvt = (vb + a.CT - 1) / a.CT;
    a.nmt = (cb + kZdM - 1) / kZdM;
    a.nunits = lines * a.nvt;
    const size_t sm = zd_smem(n, K2, nt, a.ast);
    auto kernel = nt == 96 ? zd_gemm_kernel<96> : zd_gemm_kernel<128>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    kernel<<<std::min(a.nunits, sms), kZdThreads, sm, st>>>(a, twf);
    return cudaGetLastError();
}

} // namespace gw
