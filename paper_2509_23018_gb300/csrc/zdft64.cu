// Stage (a), last-axis transform of the pair products on the BF16 tensor cores to FP64 accuracy.
//
// The product of zdft.cu (line by line, rows psi_c, columns W_q conj(psi_v), K = Re and Im of a line's
// points), with operands cut into seven balanced base-512 digits relative to the line's largest entry:
// x = 2^(E - 62) sum_{i<7} 512^(6-i) d_i, 62 bits where a double keeps 53 of each entry.  The slices hold
// the digits themselves (|d_0| <= 128, |d_i| <= 256, exact in BF16), so every accumulator holds whole
// numbers; the products with i + j <= 6 are kept, summed over at most 112 real entries in FP32: one
// accumulator per i + j, and for lines of more than 32 points two for i + j = 3 (d_1 d_2 and d_2 d_1, the
// others) and i + j = 4 (d_1 d_3 and d_3 d_1, the others), so that the sums for i + j <= 4 stay within 2^24
// (at most 64 2^18 and 112 2^17) and are exact whatever the digits.  i + j = 5 and 6 (112 5 2^16, 112 6 2^16) may be rounded by up to 4 in each of their
// 42 and 49 MMA steps where a line's digits are all near their largest with one sign: 2^-51 of the operands'
// largest product at most.  The epilogue adds them as 64-bit integers in units of 2^-40 of the leading
// group (|sum| < 2^62), 2^-54 of the operands' largest product, and rounds once, to the double
//     F = acc 2^(E_row + E_col - 56).
#include "internal.h"
#include "ptx.cuh"
#include "oz_digits.cuh"
#include "zd_tiles.cuh"

#include <algorithm>

namespace gw {

constexpr int kQdSlices = 7;
constexpr int kQdN = 96;                             // columns per tile
constexpr int kQdMaxStages = 7;                      // lines of up to 56 points
constexpr unsigned kQdASlice = kZdM * kZdKB * 2;     // 4 KB
constexpr unsigned kQdAStage = kQdSlices * kQdASlice; // 28 KB
constexpr unsigned kQdBSlice = kQdN * kZdKB * 2;     // 3 KB
constexpr unsigned kQdBStage = kQdSlices * kQdBSlice; // 21 KB
constexpr int kQdNoLine = -400, kQdMaxExpo = 390;    // exponent of a zero line; those the scaling takes
// idesc: D = F32, A = B = BF16, both K-major, N = 96, M = 128
constexpr uint32_t kQdIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kQdN >> 3) << 17) |
                              ((uint32_t)(kZdM >> 4) << 24);

// the seven digits of x 2^(62 - E), as BF16
__device__ __forceinline__ void qd_digits(double x, int E, uint16_t out[kQdSlices])
{
    const long long nb = oz_round_scaled(x, 62 - E) + oz_digit_bias<9>(kQdSlices);
    out[0] = oz_small_bf16((int)(nb >> 54));
#pragma unroll
    for (int i = 1; i < kQdSlices; ++i) out[i] = oz_small_bf16((int)((nb >> (9 * (kQdSlices - 1 - i))) & 511) - 256);
}

// exponent of a line (|x| < 2^(E - 1)) from the bits of its largest magnitude; sets *guard where the
// scaling does not hold
__device__ __forceinline__ int qd_expo(unsigned long long m, int *guard)
{
    const int E = oz_expo_bits(m, kQdNoLine);
    if (m != 0 && (E > kQdMaxExpo || E < -kQdMaxExpo)) {
        *guard = 1;
        return kQdNoLine;
    }
    return E;
}

// ------------------------------------------------------------------ row slices and column exponents
// A[l][mt][ks][slice] as in zd_rows_kernel, the rows' exponents ER[l][128 nmt] behind it: one warp per row.
__global__ void __launch_bounds__(256) zd64_rows_kernel(const double2 *__restrict__ psi, int nr, int n, int nlines,
                                                        int nmt, unsigned char *__restrict__ A, int *__restrict__ ER,
                                                        int *guard)
{
    const int lane = threadIdx.x & 31, l = blockIdx.y, r = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int nst = zd_stages(n);
    unsigned char *dst = A + ((int64_t)l * nmt + r / kZdM) * nst * kQdAStage;
    const int rt = r % kZdM;
    const double2 *row = psi + ((int64_t)min(r, nr - 1) * nlines + l) * n;
    unsigned long long m = 0;
    double2 x[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int i = lane + 32 * u;
        x[u] = i < n && r < nr ? row[i] : make_double2(0.0, 0.0);
        m = max(m, oz_absmax_bits(x[u].x, x[u].y));
    }
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    const int E = qd_expo(m, guard);
    if (lane == 0) ER[(int64_t)l * nmt * kZdM + r] = E;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int i = lane + 32 * u;
        if (i >= 8 * nst) break;
        uint16_t dr[kQdSlices], di[kQdSlices];
        qd_digits(x[u].x, E, dr);
        qd_digits(x[u].y, E, di);
        unsigned char *p = dst + (i >> 3) * kQdAStage + sw32_off(rt, 2 * (i & 7));
#pragma unroll
        for (int s = 0; s < kQdSlices; ++s)
            *(uint32_t *)(p + s * kQdASlice) = (uint32_t)dr[s] | ((uint32_t)di[s] << 16);
    }
}

// E[band][l] of a line's columns: |W_q psi| <= |Re psi| + |Im psi|
__global__ void __launch_bounds__(256) zd64_colexp_kernel(const double2 *__restrict__ psi, int nb, int n, int nlines,
                                                          int *__restrict__ E, int *guard)
{
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= (int64_t)nb * nlines) return;
    unsigned long long m = 0;
    for (int i = lane; i < n; i += 32) {
        const double2 x = psi[w * n + i];
        m = max(m, oz_dbits(fabs(x.x) + fabs(x.y)));
    }
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    const int e = qd_expo(m, guard);
    if (lane == 0) E[w] = e;
}

// ------------------------------------------------------------------ the product
// As zd_gemm_kernel: one block per SM, persistent over units (line, valence tile of CT bands), the
// column stages resident, the row stages through a ring.  A tile of 128 conduction bands x 96 columns
// runs in two passes over K, because its seven or nine accumulators of 96 columns do not fit in TMEM, five do: first the
// groups i + j = 6, 5, 4 (18 products a stage), then 3..0 (10 products, for which four of a row stage's
// seven slices are loaded; the second pass starts in the accumulator that the first leaves free).  The
// epilogue keeps the sums as 64-bit integers in between.
//  warps 0..3: TMA, MMA (and TMEM), two producers; warps 4..11: epilogue (TMEM lane quadrant
//  warp % 4, half of the columns each); warps 12..15: producers.
//
// 4.87 ms for 8192 pairs on 48^3 (8 x 1024 bands, K2 = 15), of which the products take 1.8 (4.32 with one
// accumulator per i + j, which leaves up to 3e-14 of an element where a line's digits have one sign); the
// FFT pair kernel spends most of its 55 ms on this axis, on the FP64 pipe.  The epilogue uses no FP64 instruction:
// converting and scaling 96 x 128 sums there would take longer than the tile's products.
constexpr int kQdThreads = 512;
constexpr int kQdProducers = 6;
constexpr int kQdPsiSlots = 2;
constexpr int kQdMaxRing = 3;
constexpr int kQdRounds = 2; // (band, frequency) pairs per producer lane: 48 pairs, 6 warps x 4

template <int V>
struct QdInt {
    static constexpr int value = V;
};

struct Qd64Args {
    CUtensorMap tmV;        // valence grids as FP32 [nv][lines][4N], box {4N, 1, CT}
    const unsigned char *A; // row slices of the block's cb conduction bands
    const int *ER;          // [lines][128 nmt] their exponents
    const int *E;           // [nv][lines] column exponents
    const int *kz;          // [K2] kept last-axis frequencies
    double2 *F;             // [lines][vb cb][K2P], row vl cb + cl
    const int *guard;
    int *status;
    int n, lines, nv, v0, vb, cb, K2, K2P, CT, nvt, nmt, nunits, ast;
};

// accumulator slot of the product d_i d_j.  First pass: i + j = 6, 5 in 0, 1 and 4 in 2; second pass: 3 in 4,
// then 2, 1, 0 in 0, 1, 2.  TWO: slot 3 takes d_0 d_4, d_2 d_2, d_4 d_0 in the first pass and d_0 d_3, d_3 d_0
// in the second.
constexpr int kQdSlots = 5;
template <bool TWO>
__device__ constexpr int qd_slot(int i, int j)
{
    const int g = i + j;
    if (TWO && (g == 4 ? i != 1 && i != 3 : g == 3 && i != 1 && i != 2)) return 3;
    return g == 3 ? 4 : g > 3 ? 6 - g : 2 - g;
}

// m 2^ex, m a 64-bit integer, rounded to a double from the bits (the FP64 pipe would take 2 clocks of
// the SM for each)
__device__ __forceinline__ double qd_double(long long v, int ex)
{
    const unsigned long long m0 = (unsigned long long)(v < 0 ? -v : v);
    if (m0 == 0) return 0.0;
    const int lz = __clzll((long long)m0);
    const unsigned long long m = m0 << lz;
    const unsigned long long b = ((unsigned long long)(1022 + 63 - lz + ex) << 52) + (m >> 11) + ((m >> 10) & 1ull);
    return __longlong_as_double((long long)(b | ((unsigned long long)v & 0x8000000000000000ull)));
}

template <bool TWO>
__global__ void __launch_bounds__(kQdThreads, 1) zd64_gemm_kernel(const __grid_constant__ Qd64Args a,
                                                                  const double2 *__restrict__ twg)
{
    if (*a.guard) return; // the FFT pair kernel takes the block
    extern __shared__ __align__(1024) unsigned char smraw[];
    unsigned char *sm = (unsigned char *)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
    const int nst = zd_stages(a.n), ncol = 2 * a.K2P;
    const uint32_t ast = a.ast;
    unsigned char *sA = sm;                             // ast x 28 KB
    unsigned char *sB = sA + ast * kQdAStage;           // nst x 21 KB
    double2 *ring = (double2 *)(sB + nst * kQdBStage);  // [slots][CT][N] valence line tiles
    const int rst = zd_ring_stride(a.CT, a.n);
    double2 *wt = ring + kQdPsiSlots * rst;             // [N] twiddles W^t
    int2 *ctab = (int2 *)(wt + a.n);                    // [48] column pair -> (band, F offset)
    uint64_t *bar = (uint64_t *)(ctab + kQdN / 2);
    uint64_t *aFull = bar, *aEmpty = aFull + kQdMaxRing, *bFull = aEmpty + kQdMaxRing, *bEmpty = bFull + kQdMaxStages,
             *tFull = bEmpty + kQdMaxStages, *tEmpty = tFull + 1, *pFull = tEmpty + kQdSlots, *pEmpty = pFull + kQdPsiSlots,
             *fin = pEmpty + kQdPsiSlots;
    uint32_t *tslot = (uint32_t *)(fin + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < a.n; i += blockDim.x) wt[i] = twg[i];
    for (int pi = threadIdx.x; pi < kQdN / 2; pi += blockDim.x) {
        const int vl = pi / a.K2P, q = pi - vl * a.K2P;
        ctab[pi] = make_int2(vl, vl * a.cb * a.K2P + q);
    }
    // columns that no frequency fills stay zero in every stage
    for (int i = threadIdx.x; i < nst * (int)kQdBStage / 16; i += blockDim.x)
        ((uint4 *)sB)[i] = make_uint4(0u, 0u, 0u, 0u);
    fence_async_shared();
    if (threadIdx.x == 0) {
        for (int i = 0; i < kQdMaxRing; ++i) {
            bar_init(&aFull[i], 1);
            bar_init(&aEmpty[i], 1);
        }
        for (int i = 0; i < kQdMaxStages; ++i) {
            bar_init(&bFull[i], kQdProducers);
            bar_init(&bEmpty[i], 1);
        }
        bar_init(tFull, 1);
        for (int i = 0; i < kQdSlots; ++i) bar_init(&tEmpty[i], 8);
        for (int i = 0; i < kQdPsiSlots; ++i) {
            bar_init(&pFull[i], 1);
            bar_init(&pEmpty[i], kQdProducers);
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

    // registers: 512 x 128 at launch, 176 for the epilogue warps, 80 for the other two warpgroups
    if (warp >= 4 && warp < 12) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 176;");
        // ---- epilogue: a quadrant's 32 rows (conduction bands) x 48 of the 96 columns per warp, in the
        // 16 x 256-bit load shape (see zd_gemm_kernel): registers 24 h + 4 j + 2 i + {0, 1} are row
        // 16 h + 8 i + lane / 4, entry 4 j + lane % 4
        const int q4 = warp & 3, half = (warp - 4) >> 2;
        const uint32_t ta = tbase + ((uint32_t)(q4 * 32) << 16) + half * (kQdN / 2);
        auto load = [&](int slot, uint32_t v[48]) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t t = ta + slot * kQdN + ((uint32_t)(16 * h) << 16);
                GW_TMEM_LD_16X256_X4(t, v + 24 * h);
                GW_TMEM_LD_16X256_X2(t + 32, v + 24 * h + 16);
            }
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive(&tEmpty[slot]);
        };
        // acc += (slot s0 + slot s1) mul, half of the rows at a time
        auto both = [&](int s0, int s1, uint32_t v[48], long long acc[48], int mul) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t t0 = ta + s0 * kQdN + ((uint32_t)(16 * h) << 16), t1 = t0 + (s1 - s0) * kQdN;
                GW_TMEM_LD_16X256_X4(t0, v);
                GW_TMEM_LD_16X256_X2(t0 + 32, v + 16);
                GW_TMEM_LD_16X256_X4(t1, v + 24);
                GW_TMEM_LD_16X256_X2(t1 + 32, v + 40);
                tmem_wait_ld();
                if (h == 1) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        bar_arrive(&tEmpty[s0]);
                        bar_arrive(&tEmpty[s1]);
                    }
                }
#pragma unroll
                for (int c = 0; c < 24; ++c)
                    acc[24 * h + c] += (long long)(__float2int_rn(__uint_as_float(v[c])) +
                                                   __float2int_rn(__uint_as_float(v[24 + c]))) * mul;
            }
        };
        for (int u = blockIdx.x; u < a.nunits && ok; u += gridDim.x) {
            const int l = u / a.nvt, vt = u - l * a.nvt;
            const int vmax = min(a.CT, a.vb - vt * a.CT);
            for (int mt = 0; mt < a.nmt; ++mt) {
                long long acc[48];
                uint32_t v[48];
                bool got = bar_wait(tFull, 0);
                if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                tc_fence_after();
                load(0, v); // i + j = 6
#pragma unroll
                for (int c = 0; c < 48; ++c) acc[c] = __float2int_rn(__uint_as_float(v[c]));
                load(1, v); // 5
#pragma unroll
                for (int c = 0; c < 48; ++c) {
                    acc[c] += (long long)__float2int_rn(__uint_as_float(v[c])) * 512;
                    acc[c] = (acc[c] + (1 << 13)) >> 14; // units of 2^-40
                }
                if constexpr (TWO) both(2, 3, v, acc, 16); // 4
                else {
                    load(2, v);
#pragma unroll
                    for (int c = 0; c < 48; ++c) acc[c] += (long long)__float2int_rn(__uint_as_float(v[c])) * 16;
                }
                got = bar_wait(tFull, 1);
                if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                tc_fence_after();
                load(0, v); // 2
#pragma unroll
                for (int c = 0; c < 48; ++c) acc[c] += (long long)__float2int_rn(__uint_as_float(v[c])) * (1 << 22);
                load(1, v); // 1
#pragma unroll
                for (int c = 0; c < 48; ++c) acc[c] += ((long long)__float2int_rn(__uint_as_float(v[c]))) * (1ll << 31);
                load(2, v); // 0
#pragma unroll
                for (int c = 0; c < 48; ++c) acc[c] += (long long)__float2int_rn(__uint_as_float(v[c]) * 256.0f) << 32;
                if constexpr (TWO) both(3, 4, v, acc, 1 << 13); // 3
                else {
                    load(4, v);
#pragma unroll
                    for (int c = 0; c < 48; ++c) acc[c] += (long long)__float2int_rn(__uint_as_float(v[c])) * (1 << 13);
                }

                const int64_t unit0 = ((int64_t)l * a.vb + (int64_t)vt * a.CT) * a.cb;
                const int r0 = mt * kZdM + q4 * 32 + (lane >> 2);
                int er[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) er[i] = __ldg(a.ER + (int64_t)l * a.nmt * kZdM + r0 + 8 * i) - 56;
#pragma unroll
                for (int j = 0; j < 6; ++j) {
                    const int2 cp = ctab[half * 24 + 4 * j + (lane & 3)];
                    if (cp.x >= vmax) continue;
                    const int ec = __ldg(a.E + (int64_t)(a.v0 + vt * a.CT + cp.x) * a.lines + l);
#pragma unroll
                    for (int i = 0; i < 4; ++i) { // rows r0 + 8 i
                        const int c = 24 * (i >> 1) + 4 * j + 2 * (i & 1), cl = r0 + 8 * i;
                        if (cl < a.cb) {
                            const int64_t fi = (unit0 + cl) * a.K2P + cp.y;
                            if (!GW_IN(fi, (int64_t)a.lines * a.cb * a.vb * a.K2P, a.status)) continue;
                            a.F[fi] = make_double2(qd_double(acc[c], er[i] + ec), qd_double(acc[c + 1], er[i] + ec));
                        }
                    }
                }
            }
        }
        if (!ok && lane == 0) atomicOr(a.status, kStatusTimeout);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        if (warp == 0) {
            // ---- TMA: line tiles one unit ahead, row slices stage by stage, pass by pass
            if (lane == 0) {
                uint32_t as = 0, ph = 1, it = 0, np = 0;
                const unsigned pbytes = (unsigned)a.CT * a.n * 16;
                auto lines = [&](int u) {
                    if (u >= a.nunits) return;
                    const uint32_t ps = np % kQdPsiSlots;
                    if (!bar_wait(&pEmpty[ps], ((np / kQdPsiSlots) & 1) ^ 1)) {
                        ok = false;
                        return;
                    }
                    const int l = u / a.nvt, vt = u - l * a.nvt;
                    bar_expect(&pFull[ps], pbytes);
                    tma3(ring + ps * rst, &a.tmV, &pFull[ps], 0, l, a.v0 + vt * a.CT);
                    ++np;
                };
                lines(blockIdx.x);
                for (int u = blockIdx.x; u < a.nunits && ok; u += gridDim.x) {
                    lines(u + gridDim.x);
                    const unsigned char *src = a.A + (int64_t)(u / a.nvt) * a.nmt * nst * kQdAStage;
                    for (int mt = 0; mt < a.nmt && ok; ++mt, src += nst * kQdAStage)
                        for (int ps = 0; ps < 2 && ok; ++ps) {
                            const unsigned bytes = (ps == 0 ? kQdSlices : 4) * kQdASlice;
                            for (int ks = 0; ks < nst; ++ks, ++it) {
                                if (!bar_wait(&aEmpty[as], ph)) { ok = false; break; }
                                bar_expect(&aFull[as], bytes);
                                bulk_copy(sA + as * kQdAStage, src + ks * kQdAStage, bytes, &aFull[as]);
                                if (++as == ast) {
                                    as = 0;
                                    ph ^= 1;
                                }
                            }
                        }
                }
                // every copy has landed before the block may leave
                for (uint32_t j = it > ast ? it - ast : 0; j < it; ++j) bar_wait(&aFull[j % ast], (j / ast) & 1);
                for (uint32_t j = np > kQdPsiSlots ? np - kQdPsiSlots : 0; j < np; ++j)
                    bar_wait(&pFull[j % kQdPsiSlots], (j / kQdPsiSlots) & 1);
                if (!ok) atomicOr(a.status, kStatusTimeout);
            }
        } else if (warp == 1) {
            // ---- MMA issue, the warp converged (umma_f16_run)
            {
                const uint32_t lead = elect_lane(), tb = __shfl_sync(0xffffffffu, tbase, 0);
                auto wait = [&](uint64_t *b, uint32_t parity) {
                    if (!__all_sync(0xffffffffu, bar_wait(b, parity))) ok = false;
                };
                const uint32_t ad0 = sdesc_sw32_low(su32(sA)), bd0 = sdesc_sw32_low(su32(sB));
                uint32_t as = 0, ph = 0, nu = 0;
                uint32_t e03 = 1, e4 = 1; // parities of the accumulators' next release: 0..2 (TWO: 3) every pass, 4 every tile
                if (blockIdx.x < a.nunits) {
                    wait(&bFull[0], 0);
                    wait(&aFull[0], 0);
                }
                tc_fence_after();
                // the products of group g in one slot, at a pass's first stage: the first starts the accumulator
                auto issue = [&](auto G, auto SLOT, uint32_t ad, uint32_t bd) {
                    constexpr int g = decltype(G)::value, slot = decltype(SLOT)::value;
                    uint32_t started = 0;
#pragma unroll
                    for (int i = 0; i <= g; ++i)
                        if (qd_slot<TWO>(i, g - i) == slot) {
                            umma_f16_run(lead, tb + slot * kQdN, ad + (uint32_t)((i * kQdASlice) >> 4),
                                         bd + (uint32_t)(((g - i) * kQdBSlice) >> 4), kSdescSw32High, kQdIdesc,
                                         started, 0, 1);
                            started = 1;
                        }
                };
                // A slice i with its B slices of the pass's groups g0 .. g1, one after the other: A is read once
                auto run = [&](int i, int g0, int g1, uint32_t ad, uint32_t bd) {
#pragma unroll
                    for (int j = 0; j < kQdSlices; ++j)
                        if (i + j >= g0 && i + j <= g1)
                            umma_f16_run(lead, tb + qd_slot<TWO>(i, j) * kQdN, ad + (uint32_t)((i * kQdASlice) >> 4),
                                         bd + (uint32_t)((j * kQdBSlice) >> 4), kSdescSw32High, kQdIdesc, 1u,
                                         j - (g0 > i ? g0 - i : 0), g1 - i + 1 - (g0 > i ? g0 - i : 0));
                };
                auto room = [&](int slot, uint32_t par) {
                    wait(&tEmpty[slot], par);
                    tc_fence_after();
                };
                for (int u = blockIdx.x; u < a.nunits && ok; u += gridDim.x, ++nu) {
                    const bool more = u + (int)gridDim.x < a.nunits;
                    for (int mt = 0; mt < a.nmt && ok; ++mt) {
                        const bool last = mt == a.nmt - 1;
                        for (int ps = 0; ps < 2 && ok; ++ps) {
                            for (int ks = 0; ks < nst && ok; ++ks) {
                                const uint32_t ad = ad0 + (uint32_t)((as * kQdAStage) >> 4);
                                const uint32_t bd = bd0 + (uint32_t)((ks * kQdBStage) >> 4);
                                const uint32_t cur = as;
                                if (++as == ast) {
                                    as = 0;
                                    ph ^= 1;
                                }
                                // the next stage's barriers are awaited between this stage's products
                                auto next = [&] {
                                    const bool wrap = ks + 1 == nst;
                                    if (wrap && ps == 1 && last && !more) return;
                                    const bool newb = wrap ? ps == 1 && last : ps == 0 && mt == 0;
                                    if (newb) wait(&bFull[wrap ? 0 : ks + 1], (wrap ? nu + 1 : nu) & 1);
                                    wait(&aFull[as], ph);
                                    tc_fence_after();
                                };
                                if (ks == 0 && ps == 0) {
                                    room(0, e03);
                                    issue(QdInt<6>{}, QdInt<0>{}, ad, bd);
                                    room(1, e03);
                                    issue(QdInt<5>{}, QdInt<1>{}, ad, bd);
                                    next();
                                    room(2, e03);
                                    issue(QdInt<4>{}, QdInt<2>{}, ad, bd);
                                    if constexpr (TWO) {
                                        room(3, e03);
                                        issue(QdInt<4>{}, QdInt<3>{}, ad, bd);
                                    }
                                } else if (ks == 0) {
                                    room(4, e4);
                                    issue(QdInt<3>{}, QdInt<4>{}, ad, bd);
                                    room(0, e03);
                                    issue(QdInt<2>{}, QdInt<0>{}, ad, bd);
                                    next();
                                    room(1, e03);
                                    issue(QdInt<1>{}, QdInt<1>{}, ad, bd);
                                    room(2, e03);
                                    issue(QdInt<0>{}, QdInt<2>{}, ad, bd);
                                    if constexpr (TWO) {
                                        room(3, e03);
                                        issue(QdInt<3>{}, QdInt<3>{}, ad, bd);
                                    }
                                } else if (ps == 0) {
#pragma unroll
                                    for (int i = 0; i < 4; ++i) run(i, 4, 6, ad, bd);
                                    next();
#pragma unroll
                                    for (int i = 4; i < 7; ++i) run(i, 4, 6, ad, bd);
                                } else {
                                    run(0, 0, 3, ad, bd);
                                    run(1, 0, 3, ad, bd);
                                    next();
                                    run(2, 0, 3, ad, bd);
                                    run(3, 0, 3, ad, bd);
                                }
                                if (ps == 1 && last) umma_commit_lead(lead, &bEmpty[ks]);
                                umma_commit_lead(lead, &aEmpty[cur]);
                            }
                            e03 ^= 1;
                            umma_commit_lead(lead, tFull);
                        }
                        e4 ^= 1;
                    }
                }
                umma_commit_lead(lead, fin);
                wait(fin, 0);
                if (!ok && lead) atomicOr(a.status, kStatusTimeout);
            }
        } else {
            // ---- producers: column slices of the valence tile, stage by stage.  A lane owns point
            // i2 = 8 ks + k2 (k2 = lane % 8) of up to two (band, frequency) pairs.
            const int pw = warp < 4 ? warp - 2 : warp - 10, k2 = lane & 7, npair = a.CT * a.K2;
            int vl[kQdRounds], col[kQdRounds], w0[kQdRounds], dw[kQdRounds];
#pragma unroll
            for (int j = 0; j < kQdRounds; ++j) {
                const int p = (j * kQdProducers + pw) * 4 + (lane >> 3);
                vl[j] = p < npair ? p / a.K2 : -1;
                const int q = p < npair ? p - vl[j] * a.K2 : 0, kz = a.kz[q];
                col[j] = vl[j] * ncol + 2 * q;
                w0[j] = (kz * k2) % a.n;
                dw[j] = (kz * 8) % a.n;
            }
            uint32_t nu = 0;
            for (int u = blockIdx.x; u < a.nunits && ok; u += gridDim.x, ++nu) {
                const int l = u / a.nvt, vt = u - l * a.nvt;
                const uint32_t ps = nu % kQdPsiSlots;
                const bool pgot = bar_wait(&pFull[ps], (nu / kQdPsiSlots) & 1);
                if (!__all_sync(0xffffffffu, pgot)) { ok = false; break; }
                const double2 *pl = ring + ps * rst;
                int E[kQdRounds], w[kQdRounds];
#pragma unroll
                for (int j = 0; j < kQdRounds; ++j) {
                    const int v = vt * a.CT + vl[j];
                    w[j] = w0[j];
                    E[j] = vl[j] >= 0 && v < a.vb ? __ldg(a.E + (int64_t)(a.v0 + v) * a.lines + l) : kQdNoLine;
                }
                for (int ks = 0; ks < nst; ++ks) {
                    const bool got = bar_wait(&bEmpty[ks], (nu & 1) ^ 1);
                    if (!__all_sync(0xffffffffu, got)) { ok = false; break; } // warp-uniform exit
                    unsigned char *B = sB + ks * kQdBStage;
#pragma unroll
                    for (int j = 0; j < kQdRounds; ++j) {
                        if (vl[j] < 0) continue;
                        const int i2 = ks * 8 + k2;
                        double2 x = make_double2(0.0, 0.0);
                        if (i2 < a.n && vt * a.CT + vl[j] < a.vb) x = pl[vl[j] * a.n + i2];
                        const double2 b = cmulc(x, wt[w[j]]); // conj(x) W
                        w[j] += dw[j];
                        if (w[j] >= a.n) w[j] -= a.n;
                        uint16_t dr[kQdSlices], di[kQdSlices];
                        qd_digits(b.x, E[j], dr);
                        qd_digits(b.y, E[j], di);
                        const int colr = col[j];
                        if (!GW_IN(colr + 1, kQdN, a.status)) continue;
                        // rows (Re c, Im c): Re column (Re b, -Im b); Im column (Im b, Re b), in the
                        // order that spreads the four pairs' stores over the banks (zd_gemm_kernel)
                        const bool im = (lane & 16) != 0;
                        unsigned char *p0 = B + sw32_off(colr + im, 2 * k2), *p1 = B + sw32_off(colr + !im, 2 * k2);
#pragma unroll
                        for (int sl = 0; sl < kQdSlices; ++sl) {
                            const uint32_t vr = (uint32_t)dr[sl] | ((uint32_t)(di[sl] ^ 0x8000u) << 16);
                            const uint32_t vi = (uint32_t)di[sl] | ((uint32_t)dr[sl] << 16);
                            *(uint32_t *)(p0 + sl * kQdBSlice) = im ? vi : vr;
                            *(uint32_t *)(p1 + sl * kQdBSlice) = im ? vr : vi;
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

// ------------------------------------------------------------------ host launchers
size_t zd64_row_bytes(int nr, int n, int lines)
{
    return (size_t)lines * ((nr + kZdM - 1) / kZdM) * (zd_stages(n) * (size_t)kQdAStage + kZdM * sizeof(int));
}

static int *zd64_row_expo(void *A, int nmt, int n, int lines)
{
    return (int *)((unsigned char *)A + (size_t)lines * nmt * zd_stages(n) * kQdAStage);
}

cudaError_t launch_zd64_rows(const void *psi, int nr, int n, int lines, void *A, int *guard, cudaStream_t st)
{
    const int nmt = (nr + kZdM - 1) / kZdM;
    zd64_rows_kernel<<<dim3(nmt * (kZdM / 8), lines), 256, 0, st>>>((const double2 *)psi, nr, n, lines, nmt,
                                                                    (unsigned char *)A,
                                                                    zd64_row_expo(A, nmt, n, lines), guard);
    return cudaGetLastError();
}

cudaError_t launch_zd64_colexp(const void *psi, int nb, int n, int lines, int *E, int *guard, cudaStream_t st)
{
    const int64_t warps = (int64_t)nb * lines;
    zd64_colexp_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>((const double2 *)psi, nb, n, lines, E, guard);
    return cudaGetLastError();
}

int zd64_valence_per_tile(int K2) { return std::max(1, std::min(6, kQdN / (2 * zd_row_entries(K2)))); }

static size_t zd64_smem(int n, int K2, int ast)
{
    return 1024 + ast * (size_t)kQdAStage + zd_stages(n) * (size_t)kQdBStage +
           16 * (size_t)kQdPsiSlots * zd_ring_stride(zd64_valence_per_tile(K2), n) + 16 * (size_t)n + 8 * (kQdN / 2) +
           8 * 40 + 64;
}

// Lines of 24 to 56 points (at least three stages; the column stages of longer ones leave no room for
// a ring of two row stages), at most 32 kept frequencies.
bool zd64_supported(int n, int K2)
{
    return n >= 24 && n <= 8 * kQdMaxStages && K2 >= 1 && K2 <= 32 && zd64_smem(n, K2, 2) <= (size_t)227 * 1024;
}

cudaError_t launch_zd64_gemm(const CUtensorMap &tmV, const void *A, const int *E, const int *kz, const double2 *tw, int n,
                             int lines, int nv, int v0, int vb, int cb, int K2, double2 *F, const int *guard,
                             int *status, cudaStream_t st)
{
    Qd64Args a;
    a.tmV = tmV;
    a.A = (const unsigned char *)A;
    a.E = E;
    a.kz = kz;
    a.F = F;
    a.guard = guard;
    a.status = status;
    a.n = n;
    a.lines = lines;
    a.nv = nv;
    a.v0 = v0;
    a.vb = vb;
    a.cb = cb;
    a.K2 = K2;
    a.K2P = zd_row_entries(K2);
    a.CT = zd64_valence_per_tile(K2);
    a.nvt = (vb + a.CT - 1) / a.CT;
    a.nmt = (cb + kZdM - 1) / kZdM;
    a.nunits = lines * a.nvt;
    a.ER = zd64_row_expo(const_cast<void *>(A), a.nmt, n, lines);
    a.ast = zd64_smem(n, K2, kQdMaxRing) <= (size_t)227 * 1024 ? kQdMaxRing : 2;
    const size_t sm = zd64_smem(n, K2, a.ast);
    // up to 64 real entries a sum for i + j = 4 (2^18 each at most) is exact
    auto kernel = 16 * zd_stages(n) > 64 ? zd64_gemm_kernel<true> : zd64_gemm_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    kernel<<<std::min(a.nunits, sms), kQdThreads, sm, st>>>(a, tw);
    return cudaGetLastError();
}

} // namespace gw
