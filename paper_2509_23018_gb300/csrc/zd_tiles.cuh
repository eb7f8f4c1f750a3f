// Operand tiles of the last-axis products of stage (a), two-float (zdft.cu) and FP64 (zdft64.cu).
#pragma once
#include "ptx.cuh"

namespace gw {

constexpr int kZdM = 128;                              // rows per tile
constexpr int kZdAcc = 128;                            // TMEM columns per accumulator
constexpr int kZdKB = 16;                              // real K entries per stage (8 points)
static __host__ __device__ constexpr int zd_stages(int n) { return (n + 7) / 8; }

// K-major operand tiles of both operands, 32-byte swizzling: row r of 32 bytes (16 BF16), 8-row
// atoms of 256 bytes, 16-byte chunk j of row r stored at chunk j ^ ((r % 8) >> 2).
// Low and high word of their descriptors.
__device__ __forceinline__ uint32_t sdesc_sw32_low(uint32_t addr) { return ((addr & 0x3FFFF) >> 4) | (1u << 16); }
constexpr uint32_t kSdescSw32High = (256u >> 4) | (1u << 14) | (6u << 29);
__device__ __forceinline__ uint32_t sw32_off(int r, int k) // byte offset of element k (< 16) of row r
{
    return (uint32_t)((r >> 3) * 256 + (r & 7) * 32 + ((((k >> 3) ^ ((r & 7) >> 2)) & 1) << 4) + (k & 7) * 2);
}

__device__ __forceinline__ void bulk_copy(void *dst, const void *src, unsigned bytes, uint64_t *b)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     su32(dst)),
                 "l"(src), "r"(bytes), "r"(su32(b))
                 : "memory");
}
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }


// one slot of the line-tile ring, in float4: CT lines, to 128 bytes (TMA destinations)
static __host__ __device__ int zd_ring_stride(int CT, int n) { return (CT * n + 7) / 8 * 8; }

} // namespace gw
