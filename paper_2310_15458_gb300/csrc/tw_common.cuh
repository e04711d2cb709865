// Digit operands of the tcgen05 products: stages of 32 entries of K in the no-swizzle
// K-major layout of 8-row x 16-byte core matrices, one block per digit slice, and the
// helpers that cut and move them.  Shared by the factorization and the sweeps.
#pragma once
#include <type_traits>

#include "common.cuh"

namespace {

constexpr int TW_M = 128, TW_NC = 64, TW_K = 32, TW_NT = 512;
constexpr int TW_KX = OZ_KX;                             // sums exact in FP32
constexpr int TW_KN = OZ_KN;                             // ... and below 2^22 (oz_fint)
constexpr int TW_A = OZ_S * TW_M * TW_K * 2;             // bytes of a stage: 64 KB
constexpr int TW_B = OZ_S * TW_NC * TW_K * 2;            // 32 KB
constexpr int TW_POLLS = 1 << 22, TW_DRAIN = 1 << 26;

__device__ __forceinline__ unsigned long long tw_key(double x) { return oz_abs_bits(x); }
__device__ __forceinline__ unsigned long long tw_key(zd x) { return max(oz_abs_bits(x.x), oz_abs_bits(x.y)); }
__device__ __forceinline__ unsigned long long shfl_max_u64(unsigned long long v, int lanes) {
  for (int d = 1; d < lanes; d <<= 1) v = max(v, (unsigned long long)__shfl_xor_sync(0xffffffffu, (long long)v, d));
  return v;
}

// the digits of eight entries (16-byte pieces, one per slice) at d + p * stride
__device__ __forceinline__ void tw_put8(const long long* X, unsigned char* d, size_t stride, uint32_t flip) {
  uint32_t g[4][OZ_S];
#pragma unroll
  for (int e = 0; e < 4; ++e) oz_digits2(X[2 * e], X[2 * e + 1], g[e]);
#pragma unroll
  for (int p = 0; p < OZ_S; ++p)
    *reinterpret_cast<uint4*>(d + (size_t)p * stride) =
        make_uint4(g[0][p] ^ flip, g[1][p] ^ flip, g[2][p] ^ flip, g[3][p] ^ flip);
}
// place of row (column) i, entries 8 kg .. of a stage inside a slice
__device__ __forceinline__ int tw_at(int i, int kg) { return (i / 8) * 512 + kg * 128 + (i % 8) * 16; }

// bulk copy global -> shared memory (both 16-byte aligned, a multiple of 16 bytes),
// counted on the mbarrier
__device__ __forceinline__ void bulk_g2s(void* smem, const void* gmem, uint32_t bytes, uint64_t* mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                   smem_u32(smem)),
               "l"(gmem), "r"(bytes), "r"(smem_u32(mbar))
               : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(mbar)), "r"(bytes) : "memory");
}

// warp-wide: N = 4 or 8 consecutive FP32 columns of this warp's 32 TMEM lanes
template <int N> __device__ __forceinline__ void tmem_ldn(uint32_t* v, uint32_t taddr) {
  if constexpr (N == 8) {
    tmem_ld8(v, taddr);
  } else {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(taddr));
  }
}
// eight group sums (weights u = 0 .. 7) of one output as W, its value W 2^(row and
// column exponents - 53 - X); narrow: over at most TW_KN entries of K, an FP32 addition in
// place of a conversion
template <int X, int C, bool NARROW>
__device__ __forceinline__ long long tw_join(const uint32_t (&gr)[OZ_S][C], int e, std::integral_constant<bool, NARROW>) {
  return oz_join<!NARROW, X>([&](int u) { return __uint_as_float(gr[u][e]); });
}

}  // namespace
