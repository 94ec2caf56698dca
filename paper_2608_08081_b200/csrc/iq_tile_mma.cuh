// Tiles of 128 x 128 binary16 operands on the tensor cores: what the bulk append and the reconstruction kernel share.
#pragma once
#include "iq_decode_common.cuh"

namespace iq {

constexpr int TILE_OPERAND = 128 * 128 * 2;  // bytes of an operand; K-major: two slabs of [128][64], 128-byte swizzle

__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,"
      "%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  tc_wait_ld();
}
// D[tmem] (+)= A[smem] * B[smem], binary16 operands, fp32 accumulation.
__device__ __forceinline__ void tc_mma_f16_ss(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, {%5, %6, %7, %8}, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(0), "r"(0), "r"(0), "r"(0)
      : "memory");
}
// K-major operand, 128-byte swizzle: rows of 128 bytes (64 binary16 contraction steps), 8 rows = 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_k128(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// fp32 result, binary16 operands, both K-major, N = 128, M = 128; A negated; A MN-major.
constexpr uint32_t TILE_IDESC = (1u << 4) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
constexpr uint32_t TILE_IDESC_NEG_A = 1u << 13, TILE_IDESC_MN_A = 1u << 15;

// The blocks M_b of one head in fp64, one thread each.
template <int D>
static __device__ __noinline__ void tile_build_m(const float* rot_head, double* m_s, int tid) {
  if (tid < D / 4) {
    double M[4][4];
    so4_matrix<double>(rot_head + (size_t)tid * 8, M);
#pragma unroll
    for (int r = 0; r < 4; r++)
#pragma unroll
      for (int c = 0; c < 4; c++) m_s[16 * tid + 4 * r + c] = M[r][c];
  }
}
}  // namespace iq
