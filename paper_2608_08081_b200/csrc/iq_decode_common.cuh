// Device helpers shared by the decode kernels: tcgen05 / tensor-memory wrappers, the byte-lookup dequantisation of
// a packing unit, named barriers.
#pragma once
#include "iq_common.cuh"

namespace iq {

// ---------------------------------------------------------------------------------------------- tcgen05 wrappers
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&o)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  tc_wait_ld();
#pragma unroll
  for (int i = 0; i < 16; i++) o[i] = __uint_as_float(r[i]);
}
// The same load without the wait: the registers are valid after tc_wait_ld().
__device__ __forceinline__ void tc_ld16_issue(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem descriptor]; fp16 operands, fp32 accumulate, M = 128, N and majors in idesc.
__device__ __forceinline__ void tc_mma_f16(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, {%5, %6, %7, %8}, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(0), "r"(0), "r"(0), "r"(0)
      : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem descriptor]; int8 operands, int32 accumulate, K = 32 per instruction.
__device__ __forceinline__ void tc_mma_i8(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, {%5, %6, %7, %8}, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(0), "r"(0), "r"(0), "r"(0)
      : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Shared-memory operand descriptor, MN-major, no swizzle: element (n, k) of a 16-bit operand sits at
// (n % 8) * 2 + (n / 8) * sbo + (k % 8) * 16 + (k / 8) * lbo bytes from the start address.
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) | (1ull << 46);
}
// Instruction descriptor: D = f32, A = B = f16, A K-major (TMEM), B MN-major, N = 16, M = 128.
constexpr uint32_t DEC_IDESC = (1u << 4) | (1u << 16) | ((16u >> 3) << 17) | ((128u >> 4) << 24);
// Integer path: D = s32, A = s8 (K-major, TMEM), B MN-major, N = 16 or 32, M = 128; B = s8 (query digits) or u8 (probability digits).
template <int N>
constexpr uint32_t DEC_IDESC_I8_SS = (2u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | (((uint32_t)N >> 3) << 17) | ((128u >> 4) << 24);
template <int N>
constexpr uint32_t DEC_IDESC_I8_SU = (2u << 4) | (1u << 7) | (0u << 10) | (1u << 16) | (((uint32_t)N >> 3) << 17) | ((128u >> 4) << 24);

// ---------------------------------------------------------------------------------------------- dequantisation
// The shift/logic pipe, which carries the byte permutes at half rate, bounds the lookups, so what can go elsewhere does. A 128 x 128
// tile of 3-bit codes, its loads and stores included, takes a scheduler 140 cycles (however many warps it has): 190 with the shifts
// and masks on that pipe or as high words of products (which occupy the multiplier for four cycles each), 162 with only the upper
// halves elsewhere.
// The upper half of a word of nibbles below 8 in the lower half, for the byte permutes, which take their selectors from there: an
// fp16x2 addition of -0 that reads the upper half twice. Exact: no such half is an infinity or a NaN (bit 11 is clear), and
// subnormals are kept.
__device__ __forceinline__ uint32_t upper_nibbles(uint32_t x, LookupConst c) {
  uint32_t r;
  asm("{\n\t.reg .b16 l, h;\n\t.reg .b32 t;\n\tmov.b32 {l, h}, %1;\n\tmov.b32 t, {h, h};\n\tadd.f16x2 %0, t, %2;\n\t}" : "=r"(r) : "r"(x), "r"(c.neg_zero));
  return r;
}
// w without the bits of `part` (part = w & mask), by a multiply-add.
__device__ __forceinline__ uint32_t without(uint32_t w, uint32_t part, LookupConst c) {
  uint32_t r;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(part), "r"(c.minus_one), "r"(w));
  return r;
}
// The selectors of one packing unit's 32 entries (3 bits), 8 to a word: the low three bits of the nibbles, and for the last 8, whose
// code bits sit in bit 3 of the nibbles of the three words, these put together.
__device__ __forceinline__ void unit_selectors(uint32_t w0, uint32_t w1, uint32_t w2, LookupConst c, uint32_t (&sel)[4]) {
  const uint32_t g0 = w0 & 0x88888888u, g1 = w1 & 0x88888888u, g2 = w2 & 0x88888888u;
  sel[0] = without(w0, g0, c);
  sel[1] = without(w1, g1, c);
  sel[2] = without(w2, g2, c);
  sel[3] = (g0 >> 3) | (g1 >> 2) | (g2 >> 1);
}
// One packing unit (32 codes in 3 words) -> 16 registers of two fp16 levels each, entries in natural order:
// out[r] = (level[code 2r], level[code 2r+1]). Byte lookups with prmt: 8 levels x (low byte, high byte).
__device__ __forceinline__ void dequant_unit(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t lo0, uint32_t lo1, uint32_t hi0,
                                             uint32_t hi1, LookupConst c, uint32_t (&out)[16]) {
  uint32_t sel[4];
  unit_selectors(w0, w1, w2, c, sel);
#pragma unroll
  for (int k = 0; k < 4; k++)
#pragma unroll
    for (int hh = 0; hh < 2; hh++) {
      const uint32_t x = hh ? upper_nibbles(sel[k], c) : sel[k];
      const uint32_t l = prmt(lo0, lo1, x), h = prmt(hi0, hi1, x);
      out[4 * k + 2 * hh] = prmt(l, h, 0x5140u);
      out[4 * k + 2 * hh + 1] = prmt(l, h, 0x7362u);
    }
}

// Integer path: one packing unit -> 8 registers of four int8 levels each, entries in natural order (one prmt per 4 codes).
__device__ __forceinline__ void dequant_unit8(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t l0, uint32_t l1, LookupConst c, uint32_t* out) {
  uint32_t sel[4];
  unit_selectors(w0, w1, w2, c, sel);
#pragma unroll
  for (int k = 0; k < 4; k++) {
    out[2 * k] = prmt(l0, l1, sel[k]);
    out[2 * k + 1] = prmt(l0, l1, upper_nibbles(sel[k], c));
  }
}
// ---- the same for every bit width: 32 consecutive entries of a packed run (BITS words at w) -> natural order.
// b = 2: 16 entries per word, codes in the low (entries 0..7) and high (8..15) bit pair of the nibbles: one 4-byte table.
// b = 4: 8 entries per word; a byte permute selects among 8 bytes, so the 16 levels are two tables of 8, looked up with
// the low three bits of the code and chosen byte by byte with a mask made from its top bit.
__device__ __forceinline__ uint32_t byte_select(uint32_t lo, uint32_t hi, uint32_t mask) { return (hi & mask) | (lo & ~mask); }

template <int BITS>
__device__ __forceinline__ void dequant32_i8(const uint32_t* w, const uint32_t (&t)[4], LookupConst c, uint32_t* out) {
  if constexpr (BITS == 3) {
    dequant_unit8(w[0], w[1], w[2], t[0], t[1], c, out);
  } else if constexpr (BITS == 2) {
#pragma unroll
    for (int j = 0; j < 2; j++) {
      const uint32_t g = w[j] & 0xCCCCCCCCu, a = without(w[j], g, c), b = g >> 2;
      out[4 * j] = prmt(t[0], t[0], a);
      out[4 * j + 1] = prmt(t[0], t[0], upper_nibbles(a, c));
      out[4 * j + 2] = prmt(t[0], t[0], b);
      out[4 * j + 3] = prmt(t[0], t[0], upper_nibbles(b, c));
    }
  } else {
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const uint32_t g = w[j] & 0x88888888u, s7 = without(w[j], g, c), s3 = g >> 3;
#pragma unroll
      for (int hh = 0; hh < 2; hh++) {
        const uint32_t x = hh ? upper_nibbles(s7, c) : s7, mx = hh ? upper_nibbles(s3, c) : s3;
        out[2 * j + hh] = byte_select(prmt(t[0], t[1], x), prmt(t[2], t[3], x), prmt(0x0000FF00u, 0u, mx));
      }
    }
  }
}

// fp16 levels: out[r] = (level[code 2r], level[code 2r+1]), 16 registers for the 32 entries.
template <int BITS>
__device__ __forceinline__ void dequant32_f16(const uint32_t* w, const uint32_t (&lo)[4], const uint32_t (&hi)[4], LookupConst c, uint32_t (&out)[16]) {
  if constexpr (BITS == 3) {
    dequant_unit(w[0], w[1], w[2], lo[0], lo[1], hi[0], hi[1], c, out);
  } else {
    uint32_t sel[4], top[4];  // four selectors of 8 entries each (b = 4: and the top bits of their codes)
    if constexpr (BITS == 2) {
      const uint32_t g0 = w[0] & 0xCCCCCCCCu, g1 = w[1] & 0xCCCCCCCCu;
      sel[0] = without(w[0], g0, c); sel[1] = g0 >> 2;
      sel[2] = without(w[1], g1, c); sel[3] = g1 >> 2;
      top[0] = top[1] = top[2] = top[3] = 0u;
    } else {
#pragma unroll
      for (int k = 0; k < 4; k++) { const uint32_t g = w[k] & 0x88888888u; sel[k] = without(w[k], g, c); top[k] = g >> 3; }
    }
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
      for (int hh = 0; hh < 2; hh++) {
        const uint32_t x = hh ? upper_nibbles(sel[k], c) : sel[k];
        uint32_t l, h;
        if constexpr (BITS == 2) {
          l = prmt(lo[0], lo[0], x);
          h = prmt(hi[0], hi[0], x);
        } else {
          const uint32_t m = prmt(0x0000FF00u, 0u, hh ? upper_nibbles(top[k], c) : top[k]);
          l = byte_select(prmt(lo[0], lo[1], x), prmt(lo[2], lo[3], x), m);
          h = byte_select(prmt(hi[0], hi[1], x), prmt(hi[2], hi[3], x), m);
        }
        out[4 * k + 2 * hh] = prmt(l, h, 0x5140u);
        out[4 * k + 2 * hh + 1] = prmt(l, h, 0x7362u);
      }
  }
}

// Pairs of fp32 values, one instruction for the two (each rounded like the scalar operation).
struct F32x2 {
  uint64_t v;
  __device__ __forceinline__ float lo() const { return __uint_as_float((uint32_t)v); }
  __device__ __forceinline__ float hi() const { return __uint_as_float((uint32_t)(v >> 32)); }
};
__device__ __forceinline__ F32x2 f32x2(float lo, float hi) {
  F32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ F32x2 fma2(F32x2 a, F32x2 b, F32x2 c) {
  F32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F32x2 add2(F32x2 a, F32x2 b) {
  F32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F32x2 mul2(F32x2 a, F32x2 b) {
  F32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}

// One lane of a converged warp. Issuing the MMAs / bulk copies from an elected lane of a converged warp keeps
// their operands in uniform registers; a lone divergent thread issues the same sequence about 3x slower.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred != 0;
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Named barrier `id` over the 128 compute threads of one group, with an OR reduction.
__device__ __forceinline__ bool group_bar_or(int id, bool pred) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %2, 0;\n\tbarrier.red.or.pred p, %1, 128, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(r) : "r"(id), "r"((uint32_t)pred) : "memory");
  return r != 0;
}
// The same over `count` threads.
__device__ __forceinline__ bool cta_bar_or_n(int id, int count, bool pred) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %3, 0;\n\tbarrier.red.or.pred p, %1, %2, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(r) : "r"(id), "r"(count), "r"((uint32_t)pred) : "memory");
  return r != 0;
}
// Named barrier `id` over `count` threads (a multiple of 32).
__device__ __forceinline__ void cta_bar_sync_n(int id, int count) { asm volatile("barrier.sync %0, %1;" ::"r"(id), "r"(count) : "memory"); }
__device__ __forceinline__ void group_bar_sync(int id) { asm volatile("barrier.sync %0, 128;" ::"r"(id) : "memory"); }

__device__ __forceinline__ float max3f(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// Reduction of 8 values per lane over the 32 lanes of a warp with 9 shuffles instead of 40: the lanes first trade
// halves of their value sets (xor 16: four values each way, xor 8: two, xor 4: one), so that lane l ends up with one
// value of head warp_reduce8_head(l), which two more butterfly steps complete. Every lane gets the result of its head.
__device__ __forceinline__ int warp_reduce8_head(int lane) { return ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1); }
template <typename OP>
__device__ __forceinline__ float warp_reduce8(const float (&v)[8], int lane, OP op) {
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  float a[4], c[2];
#pragma unroll
  for (int i = 0; i < 4; i++) a[i] = op(b4 ? v[i + 4] : v[i], __shfl_xor_sync(FULL, b4 ? v[i] : v[i + 4], 16));
#pragma unroll
  for (int i = 0; i < 2; i++) c[i] = op(b3 ? a[i + 2] : a[i], __shfl_xor_sync(FULL, b3 ? a[i] : a[i + 2], 8));
  float r = op(b2 ? c[1] : c[0], __shfl_xor_sync(FULL, b2 ? c[0] : c[1], 4));
  r = op(r, __shfl_xor_sync(FULL, r, 2));
  return op(r, __shfl_xor_sync(FULL, r, 1));
}
// The same for (value, row) pairs: the larger value wins, the lower row among equal values (rows < 0 mean "none").
__device__ __forceinline__ void argmax_merge(float& bv, int& bi, float ov, int oi) {
  if (ov > bv || (ov == bv && oi >= 0 && (bi < 0 || oi < bi))) { bv = ov; bi = oi; }
}
__device__ __forceinline__ void warp_argmax8(const float (&v)[8], const int (&ix)[8], int lane, float& rv, int& ri) {
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  float a[4], c[2];
  int ai[4], ci[2];
#pragma unroll
  for (int i = 0; i < 4; i++) {
    a[i] = b4 ? v[i + 4] : v[i];
    ai[i] = b4 ? ix[i + 4] : ix[i];
    argmax_merge(a[i], ai[i], __shfl_xor_sync(FULL, b4 ? v[i] : v[i + 4], 16), __shfl_xor_sync(FULL, b4 ? ix[i] : ix[i + 4], 16));
  }
#pragma unroll
  for (int i = 0; i < 2; i++) {
    c[i] = b3 ? a[i + 2] : a[i];
    ci[i] = b3 ? ai[i + 2] : ai[i];
    argmax_merge(c[i], ci[i], __shfl_xor_sync(FULL, b3 ? a[i] : a[i + 2], 8), __shfl_xor_sync(FULL, b3 ? ai[i] : ai[i + 2], 8));
  }
  rv = b2 ? c[1] : c[0];
  ri = b2 ? ci[1] : ci[0];
  argmax_merge(rv, ri, __shfl_xor_sync(FULL, b2 ? c[0] : c[1], 4), __shfl_xor_sync(FULL, b2 ? ci[0] : ci[1], 4));
  argmax_merge(rv, ri, __shfl_xor_sync(FULL, rv, 2), __shfl_xor_sync(FULL, ri, 2));
  argmax_merge(rv, ri, __shfl_xor_sync(FULL, rv, 1), __shfl_xor_sync(FULL, ri, 1));
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL, v, o));
  return v;
}

}  // namespace iq
