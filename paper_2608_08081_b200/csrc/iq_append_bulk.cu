// Bulk quantize-append (Algorithm 1 for prompts and chunks of them): the whole rotation of a tile of 128 rows as one
// contraction on the tensor cores, codes decided and packed straight out of tensor memory.
//
// Tile = (tensor, KV head, sequence, 128-row block of the cache), K and V in one launch. With the unnormalised rotation
// W = blockdiag(M_b) H_d, u s = W x. The tile X (128 rows of binary16) sits in shared memory as it came; the roles of the
// two operands are chosen so that a thread reads from its tensor-memory lane what it has to pack next to each other:
//   K: D[row][coordinate]  = X W^T   thread = row,        the words of its packed row
//   V: D[coordinate][row]  = W X^T   thread = coordinate, the words of its token-transposed record
// W is split into two binary16 terms, W_hi + W_lo (|W - W_hi - W_lo| <= 2^-22 |W|, or 2^-25 where W_lo is subnormal), the
// products with binary16 rows are exact and summed in fp32, the small terms first. W has only 4 distinct magnitudes per row (M_b times a 4-point
// transform; the rest of H_d is signs), so a CTA builds it in about a microsecond per head. d = 256: H_256 is
// [[H, H], [H, -H]], so the operand of the second half of the contraction is that of the first, negated where both
// halves are the upper ones by the instruction's negate bit: 2 x 64 KB of W instead of 256.
//
// Decision. Per threshold one fused multiply-add with saturation, sat(B x + o_j), B = 0.5 / (GUARD s): 0 below, 1 above, and a
// fraction inside a band of +-GUARD around the threshold. The code is the sum; a sum that is not a whole number (16 + code
// is kept, so its fraction bits are the same for all codes; they are OR-ed over 8 coordinates) marks a coordinate too
// close to call, which is put on a list and decided again in fp64 by eight lanes (exact +-1 sums, the norm and the block
// in fp64). Where 8 columns of a warp have many, or the list is full (rows with ties throughout: constant rows, rows whose
// Walsh-Hadamard coordinates vanish), the rows are marked instead; the group's warps share the marked rows of a tile when
// the next one has been copied in, a row at a time by a warp. 4 x 8 K constant rows, d = 128, 3 bits: 0.77 ms, every 13th row
// constant 0.28 (ordinary rows 0.081); with every warp of a V tile deciding all rows, code by code: 8.8 and 0.9.
//
// GUARD bounds the error of a sum that ends near a threshold t, so the codes are those of an fp64 evaluation. An instruction
// (16 products) aligns its products and the running sum to the largest of them, keeps two bits below the fp32 last
// place, and cuts; the result is cut to fp32 (an emulation of just this gives the same bits as the tensor core on sums of
// all kinds). So it loses at most 17 x 2^-25 of the larger of the running sum and its products, and 2^-23 of its result. The
// running sums S_i of a row of norm 1 that end at t are bounded together, by Cauchy-Schwarz on sum c_i S_i: at d = 128 the
// cuts are at most 1.9e-5 + 2.3e-6 t, with W's 2^-22 sqrt(d) and the rounding of x B 2.25e-5 + 2.3e-6 t. At d = 256 the second
// half's lower terms would each cut the sum of the first half; they come last, where it is back at t: 5.5e-5 + 9.8e-6 t
// (9.1e-5 + 7e-6 t in the other order). Rows built against it (an emulated search over prefixes along W's row, with the low bits of
// every element chosen for the largest cut) reach 7e-6 and 1.9e-5, Gaussian and outlier rows 1e-6.
// Symmetric codebooks (t_mid = 0, t_j = -t_-j): the positive thresholds against |x| plus the sign, 4 instead of 7
// multiply-adds per coordinate at 3 bits, 8 instead of 15 at 4 bits.
//
// Work split: one persistent CTA per SM takes an equal contiguous share of the tiles, ordered by head; NG groups of four
// warps (eight at d = 256), each with a tile buffer and accumulator columns of its own, take the tiles in turn. A group
// copies its next tile in (cp.async) while it packs the present one; a control warp per group finds the tiles and issues
// the MMAs. The groups run in different phases, so that copies, norms and contractions of one run under the packing of
// the others. No pipe is near its limit and issue is at 42 %. A group's phases run one after the other and the groups that fit do
// not cover them all, but that is not the whole bound: a copy without the norm, a third of that chain, took 244 us instead of 278.
//
// Measured (K and V rows of 8 KV heads, Gaussian with outlier channels), against one row in 8 or 16 lanes with butterflies
// by shuffle and a kernel per tensor: 1.6 M rows, d = 128, 3 bits: 255 us instead of 491 (1.9 TB/s of rows in and codes
// out); 262 k rows, d = 256, 4 bits: 187 instead of 457; 50 k rows in chunks of 500 per sequence: 26.0 instead of 54.5.
#include <cmath>

#include "iq_append_row.cuh"
#include "iq_decode_common.cuh"
#include "iq_kernels.h"
#include "iq_tile_mma.cuh"

namespace iq {

// Half-width of the band around a threshold in which the tile decision is not trusted (see above); t: the largest threshold.
static float bulk_guard(int head_dim, float t) { return head_dim == 128 ? 2.25e-5f + 2.3e-6f * t : 5.5e-5f + 9.8e-6f * t; }

template <int D>
struct BulkLayout {
  static constexpr int NJ = D / 128;              // 128-coordinate halves: of the contraction and of the result
  static constexpr int GT = 128 * NJ;             // threads of a packing group
  static constexpr int NG = 4 / NJ;               // packing groups: their accumulators fill the tensor memory
  static constexpr int PACK = GT * NG;            // 512 packing threads
  static constexpr int THREADS = PACK + 32 * NG;  // + a control warp per group
  static constexpr int OPERAND = TILE_OPERAND;
  static constexpr int W_BYTES = NJ * 2 * OPERAND;
  static constexpr int LIST = 48;                 // undecided coordinates a warp collects ...
  static constexpr int LIST_STEP = 12;            // ... unless 8 columns have more: rows with ties throughout, decided as a whole
  static constexpr int LIST_FLUSH = 32;           // ... and decides in fp64 after a tile that left it with this many, or at the end
  static constexpr int TILES = 4;                 // tile descriptors kept: the next, the present, and the one before (its rows are redone late)
  // shared memory: W, the groups' tile buffers (128 contraction steps), the warps' lists, the rest
  static constexpr int OFF_X = W_BYTES;
  static constexpr int OFF_LIST = OFF_X + NG * OPERAND;
  static constexpr int LIST_BYTES = 20 * LIST;    // source rows (8), destinations (8), (side, code, coordinate, entry) (4)
  static constexpr int OFF_BINV = OFF_LIST + (PACK / 32) * LIST_BYTES;  // [NG][128] 0.5 / (GUARD s) of the rows of a group's tile
  static constexpr int OFF_SS = OFF_BINV + NG * 512;                    // [NG][2][128] fp64 partial square sums (d = 256)
  static constexpr int OFF_M = OFF_SS + (NJ > 1 ? NG * 2048 : 0);       // [D][4] fp64 rows of the blocks M_b
  static constexpr int OFF_TILE = OFF_M + D * 32;                       // [NG][TILES] tile descriptors
  static constexpr int OFF_ROWS = OFF_TILE + NG * TILES * 48;           // [NG] rows to be decided again
  static constexpr int OFF_WARP = OFF_ROWS + NG * 64;                   // [16] coordinates on the warps' lists
  static constexpr int OFF_PRE = OFF_WARP + (PACK / 32) * 4;            // [THREADS + 1] int64 block counts before a slice of the batch
  static constexpr int OFF_WSUM = OFF_PRE + 8 * (THREADS + 2);
  static constexpr int OFF_TAU = OFF_WSUM + 8 * 32;                     // [2][16] 0.5 / GUARD * threshold, K and V
  static constexpr int OFF_BAR = OFF_TAU + 128;                         // [NG][5] mbarriers: tile described, copied in, norms, accumulator, drained
  static constexpr int OFF_MISC = OFF_BAR + 8 * (5 * NG + (NG & 1));
  static constexpr int SMEM = OFF_MISC + 32 + 1024;                     // + alignment of the swizzle atoms
};
static_assert(BulkLayout<128>::SMEM <= 227 * 1024 && BulkLayout<256>::SMEM <= 227 * 1024, "shared memory overflow");

struct BulkTile {       // a tile, as the control warp hands it to its group
  const __half* src;    // row 0 of its block in the input (may lie before the buffer: rows outside [c_lo, c_hi) are not read)
  size_t row0;          // row 0 of its block in the cache arrays
  int kind;             // 0: K, 1: V, -1: no more tiles for this head
  int c_lo, c_hi;       // rows of the block that are new
  int special;          // it has a row of norm zero or not finite
  int pad[4];
};
static_assert(sizeof(BulkTile) == 48, "tile descriptor");
struct BulkRows {       // rows of the group's present tile and of the one before, by its parity; set by all warps at the end of a tile
  uint32_t full[2][4];  // decided again as a whole: read by all warps when the next tile is copied in
  uint32_t near[2][4];  // with a coordinate that is decided again: counted then
};

__device__ __forceinline__ void tc_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
  tc_wait_ld();
}
__device__ __forceinline__ double half_to_double(uint32_t bits) {
  double d;
  asm("cvt.f64.f16 %0, %1;" : "=d"(d) : "h"((uint16_t)bits));
  return d;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Sets the code of entry e of a packed run (a K row or a V record) to `code`, whatever it was. Other bits of the same
// words may be set at the same time by other threads.
template <int BITS>
__device__ __forceinline__ void patch_code(uint32_t* run, int e, int code) {
  if constexpr (BITS == 3) {
    uint32_t* u = run + 3 * (e >> 5);
    const int c = e & 31;
    if (c < 24) {
      const int sh = 4 * (c & 7);
      atomicAnd(&u[c >> 3], ~(7u << sh));
      atomicOr(&u[c >> 3], (uint32_t)code << sh);
    } else {
      const int sh = 4 * (c - 24) + 3;
#pragma unroll
      for (int k = 0; k < 3; k++) {
        if ((code >> k) & 1) atomicOr(&u[k], 1u << sh);
        else atomicAnd(&u[k], ~(1u << sh));
      }
    }
  } else {
    int word, sh;
    packed_place<BITS>(e, word, sh);
    atomicAnd(&run[word], ~(((1u << BITS) - 1u) << sh));
    atomicOr(&run[word], (uint32_t)code << sh);
  }
}

// The listed coordinates in fp64, eight lanes each: z = the four outputs of the coordinate's block of H x (exact sums),
// u = its row of M_b times z, over the exact norm, against the thresholds from the first that it may not be above.
template <int D, int BITS>
static __device__ __noinline__ void bulk_redo(const QuantizeParams& p, const double* m_s, const __half* const* src_s,
                                              uint32_t* const* dst_s, const uint32_t* info_s, int n, int lane) {
  constexpr int EPL = D / 8;  // elements per lane
  const int li = lane & 7;
#pragma unroll 1
  for (int base = 0; base < n; base += 4) {
    const int e = base + (lane >> 3);
    const bool act = e < n;
    const int ee = act ? e : n - 1;
    const uint32_t info = info_s[ee];
    const int coord = info & 0xff, entry = (info >> 8) & 0xff, nearest = (info >> 16) & 15;
    const uint4* src = reinterpret_cast<const uint4*>(src_s[ee] + li * EPL);
    const int blk = coord >> 2;
    double z[4] = {0.0, 0.0, 0.0, 0.0}, ss = 0.0;
    uint4 t4[EPL / 8];
#pragma unroll
    for (int i = 0; i < EPL / 8; i++) t4[i] = src[i];
#pragma unroll
    for (int i = 0; i < EPL / 8; i++) {
      const uint32_t w[4] = {t4[i].x, t4[i].y, t4[i].z, t4[i].w};
#pragma unroll
      for (int hq = 0; hq < 2; hq++) {  // 4 elements: quad l of the row
        const float2 fa = __half22float2(*reinterpret_cast<const __half2*>(&w[2 * hq]));
        const float2 fb = __half22float2(*reinterpret_cast<const __half2*>(&w[2 * hq + 1]));
        ss += ((double)(fa.x * fa.x) + (double)(fa.y * fa.y)) + ((double)(fb.x * fb.x) + (double)(fb.y * fb.y));
        const int l = li * (EPL / 4) + 2 * i + hq;
        const double sg = (__popc(blk & l) & 1) ? -1.0 : 1.0;
        const double s01 = (double)fa.x + (double)fa.y, d01 = (double)fa.x - (double)fa.y;
        const double s23 = (double)fb.x + (double)fb.y, d23 = (double)fb.x - (double)fb.y;
        z[0] += sg * (s01 + s23);
        z[1] += sg * (d01 + d23);
        z[2] += sg * (s01 - s23);
        z[3] += sg * (d01 - d23);
      }
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
#pragma unroll
      for (int c = 0; c < 4; c++) z[c] += __shfl_xor_sync(FULL, z[c], o);
      ss += __shfl_xor_sync(FULL, ss, o);
    }
    const double* m = m_s + 4 * coord;
    const double u = (m[0] * z[0] + m[1] * z[1] + m[2] * z[2] + m[3] * z[3]) * inv_sqrt(ss);  // (rows of norm zero are not listed)
    const float* th = ((info >> 20) & 1u) ? p.thresholds_v : p.thresholds_k;
    int code = max(nearest - 1, 0);
    while (code < (1 << BITS) - 1 && u > (double)th[code]) code++;
    if (act && li == 0) patch_code<BITS>(dst_s[ee], entry, code);
  }
}

// The codes of a row in fp64 throughout (exact +-1 sums, the blocks from shared memory): lane l those of coordinates l E ...
template <int D, int BITS>
static __device__ __forceinline__ void bulk_exact_row(const __half* src_row, const double* m_s, const float (&th)[(1 << BITS) - 1], int lane, int (&code)[D / 32]) {
  constexpr int E = D / 32, NT = (1 << BITS) - 1;
  const __half2* src = reinterpret_cast<const __half2*>(src_row + lane * E);
  double v[E], ss = 0.0;
#pragma unroll
  for (int k = 0; k < E / 2; k++) {
    const float2 f = __half22float2(src[k]);
    v[2 * k] = (double)f.x;
    v[2 * k + 1] = (double)f.y;
    ss += (double)(f.x * f.x) + (double)(f.y * f.y);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(FULL, ss, o);
  wht_warp<double, E>(v, lane);
  const double inv = ss > 0.0 ? inv_sqrt(ss) : 0.0;
#pragma unroll
  for (int e = 0; e < E; e++) {
    const double* m = m_s + 4 * (lane * E + e);
    const double* z = v + (e & ~3);
    bool nb;
    code[e] = decide_code_n<double, NT>((m[0] * z[0] + m[1] * z[1] + m[2] * z[2] + m[3] * z[3]) * inv, th, nb, 0.0);
  }
}

// 8 mask bits -> the lowest bits of the 8 nibbles of a word.
__device__ __forceinline__ uint32_t spread8(uint32_t b) {
  b &= 0xffu;
  b = (b | (b << 12)) & 0x000F000Fu;
  b = (b | (b << 6)) & 0x03030303u;
  return (b | (b << 3)) & 0x11111111u;
}
// The packed words of 32 entries from their codes as four words of nibbles.
template <int BITS>
__device__ __forceinline__ void pack_nibbles(const uint32_t (&nib)[4], uint32_t* word) {
  if constexpr (BITS == 4) {
#pragma unroll
    for (int q = 0; q < 4; q++) word[q] = nib[q];
  } else if constexpr (BITS == 3) {  // entries 24..31: bit k of the code into the top bits of word k's nibbles
    word[0] = nib[0] | ((nib[3] & 0x11111111u) << 3);
    word[1] = nib[1] | ((nib[3] & 0x22222222u) << 2);
    word[2] = nib[2] | ((nib[3] & 0x44444444u) << 1);
  } else {
    word[0] = nib[0] | (nib[1] << 2);
    word[1] = nib[2] | (nib[3] << 2);
  }
}
// The bits of packed word k that belong to the entries of vm (32 bits, one per entry).
template <int BITS>
__device__ __forceinline__ uint32_t packed_mask(uint32_t vm, int k) {
  if constexpr (BITS == 4) return spread8(vm >> (8 * k)) * 15u;
  else if constexpr (BITS == 3) return spread8(vm >> (8 * k)) * 7u + spread8(vm >> 24) * 8u;
  else return spread8(vm >> (16 * k)) * 3u + spread8(vm >> (16 * k + 8)) * 12u;
}
// Which of the 32 rows from 32 u on are new, rows [c_lo, c_hi) of the block being so.
__device__ __forceinline__ uint32_t new_rows(int c_lo, int c_hi, int u) {
  const int a = min(max(c_lo - 32 * u, 0), 32), z = min(max(c_hi - 32 * u, 0), 32);
  if (a >= z) return 0u;
  return (z == 32 ? 0xFFFFFFFFu : (1u << z) - 1u) & ~((1u << a) - 1u);
}

// Rows of which the lists did not take every undecided coordinate, again as a whole, by one warp: the rows `m` of the 32 from
// 32 u on (V, d = 256: those of the 16 that are this warp's, `part`). Stores and changes that other warps make to the same
// codes are of the same values, or are changed to these by their lists; words of V have other rows' codes too, which the
// lists may be changing, so bits of part of a word are set one way and the other by atomics.
template <int D, int BITS>
static __device__ __noinline__ void bulk_redo_rows(const QuantizeParams& p, const double* m_s, const BulkTile* t, uint32_t m, int u, int part, int lane) {
  constexpr int E = D / 32, NT = (1 << BITS) - 1, NJ = D / 128;
  const bool is_v = t->kind != 0;
  float th[NT];
#pragma unroll
  for (int i = 0; i < NT; i++) th[i] = is_v ? p.thresholds_v[i] : p.thresholds_k[i];
  const uint32_t vm = m & new_rows(t->c_lo, t->c_hi, u) & (NJ == 1 || !is_v ? 0xFFFFFFFFu : (part ? 0xFFFF0000u : 0x0000FFFFu));
  const __half* src0 = t->src + (long long)(32 * u) * p.stride_t;
  int code[E];
  if (!is_v) {
    const RowSink sink{p.k_codes, p.k_scales, p.v_codes, p.v_scales, p.status, p.scale_f16};
    m = vm;
#pragma unroll 1
    while (m) {
      const int r = __ffs(m) - 1;
      m &= m - 1u;
      bulk_exact_row<D, BITS>(src0 + (long long)r * p.stride_t, m_s, th, lane, code);
      warp_store_k_row<D, BITS, false>(sink, t->row0 + 32 * u + r, code, 0.f, lane);
    }
  } else if (vm) {
    constexpr int Q = 4 / NJ;  // groups of 8 rows
    const int q0 = NJ == 1 ? 0 : 2 * part;
    uint32_t nib[E][Q];
#pragma unroll 1
    for (int q = 0; q < Q; q++) {
#pragma unroll
      for (int e = 0; e < E; e++) {
#pragma unroll
        for (int i = 0; i < Q - 1; i++) nib[e][i] = nib[e][i + 1];
        nib[e][Q - 1] = 0u;
      }
#pragma unroll 1
      for (int i = 0; i < 8; i++) {
        const int r = 8 * (q0 + q) + i;
        if (!((vm >> r) & 1u)) continue;
        bulk_exact_row<D, BITS>(src0 + (long long)r * p.stride_t, m_s, th, lane, code);
#pragma unroll
        for (int e = 0; e < E; e++) nib[e][Q - 1] |= (uint32_t)code[e] << (4 * i);
      }
    }
#pragma unroll
    for (int e = 0; e < E; e++) {
      uint32_t word[BITS];
      if constexpr (NJ == 1) {
        pack_nibbles<BITS>(nib[e], word);
      } else {
        const uint32_t n4[4] = {part ? 0u : nib[e][0], part ? 0u : nib[e][1], part ? nib[e][0] : 0u, part ? nib[e][1] : 0u};
        pack_nibbles<BITS>(n4, word);
      }
      uint32_t* d = reinterpret_cast<uint32_t*>(p.v_codes + ((t->row0 / 128) * D + lane * E + e) * (size_t)(16 * BITS)) + BITS * u;
#pragma unroll
      for (int k = 0; k < BITS; k++) {
        const uint32_t wm = packed_mask<BITS>(vm, k);
        if (wm == 0xFFFFFFFFu) {
          d[k] = word[k];
        } else if (wm) {
          atomicAnd(d + k, ~wm);
          atomicOr(d + k, word[k]);
        }
      }
    }
  }
}

// W of one head into shared memory: thread = (row i, part of the row's quads). W[i][4l + e] = +-V4[e] with
// V4[e] = sum_c M[i%4][c] (-1)^popc(c & e), the sign (-1)^popc(b & l) with b the 4-block of i inside its 128-row half.
template <int D>
static __device__ __noinline__ void bulk_build_w(const double* m_s, uint8_t* w_s, int tid) {
  using L = BulkLayout<D>;
  constexpr int PARTS = L::PACK / D;  // threads per row
  const int i = tid % D, part = tid / D;
  uint32_t hi[2], lo[2];
  {
    const double* m = m_s + 4 * i;
    const double v4[4] = {(m[0] + m[1]) + (m[2] + m[3]), (m[0] - m[1]) + (m[2] - m[3]), (m[0] + m[1]) - (m[2] + m[3]), (m[0] - m[1]) - (m[2] - m[3])};
    __half h[4], l[4];
#pragma unroll
    for (int e = 0; e < 4; e++) {
      h[e] = __double2half(v4[e]);
      l[e] = __double2half(v4[e] - (double)__half2float(h[e]));
    }
#pragma unroll
    for (int e = 0; e < 2; e++) {
      hi[e] = (uint32_t)__half_as_ushort(h[2 * e]) | ((uint32_t)__half_as_ushort(h[2 * e + 1]) << 16);
      lo[e] = (uint32_t)__half_as_ushort(l[2 * e]) | ((uint32_t)__half_as_ushort(l[2 * e + 1]) << 16);
    }
  }
  const int j = i >> 7, ii = i & 127, b = ii >> 2;
  uint8_t* base_lo = w_s + (size_t)(2 * j) * L::OPERAND;
  uint8_t* base_hi = base_lo + L::OPERAND;
#pragma unroll 4
  for (int m = part * (16 / PARTS); m < (part + 1) * (16 / PARTS); m++) {  // 16-byte chunk m: quads 2m, 2m + 1
    const uint32_t s0 = (__popc(b & (2 * m)) & 1) ? 0x80008000u : 0u, s1 = (__popc(b & (2 * m + 1)) & 1) ? 0x80008000u : 0u;
    const int off = (m >> 3) * (L::OPERAND / 2) + ii * 128 + (((m & 7) ^ (ii & 7)) * 16);
    *reinterpret_cast<uint4*>(base_hi + off) = make_uint4(hi[0] ^ s0, hi[1] ^ s0, hi[0] ^ s1, hi[1] ^ s1);
    *reinterpret_cast<uint4*>(base_lo + off) = make_uint4(lo[0] ^ s0, lo[1] ^ s0, lo[0] ^ s1, lo[1] ^ s1);
  }
}

// A group's position in the tiles of a head: K tiles of all sequences, then V tiles, each sequence's blocks in order.
struct BulkWalk {
  int is_v, b;
  long long first;   // index (within the head and tensor) of the sequence's first tile
  int n_tiles;       // tiles of the sequence
  long long blk0;    // its first block
  int pos0, n_new;
};

// How a coordinate is decided. CLOSE: thresholds may lie within one another's bands, where two fractions can add up to a
// whole number, so the thresholds below and above the band are counted; twice the instructions (4 x 32 K rows, d = 128,
// thresholds 1e-5 apart: 894 us where a warp per row takes 1790).
enum BulkMode { BULK_PLAIN, BULK_SYMMETRIC, BULK_CLOSE };

// 16 + code of one coordinate as a float, with a fraction where it lies in the band of a threshold. x: the coordinate of
// W x, b = big / s, off[j] = 0.5 - big t_j, big = 0.5 / GUARD.
template <int BITS, int MODE, int NS>
__device__ __forceinline__ float bulk_decide(float x, float b, const float (&off)[NS]) {
  if constexpr (MODE == BULK_CLOSE) {
    float lo = 16.0f, hi = 16.0f;
#pragma unroll
    for (int j = 0; j < NS; j++) {
      const float v = fmaf(x, b, off[j]);
      lo += v >= 1.0f ? 1.0f : 0.0f;
      hi += v > 0.0f ? 1.0f : 0.0f;
    }
    return hi > lo ? lo + 0.5f : lo;
  } else if constexpr (MODE == BULK_SYMMETRIC) {
    float m = __saturatef(fmaf(fabsf(x), b, off[0]));
#pragma unroll
    for (int j = 1; j < NS; j++) m += __saturatef(fmaf(fabsf(x), b, off[j]));
    return __uint_as_float(__float_as_uint(m) | (__float_as_uint(x) & 0x80000000u)) + (__saturatef(fmaf(x, b, 0.5f)) + (16.0f + (float)NS));
  } else {
    float m = __saturatef(fmaf(x, b, off[0])) + 16.0f;
#pragma unroll
    for (int j = 1; j < NS; j++) m += __saturatef(fmaf(x, b, off[j]));
    return m;
  }
}

// 32 columns of a lane: the nibble words of their codes, and per word the fraction bits of its sums OR-ed together.
// ROWS: a column is a row (V tiles), its b in shared memory; otherwise the lane is one, b0.
template <int BITS, int MODE, bool ROWS, int NS>
__device__ __forceinline__ void bulk_pack32(uint32_t taddr, const float* b_s, float b0, const float (&off)[NS], uint32_t (&nib)[4], uint32_t (&odd)[4]) {
  constexpr float MAGIC = 8388608.0f - 16.0f * 4369.0f;  // 2^23 - the 16 of four sums, one per nibble
  uint32_t xr[32];
  tc_ld32(taddr, xr);
#pragma unroll
  for (int q = 0; q < 4; q++) {
    float tt[2];
    uint32_t acc = 0u;
#pragma unroll
    for (int hq = 0; hq < 2; hq++) {
      float4 b4;
      if constexpr (ROWS) b4 = *reinterpret_cast<const float4*>(b_s + 8 * q + 4 * hq);
      else b4 = make_float4(b0, b0, b0, b0);
      const uint32_t* x = xr + 8 * q + 4 * hq;
      const float c0 = bulk_decide<BITS, MODE, NS>(__uint_as_float(x[0]), b4.x, off), c1 = bulk_decide<BITS, MODE, NS>(__uint_as_float(x[1]), b4.y, off);
      const float c2 = bulk_decide<BITS, MODE, NS>(__uint_as_float(x[2]), b4.z, off), c3 = bulk_decide<BITS, MODE, NS>(__uint_as_float(x[3]), b4.w, off);
      tt[hq] = fmaf(c3, 4096.f, fmaf(c2, 256.f, fmaf(c1, 16.f, c0 + MAGIC)));
      acc = (acc | __float_as_uint(c0) | __float_as_uint(c1));
      acc = (acc | __float_as_uint(c2) | __float_as_uint(c3));
    }
    nib[q] = prmt(__float_as_uint(tt[0]), __float_as_uint(tt[1]), 0x5410u);
    odd[q] = acc & 0x0007FFFFu;  // the fraction bits of a float in [16, 32)
  }
}

template <int D, int BITS, int MODE>
__global__ void __launch_bounds__(BulkLayout<D>::THREADS, 1) append_bulk_kernel(const __grid_constant__ QuantizeParams p, const __grid_constant__ int batch) {
  using L = BulkLayout<D>;
  constexpr int NJ = L::NJ, NG = L::NG, GT = L::GT;
  constexpr int NT = (1 << BITS) - 1;                   // thresholds
  constexpr bool SYM = MODE == BULK_SYMMETRIC;
  constexpr int NS = SYM ? (1 << (BITS - 1)) - 1 : NT;  // those compared one by one (besides zero)

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool control = tid >= L::PACK;
  const int grp = control ? warp - L::PACK / 32 : tid / GT;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::OFF_BAR);
  uint64_t* tile_bar = bars + 5 * grp;       // the next tile has been described
  uint64_t* copy_bar = bars + 5 * grp + 1;   // the tile (half) is in the buffer, the accumulator has been read
  uint64_t* norm_bar = bars + 5 * grp + 2;   // the norms are in shared memory, the buffer has been read
  uint64_t* full_bar = bars + 5 * grp + 3;   // the MMAs are done
  uint64_t* drain_bar = bars + 5 * grp + 4;  // (after a wait that gave up) all MMAs of the group are done
  BulkTile* tiles = reinterpret_cast<BulkTile*>(smem + L::OFF_TILE) + L::TILES * grp;
  uint8_t* xs = smem + L::OFF_X + grp * L::OPERAND;
  long long* pre_s = reinterpret_cast<long long*>(smem + L::OFF_PRE);
  long long* wsum_s = reinterpret_cast<long long*>(smem + L::OFF_WSUM);
  float* tau_s = reinterpret_cast<float*>(smem + L::OFF_TAU);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::OFF_MISC);
  int* zero_code_s = reinterpret_cast<int*>(smem + L::OFF_MISC + 8);    // [2] code of u = 0, K and V (+ 16: it is near a threshold)

  volatile int* started_s = reinterpret_cast<volatile int*>(smem + L::OFF_MISC + 16);  // [NG]

  // ---- set-up that reads nothing a predecessor may have written
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
  }
  if (control && lane == 0) {
    mbar_init(tile_bar, 1);
    mbar_init(copy_bar, GT);
    mbar_init(norm_bar, GT);
    mbar_init(full_bar, 1);
    mbar_init(drain_bar, 1);
    fence_mbar_init();
  }
  if (tid == L::PACK) {
    int zk = 0, zv = 0;
    for (int j = 0; j < NT; j++) {
      zk = (zk + (0.f > p.thresholds_k[j] ? 1 : 0)) | (fabsf(p.thresholds_k[j]) <= GUARD_BAND ? 16 : 0);
      zv = (zv + (0.f > p.thresholds_v[j] ? 1 : 0)) | (fabsf(p.thresholds_v[j]) <= GUARD_BAND ? 16 : 0);
    }
    zero_code_s[0] = zk;
    zero_code_s[1] = zv;
    for (int g = 0; g < NG; g++) started_s[g] = 0;
  }
  if (tid < 32) tau_s[tid] = (tid & 15) < NT ? p.big * (tid < 16 ? p.thresholds_k[tid & 15] : p.thresholds_v[tid & 15]) : 0.f;
  if (tid < L::PACK / 32) reinterpret_cast<int*>(smem + L::OFF_WARP)[tid] = 0;
  grid_dependency_wait();

  // ---- blocks of every sequence; this CTA's share of the tiles
  auto seq_blocks = [&](int b, int& pos0, int& n, long long& blk0) {
    n = min(p.n_new ? p.n_new[b] : p.n_new_max, p.n_new_max);
    pos0 = p.append_pos[b];
    if (n <= 0) { n = 0; blk0 = 0; return 0; }
    blk0 = (long long)pos0 >> 7;  // floor
    return (int)((((long long)pos0 + n - 1) >> 7) - blk0 + 1);
  };
  const int per = (batch + L::THREADS - 1) / L::THREADS;  // sequences per slice
  {
    long long sum = 0;
    for (int b = tid * per; b < min(batch, (tid + 1) * per); b++) {
      int pos0, n;
      long long blk0;
      sum += seq_blocks(b, pos0, n, blk0);
    }
    long long inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long t = __shfl_up_sync(FULL, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) wsum_s[warp] = inc;
    __syncthreads();
    long long before = 0;
    for (int w = 0; w < warp; w++) before += wsum_s[w];
    pre_s[tid] = before + inc - sum;
    if (tid == L::THREADS - 1) pre_s[L::THREADS] = before + inc;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot[0];
  const long long nb = pre_s[L::THREADS];          // tiles of one tensor of one head
  const long long total = 2 * nb * p.n_kv_heads;
  const long long lo = total * blockIdx.x / gridDim.x, hi = total * (blockIdx.x + 1) / gridDim.x;
  bool failed = false;      // a bounded wait gave up: the CTA leaves at the end of the head
  uint32_t n_redone = 0;    // (the first four threads of a group) rows with coordinates decided again
  // phases, kept over the heads: tiles described, halves copied in (= MMA batches), tiles whose norms are done
  uint32_t n_tile = 0, n_half = 0, n_norm = 0;
  bool first = true;

  long long item = lo;
  while (item < hi) {  // one head per pass
    const int h = (int)(item / (2 * nb));
    const long long head0 = 2 * nb * h;
    const long long seg_lo = item - head0, seg_hi = min(hi - head0, 2 * nb);
    const float* rot_head = p.rot + (size_t)h * (D / 4) * 8;

    if (control) {
      // ================================================================ control warp of group grp
      BulkWalk w;
      w.is_v = -1;
      w.b = 0; w.first = 0; w.n_tiles = 0; w.blk0 = 0; w.pos0 = 0; w.n_new = 0;
      long long it = seg_lo + grp;
      BulkTile nt;
      nt.kind = 0; nt.c_lo = nt.c_hi = 0; nt.row0 = 0; nt.src = nullptr; nt.special = 0;
      auto locate = [&](long long j) {  // the sequence of tile j of a tensor
        int a = 0, z = L::THREADS;
        while (z - a > 1) { const int m = (a + z) >> 1; if (pre_s[m] <= j) a = m; else z = m; }
        long long first = pre_s[a];
        for (int b = a * per;; b++) {
          w.n_tiles = seq_blocks(b, w.pos0, w.n_new, w.blk0);
          if (j < first + w.n_tiles || b + 1 >= batch) { w.b = b; w.first = first; return; }
          first += w.n_tiles;
        }
      };
      // describes the group's next tile; tiles outside the cache or without a page are counted and passed over
      auto describe_next = [&]() {
        bool found = false;
        for (; it < seg_hi && !found; it += NG) {
          const int is_v = it >= nb ? 1 : 0;
          const long long j = it - (is_v ? nb : 0);
          if (is_v != w.is_v || j >= w.first + w.n_tiles) { w.is_v = is_v; locate(j); }
          const long long t0 = (w.blk0 + (j - w.first)) * 128;
          nt.kind = is_v;
          nt.c_lo = (int)(max(t0, (long long)w.pos0) - t0);
          nt.c_hi = (int)(min(t0 + 128, (long long)w.pos0 + w.n_new) - t0);
          found = t0 >= 0 && t0 + 128 <= p.t_cap;
          if (!found && lane == 0 && p.status) atomicOr(&p.status[0], IQ_STATUS_ROW_OUT_OF_RANGE);
          if (found) found = cache_row_for_write(p.pm, w.b, h, t0, lane == 0 ? p.status : nullptr, nt.row0);
          if (found) nt.src = (is_v ? p.v_new : p.k_new) + (size_t)w.b * p.stride_b + (size_t)h * p.stride_h + (t0 - (long long)w.pos0) * p.stride_t;
          else if (lane == 0 && p.status) atomicAdd(&p.status[2], (unsigned)(nt.c_hi - nt.c_lo));
        }
        if (lane == 0) {
          BulkTile d = nt;
          d.special = 0;
          if (!found) d.kind = -1;
          tiles[n_tile % L::TILES] = d;
          mbar_arrive(tile_bar);
        }
        __syncwarp();
        n_tile++;
        return found;
      };
      bool have = describe_next();
      __syncthreads();  // W is in place
      while (have) {
        const bool is_v = nt.kind != 0;
#pragma unroll
        for (int hf = 0; hf < NJ; hf++) {
          if (!failed) failed = __any_sync(FULL, !mbar_wait_bounded(copy_bar, n_half & 1u, DEC_WAIT_LIMIT));
          n_half++;
          if (failed) continue;
          tc_fence_after();
          if (elect_one()) {
            const uint64_t xd = smem_desc_k128(smem_u32(xs));
#pragma unroll
            for (int j = 0; j < NJ; j++)
#pragma unroll
              for (int hl = 0; hl < 2; hl++) {  // W_lo, then W_hi; the second half the other way round
                const uint64_t wd = smem_desc_k128(smem_u32(smem + (2 * j + (hf ? 1 - hl : hl)) * L::OPERAND));
                const uint64_t a0 = is_v ? wd : xd, b0 = is_v ? xd : wd;
#pragma unroll
                for (int k = 0; k < 8; k++) {  // 16 contraction steps each: 32 bytes inside a 128-byte row, 4 per slab
                  const uint64_t step = (uint64_t)((k >> 2) * (L::OPERAND / 2) + (k & 3) * 32) >> 4;
                  tc_mma_f16_ss(tmem_base + grp * GT + 128 * j, a0 + step, b0 + step, (j & hf) ? TILE_IDESC | TILE_IDESC_NEG_A : TILE_IDESC, (hf | hl | k) != 0);
                }
              }
            tc_commit(full_bar);
          }
          __syncwarp();
        }
        have = describe_next();  // (into the slot of the tile four before: the group was done with it when it had the one before this copied in)
      }
    } else {
      // ================================================================ packing group: thread = tensor-memory lane (and 128-column half)
      const int gt = tid % GT, r = gt & 127, part = gt >> 7;
      const uint32_t tmem_t = tmem_base + (uint32_t)(grp * GT) + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(part * 128);
      float* binv_s = reinterpret_cast<float*>(smem + L::OFF_BINV) + grp * 128;
      double* ss_s = reinterpret_cast<double*>(smem + L::OFF_SS) + grp * 256;
      uint8_t* list = smem + L::OFF_LIST + warp * L::LIST_BYTES;
      const __half** src_s = reinterpret_cast<const __half**>(list);
      uint32_t** dst_s = reinterpret_cast<uint32_t**>(list + 8 * L::LIST);
      uint32_t* info_s = reinterpret_cast<uint32_t*>(list + 16 * L::LIST);
      int* const n_list_s = reinterpret_cast<int*>(smem + L::OFF_WARP) + warp;
      BulkRows* rows_s = reinterpret_cast<BulkRows*>(smem + L::OFF_ROWS) + grp;
      double* m_s = reinterpret_cast<double*>(smem + L::OFF_M);

      // 128-coordinate half hf of a tile's rows into the group's buffer; rows that are not new repeat the nearest one that
      // is (their results are dropped)
      auto load_half = [&](const BulkTile& t, int hf) {
        const int ch = gt & 15, c_lo = t.c_lo, c_last = t.c_hi - 1;
        const __half* src = t.src + hf * 128 + ch * 8;
        const uint32_t dst0 = smem_u32(xs) + (uint32_t)((ch >> 3) * (L::OPERAND / 2));
#pragma unroll
        for (int i = 0; i < 2048 / GT; i++) {
          const int row = (gt >> 4) + i * (GT / 16);
          const int rs = min(max(row, c_lo), c_last);
          cp_async16(dst0 + (uint32_t)(row * 128 + (((ch & 7) ^ (row & 7)) * 16)), src + (long long)rs * p.stride_t);
        }
      };
      auto copied_in = [&]() {  // this thread's copies have arrived (and its reads of the accumulator are done)
        cp_async_wait_all();
        fence_proxy_async();
        tc_fence_before();
        mbar_arrive(copy_bar);
        if (!failed) failed = !mbar_wait_bounded(copy_bar, n_half & 1u, DEC_WAIT_LIMIT);
      };
      // squares of this thread's share of row r in the buffer (exact products, summed in fp64)
      auto square_sum = [&]() {
        double s4[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int c = 0; c < 16 / NJ; c++) {
          const int ch = part * (16 / NJ) + c;
          const uint4 t4 = *reinterpret_cast<const uint4*>(xs + (ch >> 3) * (L::OPERAND / 2) + r * 128 + (((ch & 7) ^ (r & 7)) * 16));
          const uint32_t wv[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
          for (int q = 0; q < 4; q++) {
            const double a = half_to_double(wv[q]), b = half_to_double(wv[q] >> 16);
            s4[q] = fma(a, a, s4[q]);
            s4[q] = fma(b, b, s4[q]);
          }
        }
        return (s4[0] + s4[1]) + (s4[2] + s4[3]);
      };
      auto describe = [&]() -> BulkTile* {  // the group's next tile, or none
        if (!failed) failed = !mbar_wait_bounded(tile_bar, n_tile & 1u, DEC_WAIT_LIMIT);
        BulkTile* t = &tiles[n_tile % L::TILES];
        n_tile++;
        return t;
      };

      // Warp w of the group decides the rows of its quarter again that are marked in tile number `no`. d = 256 has two warps per
      // quarter: K rows go to the one or the other by turns, V rows by halves.
      auto redo_marked = [&](uint32_t no) {
        uint32_t m = __shfl_sync(FULL, rows_s->full[no & 1u][warp & 3], 0);
        if (m == 0u) return;
        const BulkTile* t = &tiles[no % L::TILES];
        if (NJ == 2 && t->kind == 0) m &= part ? 0xAAAAAAAAu : 0x55555555u;
        if (m != 0u) bulk_redo_rows<D, BITS>(p, m_s, t, m, warp & 3, part, lane);
        __syncwarp();
      };
      if (gt < 16) reinterpret_cast<uint32_t*>(rows_s)[gt] = 0u;

      tile_build_m<D>(rot_head, m_s, tid);  // (while the control warps find the first tiles)
      BulkTile* t = describe();
      int kind = failed ? -1 : t->kind;
      if (kind >= 0) load_half(*t, 0);
      cta_bar_sync_n(1, L::PACK);
      bulk_build_w<D>(m_s, smem, tid);
      fence_proxy_async();
      __syncthreads();  // W is in place

      while (!__any_sync(FULL, failed || kind < 0)) {
        copied_in();
        n_half++;
        redo_marked(n_tile - 2u);  // the tile before this one, number n_tile - 1
        if (first) {  // the groups' first norms one after the other: the conversions of all groups at once would keep one
                      // pipe busy and the others idle, tile after tile
          for (int i = 0; i < 64 && grp > 0 && started_s[grp - 1] == 0; i++) __nanosleep(64);
        }
        double ss = square_sum();
        if (first && gt == 0) started_s[grp] = 1;
        first = false;
        if constexpr (NJ == 2) {
          ss_s[part * 128 + r] = ss;
          mbar_arrive(norm_bar);  // everybody has read the first half ...
          if (!failed) failed = !mbar_wait_bounded(norm_bar, n_norm & 1u, DEC_WAIT_LIMIT);
          n_norm++;
          if (!failed) failed = !mbar_wait_bounded(full_bar, (n_half - 1) & 1u, p.wait_polls);  // ... the MMAs too
          load_half(*t, 1);
          copied_in();
          n_half++;
          ss = square_sum();
          ss_s[part * 128 + r] += ss;
          mbar_arrive(norm_bar);
          if (!failed) failed = !mbar_wait_bounded(norm_bar, n_norm & 1u, DEC_WAIT_LIMIT);
          n_norm++;
          ss = ss_s[r] + ss_s[128 + r];
        }
        const bool is_v = kind != 0;
        const BulkTile* const cur = t;  // (read where it is needed: its slot is kept, registers are short)
        float binv = 0.f;
        if (NJ == 1 || part == 0 || !is_v) {
          float s = sqrtf((float)ss);
          {  // the correctly rounded root by exact fp64 midpoint tests
            const float up = __uint_as_float(__float_as_uint(s) + 1u);
            const float dn = (s > 0.f) ? __uint_as_float(__float_as_uint(s) - 1u) : 0.f;
            const double mu = 0.5 * ((double)s + (double)up), md = 0.5 * ((double)s + (double)dn);
            if (ss > mu * mu) s = up;
            else if (s > 0.f && ss < md * md) s = dn;
          }
          const bool ordinary = s > 0.f && s < INFINITY;
          binv = ordinary ? p.big * __frcp_rn(s) : 0.f;
          if (part == 0) {
            if (is_v) binv_s[r] = binv;
            if (r >= cur->c_lo && r < cur->c_hi) {
              if (!ordinary) t->special = 1;
              store_scale(is_v ? p.v_scales : p.k_scales, cur->row0 + r, s, p.scale_f16, p.status);
            }
          }
        }
        float off[NS];
#pragma unroll
        for (int j = 0; j < NS; j++) off[j] = 0.5f - tau_s[(is_v ? 16 : 0) + (SYM ? j + (1 << (BITS - 1)) : j)];
        mbar_arrive(norm_bar);
        if (!failed) failed = !mbar_wait_bounded(norm_bar, n_norm & 1u, DEC_WAIT_LIMIT);
        n_norm++;
        if (gt < 4) {  // everybody has read the marks of the tile before; the next tile sets its own there
          n_redone += __popc(rows_s->near[n_tile & 1u][gt]);
          rows_s->full[n_tile & 1u][gt] = rows_s->near[n_tile & 1u][gt] = 0u;
        }
        if (!failed) failed = !mbar_wait_bounded(full_bar, (n_half - 1) & 1u, p.wait_polls);
        tc_fence_after();
        const bool special = t->special != 0;
        // the next tile's copy runs under the packing of this one
        t = describe();
        kind = failed ? -1 : t->kind;
        if (kind >= 0) load_half(*t, 0);

        // ---- decisions and packing: 128 columns of this thread's lane, 32 at a time
        auto run_of = [&]() {  // the record (V) or packed row (K) of this thread
          return reinterpret_cast<uint32_t*>(is_v ? p.v_codes + ((cur->row0 / 128) * D + gt) * (size_t)(16 * BITS)
                                                  : p.k_codes + (cur->row0 + r) * (size_t)(BITS * D / 8));
        };
        uint32_t word[4 * BITS];
#pragma unroll
        for (int i = 0; i < 4 * BITS; i++) word[i] = 0u;
#pragma unroll 1
        for (int ch = 0; ch < 4; ch++) {
          uint32_t nib[4], odd[4];
          if (is_v) bulk_pack32<BITS, MODE, true, NS>(tmem_t + 32 * ch, binv_s + 32 * ch, 0.f, off, nib, odd);
          else bulk_pack32<BITS, MODE, false, NS>(tmem_t + 32 * ch, nullptr, binv, off, nib, odd);
          if (__any_sync(FULL, special || ((odd[0] | odd[1]) | (odd[2] | odd[3])) != 0u)) {
            // some coordinate of the warp lies in a band (or the tile has rows to be treated apart): the words in question
            // again, with the nearest codes, and the coordinates of new rows go on the list
            const uint32_t odd_words = (odd[0] ? 1u : 0u) | (odd[1] ? 2u : 0u) | (odd[2] ? 4u : 0u) | (odd[3] ? 8u : 0u);
            const uint32_t valid = is_v ? new_rows(cur->c_lo, cur->c_hi, ch) : (r >= cur->c_lo && r < cur->c_hi ? 255u : 0u);  // the new rows
#pragma unroll 1
            for (int q = 0; q < 4; q++) {
              if (!special && !__any_sync(FULL, (odd_words >> q) & 1u)) continue;
              uint32_t x8[8], nw = 0u, near_m = 0u;  // the nearest codes, which of them are undecided (+ 8: of a zero row, at a threshold)
              float b8[8];
              tc_ld8(tmem_t + 32 * ch + 8 * q, x8);
#pragma unroll
              for (int i = 0; i < 8; i++) b8[i] = is_v ? binv_s[32 * ch + 8 * q + i] : binv;
#pragma unroll
              for (int i = 0; i < 8; i++) {
                const uint32_t cb = __float_as_uint(bulk_decide<BITS, MODE, NS>(__uint_as_float(x8[i]), b8[i], off));
                nw |= (((cb + 0x0003FFFFu) >> 19) & 15u) << (4 * i);
                if (cb & 0x0007FFFFu) near_m |= 1u << i;
              }
              if (special) {
#pragma unroll
                for (int i = 0; i < 8; i++) {
                  if (b8[i] != 0.f) continue;
                  const float z = __uint_as_float(x8[i]) * 0.f;  // a row of norm zero: u = 0; one whose norm is not finite: not a number, above no threshold
                  const uint32_t zc = (uint32_t)zero_code_s[is_v ? 1 : 0];
                  nw = (nw & ~(15u << (4 * i))) | (z != z ? 0u : (zc & 15u) << (4 * i));
                  near_m &= ~(1u << i);
                  if (z == z && zc >= 16u) near_m |= 256u << i;  // (only counted)
                }
              }
              near_m &= ((is_v ? valid >> (8 * q) : valid) & 255u) * 257u;
#pragma unroll
              for (int k = 0; k < 4; k++) nib[k] = (k == q) ? nw : nib[k];
              uint32_t rows;
              if (is_v) {
                rows = __reduce_or_sync(FULL, near_m);
                rows = ((rows | rows >> 8) & 255u) << (8 * q);
              } else {
                rows = __ballot_sync(FULL, near_m != 0u);
              }
              if (lane == 0) atomicOr(&rows_s->near[n_tile & 1u][is_v ? ch : warp & 3], rows);
              near_m &= 255u;
              const int n_list = *n_list_s, n_near = (int)__reduce_add_sync(FULL, (unsigned)__popc(near_m));
              if (n_near > L::LIST_STEP || n_list + n_near > L::LIST) {  // their rows again as a whole (the tile's number is n_tile - 2)
                if (lane == 0) atomicOr(&rows_s->full[n_tile & 1u][is_v ? ch : warp & 3], rows);
                near_m = 0u;
              }
              __syncwarp();
              while (near_m) {
                const int i = __ffs(near_m) - 1, col = 32 * ch + 8 * q + i;
                near_m &= near_m - 1u;
                const int row = is_v ? col : r, coord = is_v ? gt : part * 128 + col;
                const int k = atomicAdd(n_list_s, 1);
                src_s[k] = cur->src + (long long)row * p.stride_t;
                dst_s[k] = run_of();
                info_s[k] = (uint32_t)coord | ((uint32_t)(is_v ? row : coord) << 8) | (((nw >> (4 * i)) & 15u) << 16) | (is_v ? 1u << 20 : 0u);
              }
              __syncwarp();
            }
          }
#pragma unroll
          for (int i = 0; i < 3 * BITS; i++) word[i] = word[i + BITS];
          pack_nibbles<BITS>(nib, word + 3 * BITS);
        }
        const int c_lo = cur->c_lo, c_hi = cur->c_hi;
        uint32_t* const dst = run_of() + (is_v ? 0 : part * (4 * BITS));
        if (is_v ? (c_lo == 0 && c_hi == 128) : (r >= c_lo && r < c_hi)) {
#pragma unroll
          for (int i = 0; i < BITS; i++)
            reinterpret_cast<uint4*>(dst)[i] = make_uint4(word[4 * i], word[4 * i + 1], word[4 * i + 2], word[4 * i + 3]);
        } else if (is_v) {  // a partly new block: the other rows' codes stay
#pragma unroll
          for (int u = 0; u < 4; u++) {
            const uint32_t vm = new_rows(c_lo, c_hi, u);
            if (vm == 0u) continue;
#pragma unroll
            for (int k = 0; k < BITS; k++) {
              const uint32_t m = packed_mask<BITS>(vm, k);
              if (m == 0u) continue;
              uint32_t* d = dst + BITS * u + k;
              *d = m == 0xFFFFFFFFu ? word[BITS * u + k] : ((*d & ~m) | (word[BITS * u + k] & m));
            }
          }
        }
        __syncwarp();  // the warp's stores come before the changes made to them below
        const int n_list = *n_list_s;
        if (n_list >= L::LIST_FLUSH) {
          bulk_redo<D, BITS>(p, m_s, src_s, dst_s, info_s, n_list, lane);
          __syncwarp();
          if (lane == 0) *n_list_s = 0;
          __syncwarp();
        }
      }
      const int n_list = *n_list_s;
      if (n_list > 0) {
        bulk_redo<D, BITS>(p, m_s, src_s, dst_s, info_s, n_list, lane);
        __syncwarp();
        if (lane == 0) *n_list_s = 0;
      }
      cta_bar_sync_n(2 + grp, GT);  // the marks of the group's last tile, and the stores to it, are in place
      if (!__any_sync(FULL, failed)) redo_marked(n_tile - 2u);
      if (gt < 4) n_redone += __popc(rows_s->near[n_tile & 1u][gt]);
    }
    item = head0 + seg_hi;
    if (__syncthreads_or(failed)) { failed = true; break; }  // (W is rebuilt for the next head)
  }

  allow_dependent_launch();
  if (n_redone && p.status) atomicAdd(&p.status[1], n_redone);
  if (failed && tid == 0 && p.status) atomicOr(&p.status[0], IQ_STATUS_WAIT_TIMEOUT);
  cp_async_wait_all();
  if (failed && control) {  // MMAs may still be running: they are waited for, again with a limit, before the tensor memory goes
    if (elect_one()) tc_commit(drain_bar);
    __syncwarp();
    mbar_wait_bounded(drain_bar, 0u, DEC_WAIT_LIMIT);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512));
}

template <int D, int BITS, int MODE>
static cudaError_t launch_bulk(const QuantizeParams& p, int batch, cudaStream_t stream) {
  using L = BulkLayout<D>;
  static bool configured[64] = {};
  static int n_sm[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  auto kern = append_bulk_kernel<D, BITS, MODE>;
  if (!configured[dev]) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&n_sm[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  // no more CTAs than tiles (a sequence's rows may begin and end inside a block)
  const long long tiles = 2ll * p.n_kv_heads * batch * (((long long)p.n_new_max + 127) / 128 + 1);
  const int ctas = (int)(tiles < n_sm[dev] ? tiles : n_sm[dev]);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3(L::THREADS);
  cfg.dynamicSmemBytes = L::SMEM;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, p, batch);
}

template <int D>
static cudaError_t launch_bulk_bits(const QuantizeParams& p, BulkMode mode, int batch, cudaStream_t stream) {
  if (p.bits == 2) return launch_bulk<D, 2, BULK_PLAIN>(p, batch, stream);
  if (p.bits == 4) return mode == BULK_SYMMETRIC ? launch_bulk<D, 4, BULK_SYMMETRIC>(p, batch, stream) : launch_bulk<D, 4, BULK_PLAIN>(p, batch, stream);
  if (mode == BULK_CLOSE) return launch_bulk<D, 3, BULK_CLOSE>(p, batch, stream);
  return mode == BULK_SYMMETRIC ? launch_bulk<D, 3, BULK_SYMMETRIC>(p, batch, stream) : launch_bulk<D, 3, BULK_PLAIN>(p, batch, stream);
}

// The largest threshold that a row can come near: |u| <= sqrt(d).
static float largest_threshold(const QuantizeParams& p, int head_dim) {
  float m = 0.f;
  for (const float* t : {p.thresholds_k, p.thresholds_v})
    for (int j = 0; j < (1 << p.bits) - 1; j++) m = fmaxf(m, fabsf(t[j]));
  return fminf(m, sqrtf((float)head_dim));
}

// No coordinate reaches this (|u| <= 16): thresholds beyond it are held here, where big * t keeps fractions.
constexpr float BULK_REACH = 32.f;

// Neighbouring thresholds that the saturating sums cannot tell apart (Lloyd-Max thresholds are 0.1 and more apart).
static bool close_thresholds(const QuantizeParams& p, int head_dim) {
  const float guard = bulk_guard(head_dim, largest_threshold(p, head_dim));
  for (const float* t : {p.thresholds_k, p.thresholds_v})
    for (int j = 1; j < (1 << p.bits) - 1; j++)
      if (t[j] > -BULK_REACH && t[j - 1] < BULK_REACH && !(t[j] - t[j - 1] > 8.f * guard)) return true;
  return false;
}

// 2 and 4 bits: close thresholds stay with a warp per row, which is all that these widths had.
bool append_bulk_takes(const QuantizeParams& p, int head_dim) { return p.bits == 3 || !close_thresholds(p, head_dim); }

cudaError_t launch_append_bulk(const QuantizeParams& params, int head_dim, int batch, cudaStream_t stream) {
  QuantizeParams p = params;
  p.big = 0.5f / bulk_guard(head_dim, largest_threshold(p, head_dim));
  const int nt = (1 << p.bits) - 1, mid = nt / 2;
  BulkMode mode = close_thresholds(p, head_dim) ? BULK_CLOSE : BULK_SYMMETRIC;
  for (float* t : {p.thresholds_k, p.thresholds_v}) {
    if (mode == BULK_SYMMETRIC && t[mid] != 0.f) mode = BULK_PLAIN;
    for (int j = 1; j <= mid; j++)
      if (mode == BULK_SYMMETRIC && t[mid - j] != -t[mid + j]) mode = BULK_PLAIN;
  }
  for (float* t : {p.thresholds_k, p.thresholds_v})
    for (int j = 0; j < nt; j++) t[j] = fminf(fmaxf(t[j], -BULK_REACH), BULK_REACH);
  return head_dim == 128 ? launch_bulk_bits<128>(p, mode, batch, stream) : launch_bulk_bits<256>(p, mode, batch, stream);
}

}  // namespace iq
