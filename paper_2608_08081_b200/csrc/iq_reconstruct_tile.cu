// Reconstruct-then-compute, first half (Figure 1, top) on the tensor cores: the rows of a 128-row block as one contraction
// X = L W with W = blockdiag(M_b) H_d, L the dequantised levels (exact binary16), times scale / d per row.
//
// Tile = (tensor, KV head, sequence, 128-row block). D[row][coordinate]: A = L, written into shared memory by the threads that
// look the codes up -- K: thread = row, K-major; V: thread = coordinate of the token-transposed records, MN-major --
// B = W^T in two binary16 terms. A thread then holds a whole row (half a row at d = 256): scale, one rounding to binary16,
// through shared memory so that rows leave in whole pieces. d = 256: H_256 = [[H, H], [H, -H]], so the contraction is two of
// 128 steps, one after the other through the same buffer, and the last stage of the butterfly, a sum and a difference in fp32.
//
// Precision. The instruction aligns its 16 products and the accumulator to the largest of them, keeps two bits below the fp32
// last place, and cuts; the sum is cut to fp32 again (read off in-bounds sums of known terms). Sixteen such cuts of running
// sums would cost more than the fp32 butterflies of iq_reconstruct.cu do. So the upper term of W is W rounded to a multiple of 2^-10
// and the levels are integers of up to 7 bits and a sign times one factor: every partial sum of their products is a multiple
// of 2^-10 below 128 * 128 (Cauchy-Schwarz: the columns of W have norm sqrt(128) per half), i.e. exact in fp32. The lower
// term (|W - hi| <= 2^-11, rounded to binary16: off by at most 2^-23) goes first, where cuts are 2^-11 as large, and is then
// cut once per doubling of the sum. Levels that are binary16 values of up to 15 bits are split in two such
// integers, 256 h + m, and take three passes through the buffer: level x lower term, m x upper, h x upper. Error against
// an fp64 evaluation before the rounding to binary16, relative to the row's rms: 0.9e-7 rms (two terms of 11 free bits each, all
// products into one sum: 1.3e-7 to 1.9e-7 at d = 128, 3e-7 with binary16 levels, 4e-7 to 7e-7 at d = 256).
//
// One persistent CTA per SM, equal contiguous shares of the tiles ordered by head; groups of 128 threads (256 at d = 256)
// take them in turn and request the next tile's codes while they work on the present one. About 20 warp instructions
// per row for the lookups, 20 for the rest; its memory traffic would take 19 us where it takes 45: the groups' barriers and
// the latency of each step bound it. Measured: 4 x 8 K rows, 8 KV heads, d = 128, 3 bits (407 k K and V rows): 44.6 us
// instead of 101 with butterflies by shuffle and codes picked one by one (iq_reconstruct.cu, which takes any levels). Three
// passes, 4 sequences of up to 8 K rows at d = 128 (4 K at 256), 3 bits: 52 us (65) where one takes 39 (49) and that kernel 88 (134).
#include <cmath>

#include "iq_kernels.h"
#include "iq_tile_mma.cuh"

namespace iq {

struct ReconstructTileParams {
  ReconstructParams r;
  int batch;
  uint32_t lo[2][3][4], hi[2][3][4];  // K and V: low / high bytes of the binary16 operand values of each pass (4 per register)
  int passes[2];                      // 1: the values with both terms of W; 3: with the lower, the upper, the upper term
  LookupConst lookup;
  float factor[2];                    // level = factor * the value of the one pass, or the values of the two that meet the upper term
};

constexpr uint32_t HALF2_NAN = 0x7FFF7FFFu;

template <int D>
struct ReconLayout {
  static constexpr int NJ = D / 128, GT = 128 * NJ, NG = 4 / NJ, THREADS = GT * NG;
  static constexpr int OFF_X = NJ * 2 * TILE_OPERAND;                // after W^T: [half of the contraction][lo, hi]
  static constexpr int OFF_M = OFF_X + NG * TILE_OPERAND;            // [D][4] fp64 rows of the blocks
  static constexpr int OFF_T = OFF_M + D * 32;                       // [lo, hi][NJ][4][128] binary16: the magnitudes of W
  static constexpr int OFF_PRE = OFF_T + 2 * D * 8;                  // [THREADS + 1] int64 block counts before a slice of the batch
  static constexpr int OFF_WSUM = OFF_PRE + 8 * (THREADS + 2);
  static constexpr int OFF_BAR = OFF_WSUM + 8 * 16;                  // [NG][2] mbarriers: MMAs done; all MMAs of a group that gave up
  static constexpr int OFF_MISC = OFF_BAR + 16 * NG;
  static constexpr int SMEM = OFF_MISC + 16 + 1024;
};
static_assert(ReconLayout<128>::SMEM <= 227 * 1024 && ReconLayout<256>::SMEM <= 227 * 1024, "shared memory overflow");

// SPLIT: some side takes three passes (an instance of its own: the loop over one pass costs 3 % at d = 128).
template <int D, int BITS, bool SPLIT>
__global__ void __launch_bounds__(ReconLayout<D>::THREADS, 1) reconstruct_tile_kernel(const __grid_constant__ ReconstructTileParams q) {
  using L = ReconLayout<D>;
  constexpr int NJ = L::NJ, NG = L::NG, GT = L::GT;
  constexpr int WPH = 4 * BITS / NJ;   // packed words of a thread per half of the contraction
  constexpr int UPH = 4 / NJ;          // the same in units of 32 entries
  const ReconstructParams& p = q.r;

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int grp = tid / GT, gt = tid % GT, r = gt & 127, part = gt >> 7, bar_id = 1 + grp;
  uint8_t* xs = smem + L::OFF_X + grp * TILE_OPERAND;
  double* m_s = reinterpret_cast<double*>(smem + L::OFF_M);
  __half* t_s = reinterpret_cast<__half*>(smem + L::OFF_T);
  long long* pre_s = reinterpret_cast<long long*>(smem + L::OFF_PRE);
  long long* wsum_s = reinterpret_cast<long long*>(smem + L::OFF_WSUM);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + L::OFF_BAR) + 2 * grp;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::OFF_MISC);

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
  }
  if (gt == 0) {
    mbar_init(bar, 1);
    mbar_init(bar + 1, 1);
    fence_mbar_init();
  }
  grid_dependency_wait();

  auto len_of = [&](int b) { return max(0, min(p.seq_lens[b], min(p.t_cap, p.out_rows))); };
  const int per = (q.batch + L::THREADS - 1) / L::THREADS;  // sequences per slice
  {
    long long sum = 0;
    for (int b = tid * per; b < min(q.batch, (tid + 1) * per); b++) sum += (len_of(b) + 127) / 128;
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
  const long long nb = pre_s[L::THREADS], total = 2 * nb * p.n_kv_heads;  // tiles of a tensor of a head, all tiles
  const long long lo = total * blockIdx.x / gridDim.x, hi = total * (blockIdx.x + 1) / gridDim.x;
  const uint32_t tmem_g = tmem_base + (uint32_t)(grp * GT);
  const uint32_t tmem_t = tmem_g + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(part * 64);
  bool failed = false;  // a bounded wait gave up (the whole group knows from its next barrier on): the rows it still owes become NaN
  uint32_t phase = 0;

  long long item = lo;
  while (item < hi) {  // one head per pass
    const int h = (int)(item / (2 * nb));
    const long long head0 = 2 * nb * h;
    const long long seg_lo = item - head0, seg_hi = min(hi - head0, 2 * nb);

    // ---- the group's next tile and its packed words
    int w_v = -1, w_b = 0, w_n = 0, w_len = 0;  // tensor, sequence, its tiles and rows
    long long w_first = 0;                      // its first tile in the tensor
    long long it = seg_lo + grp;
    uint32_t words[NJ * WPH];
    float scale = 0.f;
    int blk = 0;
    auto fetch = [&]() {
      w_v = it >= nb ? 1 : 0;
      const long long j = it - (w_v ? nb : 0);
      if (j < w_first || j >= w_first + w_n) {
        int a = 0, z = L::THREADS;
        while (z - a > 1) { const int m = (a + z) >> 1; if (pre_s[m] <= j) a = m; else z = m; }
        w_first = pre_s[a];
        for (w_b = a * per;; w_b++) {
          w_len = len_of(w_b);
          w_n = (w_len + 127) / 128;
          if (j < w_first + w_n || w_b + 1 >= q.batch) break;
          w_first += w_n;
        }
      }
      blk = (int)(j - w_first);
      const size_t row0 = cache_row(p.pm, w_b, h, (long long)blk * 128, nullptr);
      const uint8_t* src = w_v ? p.v_codes + ((row0 / 128) * D + r) * (size_t)(16 * BITS) : p.k_codes + (row0 + r) * (size_t)(BITS * D / 8);
      const size_t half_step = w_v ? (size_t)128 * 16 * BITS : (size_t)16 * BITS;
#pragma unroll
      for (int hf = 0; hf < NJ; hf++)
#pragma unroll
        for (int i = 0; i < WPH / 2; i++) {
          const uint2 t = *reinterpret_cast<const uint2*>(src + hf * half_step + part * (4 * WPH) + 8 * i);
          words[hf * WPH + 2 * i] = t.x;
          words[hf * WPH + 2 * i + 1] = t.y;
        }
      scale = load_scale(w_v ? p.v_scales : p.k_scales, row0 + r, p.scale_f16);
    };
    bool have = it < seg_hi;
    if (have) fetch();

    // ---- W^T of the head: W[i][k] = +-V4_i[k % 4], sign (-1)^popc(b & l) with b the 4-block of i, l that of k, in their halves
    tile_build_m<D>(p.rot + (size_t)h * (D / 4) * 8, m_s, tid);
    __syncthreads();
    if (tid < D) {
      const double* m = m_s + 4 * tid;
      const double v4[4] = {(m[0] + m[1]) + (m[2] + m[3]), (m[0] - m[1]) + (m[2] - m[3]), (m[0] + m[1]) - (m[2] + m[3]), (m[0] - m[1]) - (m[2] - m[3])};
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const __half x = __double2half(rint(v4[e] * 1024.0) * (1.0 / 1024.0));  // |V4| <= 2: exact in binary16
        t_s[((NJ + (tid >> 7)) * 4 + e) * 128 + (tid & 127)] = x;
        t_s[((tid >> 7) * 4 + e) * 128 + (tid & 127)] = __double2half(v4[e] - (double)__half2float(x));
      }
    }
    __syncthreads();
#pragma unroll 2
    for (int c = tid; c < 2 * NJ * 2048; c += L::THREADS) {  // 16-byte chunk m of row k of operand (half, lo / hi)
      const int k = c & 127, m = (c >> 7) & 15, op = c >> 11, l = k >> 2;
      const int hf = op >> 1, hl = op & 1;
      const uint4 t = *reinterpret_cast<const uint4*>(t_s + ((hl * NJ + hf) * 4 + (k & 3)) * 128 + 8 * m);
      const uint32_t s0 = (__popc(l & (2 * m)) & 1) ? 0x80008000u : 0u, s1 = (__popc(l & (2 * m + 1)) & 1) ? 0x80008000u : 0u;
      *reinterpret_cast<uint4*>(smem + op * TILE_OPERAND + (m >> 3) * (TILE_OPERAND / 2) + k * 128 + (((m & 7) ^ (k & 7)) * 16)) =
          make_uint4(t.x ^ s0, t.y ^ s0, t.z ^ s1, t.w ^ s1);
    }
    fence_proxy_async();
    __syncthreads();

    while (have) {
      const int is_v = w_v, b = w_b, row_base = blk * 128, n_rows = min(128, w_len - row_base);
      auto out_rows = [&]() { return (is_v ? p.v_out : p.k_out) + (size_t)b * p.stride_b + (size_t)row_base * p.stride_t + (size_t)h * p.stride_h; };
      if (failed) {  // no more MMAs
        __half* const out = out_rows();
        for (int i = gt; i < n_rows * (D / 8); i += GT)
          *reinterpret_cast<uint4*>(out + (long long)(i / (D / 8)) * p.stride_t + 8 * (i % (D / 8))) = make_uint4(HALF2_NAN, HALF2_NAN, HALF2_NAN, HALF2_NAN);
        it += NG;
        have = it < seg_hi;
        if (have) fetch();
        continue;
      }
      const float f = scale * q.factor[is_v] * (1.0f / (float)D);  // 1/sqrt(d) of the dequantisation times 1/sqrt(d) of H_d
      const int passes = SPLIT ? q.passes[is_v] : 1;
#pragma unroll
      for (int hf = 0; hf < NJ; hf++)
#pragma unroll 1
      for (int ps = 0; ps < passes; ps++) {
        uint32_t l_lo[4], l_hi[4];
#pragma unroll
        for (int i = 0; i < 4; i++) { l_lo[i] = q.lo[is_v][ps][i]; l_hi[i] = q.hi[is_v][ps][i]; }
#pragma unroll
        for (int u = 0; u < UPH; u++) {  // 32 entries -> four 16-byte pieces of the operand
          uint32_t lv[16];
          dequant32_f16<BITS>(words + hf * WPH + BITS * u, l_lo, l_hi, q.lookup, lv);
#pragma unroll
          for (int k = 0; k < 4; k++) {
            const int c = part * (16 / NJ) + 4 * u + k;  // piece: 8 coordinates of the row (K), 8 rows of the coordinate (V)
            const int off = is_v ? c * 2048 + (r & 7) * 16 + (r >> 3) * 128
                                 : (c >> 3) * (TILE_OPERAND / 2) + r * 128 + (((c & 7) ^ (r & 7)) * 16);
            *reinterpret_cast<uint4*>(xs + off) = make_uint4(lv[4 * k], lv[4 * k + 1], lv[4 * k + 2], lv[4 * k + 3]);
          }
        }
        fence_proxy_async();
        tc_fence_before();
        cta_bar_sync_n(bar_id, GT);
        if (gt < 32 && elect_one()) {
          tc_fence_after();
          const uint64_t ad0 = is_v ? smem_desc_mn(smem_u32(xs), 128, 2048) : smem_desc_k128(smem_u32(xs));
          const uint32_t idesc = TILE_IDESC | (is_v ? TILE_IDESC_MN_A : 0u);
#pragma unroll
          for (int hl = 0; hl < 2; hl++) {  // W_lo, then W_hi
            if (passes > 1 && hl != (ps > 0)) continue;
            const uint64_t bd0 = smem_desc_k128(smem_u32(smem + (2 * hf + hl) * TILE_OPERAND));
#pragma unroll
            for (int k = 0; k < 8; k++) {
              const uint64_t step = (uint64_t)((k >> 2) * (TILE_OPERAND / 2) + (k & 3) * 32) >> 4;
              tc_mma_f16_ss(tmem_g + 128 * hf, ad0 + (is_v ? (uint64_t)(16 * k) : step), bd0 + step, idesc, (ps | hl | k) != 0);
            }
          }
          tc_commit(bar);
        }
        __syncwarp();
        if (hf == NJ - 1 && ps == passes - 1) {  // the next tile's codes are on their way during the rest
          it += NG;
          have = it < seg_hi;
          if (have) fetch();
        }
        if (!failed) failed = !mbar_wait_bounded(bar, phase, p.wait_polls);
        phase ^= 1u;
      }
      tc_fence_after();
      __half* const out = out_rows();

      // ---- this thread's columns of row r (d = 256: 64 of each half's result): scale, round, through the operand's buffer
      // (256 bytes per row and round)
#pragma unroll
      for (int rd = 0; rd < NJ; rd++) {
        if (rd > 0) cta_bar_sync_n(bar_id, GT);  // the round before has left the buffer
#pragma unroll
        for (int ch = 0; ch < UPH / NJ; ch++) {  // 32 columns (d = 256: of both halves, which make 64 coordinates)
          uint32_t xr[NJ][32];
          tc_ld32(tmem_t + 32 * (NJ == 1 ? ch : rd), xr[0]);
          if constexpr (NJ == 2) tc_ld32(tmem_t + 128 + 32 * rd, xr[1]);
#pragma unroll
          for (int s = 0; s < NJ; s++)
#pragma unroll
            for (int k = 0; k < 4; k++) {
              uint32_t o[4];
#pragma unroll
              for (int i = 0; i < 4; i++) {
                float y[2];
#pragma unroll
                for (int e = 0; e < 2; e++) {
                  y[e] = __uint_as_float(xr[0][8 * k + 2 * i + e]);
                  if constexpr (NJ == 2) y[e] = s ? y[e] - __uint_as_float(xr[1][8 * k + 2 * i + e]) : y[e] + __uint_as_float(xr[1][8 * k + 2 * i + e]);
                }
                o[i] = pack_half2(y[0] * f, y[1] * f);
              }
              const int c = NJ == 1 ? 4 * ch + k : 8 * part + 4 * s + k;
              *reinterpret_cast<uint4*>(xs + r * 256 + ((c ^ (r & 7)) * 16)) = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
        failed = cta_bar_or_n(bar_id, GT, failed);
        const int c = gt & 15;  // piece of the row; its coordinate
        const int coord = NJ == 1 ? 8 * c : 128 * ((c >> 2) & 1) + 64 * (c >> 3) + 32 * rd + 8 * (c & 3);
#pragma unroll
        for (int i = 0; i < 2048 / GT; i++) {
          const int row = (gt >> 4) + i * (GT / 16);
          uint4 v = *reinterpret_cast<const uint4*>(xs + row * 256 + ((c ^ (row & 7)) * 16));
          if (failed) v = make_uint4(HALF2_NAN, HALF2_NAN, HALF2_NAN, HALF2_NAN);
          if (row < n_rows) *reinterpret_cast<uint4*>(out + (long long)row * p.stride_t + coord) = v;
        }
      }
      tc_fence_before();
      cta_bar_sync_n(bar_id, GT);  // the buffer and the accumulator have been read
    }
    item = head0 + seg_hi;
    __syncthreads();  // W^T is rebuilt for the next head
  }
  allow_dependent_launch();
  if (failed && gt < 32) {  // MMAs may still be running: they are waited for, again with a limit, before the tensor memory goes
    if (elect_one()) tc_commit(bar + 1);
    __syncwarp();
    mbar_wait_bounded(bar + 1, 0u, DEC_WAIT_LIMIT);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512));
}

template <int D, int BITS, bool SPLIT>
static cudaError_t launch_one(const ReconstructTileParams& q, cudaStream_t stream) {
  using L = ReconLayout<D>;
  static bool configured[64] = {};
  static int n_sm[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  auto kern = reconstruct_tile_kernel<D, BITS, SPLIT>;
  if (!configured[dev]) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&n_sm[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  const long long rows = q.r.t_cap < q.r.out_rows ? q.r.t_cap : q.r.out_rows;
  const long long tiles = 2ll * q.r.n_kv_heads * q.batch * ((rows + 127) / 128);
  const int ctas = (int)(tiles < n_sm[dev] ? tiles : n_sm[dev]);
  return launch_after_predecessor(kern, dim3((unsigned)ctas), dim3(L::THREADS), L::SMEM, stream, q);
}

template <bool SPLIT>
static cudaError_t launch_bits(const ReconstructTileParams& q, int head_dim, cudaStream_t stream) {
  const int bits = q.r.bits;
  if (head_dim == 128) return bits == 2 ? launch_one<128, 2, SPLIT>(q, stream) : (bits == 3 ? launch_one<128, 3, SPLIT>(q, stream) : launch_one<128, 4, SPLIT>(q, stream));
  return bits == 2 ? launch_one<256, 2, SPLIT>(q, stream) : (bits == 3 ? launch_one<256, 3, SPLIT>(q, stream) : launch_one<256, 4, SPLIT>(q, stream));
}

// The operand values of one side's levels, and how many passes they take. On the 8-bit grid (factor 1/127 of the largest level) a
// level is an integer of 7 bits and a sign: one pass, if its product with the factor rounds to the level in fp32; levels
// that are off the grid by an fp32 place or two take three, with the difference as the middle one (rounded to 11 bits, 2^-33 of the
// level). Binary16 levels that are integers of 15 bits and a sign in units of a power of two: three.
static bool operand_levels(const float* lv, int n, uint32_t (&lo)[3][4], uint32_t (&hi)[3][4], int& passes, float& factor) {
  for (int t = 0; t < 3; t++)
    for (int i = 0; i < 4; i++) lo[t][i] = hi[t][i] = 0u;
  auto put = [&](int t, int i, float v) {  // false: not a binary16 value
    const __half hv = __float2half_rn(v);
    const uint32_t bits = __half_as_ushort(hv);
    lo[t][i >> 2] |= (bits & 0xffu) << (8 * (i & 3));
    hi[t][i >> 2] |= (bits >> 8) << (8 * (i & 3));
    return fabsf(v) <= 65504.f && __half2float(hv) == v;
  };
  float mx = 0.f;
  for (int i = 0; i < n; i++) mx = fmaxf(mx, fabsf(lv[i]));
  const float f0 = mx / 127.0f;
  bool near_grid = f0 > 0.f;
  for (int i = 0; i < n; i++) near_grid = near_grid && fabsf(nearbyintf(lv[i] / f0) * f0 - lv[i]) <= 2.4e-7f * fabsf(lv[i]);
  if (near_grid) {
    passes = 3;
    factor = f0;
    for (const float f : {f0, nextafterf(f0, 0.f), nextafterf(f0, INFINITY)}) {
      bool grid = true;
      for (int i = 0; i < n; i++) grid = grid && nearbyintf(lv[i] / f) * f == lv[i];
      if (grid) { passes = 1; factor = f; break; }
    }
    for (int i = 0; i < n; i++) {
      const float v = nearbyintf(lv[i] / factor);
      put(0, i, v);
      put(1, i, (float)(((double)lv[i] - (double)v * factor) / factor));
      put(2, i, v);
    }
    return true;
  }
  float unit = 1.f;  // the largest power of two (at most 1) that all levels are multiples of
  for (int i = 0; i < n; i++)
    while (unit > 1e-9f && fmodf(lv[i], unit) != 0.f) unit *= 0.5f;
  bool ok = mx / unit <= 32767.f;
  for (int i = 0; i < n && ok; i++) {
    const float h = nearbyintf(lv[i] / unit / 256.f) * 256.f * unit;
    ok = put(0, i, lv[i]) && put(1, i, lv[i] - h) && put(2, i, h);
  }
  passes = 3;
  factor = 1.f;
  return ok;
}

bool launch_reconstruct_tiles(const ReconstructParams& p, int head_dim, int batch, cudaStream_t stream, cudaError_t& e) {
  ReconstructTileParams q;
  q.r = p;
  q.batch = batch;
  q.lookup = LOOKUP_CONST;
  if (!operand_levels(p.levels_k, 1 << p.bits, q.lo[0], q.hi[0], q.passes[0], q.factor[0])) return false;
  if (!operand_levels(p.levels_v, 1 << p.bits, q.lo[1], q.hi[1], q.passes[1], q.factor[1])) return false;
  e = q.passes[0] + q.passes[1] > 2 ? launch_bits<true>(q, head_dim, stream) : launch_bits<false>(q, head_dim, stream);
  return true;
}

}  // namespace iq
