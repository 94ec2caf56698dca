// Quantize-append for few new rows (Algorithm 1: normalise, WHT, SO(4) blocks, Lloyd-Max, bit-pack; a warp per row: the
// decode step, the verification of a few drafted rows), the dispatch between it and the bulk kernel (iq_append_bulk.cu), and the calibration kernels. K rows are
// packed row-major, V rows token-transposed.
#include "iq_common.cuh"
#include "iq_kernels.h"
#include "iq_append_row.cuh"

namespace iq {

// Work mapping of the histogram kernel: a row is shared by LPR = d/16 lanes, 16 consecutive coordinates (4 whole SO(4)
// blocks) per lane, so a warp holds 32/LPR rows at a time (4 at d = 128, 2 at d = 256). The Walsh-Hadamard
// butterfly runs 4 stages inside the lane and log2(LPR) xor-shuffle stages across the row's lanes.
template <int D>
struct RowQuantizer {
  static constexpr int E = 16;
  static constexpr int LPR = D / E;        // lanes per row: 8 or 16
  static constexpr int RPW = 32 / LPR;     // rows per warp: 4 or 2
  static constexpr int NB = E / 4;         // SO(4) blocks per lane
  // The head's d/4 block matrices live in shared memory, 4 blocks (64 floats) + 4 floats of padding per lane-in-row:
  // with the padding the 8 or 16 different 16-byte rows a warp reads at a time fall into different banks. Keeping
  // them in registers (64 per thread) halves the number of resident warps.
  static constexpr int M_STRIDE = NB * 16 + 4;
  static constexpr int M_FLOATS = LPR * M_STRIDE;
  const float4* Ms;        // this lane's NB matrices in shared memory, row-major

  // Called by every thread of the CTA (then __syncthreads()): the matrices of the head's blocks into m_smem.
  __device__ __forceinline__ static void fill_matrices(const float* rot_head, float* m_smem, int tid, int n_threads) {
    for (int blk = tid; blk < D / 4; blk += n_threads) {
      float Mt[4][4];
      so4_matrix<float>(rot_head + (size_t)blk * 8, Mt);
      float* dst = m_smem + (blk / NB) * M_STRIDE + (blk % NB) * 16;
#pragma unroll
      for (int r = 0; r < 4; r++) *reinterpret_cast<float4*>(dst + 4 * r) = make_float4(Mt[r][0], Mt[r][1], Mt[r][2], Mt[r][3]);
    }
  }

  __device__ __forceinline__ void init(int lane, const float* m_smem) {
    Ms = reinterpret_cast<const float4*>(m_smem + (lane % LPR) * M_STRIDE);
  }

  // butterflies across the lanes of one row (strides 16, 32, ...): lane bit b of (lane % LPR) <-> stride 16 << b
  template <typename T>
  __device__ __forceinline__ static void wht(T (&v)[E], int lane) {
#pragma unroll
    for (int s = 1; s < E; s <<= 1)
#pragma unroll
      for (int i = 0; i < E; i++)
        if ((i & s) == 0) {
          const T a = v[i], c = v[i + s];
          v[i] = a + c;
          v[i + s] = a - c;
        }
#pragma unroll
    for (int o = 1; o < LPR; o <<= 1) {
      const T sgn = (lane & o) ? T(-1) : T(1);  // the upper lane of a pair keeps (other - own)
#pragma unroll
      for (int i = 0; i < E; i++) {
        const T other = shfl_xor_t<T>(v[i], o);
        v[i] = sgn * v[i] + other;  // one fused multiply-add, exact: sgn is +-1
      }
    }
  }

  __device__ __forceinline__ static void unpack16(const uint4& r0, const uint4& r1, float (&x)[E]) {
    const uint32_t r[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const __half2 hh = *reinterpret_cast<const __half2*>(&r[k]);
      x[2 * k] = __low2float(hh);
      x[2 * k + 1] = __high2float(hh);
    }
  }

  // Algorithm 1, steps 1-2 for the row this lane belongs to (r0, r1 = this lane's 16 fp16 values, zeros for the lanes
  // of a row that is not used; those lanes still take part in the shuffles): returns the fp32 scale s (and its fp64
  // square sum) and leaves M_b (H x) -- u * s, the rotated coordinates before the division by the norm -- in x.
  __device__ __forceinline__ float rotate(const uint4& r0, const uint4& r1, int lane, float (&x)[E], double& ss_out) const {
    unpack16(r0, r1, x);
    // Step 1: s = ||x||_2. Squares of fp16 values are exact in fp32 (22 bits); they are summed in fp64 so that the
    // stored fp32 scale is the correctly rounded norm.
    double ss = 0.0;
#pragma unroll
    for (int e = 0; e < E; e += 2) ss += (double)(x[e] * x[e]) + (double)(x[e + 1] * x[e + 1]);
#pragma unroll
    for (int o = 1; o < LPR; o <<= 1) ss += __shfl_xor_sync(FULL, ss, o);
    float s = sqrtf((float)ss);
    {  // correct the fp32 estimate with exact fp64 midpoint tests instead of a double-precision square root
      const float up = __uint_as_float(__float_as_uint(s) + 1u);
      const float dn = (s > 0.f) ? __uint_as_float(__float_as_uint(s) - 1u) : 0.f;
      const double mu = 0.5 * ((double)s + (double)up), md = 0.5 * ((double)s + (double)dn);
      if (ss > mu * mu) s = up;
      else if (s > 0.f && ss < md * md) s = dn;
    }
    ss_out = ss;
    // Step 2: u = sqrt(d) * R x^ = M_b (H_unnormalised x) / s  (the two sqrt(d) factors cancel)
    wht<float>(x, lane);
#pragma unroll
    for (int j = 0; j < NB; j++) {
      const float x0 = x[4 * j], x1 = x[4 * j + 1], x2 = x[4 * j + 2], x3 = x[4 * j + 3];
#pragma unroll
      for (int r = 0; r < 4; r++) {
        const float4 m = Ms[4 * j + r];
        x[4 * j + r] = m.x * x0 + m.y * x1 + m.z * x2 + m.w * x3;
      }
    }

    return s;
  }
};

// ---------------------------------------------------------------------------------------------------------
// Few new rows per sequence (the decode step appends one): latency matters, not throughput. One warp per
// (sequence, KV head, tensor) with the whole warp on a row -- lane l owns coordinates l*d/32 .. (one or two SO(4)
// blocks), five shuffle stages of the butterfly -- a short instruction stream and no shared memory. The V row goes
// straight into its transposed records with one read-modify-write per touched word.
// ---------------------------------------------------------------------------------------------------------
template <int D, int BITS, bool MANY>
__global__ void __launch_bounds__(32) quantize_append_few_kernel(const __grid_constant__ QuantizeParams p) {
  constexpr int E = D / 32;
  grid_dependency_wait();
  allow_dependent_launch();
  const int lane = threadIdx.x;
  const bool is_v = (blockIdx.x & 1) != 0;
  const int chunk = blockIdx.x >> 1;  // the warp takes the rows that fall into one 128-row block of the cache
  const int h = blockIdx.y, b = blockIdx.z;
  int n_new = p.n_new ? p.n_new[b] : p.n_new_max;
  n_new = min(n_new, p.n_new_max);
  if (n_new <= 0) return;
  const long long pos0 = p.append_pos[b];
  // rows i with floor((pos0 + i) / 128) == floor(pos0 / 128) + chunk (rows at negative positions: chunk 0, they are refused below)
  const long long blk0 = pos0 >= 0 ? pos0 / 128 : 0;
  const long long lo = max(0ll, (blk0 + chunk) * 128 - pos0), hi = min((long long)n_new, (blk0 + chunk + 1) * 128 - pos0);
  const int i_lo = (int)((chunk == 0) ? 0 : lo), i_hi = (int)hi;
  if (i_lo >= i_hi) return;
  const __half* src_base = (is_v ? p.v_new : p.k_new) + (size_t)b * p.stride_b + (size_t)h * p.stride_h + lane * E;
  __half2 raw[E / 2];  // the first row is requested before the rotation blocks are set up: two latencies in one
#pragma unroll
  for (int k = 0; k < E / 2; k++) raw[k] = reinterpret_cast<const __half2*>(src_base + (size_t)i_lo * p.stride_t)[k];
  WarpRowQuantizer<D, BITS, MANY> rq;
  const RowSink sink{p.k_codes, p.k_scales, p.v_codes, p.v_scales, p.status, p.scale_f16};
  rq.init(p.rot + (size_t)h * (D / 4) * 8, is_v ? p.thresholds_v : p.thresholds_k, lane);
  // Several V rows: the codes of consecutive rows that share words of the records (one word of 8 or 16 rows at 4 and 2 bits,
  // three words of 32 rows at 3) are collected in registers and the words are written once -- whole when every entry is
  // new, merged with the old word otherwise -- instead of one read-modify-write per row.
  constexpr int PW = BITS == 3 ? 3 : 1;  // words collected
  uint32_t pend[E][PW], pend_mask[PW];
  int pend_word = -1;                    // the first of them within the record
  size_t pend_blk = 0;
#pragma unroll
  for (int w = 0; w < PW; w++) {
    pend_mask[w] = 0u;
#pragma unroll
    for (int e = 0; e < E; e++) pend[e][w] = 0u;
  }
  auto flush_pending = [&]() {
    if (pend_word >= 0) {
#pragma unroll
      for (int e = 0; e < E; e++) {
        uint32_t* dst = reinterpret_cast<uint32_t*>(p.v_codes + (pend_blk * D + lane * E + e) * (size_t)(16 * BITS)) + pend_word;
#pragma unroll
        for (int w = 0; w < PW; w++) {
          if (pend_mask[w] != 0u) dst[w] = (pend_mask[w] == 0xFFFFFFFFu) ? pend[e][w] : ((dst[w] & ~pend_mask[w]) | pend[e][w]);
          pend[e][w] = 0u;
        }
      }
    }
#pragma unroll
    for (int w = 0; w < PW; w++) pend_mask[w] = 0u;
    pend_word = -1;
  };
  for (int i = i_lo; i < i_hi; i++) {
    __half2 nxt[E / 2];  // the next row is requested before this one is worked on
    if (i + 1 < i_hi) {
#pragma unroll
      for (int k = 0; k < E / 2; k++) nxt[k] = reinterpret_cast<const __half2*>(src_base + (size_t)(i + 1) * p.stride_t)[k];
    }
    const long long t = pos0 + i;
    bool ok = true;
    size_t row = 0;  // the row's place in the cache arrays
    if (t < 0 || t >= p.t_cap) {
      if (lane == 0 && p.status) {  // counted per (row, KV head, tensor), like the bulk kernels
        atomicOr(&p.status[0], IQ_STATUS_ROW_OUT_OF_RANGE);
        atomicAdd(&p.status[2], 1u);
      }
      ok = false;
    } else if (!cache_row_for_write(p.pm, b, h, t, p.status, row)) {  // no such page: skipped and counted
      if (lane == 0 && p.status) atomicAdd(&p.status[2], 1u);
      ok = false;
    }
    if (ok) {
      int code[E];
      const float s = rq.run(raw, lane, code, p.status);
      if (!is_v) {
        warp_store_k_row<D, BITS>(sink, row, code, s, lane);
      } else if constexpr (!MANY) {
        warp_store_v_row<D, BITS>(sink, row, t, code, s, lane);
      } else {
        int word, sh;
        if constexpr (BITS == 3) word = 3 * ((int)(t % 128) / 32);
        else packed_place<BITS>((int)(t % 128), word, sh);
        if (word != pend_word || row / 128 != pend_blk) {
          flush_pending();
          pend_word = word;
          pend_blk = row / 128;
        }
        if constexpr (BITS == 3) {  // entry r of the unit: word r / 8, or for the last 8 a bit of each
          const int r = (int)(t % 32);
          sh = r < 24 ? 4 * (r & 7) : 4 * (r - 24) + 3;
#pragma unroll
          for (int w = 0; w < 3; w++) {
            const uint32_t bits = r < 24 ? (r >> 3 == w ? 7u : 0u) : 1u;
            pend_mask[w] |= bits << sh;
#pragma unroll
            for (int e = 0; e < E; e++) pend[e][w] |= (((uint32_t)code[e] >> (r < 24 ? 0 : w)) & bits) << sh;
          }
        } else {
#pragma unroll
          for (int e = 0; e < E; e++) pend[e][0] |= (uint32_t)code[e] << sh;
          pend_mask[0] |= ((1u << BITS) - 1u) << sh;
        }
        if (lane == 0) store_scale(p.v_scales, row, s, p.scale_f16, p.status);
      }
    }
    if (i + 1 < i_hi) {
#pragma unroll
      for (int k = 0; k < E / 2; k++) raw[k] = nxt[k];
    }
  }
  if constexpr (MANY) flush_pending();
}

// ---------------------------------------------------------------------------------------------------------
// Calibration: histogram of the rotated, normalised coordinates u = sqrt(d) R x^ of a set of rows -- the empirical
// marginal that Step 3's Lloyd-Max codebook is fitted to. Same row mapping as the K kernel; the CTA counts into a
// histogram in shared memory and adds its non-empty bins to the caller's at the end. Zero rows are left out.
// ---------------------------------------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(QA_WARPS * 32, 4) rotated_histogram_kernel(const __grid_constant__ HistogramParams p) {
  using RQ = RowQuantizer<D>;
  constexpr int LPR = RQ::LPR, RPW = RQ::RPW;
  __shared__ uint32_t hist_s[HIST_MAX_BINS];
  __shared__ __align__(16) float m_s[RQ::M_FLOATS];
  grid_dependency_wait();
  allow_dependent_launch();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.z, h = blockIdx.y;
  int n_rows = p.n_rows ? p.n_rows[b] : p.n_rows_max;
  n_rows = min(n_rows, p.n_rows_max);
  const int cta_begin = blockIdx.x * QA_WARPS * HIST_ROWS_PER_WARP;
  if (cta_begin >= n_rows) return;
  for (int i = tid; i < p.bins; i += QA_WARPS * 32) hist_s[i] = 0u;
  RQ::fill_matrices(p.rot + (size_t)h * (D / 4) * 8, m_s, tid, QA_WARPS * 32);
  __syncthreads();
  RQ rq;
  rq.init(lane, m_s);
  const int li = lane % LPR, sub = lane / LPR;
  const __half* src_base = p.x + (size_t)b * p.stride_b + (size_t)h * p.stride_h + li * 16;
  const int row_begin = cta_begin + warp * HIST_ROWS_PER_WARP, row_end = min(n_rows, row_begin + HIST_ROWS_PER_WARP);
  const float to_bin = (float)p.bins / (2.f * p.range);
  for (int i0 = row_begin; i0 < row_end; i0 += RPW) {
    const int i = i0 + sub;
    const bool active = i < row_end;
    uint4 r0 = make_uint4(0u, 0u, 0u, 0u), r1 = r0;
    if (active) {
      const uint4* src = reinterpret_cast<const uint4*>(src_base + (size_t)i * p.stride_t);
      r0 = __ldg(src);
      r1 = __ldg(src + 1);
    }
    float x[16];
    double ss;
    const float s = rq.rotate(r0, r1, lane, x, ss);
    if (active && s > 0.f) {
      const float inv_s = __frcp_rn(s);
#pragma unroll
      for (int e = 0; e < 16; e++) {
        const int bin = (int)floorf((x[e] * inv_s + p.range) * to_bin);
        atomicAdd(&hist_s[min(max(bin, 0), p.bins - 1)], 1u);
      }
    }
  }
  __syncthreads();
  for (int i = tid; i < p.bins; i += QA_WARPS * 32)
    if (hist_s[i]) atomicAdd(&p.hist[i], hist_s[i]);
}

cudaError_t launch_rotated_histogram(const HistogramParams& p, int head_dim, int batch, cudaStream_t stream) {
  if (p.n_rows_max <= 0 || batch <= 0) return cudaSuccess;
  const int rows_per_cta = QA_WARPS * HIST_ROWS_PER_WARP;
  dim3 grid((p.n_rows_max + rows_per_cta - 1) / rows_per_cta, p.n_kv_heads, batch);
  return head_dim == 128 ? launch_after_predecessor(rotated_histogram_kernel<128>, grid, dim3(QA_WARPS * 32), 0, stream, p)
                         : launch_after_predecessor(rotated_histogram_kernel<256>, grid, dim3(QA_WARPS * 32), 0, stream, p);
}

// Calibration of the rotation: z = sqrt(d) H_d x^ (Algorithm 1, lines 1-2, in the unit-variance units of the codebook) of
// a set of rows, written out as fp32. One warp per row, lane l holds coordinates l E .. l E + E - 1.
template <int D>
__global__ void __launch_bounds__(QA_WARPS * 32) wht_coordinates_kernel(const __grid_constant__ WhtParams p) {
  constexpr int E = D / 32;
  grid_dependency_wait();
  allow_dependent_launch();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.z, h = blockIdx.y;
  const int t = blockIdx.x * QA_WARPS + warp;
  int n_rows = p.n_rows ? p.n_rows[b] : p.n_rows_max;
  n_rows = min(n_rows, p.n_rows_max);
  if (t >= n_rows) return;
  const __half* src = p.x + (size_t)b * p.stride_b + (size_t)t * p.stride_t + (size_t)h * p.stride_h + lane * E;
  float v[E];
  double ss = 0.0;  // squares of fp16 values are exact in fp32
#pragma unroll
  for (int e = 0; e < E; e++) {
    v[e] = __half2float(src[e]);
    ss += (double)(v[e] * v[e]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(FULL, ss, o);
  wht_warp<float, E>(v, lane);  // unnormalised: the 1/sqrt(d) of H_d and the sqrt(d) of the units cancel
  const float inv_s = ss > 0.0 ? (float)(1.0 / sqrt(ss)) : 0.f;
  float* dst = p.z + (((size_t)b * p.n_rows_max + t) * p.n_kv_heads + h) * D + lane * E;
#pragma unroll
  for (int e = 0; e < E; e++) dst[e] = v[e] * inv_s;
}

cudaError_t launch_wht_coordinates(const WhtParams& p, int head_dim, int batch, cudaStream_t stream) {
  if (p.n_rows_max <= 0 || batch <= 0) return cudaSuccess;
  dim3 grid((p.n_rows_max + QA_WARPS - 1) / QA_WARPS, p.n_kv_heads, batch);
  return head_dim == 128 ? launch_after_predecessor(wht_coordinates_kernel<128>, grid, dim3(QA_WARPS * 32), 0, stream, p)
                         : launch_after_predecessor(wht_coordinates_kernel<256>, grid, dim3(QA_WARPS * 32), 0, stream, p);
}

template <int D, int BITS, bool MANY>
static cudaError_t launch_few_rows(const QuantizeParams& p, int batch, cudaStream_t stream) {
  // x = 2 * chunk + (0: the K rows, 1: the V rows) of (sequence, KV head); a chunk is the part of the new rows inside
  // one 128-row block of the cache (+1: the first row may sit in the middle of a block)
  dim3 grid(2 * ((p.n_new_max + 127) / 128 + 1), p.n_kv_heads, batch);
  return launch_after_predecessor(quantize_append_few_kernel<D, BITS, MANY>, grid, dim3(32), 0, stream, p);
}
template <int D, int BITS>
static cudaError_t launch_few(const QuantizeParams& p, int batch, cudaStream_t stream) {
  return p.n_new_max > 1 ? launch_few_rows<D, BITS, true>(p, batch, stream) : launch_few_rows<D, BITS, false>(p, batch, stream);
}

cudaError_t launch_quantize_append(const QuantizeParams& p, int head_dim, int batch, cudaStream_t stream) {
  if (p.n_new_max <= 0 || batch <= 0) return cudaSuccess;
  // Few rows per sequence: a warp for the rows that fall into a block, one after the other (5 us for one row, 0.7 - 1.6 us for each
  // more). More: the bulk kernel, which takes a whole tile for a block however few of its rows are new, unless two thresholds
  // of a 2- or 4-bit codebook are too close together for its decision. The line lies where the two met at 2, 3 and 4 bits, in us
  // for 8 rows / at the line (warp per block, bulk), 8 KV heads, 1 - 8 / 32 / 128 sequences:
  //   d = 128: 10 - 15 / 11 - 15 / 20 - 26 and 13 - 17 at 10 / 23 - 30 at 20 / 49 - 66 at 24; bulk 12 - 26 / 24 - 33 / 53 - 79
  //   d = 256: 14 - 22 / 17 - 25 / 31 - 45 and 20 - 36 at 14 / 40 - 66 at 28 / 110 - 180 at 42; bulk 20 - 35 / 46 - 68 / 122 - 190
  const long long pairs = (long long)batch * p.n_kv_heads;
  const int line = head_dim == 128 ? (pairs < 128 ? 10 : (pairs < 512 ? 20 : 24)) : (pairs < 128 ? 14 : (pairs < 512 ? 28 : 42));
  if (p.n_new_max > line && append_bulk_takes(p, head_dim)) return launch_append_bulk(p, head_dim, batch, stream);
  if (p.bits == 2) return head_dim == 128 ? launch_few<128, 2>(p, batch, stream) : launch_few<256, 2>(p, batch, stream);
  if (p.bits == 4) return head_dim == 128 ? launch_few<128, 4>(p, batch, stream) : launch_few<256, 4>(p, batch, stream);
  return head_dim == 128 ? launch_few<128, 3>(p, batch, stream) : launch_few<256, 3>(p, batch, stream);
}

}  // namespace iq
