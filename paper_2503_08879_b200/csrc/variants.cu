// Kernels of the comparison paths that sit beside the four steps of the method:
//   - StreamLLM_R (Section 3.1 "Baselines", Appendix A.1): the sink + recent + last rows of a PRE-RoPE key cache,
//     each key rotated by its index inside the kept window while it is copied; values copied verbatim.
//   - the pooled reading of Step 2: the score rows of a KV head's G query heads summed into one row.
//   - a Quest-style comparator (Section 3.1 "Baselines"): per block of 16 tokens the element-wise minimum and
//     maximum of the keys (built once), and per decode step an upper bound of every block's attention logit.
// Both are plain streaming kernels (HBM-bound, no reuse): one warp per 256-byte row, 16-byte accesses.
#include "common.cuh"

namespace sagekv {

// ---- StreamLLM_R ---------------------------------------------------------------------------------------------
// Row r of the reduced cache (r < S: sink token r; otherwise token N - (S + R + 1) + r, i.e. the R recent tokens
// and the last one) gets  y[i] = x[i] cos(a_i) - x[i + 64] sin(a_i),  y[i + 64] = x[i + 64] cos(a_i) + x[i] sin(a_i),
// a_i = r * theta^(-2i/128): dimension i is paired with i + 64, as in the Llama and Qwen models.  Angles, sines
// and cosines are taken in double precision (positions reach thousands of radians at the low dimensions, and the
// kernel moves a few hundred rows), the products in double, one rounding to bf16 at the end.
__global__ void __launch_bounds__(256) compact_window_rope_kernel(const WindowRopeParams p) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  wait_for_predecessor();
  const int L = p.S + p.R + 1;
  const int64_t n_rows = (int64_t)p.B * p.H_kv * L;
  const double log2_theta = log2((double)p.theta);
  for (int64_t it = (int64_t)blockIdx.x * 8 + warp; it < n_rows; it += (int64_t)gridDim.x * 8) {
    const int r = (int)(it % L);
    const int bk = (int)(it / L), b = bk / p.H_kv, kvh = bk - b * p.H_kv;
    const int64_t tok = r < p.S ? r : (int64_t)p.N - L + r;
    if (!SAGEKV_OK_INDEX(p.status, tok >= 0 && tok < p.N)) continue;
    const int64_t src = (int64_t)b * p.ks.batch_stride + (int64_t)kvh * p.ks.head_stride + tok * p.ks.token_stride;
    const int64_t dst = (int64_t)b * p.cs.batch_stride + (int64_t)kvh * p.cs.head_stride + (int64_t)r * p.cs.token_stride;
    // lanes 0-15 hold dims 4*lane .. +3 and their partners 64 + 4*lane .. +3 of K; lanes 16-31 copy V (16 bytes each)
    if (lane < 16) {
      const uint2 lo = *reinterpret_cast<const uint2 *>(p.K + src + 4 * lane);
      const uint2 hi = *reinterpret_cast<const uint2 *>(p.K + src + 64 + 4 * lane);
      const uint32_t xl[2] = {lo.x, lo.y}, xh[2] = {hi.x, hi.y};
      uint32_t yl[2], yh[2];
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        float ol[2], oh[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int i = 4 * lane + 2 * w + e;
          const double x1 = (double)__uint_as_float(((xl[w] >> (16 * e)) & 0xffffu) << 16);
          const double x2 = (double)__uint_as_float(((xh[w] >> (16 * e)) & 0xffffu) << 16);
          const double ang = (double)r * exp2(-(double)(2 * i) / (double)kHeadDim * log2_theta);
          double sn, cn;
          sincos(ang, &sn, &cn);
          ol[e] = (float)(x1 * cn - x2 * sn);
          oh[e] = (float)(x2 * cn + x1 * sn);
        }
        yl[w] = pack_bf16x2(ol[0], ol[1]);
        yh[w] = pack_bf16x2(oh[0], oh[1]);
      }
      *reinterpret_cast<uint2 *>(p.Kc + dst + 4 * lane) = make_uint2(yl[0], yl[1]);
      *reinterpret_cast<uint2 *>(p.Kc + dst + 64 + 4 * lane) = make_uint2(yh[0], yh[1]);
    } else {
      const int piece = (lane - 16) * 8;
      st_v4(p.Vc + dst + piece, ld_stream_v4(p.V + src + piece));
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *p.d_step = 0;
}

cudaError_t launch_compact_window_rope(const WindowRopeParams &p, int n_sm, cudaStream_t stream) {
  const int64_t n_rows = (int64_t)p.B * p.H_kv * (p.S + p.R + 1);
  int64_t blocks = (n_rows + 7) / 8;
  if (blocks > 4 * (int64_t)n_sm) blocks = 4 * (int64_t)n_sm;
  if (blocks < 1) blocks = 1;
  return launch_next(compact_window_rope_kernel, dim3((unsigned)blocks), 256, 0, stream, 0, p);
}

// ---- pooled scores -------------------------------------------------------------------------------------------
// pooled[b, g, i] = sum over j < G of scores[b, g*G + j, i], added in head order in fp32.
__global__ void __launch_bounds__(256) pool_scores_kernel(const float *scores, int64_t row_stride, float *pooled,
                                                          int64_t pooled_stride, int E, int G, int n_groups) {
  wait_for_predecessor();
  const int n_vec = E >> 2;
  for (int g = blockIdx.y; g < n_groups; g += gridDim.y) {
    const float *src = scores + (int64_t)g * G * row_stride;
    float *dst = pooled + (int64_t)g * pooled_stride;
    for (int v = blockIdx.x * 256 + threadIdx.x; v < n_vec; v += gridDim.x * 256) {
      float4 acc = *reinterpret_cast<const float4 *>(src + 4 * v);
      for (int j = 1; j < G; ++j) {
        const float4 x = *reinterpret_cast<const float4 *>(src + (int64_t)j * row_stride + 4 * v);
        acc.x += x.x; acc.y += x.y; acc.z += x.z; acc.w += x.w;
      }
      *reinterpret_cast<float4 *>(dst + 4 * v) = acc;
    }
    if (blockIdx.x == 0 && (int)threadIdx.x < E - 4 * n_vec) {
      const int i = 4 * n_vec + threadIdx.x;
      float acc = src[i];
      for (int j = 1; j < G; ++j) acc += src[(int64_t)j * row_stride + i];
      dst[i] = acc;
    }
  }
}

cudaError_t launch_pool_scores(const float *scores, int64_t row_stride, float *pooled, int64_t pooled_stride, int E, int G,
                               int n_groups, int n_sm, cudaStream_t stream) {
  if (E <= 0 || n_groups <= 0) return cudaSuccess;
  int bx = (E / 4 + 256 * 4 - 1) / (256 * 4);
  const int want = (4 * n_sm + n_groups - 1) / n_groups;
  if (bx > want) bx = want;
  if (bx < 1) bx = 1;
  return launch_next(pool_scores_kernel, dim3((unsigned)bx, (unsigned)(n_groups < 65535 ? n_groups : 65535)), 256, 0, stream, 0,
                     scores, row_stride, pooled, pooled_stride, E, G, n_groups);
}

// ---- Quest-style block summaries -----------------------------------------------------------------------------
// One warp per block of 16 tokens of the eviction region: the two half-warps take alternate rows, 16 bytes (8
// dims) per lane, and are merged with one shuffle.  Minima and maxima of bf16 values are bf16 values: exact.
__device__ __forceinline__ void minmax_bf16x8(uint4 v, float (&lo)[8], float (&hi)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float a = __uint_as_float(w[i] << 16), b = __uint_as_float(w[i] & 0xffff0000u);
    lo[2 * i] = fminf(lo[2 * i], a); hi[2 * i] = fmaxf(hi[2 * i], a);
    lo[2 * i + 1] = fminf(lo[2 * i + 1], b); hi[2 * i + 1] = fmaxf(hi[2 * i + 1], b);
  }
}

__global__ void __launch_bounds__(256) quest_build_kernel(const uint16_t *K, sagekv_strides ks, uint16_t *kmin, uint16_t *kmax,
                                                          int S, int E, int n_blocks, int H_kv) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int kvh = blockIdx.y, b = blockIdx.z;
  wait_for_predecessor();
  const uint16_t *Kh = K + (int64_t)b * ks.batch_stride + (int64_t)kvh * ks.head_stride + (int64_t)S * ks.token_stride;
  for (int blk = blockIdx.x * 8 + warp; blk < n_blocks; blk += gridDim.x * 8) {
    float lo[8], hi[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) { lo[i] = INFINITY; hi[i] = -INFINITY; }
    const int t0 = blk * kQuestBlock, t1 = min(E, t0 + kQuestBlock);
#pragma unroll
    for (int u = 0; u < kQuestBlock / 2; ++u) {
      const int t = t0 + 2 * u + (lane >> 4);
      if (t < t1) minmax_bf16x8(ld_stream_v4(Kh + (int64_t)t * ks.token_stride + (lane & 15) * 8), lo, hi);
    }
    uint32_t olo[4], ohi[4];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      lo[i] = fminf(lo[i], __shfl_xor_sync(0xffffffffu, lo[i], 16));
      hi[i] = fmaxf(hi[i], __shfl_xor_sync(0xffffffffu, hi[i], 16));
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) { olo[i] = pack_bf16x2(lo[2 * i], lo[2 * i + 1]); ohi[i] = pack_bf16x2(hi[2 * i], hi[2 * i + 1]); }
    const int64_t o = (((int64_t)b * H_kv + kvh) * n_blocks + blk) * kHeadDim + (lane & 15) * 8;
    if (lane < 16) st_v4(kmin + o, make_uint4(olo[0], olo[1], olo[2], olo[3]));
    else st_v4(kmax + o, make_uint4(ohi[0], ohi[1], ohi[2], ohi[3]));
  }
}

cudaError_t launch_quest_build(const uint16_t *K, sagekv_strides ks, uint16_t *kmin, uint16_t *kmax, int S, int E, int H_kv,
                               int B, int n_sm, cudaStream_t stream) {
  const int n_blocks = (E + kQuestBlock - 1) / kQuestBlock;
  if (n_blocks <= 0) return cudaSuccess;
  int gx = (n_blocks + 7) / 8;
  const int want = (8 * n_sm + H_kv * B - 1) / (H_kv * B);
  if (gx > want) gx = want;
  return launch_next(quest_build_kernel, dim3((unsigned)gx, (unsigned)H_kv, (unsigned)B), 256, 0, stream, 0, K, ks, kmin, kmax, S, E,
                     n_blocks, H_kv);
}

// u[b, h, blk] = scale * sum_c max(q[b,h,c] * kmin[b, h/G, blk, c], q[b,h,c] * kmax[...]), fp32.  For finite summaries
// (kmin <= kmax) the larger product is the one with kmax where q is positive and with kmin where it is negative, so a
// bound is a dot product over 256 terms: (max(q, 0), min(q, 0)) . (kmax, kmin), every term an exact bf16 product.  That
// puts the G heads of a KV head on the tensor cores: a warp takes 16 blocks as the rows of its tiles and the heads (padded
// to 8) as the columns, and because a dot product does not care in which order its terms are added, the fragments are
// filled from plain 16-byte loads with the summaries and the query in the same column order.
// Bound by memory: 33.5 MB of summaries (8 KV heads x 8183 blocks) take 19.1 us with one product, one maximum and one
// addition per head and element, 8.2 on the tensor cores in CTAs of eight warps (two of them per SM) and 6.8 in CTAs of four
// (five per SM: the last wave is shorter).
__device__ __forceinline__ float bf16_at(const uint16_t *p) { return __uint_as_float((uint32_t)*p << 16); }

// a <= b for all eight pairs (false for NaN)
__device__ __forceinline__ bool le_bf16x8(uint4 a, uint4 b) {
  auto le = [](uint32_t x, uint32_t y) {
    uint32_t r;
    asm("set.le.u32.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(y));
    return r;
  };
  return (le(a.x, b.x) & le(a.y, b.y) & le(a.z, b.z) & le(a.w, b.w)) == 0xffffffffu;
}

constexpr int kBoundsWarps = 4;

__global__ void __launch_bounds__(kBoundsWarps * 32, 5) quest_bounds_kernel(const uint16_t *q, const uint16_t *kmin, const uint16_t *kmax, float *u,
                                                           int64_t u_stride, int n_blocks, int G, int H_q, int H_kv, float scale) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, c = lane & 3;
  const int kvh = blockIdx.y, b = blockIdx.z;
  const int first = (blockIdx.x * kBoundsWarps + warp) * 16;
  wait_for_predecessor();
  if (first >= n_blocks) return;
  // lane (g, c) holds, of blocks first + g and first + g + 8, the 16-byte pieces at columns j*32 + c*8 of both summaries
  const int64_t base = ((int64_t)b * H_kv + kvh) * n_blocks;
  const int64_t o0 = (base + min(first + g, n_blocks - 1)) * kHeadDim + c * 8, o1 = (base + min(first + g + 8, n_blocks - 1)) * kHeadDim + c * 8;
  uint4 a0[2][4], a1[2][4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    a0[0][j] = ld_stream_v4(kmax + o0 + j * 32);
    a1[0][j] = ld_stream_v4(kmax + o1 + j * 32);
    a0[1][j] = ld_stream_v4(kmin + o0 + j * 32);
    a1[1][j] = ld_stream_v4(kmin + o1 + j * 32);
  }
  uint4 qf[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) qf[j] = make_uint4(0u, 0u, 0u, 0u);
  if (g < G) {
    const uint16_t *qrow = q + ((int64_t)b * H_q + kvh * G + g) * kHeadDim + c * 8;
#pragma unroll
    for (int j = 0; j < 4; ++j) qf[j] = *reinterpret_cast<const uint4 *>(qrow + j * 32);
  }
  // the elements of a word with their sign bit clear, and those with it set; the others become zero
  auto negative = [](uint32_t w) { return w & (((w >> 15) & 0x00010001u) * 0xffffu); };
  bool ordered = true;                                   // kmin <= kmax everywhere (and no NaN)
#pragma unroll
  for (int j = 0; j < 4; ++j) ordered &= le_bf16x8(a0[1][j], a0[0][j]) && le_bf16x8(a1[1][j], a1[0][j]);
  float d[2][4];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    d[s][0] = d[s][1] = d[s][2] = d[s][3] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t nx = negative(qf[j].x), ny = negative(qf[j].y), nz = negative(qf[j].z), nw = negative(qf[j].w);
      const uint32_t bx = s == 0 ? qf[j].x ^ nx : nx, by = s == 0 ? qf[j].y ^ ny : ny;
      const uint32_t bz = s == 0 ? qf[j].z ^ nz : nz, bw = s == 0 ? qf[j].w ^ nw : nw;
      mma_bf16_16816(d[s][0], d[s][1], d[s][2], d[s][3], a0[s][j].x, a1[s][j].x, a0[s][j].y, a1[s][j].y, bx, by);
      mma_bf16_16816(d[s][0], d[s][1], d[s][2], d[s][3], a0[s][j].z, a1[s][j].z, a0[s][j].w, a1[s][j].w, bz, bw);
    }
  }
  // lane (g, c) has blocks first + g (elements 0, 1) and first + g + 8 (2, 3) of heads 2c and 2c + 1
  float *row = u + ((int64_t)b * H_q + kvh * G + 2 * c) * u_stride + first + g;
  // (a non-finite term, even times zero, leaves a non-finite sum: such sums, and summaries that are no minima and
  // maxima, are taken again term by term)
  const bool all_ordered = __all_sync(0xffffffffu, ordered);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int h = 2 * c + (e & 1), blk = first + g + 8 * (e >> 1);
    if (h >= G || blk >= n_blocks) continue;
    float sum = d[0][e] + d[1][e];
    if (!all_ordered || !(fabsf(sum) <= 3.0e38f)) {
      sum = 0.f;
      for (int i = 0; i < kHeadDim; ++i) {
        const float qv = bf16_at(q + ((int64_t)b * H_q + kvh * G + h) * kHeadDim + i);
        sum += fmaxf(qv * bf16_at(kmin + (base + blk) * kHeadDim + i), qv * bf16_at(kmax + (base + blk) * kHeadDim + i));
      }
    }
    row[(e & 1) * u_stride + 8 * (e >> 1)] = sum * scale;
  }
}

cudaError_t launch_quest_bounds(const uint16_t *q, const uint16_t *kmin, const uint16_t *kmax, float *u, int64_t u_stride,
                                int n_blocks, int G, int H_q, int H_kv, int B, float scale, int n_sm, cudaStream_t stream) {
  if (n_blocks <= 0) return cudaSuccess;
  const int per_cta = kBoundsWarps * 16;
  return launch_next(quest_bounds_kernel, dim3((unsigned)((n_blocks + per_cta - 1) / per_cta), (unsigned)H_kv, (unsigned)B),
                     kBoundsWarps * 32, 0, stream, 0, q, kmin, kmax, u, u_stride, n_blocks, G, H_q, H_kv, scale);
}

}  // namespace sagekv
