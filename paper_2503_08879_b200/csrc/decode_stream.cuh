// Decode attention for launches with many tiles: the same attention as decode_attn_kernel, as a stream.
//
// A CTA takes either one part of a KV head (`split` CTAs per head, merged across their cluster) or whole heads one
// after another.  Its 16-row tiles are dealt to its four warps in turn, and each warp works for itself: its tiles come
// through a private ring of kStStages stages (K and V of one tile, tensor copies counted on an mbarrier of the
// stage), it keeps a running maximum, the sums and the whole 128-column result of its tiles in registers, and
// refills a stage as soon as it has read it.  No block barrier is passed until the head (or the part) is finished;
// then the warps' results are merged in shared memory and, with several CTAs per head, the CTAs' results over
// distributed shared memory, every CTA finishing a slice of the columns.
//
// What bounds it: HBM where all SMs are full (256 heads x 2049 rows: 42.8 us per launch, 6.3 TB/s; decode_attn_kernel,
// whose whole-SM CTAs load, compute and merge one after another, took 84.8), else the tiles a warp takes one after
// another at 0.6 us each, three in flight per warp (8 heads x 8193 rows over 16 CTAs per head: 8.7 us against 11.0).
// Two CTAs per SM, so that a launch's copies start while its predecessor still computes and merges; 4 warps x 3 stages,
// 8 warps with single slots and a first product one tile ahead measured the same within 3 %.
#pragma once

namespace sagekv {

constexpr int kStWarps = 4;
constexpr int kStThreads = kStWarps * 32;
constexpr int kStStages = 3;                       // 96 KB of tiles per CTA, so that two CTAs fit on an SM
constexpr int kStStageBytes = 2 * kSlotBytes;      // a K and a V tile
constexpr int kStMaxCluster = 16;
constexpr int kStHeadStride = kHeadDim + 4;        // floats between the heads of a warp's result: the 32 lanes of a store fall into 32 banks

struct StShared {
  unsigned char ring[kStWarps][kStStages][kStStageBytes];   // tensor copies with the 128-byte swizzle: 1024-byte boundaries
  union {
    float o[kStWarps][kMaxGroup * kStHeadStride];           // results of the warps (a CTA with whole heads)
    struct {
      float o[kHeadDim * kMaxGroup];                        // [source CTA][head][my column]: what the CTAs of the cluster send
      float2 ml[kStMaxCluster][kMaxGroup];                  // [source CTA][head] (max, sum)
    } inbox;
  };
  float2 ml[kStWarps][kMaxGroup];                           // (max, sum) of a warp's tiles
  unsigned long long bar[kStWarps][kStStages];
  unsigned long long inbox_bar;
};
static_assert(kStStages * kStStageBytes >= kMaxGroup * kStHeadStride * 4, "a warp's result fits into its ring");

// transposes an 8x8 matrix of 16-bit elements held by the warp (lane (g, c): row g, columns 2c and 2c + 1)
__device__ __forceinline__ uint32_t movmatrix(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

// split > 1 (a power of two): CTA i takes part i % split of head i / split, a cluster is the split CTAs of a head.
// split = 1: CTA i takes the whole heads [i * per_cta, (i + 1) * per_cta).
__global__ void __launch_bounds__(kStThreads, 2)
decode_stream_kernel(const DecodeParams p, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                     const int split, const int per_cta) {
  extern __shared__ __align__(1024) unsigned char st_smem[];
  StShared &sh = *reinterpret_cast<StShared *>(st_smem);
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, c = lane & 3, h0 = 2 * c, h1 = 2 * c + 1;
  const bool append = p.k_new != nullptr;
  const int n_tiles = (p.L + 15) >> 4, heads = p.B * p.H_kv;
  int first_head, first_tile, n, rank = 0;                     // my tiles: n of them from tile first_tile of head first_head on
  if (split > 1) {
    first_head = (int)blockIdx.x / split;
    rank = (int)blockIdx.x - first_head * split;
    first_tile = n_tiles * rank / split;
    n = n_tiles * (rank + 1) / split - first_tile;
  } else {
    first_head = (int)blockIdx.x * per_cta;
    first_tile = 0;
    n = min(per_cta, heads - first_head) * n_tiles;
  }
  SAGEKV_TRACE_BEGIN
  SAGEKV_STAMP(0);
  const int cols_log = 7 - (31 - __clz(split)), cols = 1 << cols_log;   // columns each CTA of a cluster finishes: 128 / split

  const uint32_t ring = smem_u32(&sh.ring[warp][0][0]), bars = smem_u32(&sh.bar[warp][0]), inbox_bar = smem_u32(&sh.inbox_bar);
  if (lane == 0) {
#pragma unroll
    for (int s = 0; s < kStStages; ++s) mbar_init(bars + 8u * s, 1);
    if (warp == 0 && split > 1) mbar_init(inbox_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_k) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_v) : "memory");
    if (warp == 0 && split > 1)                          // from every CTA of the cluster: my columns and the (max, sum) pairs
      mbar_expect_tx(inbox_bar, (uint32_t)(split * p.G * (cols * 4 + 8)));
  }
  __syncwarp();
  if (split > 1) cluster.barrier_arrive();               // waited for before the first store into a peer: its barrier is set up
  if (p.pdl_mode < 2) {                                  // (see decode_attn_kernel: nothing is read or written before the wait, but for mode 2)
    wait_for_predecessor();
    // (mode 0: a successor waiting on the SMs from the start costs a launch that fills them, 256 heads x 2049 rows in four
    // layers 177.6 -> 181.0 us)
    if (p.pdl_mode == 1) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }

  // the next tile to request: index rx in my range, tile rt of head rk of batch entry rb
  int rx = warp, rt = first_tile + warp, rb = first_head / p.H_kv, rk = first_head - rb * p.H_kv;
  uint64_t stream_policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(stream_policy));
  auto request = [&](int s) {                            // lanes 0..3: one box each
    if (rx >= n) return;
    while (rt >= n_tiles) {
      rt -= n_tiles;
      if (++rk == p.H_kv) { rk = 0; ++rb; }
    }
    const uint32_t bar = bars + 8u * s;
    if (lane == 0) mbar_expect_tx(bar, kStStageBytes);
    __syncwarp();
    if (lane < 4)
      tensor_copy_4d(ring + (uint32_t)(s * kStStageBytes + lane * kHalfBytes), lane < 2 ? &map_k : &map_v, (lane & 1) * 64, rt << 4, rk, rb,
                     bar, stream_policy);
    rx += kStWarps;
    rt += kStWarps;
  };
#pragma unroll
  for (int s = 0; s < kStStages; ++s) request(s);

  // fragment addresses within a stage
  const int mi = lane >> 3, l8 = lane & 7;
  uint32_t k_off[8], v_off[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    k_off[j] = tile_offset((mi & 1) * 8 + l8, 2 * j + (mi >> 1));
    v_off[j] = kSlotBytes + tile_offset((mi >> 1) * 8 + l8, 2 * j + (mi & 1));
  }
  const int win_lo = p.S + p.n_sel;
  const int seg0 = p.S + (p.pooled ? 0 : h0 * p.k_q), seg1 = p.S + (p.pooled ? 0 : h1 * p.k_q);
  const bool in0 = h0 < p.G, in1 = h1 < p.G;
  // how many of my tiles hold window rows: only a warp that has some reads the step counter
  int my_win = 0;
  if (append)
    for (int hx = -first_tile; hx < n; hx += n_tiles) {
      const int a = max(0, hx + (win_lo >> 4)), z = min(n, hx + n_tiles);        // indices of the head's window tiles in my range
      const int first = a + ((warp - a) & (kStWarps - 1));
      if (first < z) my_win += (z - 1 - first) / kStWarps + 1;
    }

  // Mode 2: when the successor may start.  Its copies compete with this launch's own as long as there are any to request, and
  // later, while this launch merges, the memory would be idle: a part of more than twice the ring releases it with its
  // last requests.  (us per launch at once / so: 8 heads x 8193 rows 9.18 / 8.74, 16 x 4097 9.43 / 8.71, 24 x 8193
  // 17.95 / 17.22; but 17 tiles per CTA, 8 x 4097, 5.69 / 5.91, and whole heads, 256 x 2049, 42.1 / 42.7)
  const bool release_late = split > 1 && n_tiles > 2 * kStWarps * kStStages * split;
  SAGEKV_STAMP(1);
  if (p.pdl_mode >= 2) {
    wait_for_predecessor();
    if (!release_late) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }

  const uint32_t ring_magic = 0xffffffffu / (uint32_t)max(p.ring_len, 1);   // (no division behind the wait)
  SAGEKV_STAMP(2);
  bool timed_out = false;
  int stage = 0, step = 0, my_ticket = -1, win_row = -1; // ring stage of my next tile; step counter; the replaced row of the window
  if (my_win > 0) asm volatile("ld.volatile.global.s32 %0, [%1];" : "=r"(step) : "l"(p.d_step));   // (ahead of the query's loads)
  uint32_t phase = 0;
  int x = warp;                                          // my next tile, as an index into the CTA's range
  int b = first_head / p.H_kv, kvh = first_head - b * p.H_kv;
  int head_x0 = -first_tile;                             // index (may be negative) of the head's tile 0 in the range
  for (; head_x0 < n; head_x0 += n_tiles) {
    const int x_end = min(n, head_x0 + n_tiles);
    // B fragments of Q^T: lane (g, c) holds head g's dims 16ks + 2c, +1 and 16ks + 8 + 2c, +1
    uint32_t qb[8][2];
    {
      const uint16_t *q_lane = p.q + ((int64_t)b * p.H_q + kvh * p.G + min(g, p.G - 1)) * kHeadDim + 2 * c;
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        qb[ks][0] = qb[ks][1] = 0u;
        if (g < p.G) {
          asm volatile("ld.global.b32 %0, [%1];" : "=r"(qb[ks][0]) : "l"(q_lane + 16 * ks));
          asm volatile("ld.global.b32 %0, [%1];" : "=r"(qb[ks][1]) : "l"(q_lane + 16 * ks + 8));
        }
      }
    }
    uint4 new_row = make_uint4(0u, 0u, 0u, 0u);          // lanes 0-15: 16 bytes of k_new, lanes 16-31: of v_new
    if (my_win > 0) {
      new_row = ld_v4((lane < 16 ? p.k_new : p.v_new) + ((int64_t)b * p.H_kv + kvh) * kHeadDim + (lane & 15) * 8);
      if (win_row < 0) {
        // a ticket per window tile, taken once the counter has been read (the increment depends on the value: see decode_attn_kernel)
        if (lane == 0)
          asm volatile("{ .reg .b32 inc; shr.u32 inc, %2, 31; add.u32 inc, inc, %3; atom.add.relaxed.gpu.global.s32 %0, [%1], inc; }"
                       : "=r"(my_ticket) : "l"(p.tickets + heads), "r"(step), "r"(my_win) : "memory");
        uint32_t r = (uint32_t)step - __umulhi((uint32_t)step, ring_magic) * (uint32_t)p.ring_len;
        while (r >= (uint32_t)p.ring_len) r -= (uint32_t)p.ring_len;
        win_row = win_lo + (int)r;
      }
    }
    const int patch_x = win_row >= 0 ? head_x0 + (win_row >> 4) : -1;

    float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
    float acc[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;

    for (; x < x_end; x += kStWarps) {
      const uint32_t tb = ring + (uint32_t)(stage * kStStageBytes);
      if (!mbar_wait(bars + 8u * stage, phase)) timed_out = true;
      if (x == 0) SAGEKV_STAMP(3);
      const bool patch = x == patch_x;                   // the staged copy of the replaced row is stale
      if (patch) {
        const uint32_t dst = tb + (lane < 16 ? 0u : (uint32_t)kSlotBytes) + tile_offset(win_row & 15, lane & 15);
        asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(new_row.x), "r"(new_row.y), "r"(new_row.z), "r"(new_row.w) : "memory");
        if (SAGEKV_OK_INDEX(p.status, win_row >= 0 && win_row < p.L && b < p.B)) {
          uint16_t *gdst = (lane < 16 ? p.Kc : p.Vc) + (int64_t)b * p.cs.batch_stride + (int64_t)kvh * p.cs.head_stride +
                           (int64_t)win_row * p.cs.token_stride + (lane & 15) * 8;
          st_v4(gdst, new_row);
        }
        __syncwarp();
      }
      // ---- S = K Q^T, 16 rows x 8 heads, four accumulator chains: lane (g, c) gets rows g, g + 8 of heads 2c, 2c + 1 ----
      float ch[4][4];
      uint32_t fa[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) ldmatrix_x4(tb + k_off[j], fa[j][0], fa[j][1], fa[j][2], fa[j][3]);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        mma_first(ch[j][0], ch[j][1], ch[j][2], ch[j][3], fa[j][0], fa[j][1], fa[j][2], fa[j][3], qb[j][0], qb[j][1]);
#pragma unroll
      for (int j = 0; j < 4; ++j) ldmatrix_x4(tb + k_off[4 + j], fa[j][0], fa[j][1], fa[j][2], fa[j][3]);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        mma_bf16_16816(ch[j][0], ch[j][1], ch[j][2], ch[j][3], fa[j][0], fa[j][1], fa[j][2], fa[j][3], qb[4 + j][0], qb[4 + j][1]);
      uint32_t va[8][4];
#pragma unroll
      for (int j = 0; j < 8; ++j) ldmatrix_x4_trans(tb + v_off[j], va[j][0], va[j][1], va[j][2], va[j][3]);
      // ---- softmax weights ----
      const int ra = ((x - head_x0) << 4) + g, rb2 = ra + 8;
      const bool ca = ra < p.S || (ra >= win_lo && ra < p.L), cb = rb2 < p.S || (rb2 >= win_lo && rb2 < p.L);
      float sv[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) sv[e] = ((ch[0][e] + ch[1][e]) + (ch[2][e] + ch[3][e])) * p.scale_log2;
      sv[0] = in0 && (ca || (uint32_t)(ra - seg0) < (uint32_t)p.k_q) ? sv[0] : -INFINITY;
      sv[1] = in1 && (ca || (uint32_t)(ra - seg1) < (uint32_t)p.k_q) ? sv[1] : -INFINITY;
      sv[2] = in0 && (cb || (uint32_t)(rb2 - seg0) < (uint32_t)p.k_q) ? sv[2] : -INFINITY;
      sv[3] = in1 && (cb || (uint32_t)(rb2 - seg1) < (uint32_t)p.k_q) ? sv[3] : -INFINITY;
      float t0 = fmaxf(sv[0], sv[2]), t1 = fmaxf(sv[1], sv[3]);
      if (__any_sync(0xffffffffu, t0 > m0 || t1 > m1)) {   // a new maximum: seldom after the first tiles
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
          t0 = fmaxf(t0, __shfl_xor_sync(0xffffffffu, t0, o));
          t1 = fmaxf(t1, __shfl_xor_sync(0xffffffffu, t1, o));
        }
        t0 = fmaxf(t0, m0); t1 = fmaxf(t1, m1);
        const float f0 = t0 == -INFINITY ? 1.f : fast_exp2(m0 - t0), f1 = t1 == -INFINITY ? 1.f : fast_exp2(m1 - t1);
        m0 = t0; m1 = t1;
        l0 *= f0; l1 *= f1;
#pragma unroll
        for (int j = 0; j < 8; ++j) { acc[j][0] *= f0; acc[j][1] *= f1; acc[j][2] *= f0; acc[j][3] *= f1; }
      }
      const float s0 = m0 == -INFINITY ? 0.f : m0, s1 = m1 == -INFINITY ? 0.f : m1;
      const uint32_t pa = pack_bf16x2(fast_exp2(sv[0] - s0), fast_exp2(sv[1] - s1));   // row g, heads 2c and 2c + 1
      const uint32_t pb = pack_bf16x2(fast_exp2(sv[2] - s0), fast_exp2(sv[3] - s1));   // row g + 8
      l0 += __uint_as_float(pa << 16) + __uint_as_float(pb << 16);                     // the weights as rounded
      l1 += __uint_as_float(pa & 0xffff0000u) + __uint_as_float(pb & 0xffff0000u);
      const uint32_t b0 = movmatrix(pa), b1 = movmatrix(pb);                           // head g, rows 2c, 2c + 1 and 2c + 8, 2c + 9
      // ---- O^T += V^T P: lane (g, c) holds columns 16j + g and 16j + g + 8 of heads 2c and 2c + 1 ----
#pragma unroll
      for (int j = 0; j < 8; ++j)
        mma_bf16_16816(acc[j][0], acc[j][1], acc[j][2], acc[j][3], va[j][0], va[j][1], va[j][2], va[j][3], b0, b1);
      __syncwarp();                                      // every lane has its fragments: the stage may be refilled
      if (patch) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      request(stage);
      if (release_late && rx >= n && p.pdl_mode >= 2) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
      if (++stage == kStStages) { stage = 0; phase ^= 1u; }
    }

    SAGEKV_STAMP_AFTER(4, acc[0][0] + acc[7][3]);
    // ---- the head (or my part of it) is done: merge the four warps ----
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
      l0 += __shfl_xor_sync(0xffffffffu, l0, o);
      l1 += __shfl_xor_sync(0xffffffffu, l1, o);
    }
    // with a cluster this is the CTA's only head: every copy it asked for has been read, its rings hold the results
    // (the inbox of the cluster takes the place of sh.o)
    float *const my_o = split > 1 ? reinterpret_cast<float *>(sh.ring[warp]) : sh.o[warp];
    const float *const all_o = split > 1 ? reinterpret_cast<const float *>(sh.ring) : sh.o[0];
    const int o_stride = split > 1 ? kStStages * kStStageBytes / 4 : kMaxGroup * kStHeadStride;
    if (split == 1) __syncthreads();                     // the previous head's results have been read
    if (g == 0) { sh.ml[warp][h0] = make_float2(m0, l0); sh.ml[warp][h1] = make_float2(m1, l1); }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float *o0 = my_o + h0 * kStHeadStride + 16 * j + g, *o1 = o0 + kStHeadStride;
      o0[0] = acc[j][0]; o1[0] = acc[j][1]; o0[8] = acc[j][2]; o1[8] = acc[j][3];
    }
    if (split > 1) cluster.barrier_wait();
    __syncthreads();
    SAGEKV_STAMP(5);
    const int64_t row0 = (int64_t)b * p.H_q + kvh * p.G;   // the head's first row of out and lse
    const bool rows_ok = SAGEKV_OK_INDEX(p.status, b >= 0 && b < p.B && kvh >= 0 && (kvh + 1) * p.G <= p.H_q);
    for (int item = tid; item < p.G * (kHeadDim / 4); item += kStThreads) {
      const int h = item >> 5, col = (item & 31) * 4;
      float2 ml[kStWarps];
      float M = -INFINITY;
#pragma unroll
      for (int w = 0; w < kStWarps; ++w) { ml[w] = sh.ml[w][h]; M = fmaxf(M, ml[w].x); }
      float l = 0.f;
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int w = 0; w < kStWarps; ++w) {
        const float f = M == -INFINITY ? 0.f : fast_exp2(ml[w].x - M);
        const float4 v = *reinterpret_cast<const float4 *>(all_o + w * o_stride + h * kStHeadStride + col);
        l += ml[w].y * f;
        o.x += v.x * f; o.y += v.y * f; o.z += v.z * f; o.w += v.w * f;
      }
      if (split == 1) {
        const float inv = l > 0.f ? 1.f / l : 0.f;
        if (rows_ok)
          *reinterpret_cast<uint2 *>(p.out + (row0 + h) * kHeadDim + col) =
              make_uint2(pack_bf16x2(o.x * inv, o.y * inv), pack_bf16x2(o.z * inv, o.w * inv));
        if (rows_ok && p.lse != nullptr && col == 0) p.lse[row0 + h] = l > 0.f ? (M + log2f(l)) * kLn2 : -INFINITY;
      } else {
        // to the CTA that finishes these columns, data and byte count travelling together
        const uint32_t own = (uint32_t)(col >> cols_log);
        uint32_t dst, rbar;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(smem_u32(&sh.inbox.o[((rank * p.G + h) << cols_log) + (col & (cols - 1))])), "r"(own));
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rbar) : "r"(inbox_bar), "r"(own));
        asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                     ::"r"(dst), "f"(o.x), "f"(o.y), "f"(o.z), "f"(o.w), "r"(rbar) : "memory");
        if ((item & 31) < split) {
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(smem_u32(&sh.inbox.ml[rank][h])), "r"(item & 31));
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rbar) : "r"(inbox_bar), "r"(item & 31));
          asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];"
                       ::"r"(dst), "f"(M), "f"(l), "r"(rbar) : "memory");
        }
      }
    }
    SAGEKV_STAMP(6);
    if (split > 1) {
      // ---- finish my columns from the inbox, two per thread ----
      if (!mbar_wait(inbox_bar, 0u)) timed_out = true;
      SAGEKV_STAMP(7);
      for (int item = tid; item < (p.G << cols_log) >> 1; item += kStThreads) {
        const int h = item >> (cols_log - 1), lc = (item & ((cols >> 1) - 1)) * 2, col = rank * cols + lc;
        float2 ml[kStMaxCluster], v[kStMaxCluster];
        float M = -INFINITY, l = 0.f, ox = 0.f, oy = 0.f;
#pragma unroll
        for (int s = 0; s < kStMaxCluster; ++s) {
          ml[s] = make_float2(-INFINITY, 0.f); v[s] = make_float2(0.f, 0.f);
          if (s < split) {
            ml[s] = sh.inbox.ml[s][h];
            v[s] = *reinterpret_cast<const float2 *>(&sh.inbox.o[((s * p.G + h) << cols_log) + lc]);
          }
          M = fmaxf(M, ml[s].x);
        }
#pragma unroll
        for (int s = 0; s < kStMaxCluster; ++s) {
          const float f = M == -INFINITY ? 0.f : fast_exp2(ml[s].x - M);
          l += ml[s].y * f;
          ox += v[s].x * f; oy += v[s].y * f;
        }
        const float inv = l > 0.f ? 1.f / l : 0.f;
        const bool ok = rows_ok && SAGEKV_OK_INDEX(p.status, h < p.G && col >= 0 && col + 2 <= kHeadDim);
        if (ok) *reinterpret_cast<uint32_t *>(p.out + (row0 + h) * kHeadDim + col) = pack_bf16x2(ox * inv, oy * inv);
        if (ok && p.lse != nullptr && col == 0) p.lse[row0 + h] = l > 0.f ? (M + log2f(l)) * kLn2 : -INFINITY;
      }
    }
    if (++kvh == p.H_kv) { kvh = 0; ++b; }
  }
#if defined(SAGEKV_TRACE)
  if (split == 1) trace_t[7] = trace_t[6];
#endif
  SAGEKV_STAMP(8);
  if (timed_out) atomicOr(p.status, kStatusWaitTimeout);
  if (my_win > 0 && lane == 0 && my_ticket + my_win == heads * (n_tiles - (win_lo >> 4))) {   // every reader has read the counter
    p.tickets[heads] = 0;
    *p.d_step = step + 1;
  }
  SAGEKV_STAMP(9);
  SAGEKV_TRACE_END(p.out);
}

}  // namespace sagekv
