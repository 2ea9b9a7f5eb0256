// Step 4: append the new token to the recent window, then attention of every query head over its view
// of the reduced cache (sink + its own selected segment + window).
//
// Flash-decoding on thread-block clusters.  The L rows of one KV head are cut into 16-row tiles that are
// dealt evenly, as contiguous ranges, to the CTAs of one cluster.  A CTA brings its K and V tiles into shared
// memory with tensor copies (one 16-row x 64-column box per request, 128-byte swizzle, completion counted on
// an mbarrier), issued by a ninth warp that does nothing else, or by all nine (decode_shares_issue).  The staging area has 50
// slots of one tile (K or V) each.  All K tiles of the range are resident from the start; so are the V tiles while slots last,
// and the remaining V tiles take over the K slots as soon as the first product is done.  There is one pass:
//   S = K Q^T     16 rows x 8 heads per mma, a tile per warp in turn (the scores of all its tiles stay in
//                 registers).  A fragments come from the swizzled tile with ldmatrix, the query (B fragments)
//                 sits in registers.
//   softmax       one maximum per head and warp, over all its tiles (two block barriers in all), so nothing is ever
//                 rescaled; the weights, rounded to bf16, go to shared memory for all tiles.
//   O^T = V^T P   split by COLUMNS: warp w accumulates columns 16w..16w+15 of all heads over all rows
//                 (transposing ldmatrix for V, the weights as B fragments), the rows of each warp's weights by themselves,
//                 and brings the eight sums to the CTA's maximum.  The warps' results are disjoint, so nothing is
//                 exchanged inside the CTA.
// Every head masks the rows of the other heads' segments.  The CTAs of a cluster are merged through
// distributed shared memory: each warp sends its 16 columns straight from registers into the inbox of the
// CTA that finishes those columns with asynchronous stores counted on that CTA's barrier (one way, no
// cluster barrier), and each CTA writes its slice of the 128 output columns.  With several clusters per
// head (caches beyond 44 tiles per CTA: a warp keeps the scores of at most six) the cluster results go to scratch and the CTA that arrives last
// (one atomic ticket, no waiting) merges them.
// The staged copy of the window row that the new token replaces is overwritten in shared memory from
// k_new / v_new once it has landed, and the CTA owning that row stores the new token into the cache.
// Every wait on a copy barrier is bounded: a wait that runs out sets kStatusWaitTimeout in the context's status
// word and the CTA runs on with whatever its shared memory holds, so every block and cluster barrier is still
// reached and the kernel ends; the output of such a launch is meaningless and the status word says so.
#include <cooperative_groups.h>
#include <cuda.h>
#include <math.h>

#include <atomic>
#include <mutex>

#include "common.cuh"
#include "trace.cuh"

namespace cg = cooperative_groups;

namespace sagekv {

constexpr int kDecodeThreads = (kDecodeWarps + 1) * 32;   // eight consumer warps and the warp that issues the copies
constexpr int kConsumerThreads = kDecodeWarps * 32;
constexpr int kDecodeBaseCluster = 8;          // the cluster size tried first (the portable limit)
constexpr int kSlotBytes = 16 * 256;           // a slot of the staging area: 16 rows of K or of V
constexpr int kHalfBytes = 16 * 128;           // 16 rows x 64 columns: one box of the tensor copy
constexpr int kPHeadWords = 12;                // 32-bit words per (tile, head) of the weight buffer: 8 used, 4 spread the banks
constexpr int kPTileWords = kMaxGroup * kPHeadWords;
constexpr int kQkGroup = 3;                    // tiles of the first product a warp works on at once
constexpr int kQkTiles = (kDecodeMaxTiles + kDecodeWarps - 1) / kDecodeWarps;   // tiles a warp may get in the first product (6)
constexpr uint32_t kWaitLimit = 1u << 22;      // polls of a copy barrier before giving up (each poll already blocks for a while)

struct DecShared {
  // softmax weights: [tile][head][row pair g: rows 2g, 2g + 1]; the tensor-memory variant keeps its two small
  // operands here instead (12 KB of weights, 4 KB of queries, both in the 128-byte-swizzled operand layout, which
  // wants 1024-byte alignment: the struct sits behind the staging area, on such a boundary)
  alignas(1024) uint32_t P[kDecodeMaxTiles * kPTileWords];
  unsigned long long bar[5];                                   // K landed, early V landed, late V landed; scores ready, outputs ready (tensor-memory variant)
  unsigned long long inbox_bar;                                // every CTA's share for this CTA's columns has landed
  unsigned long long ml_bar;                                   // every CTA's (max, sum) pairs have landed (they travel ahead of the columns)
  int last;
  uint32_t tmem_base;                                          // tensor-memory variant: first column of the CTA's allocation
  int pad_[2];
  float warp_m[kDecodeWarps][kMaxGroup];                       // maxima of the warps' rows
  float warp_l[kDecodeWarps][kMaxGroup];                       // sums of the warps' (rounded) weights, in units of the CTA's maxima
  float warp_f[kDecodeWarps][kMaxGroup];                       // what brings a warp's weights to these units
  float2 inbox_ml[kDecodeMaxCluster][kMaxGroup];               // [source CTA][head] (max, sum)
  float inbox_o[(kHeadDim + 4 * kDecodeMaxCluster) * kMaxGroup];   // [source CTA][my column][head]; cluster size x columns <= 160
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// false: the wait ran out
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (uint32_t i = 0; i < kWaitLimit; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// one box of a [batch, head, row, column] bf16 tensor -> shared memory; the copy reads this GPU's memory only
// (the cache rows are read once per call: they are marked evict-first in L2, so that the small operands every
// call reads after its dependency wait, q and the step counter, tend to stay there)
__device__ __forceinline__ void tensor_copy_4d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, int w, uint32_t bar,
                                               uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
// D(16x8, fp32) = A(16x16, bf16, row) * B(16x8, bf16, col): the first link of an accumulator chain
__device__ __forceinline__ void mma_first(float &d0, float &d1, float &d2, float &d3, uint32_t a0, uint32_t a1, uint32_t a2,
                                          uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d0), "=f"(d1), "=f"(d2), "=f"(d3)
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// Byte offset, inside a staged K or V tile (two 2 KB boxes: columns 0..63 and 64..127), of the 16-byte piece
// `piece` (0..15) of row `row` (0..15): the 128-byte swizzle of the tensor copy XORs the piece index within a
// 128-byte line with the line index modulo 8 (the boxes start on 1024-byte boundaries).
__device__ __forceinline__ uint32_t tile_offset(int row, int piece) {
  return (uint32_t)((piece >> 3) * kHalfBytes + row * 128 + (((piece & 7) ^ (row & 7)) << 4));
}

// keeps a value that was worked out early in a register, so that the work is not redone (later) where it is used
__device__ __forceinline__ void pin(uint32_t &x) { asm volatile("" : "+r"(x)); }
__device__ __forceinline__ void pin(int &x) { asm volatile("" : "+r"(x)); }

__device__ __forceinline__ void bar_sync(int id, int n_threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n_threads) : "memory");
}

// n_slots: slots of this launch's staging area (min(2 * most tiles of a CTA, kDecodeSlots)).
// kLong: a CTA may have more tiles than half the slots (part of V arrives late, a warp may have up to six tiles in
// the first product); false keeps the common case free of that.  kShared: all nine warps ask for the copies at the start, each for
// a ninth of the boxes (the bytes to expect are set before they do); late V tiles are the ninth warp's in any case.
template <bool kLong, bool kShared>
__global__ void __launch_bounds__(kDecodeThreads, 1)
decode_attn_kernel(const DecodeParams p, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                   const int n_slots) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t stage = (raw + 1023u) & ~1023u;                 // the slots: boxes on 1024-byte boundaries
  DecShared &sh = *reinterpret_cast<DecShared *>(smem_raw + (stage - raw) + (size_t)n_slots * kSlotBytes);

  cg::cluster_group cluster = cg::this_cluster();
  const int cs = cluster.num_blocks();
  const int rank = cluster.block_rank();
  const int ci = blockIdx.x, kvh = blockIdx.y, b = blockIdx.z;    // ci: CTA index within the head
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, c = lane & 3;
  const int h0 = 2 * c, h1 = 2 * c + 1;                           // the two heads a lane's accumulators belong to
  const bool producer = warp == kDecodeWarps;
  const bool append = p.k_new != nullptr;
  SAGEKV_TRACE_BEGIN
  SAGEKV_STAMP(0);

  // tiles of this CTA: an even deal of the head's n_tiles over the gridDim.x CTAs, contiguous ranges
  const int n_tiles = (p.L + 15) >> 4;
  const int base_n = n_tiles / (int)gridDim.x, rem = n_tiles % (int)gridDim.x;
  const int first_tile = ci * base_n + min(ci, rem);
  const int n = base_n + (ci < rem ? 1 : 0);                      // my tiles: K tile t in slot t
  // V tile t sits in slot n + t while slots last (the early ones, requested at once); the others (late) take
  // slot n + t - n_slots, a K slot, once the first product is done
  constexpr int kQk = kLong ? kQkTiles : kQkGroup;           // tiles of the first product a warp may have
  const int n_early = kLong ? min(n, n_slots - n) : n, n_late = n - n_early;
  auto v_slot = [&](int t) { return (!kLong || t < n_early) ? n + t : n + t - n_slots; };

  // columns each CTA of the cluster finishes: a multiple of 4, the last CTA may get fewer
  const int cols = ((kHeadDim + cs - 1) / cs + 3) & ~3;
  const int my_cols = max(0, min(cols, kHeadDim - rank * cols));
  const int n_pairs = (p.G + 1) >> 1;                             // head pairs in use

  const uint32_t kbar = smem_u32(&sh.bar[0]), vbar_e = smem_u32(&sh.bar[1]), vbar_l = smem_u32(&sh.bar[2]);
  const uint32_t inbox_bar = smem_u32(&sh.inbox_bar);
  const uint32_t ml_bar = smem_u32(&sh.ml_bar);
  if (tid == 0) {
    mbar_init(kbar, 1);
    mbar_init(vbar_e, 1);
    mbar_init(vbar_l, 1);
    mbar_init(inbox_bar, 1);
    mbar_init(ml_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_k) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_v) : "memory");
    // from every CTA of the cluster: 8 bytes per (own column, head pair in use) and 64 bytes of (max, sum) pairs
    mbar_expect_tx(inbox_bar, (uint32_t)(cs * my_cols * n_pairs * 8));
    mbar_expect_tx(ml_bar, (uint32_t)(cs * 64));
    if (kShared) {
      mbar_expect_tx(kbar, (uint32_t)n * kSlotBytes);
      mbar_expect_tx(vbar_e, (uint32_t)n_early * kSlotBytes);
    }
  }
  __syncthreads();
  cluster.barrier_arrive();                              // waited for just before the first store into a peer: its barrier is set up

  // Programmatic dependent launch: until the wait returns, nothing that an earlier kernel on the stream may
  // still be writing is read (q, k_new, v_new, the step counter) and nothing at all is written to global
  // memory.  In prefetch mode the rows of the reduced cache are requested first: the caller has promised that
  // the kernel directly before this one does not write this layer's cache.  The successor is released only
  // after the wait, so at most one kernel runs ahead of its dependency.
  if (p.pdl_mode < 2) {
    wait_for_predecessor();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }

  // ---- the copies, two boxes per tile: requests op_lo + who, op_lo + who + step, ... of a range of tiles ----
  uint64_t stream_policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(stream_policy));
  auto request = [&](const CUtensorMap *map, int t_lo, int t_hi, bool is_v, uint32_t bar, int who, int step) {   // tiles [t_lo, t_hi)
    for (int op = 2 * t_lo + who; op < 2 * t_hi; op += step) {
      const int t = op >> 1, hf = op & 1;
      const uint32_t dst = stage + (uint32_t)((is_v ? v_slot(t) : t) * kSlotBytes + hf * kHalfBytes);
      tensor_copy_4d(dst, map, hf * 64, (first_tile + t) << 4, kvh, b, bar, stream_policy);
    }
  };
  if (kShared) {                                         // (the byte counts are set above)
    const int who = lane * (kDecodeWarps + 1) + (producer ? 0 : warp + 1);
    request(&map_k, 0, n, false, kbar, who, kDecodeThreads);
    request(&map_v, 0, n_early, true, vbar_e, who, kDecodeThreads);
  }
  // ---- the warp that issues the copies: lane i takes requests i, i + 32, ... ----
  if (producer) {
    auto issue = [&](const CUtensorMap *map, int t_lo, int t_hi, bool is_v, uint32_t bar) {   // tiles [t_lo, t_hi)
      if (lane == 0 && t_hi > t_lo) mbar_expect_tx(bar, (uint32_t)(t_hi - t_lo) * kSlotBytes);
      __syncwarp();
      request(map, t_lo, t_hi, is_v, bar, lane, 32);
    };
    // (In prefetch mode this warp never waits for the predecessor: it reads nothing of it, and what it requests
    // after barrier A comes after the consumers' wait.  It leaves the release of the successor to the consumers,
    // who give it after their wait: a release from here would let a second launch run ahead.)
    if (!kShared) {
      issue(&map_k, 0, n, false, kbar);
      issue(&map_v, 0, n_early, true, vbar_e);
    }
    bar_sync(1, kDecodeThreads);                         // A: every consumer warp is done with the K slots
    if (kLong && n_late > 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // their reads (and a patched row) precede the refill
      issue(&map_v, n_early, n, true, vbar_l);
    }
    return;                                              // (its cluster arrival at entry stands; it takes part in nothing else)
  }

  // ---- everything that does not depend on the predecessor's results is worked out before the wait ----
  // The instructions after the wait form one long dependent chain per warp, so every address, mask and index
  // that can be known now is computed now and kept in a register.
  // (1) which of this lane's score elements are visible to their heads (sink, own segment, window): bit 4i + e
  //     for the warp's i-th tile, element e of the accumulator
  // Row order of the K fragments: A row m of the mma (m < 8) holds token 2m (m < 4) or 2m + 1, A row m + 8 the
  // other token of the pair (2m, 2m + 1).  So a lane's accumulators belong to two neighbouring tokens, whose
  // weights make one 32-bit word of the second product's B fragment, and the eight rows one ldmatrix phase
  // reads still fall into eight different bank groups of the swizzled tile.
  const int win_lo = p.S + p.n_sel;
  const int seg0_lo = p.S + (p.pooled ? 0 : h0 * p.k_q), seg0_hi = seg0_lo + p.k_q;
  const int seg1_lo = p.S + (p.pooled ? 0 : h1 * p.k_q), seg1_hi = seg1_lo + p.k_q;
  uint32_t vis = 0;
#pragma unroll
  for (int i = 0; i < kQk; ++i) {
    const int r0 = ((first_tile + warp + kDecodeWarps * i) << 4) + 2 * g;
    const int ra = r0 + (g >= 4 ? 1 : 0), rb = r0 + (g >= 4 ? 0 : 1);   // tokens of accumulator elements 0, 1 and 2, 3
    const bool va = ra < p.L, vb = rb < p.L;
    const bool sa = ra < p.S || ra >= win_lo, sb = rb < p.S || rb >= win_lo;
    vis |= (va && h0 < p.G && (sa || (ra >= seg0_lo && ra < seg0_hi)) ? 1u : 0u) << (4 * i);
    vis |= (va && h1 < p.G && (sa || (ra >= seg1_lo && ra < seg1_hi)) ? 2u : 0u) << (4 * i);
    vis |= (vb && h0 < p.G && (sb || (rb >= seg0_lo && rb < seg0_hi)) ? 4u : 0u) << (4 * i);
    vis |= (vb && h1 < p.G && (sb || (rb >= seg1_lo && rb < seg1_hi)) ? 8u : 0u) << (4 * i);
  }
  // (2) fragment addresses: K rows for the first product (ldmatrix), V for the second (transposing ldmatrix), the
  //     weight words this lane writes and reads
  const int mi = lane >> 3, l8 = lane & 7;
  const int arow = 2 * l8 + (((mi & 1) != 0) != (l8 >= 4) ? 1 : 0);
  uint32_t k_off[8];                                     // k-step ks of a tile: slot base + k_off[ks]
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) k_off[ks] = tile_offset(arow, 2 * ks + (mi >> 1));
  const uint16_t *q_lane = p.q + ((int64_t)b * p.H_q + kvh * p.G + min(g, p.G - 1)) * kHeadDim + 2 * c;   // this lane's first query element
  uint32_t v_off = tile_offset((mi >> 1) * 8 + l8, 2 * warp + (mi & 1));
  uint32_t pw_addr = smem_u32(sh.P) + (uint32_t)((h0 * kPHeadWords + g) * 4);   // + tile * kPTileWords * 4; head h1: + kPHeadWords * 4
  uint32_t pr_addr = smem_u32(sh.P) + (uint32_t)((g * kPHeadWords + c) * 4);    // + tile * kPTileWords * 4; rows 2c+8, 2c+9: + 16
  // (3) where this lane's results go: the owners of its two columns, as addresses in their shared memory
  const int col_a = 16 * warp + g, col_b = col_a + 8;
  const int own_a = col_a / cols, own_b = col_b / cols;
  uint32_t dst_a, dst_b, bar_a, bar_b, dst_ml = 0, bar_ml = 0;
  {
    const uint32_t inbox = smem_u32(sh.inbox_o);
    const uint32_t la = inbox + (uint32_t)(((rank * cols + (col_a - own_a * cols)) * kMaxGroup + h0) * 4);
    const uint32_t lb = inbox + (uint32_t)(((rank * cols + (col_b - own_b * cols)) * kMaxGroup + h0) * 4);
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst_a) : "r"(la), "r"(own_a));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst_b) : "r"(lb), "r"(own_b));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar_a) : "r"(inbox_bar), "r"(own_a));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar_b) : "r"(inbox_bar), "r"(own_b));
    if (warp == 0 && g < cs) {                           // lane (g, c) of warp 0 tells CTA g the (max, sum) of heads 2c, 2c+1
      const uint32_t lm = smem_u32(&sh.inbox_ml[rank][h0]);
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst_ml) : "r"(lm), "r"(g));
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar_ml) : "r"(ml_bar), "r"(g));
    }
  }
  // (4) integer divisions cost a hundred instructions apiece: the ones the tail needs are done here, and the step
  //     counter is reduced modulo the ring length with a reciprocal worked out here
  int n_clusters = (int)gridDim.x / cs, cl = ci / cs;
  uint32_t ring_magic = 0xffffffffu / (uint32_t)max(p.ring_len, 1);
  pin(n_clusters); pin(cl); pin(ring_magic);
  // (5) the finishing stage: one thread per output value (own column lc, head fh)
  const int fin_items = my_cols * p.G, n_src = cs;
  int fin_lc = tid / p.G, fin_h = tid - fin_lc * p.G;
  uint16_t *fin_out = p.out + ((int64_t)b * p.H_q + kvh * p.G + fin_h) * kHeadDim + rank * cols + fin_lc;
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) pin(k_off[ks]);
  asm volatile("" : "+l"(q_lane)); pin(v_off); pin(pw_addr); pin(pr_addr); pin(dst_a); pin(dst_b); pin(bar_a); pin(bar_b); pin(dst_ml); pin(bar_ml);
  pin(vis); pin(fin_lc); pin(fin_h); asm volatile("" : "+l"(fin_out));

  SAGEKV_STAMP(1);
  if (p.pdl_mode >= 2) {
    wait_for_predecessor();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  SAGEKV_STAMP(2);

  // What the predecessor may have written is read now, all requests issued back to back (query first: the first
  // product needs it; the step counter last: only the patch of the replaced row needs it), so the round trips to
  // L2 overlap instead of queueing behind one another.
  uint32_t qb[8][2];                      // B fragments of Q^T: lane (g, c) holds head g's dims 16ks + 2c, +1 and 16ks + 8 + 2c, +1
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) qb[ks][0] = qb[ks][1] = 0u;
  if (g < p.G) {
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      asm volatile("ld.global.b32 %0, [%1];" : "=r"(qb[ks][0]) : "l"(q_lane + 16 * ks));
      asm volatile("ld.global.b32 %0, [%1];" : "=r"(qb[ks][1]) : "l"(q_lane + 16 * ks + 8));
    }
  }
  const uint16_t *kn = append ? p.k_new + ((int64_t)b * p.H_kv + kvh) * kHeadDim : nullptr;
  const uint16_t *vn = append ? p.v_new + ((int64_t)b * p.H_kv + kvh) * kHeadDim : nullptr;
  uint4 new_row = make_uint4(0u, 0u, 0u, 0u);            // lanes 0-15: 16 bytes of k_new, lanes 16-31: of v_new
  int step = 0, my_ticket = -1;
  if (append) {
    new_row = ld_v4((lane < 16 ? kn : vn) + (lane & 15) * 8);
    asm volatile("ld.volatile.global.s32 %0, [%1];" : "=r"(step) : "l"(p.d_step));
    // One ticket per CTA, taken once the counter has been read, by a thread of the warp with the fewest tiles.
    // The increment is computed from the value read (its sign bit, never set, plus one), so the atomic cannot
    // be issued before the load has returned; a release fence in its place held the warp for 0.5 us, and the
    // block barrier after the first product with it.  The answer is looked at only when the CTA is done.
    if (tid == kConsumerThreads - 1)
      asm volatile("{ .reg .b32 inc; shr.u32 inc, %2, 31; add.u32 inc, inc, 1; atom.add.relaxed.gpu.global.s32 %0, [%1], inc; }"
                   : "=r"(my_ticket) : "l"(p.tickets + p.B * p.H_kv), "r"(step) : "memory");
  }

  bool timed_out = false;                 // a copy never arrived: reported through the status word; the CTA runs on (its output is then meaningless)
  if (n > 0 && !mbar_wait(kbar, 0u)) timed_out = true;
  SAGEKV_STAMP(3);

  // the staged copy of the replaced row is stale: the warp that works on its tile patches K now, and V as soon as
  // the tile's V copy is here (now, for an early tile; after the first product, for a late one)
  int slot = -1, st = -1;                 // the replaced window row and its CTA-local tile (if 0 <= st < n)
  if (append) {
    uint32_t r = (uint32_t)step - __umulhi((uint32_t)step, ring_magic) * (uint32_t)p.ring_len;   // the quotient may be one short
    while (r >= (uint32_t)p.ring_len) r -= (uint32_t)p.ring_len;
    slot = p.S + p.n_sel + (int)r;
    st = (slot >> 4) - first_tile;
  }
  const bool patcher = append && st >= 0 && st < n && (st & (kDecodeWarps - 1)) == warp;
  auto patch = [&](bool is_v) {           // lanes 0-15 hold the new K row, lanes 16-31 the new V row
    if ((lane >= 16) == is_v) {
      const int row = slot & 15, piece = lane & 15;
      const uint32_t dst = stage + (uint32_t)((is_v ? v_slot(st) : st) * kSlotBytes) + tile_offset(row, piece);
      asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(new_row.x), "r"(new_row.y), "r"(new_row.z), "r"(new_row.w) : "memory");
    }
  };
  if (patcher) {
    patch(false);
    if (st < n_early) {
      if (!mbar_wait(vbar_e, 0u)) timed_out = true;
      patch(true);
    }
    if (SAGEKV_OK_INDEX(p.status, slot >= 0 && slot < p.L)) {
      uint16_t *gdst = (lane < 16 ? p.Kc : p.Vc) + (int64_t)b * p.cs.batch_stride + (int64_t)kvh * p.cs.head_stride +
                       (int64_t)slot * p.cs.token_stride + (lane & 15) * 8;
      st_v4(gdst, new_row);
    }
    __syncwarp();
  }

  // ---- S = K Q^T: this warp's tiles are warp, warp + 8, ...; three at a time ----
  // An mma takes far longer than its issue slot, so the work is laid out as short independent chains: per
  // tile four accumulators (k-steps j and j + 4), the fragments requested ahead of the mmas.
  float sv[kQk][4];
  float wm0 = -INFINITY, wm1 = -INFINITY;
#pragma unroll
  constexpr int kGrp = kLong ? 2 : kQkGroup;                // tiles at once: two where the scores of six tiles stay in registers
  for (int grp = 0; grp < kQk / kGrp; ++grp) {
    if (warp + kDecodeWarps * kGrp * grp < n) {
      float ch[kGrp][4][4];
      uint32_t fa[kGrp][4][4];
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {                   // k-steps 0..3, then 4..7
#pragma unroll
        for (int i = 0; i < kGrp; ++i) {
          const int t = warp + kDecodeWarps * (kGrp * grp + i);
          if (t < n) {
            const uint32_t tb = stage + (uint32_t)(t * kSlotBytes);
#pragma unroll
            for (int j = 0; j < 4; ++j) ldmatrix_x4(tb + k_off[4 * hf + j], fa[i][j][0], fa[i][j][1], fa[i][j][2], fa[i][j][3]);
          }
        }
#pragma unroll
        for (int i = 0; i < kGrp; ++i) {
          if (warp + kDecodeWarps * (kGrp * grp + i) < n) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              if (hf == 0)
                mma_first(ch[i][j][0], ch[i][j][1], ch[i][j][2], ch[i][j][3], fa[i][j][0], fa[i][j][1], fa[i][j][2], fa[i][j][3],
                          qb[j][0], qb[j][1]);
              else
                mma_bf16_16816(ch[i][j][0], ch[i][j][1], ch[i][j][2], ch[i][j][3], fa[i][j][0], fa[i][j][1], fa[i][j][2], fa[i][j][3],
                               qb[4 + j][0], qb[4 + j][1]);
            }
          }
        }
      }
#pragma unroll
      for (int i = 0; i < kGrp; ++i) {
        const int ti = kGrp * grp + i;
        const bool have = warp + kDecodeWarps * ti < n;
        const uint32_t vb4 = have ? (vis >> (4 * ti)) & 15u : 0u;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float x = have ? (ch[i][0][e] + ch[i][1][e]) + (ch[i][2][e] + ch[i][3][e]) : 0.f;
          sv[ti][e] = ((vb4 >> e) & 1u) ? x * p.scale_log2 : -INFINITY;
        }
        wm0 = fmaxf(wm0, fmaxf(sv[ti][0], sv[ti][2]));
        wm1 = fmaxf(wm1, fmaxf(sv[ti][1], sv[ti][3]));
      }
    } else {
#pragma unroll
      for (int i = 0; i < kGrp; ++i)
        sv[kGrp * grp + i][0] = sv[kGrp * grp + i][1] = sv[kGrp * grp + i][2] = sv[kGrp * grp + i][3] = -INFINITY;
    }
  }
  // over the eight lanes that hold the same heads (equal c)
  // (three exchange steps: measured, redux.sync.max.f32 over such a partial lane mask took 0.2 us apiece)
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    wm0 = fmaxf(wm0, __shfl_xor_sync(0xffffffffu, wm0, o));
    wm1 = fmaxf(wm1, __shfl_xor_sync(0xffffffffu, wm1, o));
  }
  if (g == 0) { sh.warp_m[warp][h0] = wm0; sh.warp_m[warp][h1] = wm1; }
  // Each warp's weights are taken relative to its own maximum, which so gets a weight of exactly 1: with one maximum for all rows of the
  // CTA the largest weights of seven warps were rounded too, and the outputs further from 64-bit ones (relative 2.18e-3, now and in
  // the streamed kernel 2.0e-3, at 16 heads x 2049 rows, G = 7; the bf16 output alone is 1.7e-3).
  const float s0 = wm0 == -INFINITY ? 0.f : wm0, s1 = wm1 == -INFINITY ? 0.f : wm1;
  // the weights enter the second product as bf16: one word per (tile, head, row pair g: rows 2g and 2g + 1);
  // their sums per head are taken from the rounded values, so that numerator and denominator agree
  float ls0 = 0.f, ls1 = 0.f;
#pragma unroll
  for (int i = 0; i < kQk; ++i) {
    const int t = warp + kDecodeWarps * i;
    if (t < n) {
      const float x0 = fast_exp2(sv[i][0] - s0), x2 = fast_exp2(sv[i][2] - s0);              // head h0: elements 0 and 2
      const float x1 = fast_exp2(sv[i][1] - s1), x3 = fast_exp2(sv[i][3] - s1);              // head h1: elements 1 and 3
      const uint32_t p0 = g < 4 ? pack_bf16x2(x0, x2) : pack_bf16x2(x2, x0);                 // (row 2g in the low half)
      const uint32_t p1 = g < 4 ? pack_bf16x2(x1, x3) : pack_bf16x2(x3, x1);
      ls0 += __uint_as_float(p0 << 16) + __uint_as_float(p0 & 0xffff0000u);                  // the weights as rounded
      ls1 += __uint_as_float(p1 << 16) + __uint_as_float(p1 & 0xffff0000u);
      const uint32_t wa = pw_addr + (uint32_t)(t * kPTileWords * 4);
      asm volatile("st.shared.u32 [%0], %1;" ::"r"(wa), "r"(p0) : "memory");
      asm volatile("st.shared.u32 [%0], %1;" ::"r"(wa + kPHeadWords * 4), "r"(p1) : "memory");
    }
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    ls0 += __shfl_xor_sync(0xffffffffu, ls0, o);
    ls1 += __shfl_xor_sync(0xffffffffu, ls1, o);
  }
  bar_sync(1, kDecodeThreads);   // A: the maxima are complete, and nobody reads a K slot any more (the copy warp refills them)

  float M0, M1;                  // maxima of heads 2c, 2c+1 over the CTA's rows (log2 units)
  {
    float a0[kDecodeWarps], a1[kDecodeWarps];
#pragma unroll
    for (int w = 0; w < kDecodeWarps; ++w) { a0[w] = sh.warp_m[w][h0]; a1[w] = sh.warp_m[w][h1]; }
#pragma unroll
    for (int s2 = kDecodeWarps / 2; s2 > 0; s2 >>= 1)   // a tree, not a chain
#pragma unroll
      for (int w = 0; w < s2; ++w) { a0[w] = fmaxf(a0[w], a0[w + s2]); a1[w] = fmaxf(a1[w], a1[w + s2]); }
    M0 = a0[0]; M1 = a1[0];
  }
  SAGEKV_STAMP_AFTER(4, M0 + M1);
  if (g == 0) {
    const float f0 = M0 == -INFINITY ? 0.f : fast_exp2(wm0 - M0), f1 = M1 == -INFINITY ? 0.f : fast_exp2(wm1 - M1);
    sh.warp_f[warp][h0] = f0; sh.warp_f[warp][h1] = f1;
    sh.warp_l[warp][h0] = ls0 * f0; sh.warp_l[warp][h1] = ls1 * f1;
  }
  bar_sync(2, kConsumerThreads);   // B: the weights are in shared memory (and a patched early V row is visible)
  SAGEKV_STAMP(5);
  // The (max, sum) pairs of the CTA go to every CTA of the cluster now, ahead of the second product, with
  // asynchronous stores that count their bytes on a barrier of their own at the receiver: the finishing stage
  // has its weights ready before the columns arrive.
  cluster.barrier_wait();                                // pairs with the arrive at kernel entry: every peer runs, its barriers are set up
  auto send2 = [&](uint32_t addr, uint32_t rbar, float x, float y) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];"
                 ::"r"(addr), "f"(x), "f"(y), "r"(rbar) : "memory");
  };
  if (warp == 0 && g < cs) {
    float L0 = 0.f, L1 = 0.f;            // sums of the (bf16-rounded) weights of heads 2c, 2c+1 over the CTA's rows
#pragma unroll
    for (int w = 0; w < kDecodeWarps; ++w) { L0 += sh.warp_l[w][h0]; L1 += sh.warp_l[w][h1]; }
    send2(dst_ml, bar_ml, M0, L0);
    send2(dst_ml + 8u, bar_ml, M1, L1);
  }

  // ---- O^T = V^T P: columns 16*warp .. +15 over all rows, the early V tiles first ----
  // A B fragment is two of the weight words (rows 2c, 2c+1 and 2c+8, 2c+9 of head g).  Eight tiles per step, one of each warp's in
  // the first product on an accumulator chain of its own, which is brought to the CTA's maxima at the end; all fragments
  // requested before the mmas.  (An mma's result takes about 130 cycles: the sums of the weights used to come from a second
  // mma per tile against a fragment of ones, on two chains eleven links long, and those chains alone took 0.75 us; they are
  // summed in registers now.)
  float xc[kDecodeWarps][4];              // O^T of warp u's rows: (col_a, h0) (col_a, h1) (col_b, h0) (col_b, h1)
#pragma unroll
  for (int u = 0; u < kDecodeWarps; ++u) xc[u][0] = xc[u][1] = xc[u][2] = xc[u][3] = 0.f;
  auto eight_tiles = [&](int t8, int t_hi, bool late) {  // of tiles [t8, t8 + 8) those below t_hi, and with `late` those that came late
    uint32_t va[kDecodeWarps][4], pb[kDecodeWarps][2];
#pragma unroll
    for (int u = 0; u < kDecodeWarps; ++u) {
      if (t8 + u < t_hi && (!late || t8 + u >= n_early)) {
        ldmatrix_x4_trans(stage + (uint32_t)(v_slot(t8 + u) * kSlotBytes) + v_off, va[u][0], va[u][1], va[u][2], va[u][3]);
        const uint32_t ra = pr_addr + (uint32_t)((t8 + u) * kPTileWords * 4);
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(pb[u][0]) : "r"(ra));
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(pb[u][1]) : "r"(ra + 16));
      }
    }
#pragma unroll
    for (int u = 0; u < kDecodeWarps; ++u)
      if (t8 + u < t_hi && (!late || t8 + u >= n_early))
        mma_bf16_16816(xc[u][0], xc[u][1], xc[u][2], xc[u][3], va[u][0], va[u][1], va[u][2], va[u][3], pb[u][0], pb[u][1]);
  };
  if (n_early > 0 && !mbar_wait(vbar_e, 0u)) timed_out = true;
  for (int t8 = 0; t8 < n_early; t8 += kDecodeWarps) eight_tiles(t8, n_early, false);
  if (kLong && n_late > 0) {                             // (the same for every thread of the CTA)
    if (!mbar_wait(vbar_l, 0u)) timed_out = true;
    if (patcher && st >= n_early) patch(true);
    bar_sync(2, kConsumerThreads);                       // a patched late V row is visible
    for (int t8 = n_early & ~(kDecodeWarps - 1); t8 < n; t8 += kDecodeWarps) eight_tiles(t8, n, true);
  }
  float2 wf[kDecodeWarps];                // the warps' factors, asked for while the last products are on their way
#pragma unroll
  for (int u = 0; u < kDecodeWarps; ++u) wf[u] = *reinterpret_cast<const float2 *>(&sh.warp_f[u][h0]);
  float acc[4];                           // (col_a, h0) (col_a, h1) (col_b, h0) (col_b, h1)
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float a[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) a[u] = xc[u][e] * ((e & 1) ? wf[u].y : wf[u].x) + xc[u + 4][e] * ((e & 1) ? wf[u + 4].y : wf[u + 4].x);
    acc[e] = (a[0] + a[1]) + (a[2] + a[3]);
  }
  if (timed_out) atomicOr(p.status, kStatusWaitTimeout);
  SAGEKV_STAMP_AFTER(6, acc[0] + acc[1] + acc[2] + acc[3]);

  // ---- merge the CTAs of the cluster: the owner of a column slice receives it from every CTA ----
  // Every warp sends its 16 columns straight from registers into the owners' inboxes with asynchronous stores
  // that count their bytes on the owner's barrier: data and signal travel together and nobody waits for an
  // acknowledgement or for a cluster-wide barrier; a CTA only waits for its own inbox to fill.
  if (h0 < p.G) {
    send2(dst_a, bar_a, acc[0], acc[1]);
    send2(dst_b, bar_b, acc[2], acc[3]);
  }
  SAGEKV_STAMP(7);
  // the weights of the sources for this thread's first output: worked out while the columns are still on their way
  float fin_w[kDecodeMaxCluster], fin_M = -INFINITY, fin_inv = 0.f, fin_l = 0.f;
  auto source_weights = [&](int h) {
    float mx[kDecodeMaxCluster], lsum[kDecodeMaxCluster];
#pragma unroll
    for (int sI = 0; sI < kDecodeMaxCluster; ++sI) {
      const float2 ml = sI < n_src ? sh.inbox_ml[sI][h] : make_float2(-INFINITY, 0.f);
      mx[sI] = ml.x; lsum[sI] = ml.y;
    }
    float tm[kDecodeMaxCluster];
#pragma unroll
    for (int sI = 0; sI < kDecodeMaxCluster; ++sI) tm[sI] = mx[sI];
#pragma unroll
    for (int w2 = kDecodeMaxCluster / 2; w2 > 0; w2 >>= 1)
#pragma unroll
      for (int sI = 0; sI < w2; ++sI) tm[sI] = fmaxf(tm[sI], tm[sI + w2]);
    fin_M = tm[0];
#pragma unroll
    for (int sI = 0; sI < kDecodeMaxCluster; ++sI) {
      fin_w[sI] = fin_M == -INFINITY ? 0.f : fast_exp2(mx[sI] - fin_M);
      lsum[sI] *= fin_w[sI];
    }
#pragma unroll
    for (int w2 = kDecodeMaxCluster / 2; w2 > 0; w2 >>= 1)
#pragma unroll
      for (int sI = 0; sI < w2; ++sI) lsum[sI] += lsum[sI + w2];
    fin_l = lsum[0];
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(fin_inv) : "f"(fin_l));   // the output is rounded to bf16: an approximate reciprocal is ample
  };
  if (!mbar_wait(ml_bar, 0u) && tid == 0) atomicOr(p.status, kStatusWaitTimeout);
  if (tid < fin_items) source_weights(fin_h);
  if (!mbar_wait(inbox_bar, 0u) && tid == 0) atomicOr(p.status, kStatusWaitTimeout);
  SAGEKV_STAMP(8);

  // ---- finish columns [rank*cols, rank*cols + my_cols) of every head from the inbox ----
  const int bk = b * p.H_kv + kvh;
  float *part = p.partials + ((int64_t)bk * n_clusters + cl) * kPartialStride;
  for (int item = tid; item < fin_items; item += kConsumerThreads) {
    if (item != tid) {
      fin_lc = item / p.G;
      fin_h = item - fin_lc * p.G;
      fin_out = p.out + ((int64_t)b * p.H_q + kvh * p.G + fin_h) * kHeadDim + rank * cols + fin_lc;
    }
    if (item != tid) source_weights(fin_h);
    const int lc = fin_lc, h = fin_h, col = rank * cols + lc;
    float ov[kDecodeMaxCluster];
#pragma unroll
    for (int sI = 0; sI < kDecodeMaxCluster; ++sI)       // the loads of all sources are in flight together
      ov[sI] = sI < n_src ? sh.inbox_o[(sI * cols + lc) * kMaxGroup + h] * fin_w[sI] : 0.f;
#pragma unroll
    for (int w2 = kDecodeMaxCluster / 2; w2 > 0; w2 >>= 1)
#pragma unroll
      for (int sI = 0; sI < w2; ++sI) ov[sI] += ov[sI + w2];
    const float o = ov[0], l = fin_l, M = fin_M;
    if (n_clusters == 1) {
      const float outv = l > 0.f ? o * fin_inv : 0.f;
      *fin_out = (uint16_t)(pack_bf16x2(outv, 0.f) & 0xffffu);
      if (p.lse != nullptr && col == 0)
        p.lse[(int64_t)b * p.H_q + kvh * p.G + h] = l > 0.f ? (M + log2f(l)) * kLn2 : -INFINITY;
    } else {
      part[h * kHeadDim + col] = o;
      if (col == 0) {
        part[kMaxGroup * kHeadDim + h] = M;
        part[kMaxGroup * kHeadDim + kMaxGroup + h] = l;
      }
    }
  }

  if (n_clusters > 1) {
    // ---- several clusters per head: the last CTA to arrive merges the cluster results ----
    __threadfence();
    bar_sync(2, kConsumerThreads);
    if (tid == 0) sh.last = atomicAdd(&p.tickets[bk], 1) == (int)gridDim.x - 1;
    bar_sync(2, kConsumerThreads);
    if (sh.last != 0) {
      __threadfence();
      const float *all = p.partials + (int64_t)bk * n_clusters * kPartialStride;
      for (int item = tid; item < p.G * kHeadDim; item += kConsumerThreads) {
        const int h = item >> 7, col = item & 127;
        float M = -INFINITY;
        for (int i = 0; i < n_clusters; ++i) M = fmaxf(M, __ldcg(all + i * kPartialStride + kMaxGroup * kHeadDim + h));
        float o = 0.f, l = 0.f;
        for (int i = 0; i < n_clusters; ++i) {
          const float *pi = all + i * kPartialStride;
          const float wgt = M == -INFINITY ? 0.f : fast_exp2(__ldcg(pi + kMaxGroup * kHeadDim + h) - M);
          o += __ldcg(pi + h * kHeadDim + col) * wgt;
          l += __ldcg(pi + kMaxGroup * kHeadDim + kMaxGroup + h) * wgt;
        }
        const float outv = l > 0.f ? o / l : 0.f;
        p.out[((int64_t)b * p.H_q + kvh * p.G + h) * kHeadDim + col] = (uint16_t)(pack_bf16x2(outv, 0.f) & 0xffffu);
        if (p.lse != nullptr && col == 0)
          p.lse[(int64_t)b * p.H_q + kvh * p.G + h] = l > 0.f ? (M + log2f(l)) * kLn2 : -INFINITY;
      }
      if (tid == 0) p.tickets[bk] = 0;
    }
  }
  // ---- the step counter: whoever took the last ticket of the launch knows that every CTA has read it ----
  if (append && tid == kConsumerThreads - 1 && my_ticket == (int)(gridDim.x * gridDim.y * gridDim.z) - 1) {
    p.tickets[p.B * p.H_kv] = 0;
    *p.d_step = step + 1;
  }
  SAGEKV_STAMP(9);
  SAGEKV_TRACE_END(p.out);
}

}  // namespace sagekv

#include "decode_attn_tc.cuh"
#include "decode_stream.cuh"

namespace sagekv {

static size_t decode_tc_smem_bytes(int per_cta) {
  return 1024 + (size_t)((per_cta + 7) / 8) * kTcBlockBytes + (size_t)per_cta * kSlotBytes + sizeof(DecShared);
}

static_assert(kStreamCtasPerSm * (sizeof(StShared) + 1024) <= 233472, "two CTAs of the stream kernel fit on one SM");
static_assert(1024 + (size_t)kDecodeSlots * kSlotBytes + sizeof(DecShared) <= 232448, "the staging area and the rest fit into 227 KB");
static int decode_slots(int per_cta) { return 2 * per_cta < kDecodeSlots ? 2 * per_cta : kDecodeSlots; }
static size_t decode_smem_bytes(int per_cta) {
  return 1024 + (size_t)decode_slots(per_cta) * kSlotBytes + sizeof(DecShared);
}

// How many clusters of `c` CTAs of a kernel can be on the device at once (a cluster must fit into one GPC, so this is
// not n_sm / c: on this part 15 clusters of 8 whole-SM CTAs but 22 of 6).  Asked of the runtime once per slot of the
// caller's table and remembered there as answer + 1 (two threads may both ask: they get the same answer).  0: unknown.

template <typename Kernel>
static int cluster_capacity(Kernel kernel, int threads, size_t smem, int c, std::atomic<int> *slot) {
  int known = slot->load(std::memory_order_relaxed);
  if (known == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(c * 64), 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = c;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nn = 0;
    if (cudaOccupancyMaxActiveClusters(&nn, kernel, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      nn = 0;
    }
    known = nn + 1;
    slot->store(known, std::memory_order_relaxed);
  }
  return known - 1;
}

static int resident_capacity(int device, int c, int tiles) {   // of decode_attn_kernel, `tiles` tiles per CTA
  static std::atomic<int> table[64][kDecodeMaxCluster + 1][kDecodeMaxTiles + 1];
  if (device < 0 || device >= 64 || c < 1 || c > kDecodeMaxCluster || tiles < 0 || tiles > kDecodeMaxTiles) return 0;
  return cluster_capacity(decode_attn_kernel<true, false>, kDecodeThreads, decode_smem_bytes(tiles), c, &table[device][c][tiles]);
}

static int stream_capacity(int device, int c) {                // of decode_stream_kernel, clusters of c CTAs
  static std::atomic<int> table[64][kStMaxCluster + 1];
  if (device < 0 || device >= 64 || c < 1 || c > kStMaxCluster) return 0;
  return cluster_capacity(decode_stream_kernel, kStThreads, sizeof(StShared), c, &table[device][c]);
}

// What moving the launch's rows takes next to a kernel's own time of `us` (the larger one dominates, and the other is
// not hidden completely): fitted as the cube root of the sum of cubes.
static float with_traffic(float us, int heads, int L) {
  const float t = 1.f + (float)heads * (float)L * (4.f * kHeadDim) / 6.4e6f;   // 6.4 TB/s
  return cbrtf(us * us * us + t * t * t);
}

cudaError_t decode_setup(DeviceInfo *dev) {
  (void)dev;
  for (auto kernel : {decode_attn_kernel<false, false>, decode_attn_kernel<false, true>, decode_attn_kernel<true, false>, decode_attn_kernel<true, true>}) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)decode_smem_bytes(kDecodeMaxTiles));
    if (e != cudaSuccess) return e;
  }
  cudaError_t e3 = cudaFuncSetAttribute(decode_stream_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(StShared));
  if (e3 == cudaSuccess) e3 = cudaFuncSetAttribute(decode_stream_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);   // clusters of 16
  if (e3 != cudaSuccess) return e3;
  return cudaFuncSetAttribute(decode_attn_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)decode_tc_smem_bytes(kTcMaxTiles));
}

// In modes 0 and 1 launches of this many KV heads keep the older, coarser costs of both kernels: two launches' clusters of six, the
// size that suits most of them, no longer fit on the device together, which the newer ones do not follow (us per launch with the older /
// newer: 17 x 2557 rows, G = 8, 7.0 / 8.1; 19 x 2557 7.1 / 8.6; 19 x 1021 4.9 / 5.6; 24 x 2561 8.5 / 9.1; but 18 x 4097 11.2 / 10.0; of 2892 launches of
// 1 to 64 heads timed both ways 55 took over 4 % longer with the newer ones from 20 heads on, 11 from 17 on.)
constexpr int kDecodeManyHeads = 17;

// Whether all nine warps of a CTA ask for its copies, or the ninth alone.  Sharing takes the copies' issue time off the launch, which
// counts where they are asked for behind the dependency wait, or late because the predecessor's clusters are in the way (us per launch
// alone / shared: mode 0, 8 heads x 2049 rows 6.5 / 5.0, 1025 rows 4.7 / 4.1; mode 2, 8 x 2049 3.96 / 3.74, 16 x 2049 5.7 / 5.0, 8 x 3000
// 5.3 / 4.4).  In modes 0 and 1 the eight warps have the query to ask for meanwhile, and few copies are soon asked for by one (8 x
// 513 3.60 / 3.75, 1 x 4 heads with 7 tiles per CTA 3.61 / 3.75, with 9 3.97 / 3.90; with 64 CTAs and 7 tiles 4.07 / 3.88); nor does it
// help where V tiles wait for K slots in many CTAs (16 x 3073 8.20 / 8.52), or several clusters per head (8 x 8193 12.0 / 12.4).
static bool decode_shares_issue(int mode, int ctas, int per_cta, int units, int n_clusters) {
  if (n_clusters > 1) return false;
  if (mode == 2) return true;
  return units < kDecodeManyHeads && per_cta >= (ctas >= 56 ? 7 : 9) && !(2 * per_cta > kDecodeSlots && units >= 12);
}

// Launch geometry for a reduced cache of L rows: nc clusters of c CTAs per KV head, a CTA taking at most
// kDecodeMaxTiles tiles (its K tiles must all be resident); nc > 1 only beyond that, the clusters' results then
// merged through scratch by the last CTA to arrive.  heads = batch x KV heads of the launch (0, or dev null: not
// known; then clusters of 8).  Back-to-back launches overlap (the next one fetches its rows while this one
// computes), which only works if the clusters of two launches fit on the device together, so the cluster sizes
// are compared by a cost fitted to measurements (below).
// (15 clusters of 8 whole-SM CTAs fit at once, 22 of 6, 26 of 5, 33 of 4.)
float decode_geometry(int L, int heads, int G, const DeviceInfo *dev, int mode, int *n_clusters, int *cs, int *per_cta_tiles,
                      int *smem_bytes) {
  const int n_tiles = (L + 15) / 16;
  int c = 1;
  while (c < kDecodeBaseCluster && c * 2 <= n_tiles) c <<= 1;                   // cluster size 1, 2, 4 or 8
  int nc = (n_tiles + c * kDecodeMaxTiles - 1) / (c * kDecodeMaxTiles);          // the fewest clusters per head
  float best = 0.f;
  const bool many = mode != 2 && heads >= kDecodeManyHeads;
  int best_waves = 1;
  if (dev != nullptr && heads > 0) {
    int best_c = c, best_nc = nc;
    const float bytes = (float)heads * (float)L * (4.f * kHeadDim);
    // up to kDecodeExtraClusters more clusters per head than needed: beyond one cluster the results are merged
    // through scratch anyway, and more, smaller clusters leave fewer V tiles waiting for a K slot
    for (int n_try = nc; n_try <= (nc > 1 ? nc + kDecodeExtraClusters : nc); ++n_try) {
      for (int cand = c; cand >= (c == kDecodeBaseCluster ? 4 : c); --cand) {
        const int per = (n_tiles + cand * n_try - 1) / (cand * n_try);
        if (per > kDecodeMaxTiles) continue;
        const int cap = resident_capacity(dev->device, cand, per);
        if (cap <= 0) continue;
        // Fitted to every cluster size (4 to 8) at 1 to 48 heads x 129 .. 4097 rows in all overlap modes, G = 4 (us per launch): a time
        // per tile of a CTA, 0.3 - 0.5 and a time per V tile that waits for a K slot where some do (one warp asking for the copies: less by
        // 0.7, timed at 12 to 16 heads x 2561 .. 5121 rows), more where the clusters of two launches do not fit on the device together, up
        // to as much again as they overfill it; beside that what moving the rows takes; and for the merge through scratch a time per query
        // head, whose results it moves (1 to 24 heads x 5697 .. 12289 rows, G = 1, 4, 8: a fixed 3.4 took one head x 12285 rows, G = 8, to 11.1
        // in place of 9.2, and kept 2 x 8193, G = 1, from 6.2, at 7.0).  (Over 1716 launches in modes 0 and 1, G = 1 to 8, what these rules and
        // those for the streamed launches choose is on average 1.1 % slower than the best that could be forced; over 1176 at lengths
        // and numbers of heads between the fitted ones 1.5 %.)
        const int late = 2 * per > kDecodeSlots ? 2 * per - kDecodeSlots : 0, units = heads * n_try;
        const int waves = (units + cap - 1) / cap;                              // of one launch
        const bool is_long = per > kQkGroup * kDecodeWarps;
        const float over = 2 * units > cap ? (float)((units < cap ? 2 * units : 2 * cap) - cap) / (float)cap : -1.f;
        const float share = (float)n_tiles / (float)(cand * n_try);
        float one, cost;
        if (many) {
          one = 2.97f + 0.0445f * (float)per * (2 * units <= cap ? 1.f : 2.f) + 0.084f * (float)late;
        } else if (mode == 2) {
          one = 2.89f + 0.035f * (float)per + (is_long ? 0.26f + 0.056f * (float)late : 0.f) + (over >= 0.f ? 0.31f + 0.59f * over : 0.f);
        } else {
          one = decode_shares_issue(mode, units * cand, per, units, n_try) ? 3.11f + 0.073f * share + (is_long ? 0.49f + 0.04f * (float)late : 0.f)
                                                                           : 3.f + 0.057f * share + 0.072f * (share > 6.f ? share - 6.f : 0.f) - (is_long ? 0.7f - 0.03f * (float)late : 0.f);
          one += over >= 0.f ? 0.21f + 0.28f * over : 0.f;
        }
        if (n_try > 1) one += many ? 3.4f : (mode == 2 ? 2.2f + 0.35f * (float)G : 2.4f + 0.4f * (float)G);
        one = (float)waves * one + (many ? 0.f : 0.5f * (float)(waves - 1));
        if (many) {
          cost = one;
        } else if (mode == 2) {
          const float t = 1.f + bytes / 5.3e6f;
          cost = powf(powf(one, 2.9f) + powf(t, 2.9f), 1.f / 2.9f);
        } else {
          const float t = 1.f + bytes / 7.3e6f;
          cost = sqrtf(one * one + t * t);
        }
        if (best == 0.f || cost < best) { best = cost; best_c = cand; best_nc = n_try; best_waves = waves; }
      }
    }
    c = best_c;
    nc = best_nc;
  } else if (nc > 1) {
    nc += kDecodeExtraClusters;                          // (context set-up: the most clusters per head a launch may choose)
  }
  const int per_cta = (n_tiles + c * nc - 1) / (c * nc);                         // most tiles a CTA gets
  *n_clusters = nc;
  *cs = c;
  *per_cta_tiles = per_cta;
  *smem_bytes = (int)decode_smem_bytes(per_cta);
  if (many && best > 0.f) best = with_traffic((float)best_waves * (3.9f + 0.14f * (float)per_cta + (nc > 1 ? 3.4f : 0.f)), heads, L);
  return best;
}

// The best launch of decode_stream_kernel: CTAs per head, heads per CTA, and its cost in us (0: none).  Mode 2, fitted to forced launches
// of every split, 1 to 128 heads x 125 .. 8193 rows x 1 to 8 query heads per KV head (G): 1.75 plus 0.017 per CTA of a
// cluster, 0.47 per tile of a warp (the ring's three tiles per warp in flight against the latency of a copy; 0.6 where a CTA takes
// whole heads), 0.06 per query head, 0.41 per round of the finishing stage (a thread takes two columns of a head: a cluster of 2 with
// G = 8 needs two), 0.8 per further head of a CTA; up to 1.1 more when two launches' CTAs do not fit on the device together.  A second
// wave costs a whole time again.  Modes 0 and 1, fitted against the resident kernel as it is now (1 to 48 heads x 129 .. 4097 rows):
// 3.47 and 2.69, 0.52 and 0.62 per tile of a warp, 1 % per query head beyond four.
static float stream_geometry(int L, int heads, int G, const DeviceInfo &dev, int mode, int *split, int *per_cta) {
  const int n_tiles = (L + 15) / 16;
  if ((int64_t)n_tiles * heads > (int64_t)1 << 30) return 0.f;
  const bool overlap = mode == 2, many = heads >= kDecodeManyHeads;
  const float base = many ? 3.9f : (mode == 0 ? 3.47f : 2.69f), per_s = many ? 0.025f : 0.006f, per_round = many ? 0.6f : (mode == 0 ? 0.52f : 0.62f);
  float best = 0.f;
  for (int s = 1; s <= kStMaxCluster && s <= n_tiles; s <<= 1) {
    const int cap = s == 1 ? kStreamCtasPerSm * dev.n_sm : s * stream_capacity(dev.device, s);
    if (cap <= 0) continue;
    const int per = s == 1 ? (heads + cap - 1) / cap : 1;
    const int ctas = s == 1 ? (heads + per - 1) / per : heads * s;
    const int waves = (ctas + cap - 1) / cap;
    const int rounds = (per * ((n_tiles + s - 1) / s) + kStWarps - 1) / kStWarps;
    const int finish = s == 1 ? 0 : (G * (kHeadDim / 2) + s * kStThreads - 1) / (s * kStThreads);   // (s == 1: no such stage)
    const float one = overlap ? 1.75f + 0.017f * (float)s + (s > 1 ? 0.47f : 0.6f) * (float)rounds + 0.06f * (float)G + 0.41f * (float)finish + 0.8f * (float)(per - 1)
                              : (base + per_s * (float)s + per_round * (float)rounds + 0.8f * (float)(per - 1)) *
                                    (1.f + 0.01f * (float)(G > 4 ? G - 4 : 0));
    float cost = with_traffic((float)waves * one, heads, L);
    if (2 * ctas > cap) cost += (overlap ? 0.13f : 0.3f) + (overlap ? 0.95f : 1.2f) * (float)(2 * (ctas < cap ? ctas : cap) - cap) / (float)cap;
    if (best == 0.f || cost < best) { best = cost; *split = s; *per_cta = per; }
  }
  return best;
}

// cuTensorMapEncodeTiled, looked up through the runtime (the library does not link against the driver)
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled_fn() {
  static std::once_flag once;
  static EncodeTiledFn fn = nullptr;
  std::call_once(once, [] {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(f);
    else
      (void)cudaGetLastError();
  });
  return fn;
}

// [B, H_kv, L, 128] bf16 through the cache strides, boxes of 16 rows x 64 columns with the 128-byte swizzle;
// rows at and beyond L read as zeros
static bool make_cache_map(CUtensorMap *map, const uint16_t *base, const DecodeParams &p) {
  EncodeTiledFn enc = encode_tiled_fn();
  if (enc == nullptr) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)kHeadDim, (cuuint64_t)p.L, (cuuint64_t)p.H_kv, (cuuint64_t)p.B};
  const cuuint64_t strides[3] = {(cuuint64_t)p.cs.token_stride * 2, (cuuint64_t)p.cs.head_stride * 2,
                                 (cuuint64_t)p.cs.batch_stride * 2};
  const cuuint32_t box[4] = {64, 16, 1, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<uint16_t *>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t launch_decode(const DecodeParams &p, const DeviceInfo &dev, cudaStream_t stream) {
  int n_clusters, cs, per_cta, smem, split = 1, heads_per_cta = 1;
  const int mode = p.overlapping ? 2 : p.pdl_mode;
  const float cost = decode_geometry(p.L, p.B * p.H_kv, p.G, &dev, mode, &n_clusters, &cs, &per_cta, &smem);
  const bool tc = p.variant == 2 && n_clusters == 1 && per_cta <= kTcMaxTiles;
  // Caches that fill the SMs more than once, and long ones, are streamed; short ones are brought in whole.  (us per
  // launch whole / streamed, overlapping: 8 heads x 2049 rows 3.9 / 4.7, 8 x 8193 10.8 / 8.5, 16 x 8193 21.0 / 13.1, 256 x 2049 84.8 / 42.8)
  const float stream_cost = tc ? 0.f : stream_geometry(p.L, p.B * p.H_kv, p.G, dev, mode, &split, &heads_per_cta);
  const bool streamed = stream_cost > 0.f && cost > 0.f && stream_cost < cost;
  CUtensorMap map_k, map_v;
  if (!make_cache_map(&map_k, p.Kc, p) || !make_cache_map(&map_v, p.Vc, p)) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = streamed ? split : cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (streamed) {
    const int heads = p.B * p.H_kv;
    cfg.gridDim = dim3((unsigned)(split > 1 ? heads * split : (heads + heads_per_cta - 1) / heads_per_cta), 1, 1);
    cfg.blockDim = dim3(kStThreads, 1, 1);
    cfg.dynamicSmemBytes = sizeof(StShared);
    return cudaLaunchKernelEx(&cfg, decode_stream_kernel, p, map_k, map_v, split, heads_per_cta);
  }
  cfg.gridDim = dim3((unsigned)(n_clusters * cs), (unsigned)p.H_kv, (unsigned)p.B);
  cfg.blockDim = dim3(kDecodeThreads, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  // the tensor-memory variant where it applies: one cluster per head, every tile resident twice over
  if (tc) {
    cfg.dynamicSmemBytes = decode_tc_smem_bytes(per_cta);
    return cudaLaunchKernelEx(&cfg, decode_attn_tc_kernel, p, map_k, map_v, per_cta);
  }
  // the short instance keeps three tiles' scores per warp and has every V tile resident from the start
  const bool is_long = 2 * per_cta > kDecodeSlots || per_cta > kQkGroup * kDecodeWarps;
  const bool shared = decode_shares_issue(mode, (int)(cfg.gridDim.x * cfg.gridDim.y * cfg.gridDim.z), per_cta, p.B * p.H_kv * n_clusters, n_clusters);
  const auto kernel = is_long ? (shared ? decode_attn_kernel<true, true> : decode_attn_kernel<true, false>)
                              : (shared ? decode_attn_kernel<false, true> : decode_attn_kernel<false, false>);
  return cudaLaunchKernelEx(&cfg, kernel, p, map_k, map_v, decode_slots(per_cta));
}

}  // namespace sagekv

SAGEKV_TRACE_READER(sagekv_trace_read)
