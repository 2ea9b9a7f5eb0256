// Selection from short rows: every CTA holds the whole score row in registers and selects by itself.
//
// A row of up to 32768 scores fits the registers of one CTA of 512 threads, so nothing is exchanged: the CTAs of a row (more than one
// only where the gather is worth spreading) all make the same selection and each writes and gathers a share of its slots.  Which rows
// take this way: short_rows_apply.
// Up to four vectors of four scores per thread (and wherever the shorter way below does not apply):
//   1. thread maxima give a bound below which no score can be selected (where there are at least k_q of them), and
//   2. one histogram of 2048 bins between that bound and the row's maximum finds the bin of the k_q-th largest score; as long as
//      that bin holds more than kShortBorder scores its keys are spread over the bins once more, by their next bits;
//   3. scores in higher bins are kept, the few of the bin ranked exactly (equal scores by position);
//   4. one prefix sum in position order gives the slots.
// Rows of equal scores and any k_q up to the row's length are selected the same way.
// More scores per thread: as the prefilter of the long rows, without its exchanges.  The histogram is taken of the maxima of
// groups of scores first, which gives a bound that few more than k_q scores reach; these are written out in position order and
// decided upon by fast_decide.
#pragma once

namespace sagekv {

constexpr int kShortBins = 2048;
constexpr int kShortBorder = 32;          // scores of the cut's bin that are ranked one against another
constexpr int kShortMaxE = 16 * 4 * kSelThreads;

// Element 4u + e of a thread is element e of vector (warp * kVec + u) * 32 + lane of the row, so that (warp, u, lane, e) order is
// position order; the first n of a thread's elements exist.  Key 0, below the key of every number, stands for none.
template <int kVec, bool kKeys>
struct ShortRow {
  uint32_t w[4 * kVec];                   // keys, or (kKeys = false) scores whose keys are worked out where they are needed
  int n;
  __device__ __forceinline__ void set(int i, float x) { w[i] = kKeys ? (i < n ? number_key(x) : 0u) : __float_as_uint(x); }
  __device__ __forceinline__ float score(int i) const { return __uint_as_float(w[i]); }
  __device__ __forceinline__ uint32_t key(int i) const { return kKeys ? w[i] : (i < n ? number_key(__uint_as_float(w[i])) : 0u); }
};

template <int kVec>
constexpr int kMaskWords = (4 * kVec + 31) / 32;

// For masks of the threads' elements (bit i & 31 of word i >> 5 for element i): how many bits are set before each of the thread's
// vectors, in position order, and in all.  tmp: one word per warp, written here.  Holds one block barrier, between the writing and
// the reading of tmp.
template <int kVec>
__device__ __forceinline__ int ordered_prefix(const uint32_t (&mask)[kMaskWords<kVec>], int *tmp, int (&before)[kVec]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kWords = (kVec + 3) / 4;
  uint32_t cnt[kWords], inc[kWords];                     // a byte per vector: at most 128 per warp
#pragma unroll
  for (int w = 0; w < kWords; ++w) {
    uint32_t m = (w & 1) == 0 ? mask[w >> 1] & 0xffffu : mask[w >> 1] >> 16;
    m = m - ((m >> 1) & 0x5555u);
    m = (m & 0x3333u) + ((m >> 2) & 0x3333u);            // every nibble holds its bit count
    m = (m | (m << 8)) & 0x00ff00ffu;
    cnt[w] = (m | (m << 4)) & 0x0f0f0f0fu;
    inc[w] = cnt[w];
  }
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
#pragma unroll
    for (int w = 0; w < kWords; ++w) {
      const uint32_t n = __shfl_up_sync(0xffffffffu, inc[w], off);
      if (lane >= off) inc[w] += n;
    }
  }
  uint32_t total[kWords];
  int sum = 0;
#pragma unroll
  for (int w = 0; w < kWords; ++w) {
    total[w] = __shfl_sync(0xffffffffu, inc[w], 31);
    sum += (int)((total[w] & 0xffu) + ((total[w] >> 8) & 0xffu) + ((total[w] >> 16) & 0xffu) + (total[w] >> 24));
  }
  if (lane == 0) tmp[warp] = sum;
  __syncthreads();
  const int t = lane < kSelWarps ? tmp[lane] : 0;
  int base = __reduce_add_sync(0xffffffffu, lane < warp ? t : 0);
  const int all = __reduce_add_sync(0xffffffffu, t);
#pragma unroll
  for (int u = 0; u < kVec; ++u) {
    const int s = 8 * (u & 3);
    before[u] = base + (int)(((inc[u >> 2] - cnt[u >> 2]) >> s) & 0xffu);
    base += (int)((total[u >> 2] >> s) & 0xffu);
  }
  return all;
}

// In `hist`, the bin in which the wanted-th largest key falls: found = bin, the key's rank in it, the keys in it.  Begins and ends
// with a barrier.
__device__ __forceinline__ void short_cut(const uint32_t *hist, int wanted, int *tmp, int *found) {
  __syncthreads();
  const int tid = threadIdx.x;
  const uint4 c4 = *reinterpret_cast<const uint4 *>(&hist[kShortBins - 4 - 4 * tid]);   // thread 0 has the top four bins
  const int cnt[4] = {(int)c4.w, (int)c4.z, (int)c4.y, (int)c4.x};
  int above = block_exclusive_scan(cnt[0] + cnt[1] + cnt[2] + cnt[3], tmp);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if (above < wanted && above + cnt[e] >= wanted) {
      found[0] = kShortBins - 1 - (4 * tid + e); found[1] = wanted - above; found[2] = cnt[e];
    }
    above += cnt[e];
  }
  __syncthreads();
}

// kPre: the maxima of groups of `per` vectors of a thread are counted first (per = 0: not in this launch).
template <int kVec, bool kPre>
__global__ void __launch_bounds__(kSelThreads + 64, kVec > 4 ? 1 : 2)
    select_short_kernel(const SelectParams p, int behind_static, int cs, int share, int per, int cand_cap) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int2 *list = reinterpret_cast<int2 *>(smem_raw);       // (slot, position) of the rows this CTA gathers
  __shared__ __align__(16) uint32_t hist[kShortBins];
  __shared__ uint32_t red[2][kSelWarps];
  __shared__ int tmp[4][kSelWarps];
  __shared__ int found[3];
  __shared__ unsigned long long border[kShortBorder];
  __shared__ int n_border;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int32_t ready = 0;
  if (behind_static && tid == 0) asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(ready) : "l"(p.ready) : "memory");
  const int row = (int)blockIdx.x / cs, rank = (int)blockIdx.x - row * cs;
  const int b = row / p.H_q, h = row - b * p.H_q, kvh = h / p.G, j = h - kvh * p.G;
  const float *grow = p.scores + (int64_t)row * p.row_stride;
  *reinterpret_cast<uint4 *>(&hist[4 * tid]) = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) n_border = 0;
  const int n_vec = p.E >> 2, rest = p.E & 3, n_all = n_vec + (rest != 0 ? 1 : 0);
  const int v0 = warp * kVec * 32 + lane;
  const int nu = min(kVec, max(0, (n_vec - v0 + 31) >> 5));   // the thread's full vectors
  const bool has_rest = rest != 0 && nu < kVec && v0 + nu * 32 == n_vec;
  // threads that have a score: those of the full warps, and the first ones of the last
  const int last_warp = n_all / (kVec * 32), in_last = n_all - last_warp * kVec * 32;
  const bool enough = last_warp * 32 + min(32, in_last) >= p.k_q;
  asm volatile("" ::"r"(b), "r"(kvh), "r"(j), "l"(grow), "r"(last_warp), "r"(nu));   // (worked out while the predecessor drains)
  bool waited = behind_static && __syncthreads_or(ready) != 0;   // (see copy_static_kernel and select_compact_kernel)
  if (!waited) {
    wait_for_predecessor();
    waited = true;
  }

  // ---- the row ----
  ShortRow<kVec, !kPre> r;
  r.n = 4 * nu + (has_rest ? rest : 0);
  {
    float4 x[kVec];
    const bool ok = SAGEKV_OK_INDEX(p.status, row < p.B * p.H_q && (int64_t)p.E <= p.row_stride);
#pragma unroll
    for (int u = 0; u < kVec; ++u) {
      x[u] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      if (ok && u < nu)
        asm volatile("ld.global.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(x[u].x), "=f"(x[u].y), "=f"(x[u].z), "=f"(x[u].w) : "l"(grow + 4 * (v0 + u * 32)));
      if (ok && u == nu && has_rest) {                   // the last, incomplete vector
        x[u].x = grow[4 * n_vec];
        if (rest > 1) x[u].y = grow[4 * n_vec + 1];
        if (rest > 2) x[u].z = grow[4 * n_vec + 2];
      }
    }
#pragma unroll
    for (int u = 0; u < kVec; ++u) { r.set(4 * u, x[u].x); r.set(4 * u + 1, x[u].y); r.set(4 * u + 2, x[u].z); r.set(4 * u + 3, x[u].w); }
  }
  const int slot_lo = min(p.k_q, rank * share), slot_hi = min(p.k_q, slot_lo + share);
  int32_t *idx_row = p.idx + (int64_t)row * p.k_q;
  auto min_max = [&](uint32_t mn, uint32_t mx, uint32_t &kmin, uint32_t &kmax) {   // over the CTA; holds a barrier
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) { red[0][warp] = mn; red[1][warp] = mx; }
    __syncthreads();
    kmin = __reduce_min_sync(0xffffffffu, lane < kSelWarps ? red[0][lane] : 0xffffffffu);
    kmax = __reduce_max_sync(0xffffffffu, lane < kSelWarps ? red[1][lane] : 0u);
  };
  uint32_t kmin, kmax;
  bool done = false;

  if (kPre && per > 0) {
    __shared__ SelShared sh;                             // what fast_decide works with
    sh.hist_fast[tid] = 0u;
    if (tid == 0) sh.n_border = 0;
    uint32_t gk[kVec];                                   // keys of the group maxima, each at its group's last vector
    uint32_t mn = 0xffffffffu, mx = 0u;
    {
      float m = -INFINITY;
#pragma unroll
      for (int u = 0; u < kVec; ++u) {
        m = fmaxf(fmaxf(m, fmaxf(r.score(4 * u), r.score(4 * u + 1))), fmaxf(r.score(4 * u + 2), r.score(4 * u + 3)));
        gk[u] = 0u;
        if (((u + 1) & (per - 1)) == 0) {                // (the group's first vector decides whether it has scores)
          if (4 * (u + 1 - per) < r.n) { gk[u] = score_key(m); mn = min(mn, gk[u]); mx = max(mx, gk[u]); }
          m = -INFINITY;
        }
      }
    }
    min_max(mn, mx, kmin, kmax);
    const uint32_t diff = kmax ^ kmin;
    const int shift = max(0, (diff ? 31 - __clz(diff) : 0) - 10);   // (kmax >> shift) - (kmin >> shift) < 2048
    const uint32_t base = kmin >> shift;
#pragma unroll
    for (int u = 0; u < kVec; ++u)
      if (gk[u] != 0u) atomicAdd(&hist[(gk[u] >> shift) - base], 1u);
    short_cut(hist, p.k_q, tmp[0], found);               // (there are more groups than k_q: see the launch)
    const uint32_t T0 = (base + (uint32_t)found[0]) << shift;
    const float T0f = key_to_score(T0);
    uint32_t hit[kMaskWords<kVec>];
#pragma unroll
    for (int w = 0; w < kMaskWords<kVec>; ++w) {
      hit[w] = 0u;
#pragma unroll
      for (int i = 0; i < 32 && 32 * w + i < 4 * kVec; ++i) hit[w] |= (r.score(32 * w + i) >= T0f ? 1u : 0u) << i;
      const int n = r.n - 32 * w;
      if (n < 32) hit[w] &= n > 0 ? (1u << n) - 1u : 0u;
    }
    int before[kVec];
    const int M = ordered_prefix<kVec>(hit, tmp[1], before);
    if (M <= cand_cap && M >= p.k_q) {
      SelCtx c;
      c.cs = cs; c.rank = rank; c.row = row;
      c.list = list; c.list_cap = share;
      c.cand_cap = cand_cap;
      unsigned long long *cand = reinterpret_cast<unsigned long long *>(smem_raw + (((size_t)share * sizeof(int2) + 15) & ~(size_t)15));
#pragma unroll
      for (int u = 0; u < kVec; ++u) {
        uint32_t m = (hit[u >> 3] >> (4 * (u & 7))) & 15u;
        int at = before[u];
        while (m) {
          const int pos = 4 * (v0 + u * 32) + __ffs(m) - 1;
          m &= m - 1;
          if (SAGEKV_OK_INDEX(p.status, pos < p.E && at < cand_cap))
            cand[at] = ((unsigned long long)score_key(grow[pos]) << 32) | (0xffffffffu - (uint32_t)pos);   // (an L1 hit)
          ++at;
        }
      }
      __syncthreads();
      cg::cluster_group cluster = cg::this_cluster();    // (not used: no arrival is pending)
      done = fast_decide(cluster, sh, p, c, cand, T0, kmax, M, false) == kFastDone;
    }
    if (!done) {                                         // many equal scores, or large ones side by side: from the start
      *reinterpret_cast<uint4 *>(&hist[4 * tid]) = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();
    }
  }

  if (!done) {
    // 1. the row's maximum, and the least thread maximum (of all scores, where there are too few threads)
    {
      uint32_t mx = 0u, mn = 0xffffffffu;
#pragma unroll
      for (int i = 0; i < 4 * kVec; ++i) mx = max(mx, r.key(i));
      if (enough) {
        if (mx != 0u) mn = mx;
      } else {
#pragma unroll
        for (int i = 0; i < 4 * kVec; ++i) mn = min(mn, r.key(i) - 1u);   // (no score: wraps to the largest)
        mn = mn == 0xffffffffu ? mn : mn + 1u;
      }
      min_max(mn, mx, kmin, kmax);
    }

    // 2. the bin of the k_q-th largest score
    const uint32_t diff = kmax ^ kmin;
    int shift = max(0, (diff ? 31 - __clz(diff) : 0) - 10);
    uint32_t base = kmin >> shift, cut;
    int wanted = p.k_q, in_cut;                          // the score looked for is the `wanted`-th largest of those that are counted
#pragma unroll
    for (int i = 0; i < 4 * kVec; ++i) {
      const uint32_t k = r.key(i);
      if (k >= kmin) atomicAdd(&hist[(k >> shift) - base], 1u);
    }
    while (true) {
      short_cut(hist, wanted, tmp[0], found);
      cut = base + (uint32_t)found[0]; wanted = found[1]; in_cut = found[2];
      if (in_cut == wanted || in_cut <= kShortBorder || shift == 0) break;
      // too many to rank: their next eleven bits
      const int next = max(0, shift - 11);
      *reinterpret_cast<uint4 *>(&hist[4 * tid]) = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();
#pragma unroll
      for (int i = 0; i < 4 * kVec; ++i) {
        const uint32_t k = r.key(i);
        if (k >= kmin && (k >> shift) == cut) atomicAdd(&hist[(k >> next) - (cut << (shift - next))], 1u);
      }
      base = cut << (shift - next);
      shift = next;
    }

    // 3. which scores are kept
    uint32_t kept[kMaskWords<kVec>], edge[kMaskWords<kVec>], any_edge = 0u;
#pragma unroll
    for (int w = 0; w < kMaskWords<kVec>; ++w) {
      kept[w] = edge[w] = 0u;
#pragma unroll
      for (int i = 0; i < 32 && 32 * w + i < 4 * kVec; ++i) {
        const uint32_t k = r.key(32 * w + i);
        kept[w] |= ((k >> shift) > cut ? 1u : 0u) << i;
        edge[w] |= ((k >> shift) == cut && k >= kmin ? 1u : 0u) << i;   // (what the histograms counted)
      }
      any_edge |= edge[w];
    }
    if (in_cut == wanted) {
#pragma unroll
      for (int w = 0; w < kMaskWords<kVec>; ++w) kept[w] |= edge[w];
    } else if (in_cut <= kShortBorder) {
      auto entry = [&](int i) {                          // larger: a larger score, or an equal one further ahead
        return ((unsigned long long)r.key(i) << 32) | (0xffffffffu - (uint32_t)(4 * (v0 + (i >> 2) * 32) + (i & 3)));
      };
#pragma unroll
      for (int i = 0; i < 4 * kVec; ++i)
        if ((edge[i >> 5] >> (i & 31)) & 1u) border[atomicAdd(&n_border, 1)] = entry(i);
      __syncthreads();
      if (any_edge != 0u) {
#pragma unroll
        for (int i = 0; i < 4 * kVec; ++i) {
          if ((edge[i >> 5] >> (i & 31)) & 1u) {
            const unsigned long long mine = entry(i);
            int larger = 0;
            for (int q = 0; q < in_cut; ++q) larger += border[q] > mine ? 1 : 0;
            if (larger < wanted) kept[i >> 5] |= 1u << (i & 31);
          }
        }
      }
    } else {                                             // equal scores: the first `wanted` of them
      int before[kVec];
      (void)ordered_prefix<kVec>(edge, tmp[2], before);
#pragma unroll
      for (int i = 0; i < 4 * kVec; ++i) {
        const uint32_t e = edge[i >> 5];
        if (((e >> (i & 31)) & 1u) && before[i >> 2] + __popc((e >> (i & 28)) & ((1u << (i & 3)) - 1u)) < wanted) kept[i >> 5] |= 1u << (i & 31);
      }
    }

    // 4. slots in position order; the CTA's share of them
    int before[kVec];
    (void)ordered_prefix<kVec>(kept, tmp[3], before);
#pragma unroll
    for (int u = 0; u < kVec; ++u) {
      uint32_t m = (kept[u >> 3] >> (4 * (u & 7))) & 15u;
      int slot = before[u];
      while (m) {
        const int pos = p.S + 4 * (v0 + u * 32) + __ffs(m) - 1;
        m &= m - 1;
        if (slot >= slot_lo && slot < slot_hi && SAGEKV_OK_INDEX(p.status, pos >= p.S && pos < p.S + p.E)) {
          idx_row[slot] = pos;
          list[slot - slot_lo] = make_int2(slot, pos);
        }
        ++slot;
      }
    }
    __syncthreads();
  }
  gather_rows<(kVec > 4 ? 8 : 4)>(p, b, kvh, j, cs, rank, list, slot_hi - slot_lo, behind_static, waited);
  if (behind_static) wait_for_predecessor();             // this kernel's end stands for the whole call's
  if (blockIdx.x == 0 && tid == 0 && p.d_step != nullptr) *p.d_step = 0;
}

struct ShortPlan {
  int cs, per;       // CTAs per row; see short_group
  bool beside;       // the sink, recent and last rows are copied by a kernel of their own (see launch_select_compact)
};

template <int kVec, bool kPre>
static cudaError_t launch_select_short_vec(const SelectParams &p, int n_rows, const ShortPlan &plan, cudaStream_t stream) {
  const int share = (p.k_q + plan.cs - 1) / plan.cs, cand_cap = plan.per > 0 ? list_cand_cap(p.k_q) : 0;
  const size_t smem = (((size_t)share * sizeof(int2) + 15) & ~(size_t)15) + (size_t)cand_cap * 9 + 32;
  return launch_next(select_short_kernel<kVec, kPre>, dim3((unsigned)(n_rows * plan.cs)), kSelThreads, smem, stream, 0, p, (int)plan.beside, plan.cs,
                     share, plan.per, cand_cap);
}

static cudaError_t select_short_setup() {
  const int most = kSelSmemLimit - 16 * 1024;            // (the kernels' own arrays)
  cudaError_t e = cudaFuncSetAttribute(select_short_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(select_short_kernel<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(select_short_kernel<4, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(select_short_kernel<4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(select_short_kernel<8, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(select_short_kernel<16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  return e;
}

// vectors of a thread per group of the first histogram: as many as leave twice k_q groups (0: there are too few)
static int short_group(const SelectParams &p, int vecs) {
  int per = vecs;
  while (per > 1 && (int64_t)(p.E >> 2) < 2 * (int64_t)p.k_q * per) per >>= 1;
  return (int64_t)(p.E >> 2) < 2 * (int64_t)p.k_q * per ? 0 : per;
}

// CTAs per row: without a gather one.  With one, as many as bring a CTA to every SM, of at least 16 rows; more rows than half
// the SMs: two CTAs to every SM, of at least 64 rows, where two fit.  (us per launch with 1 / 2 / 4 / 8 CTAs per row: 32 rows of 8000,
// k_q = 240, 10.8 / 7.6 / 6.9 / 8.7; 64 rows 11.3 / 7.9 / 9.1; 128 rows 12.2 / 10.9.)
static ShortPlan short_plan(const SelectParams &p, int n_sm) {
  const int n_rows = p.B * p.H_q, n_static = p.Kc != nullptr ? p.S + p.R + 1 : 0;
  ShortPlan plan = {1, 0, false};
  if (p.Kc != nullptr) {
    const int room = n_sm / n_rows;
    plan.cs = room >= 2 ? min(room, (p.k_q + 15) / 16) : (p.E <= 4 * 4 * kSelThreads ? min(2 * n_sm / n_rows, (p.k_q + 63) / 64) : 1);
    if (plan.cs < 1) plan.cs = 1;
    while (plan.cs < room && n_static > kStaticPerWarp * p.G * plan.cs * kSelWarps) ++plan.cs;   // (rather than a second kernel)
  }
  plan.beside = n_static > kStaticPerWarp * p.G * plan.cs * kSelWarps;
  if (p.E > 2 * 4 * kSelThreads) plan.per = short_group(p, p.E <= 4 * 4 * kSelThreads ? 4 : (p.E <= 8 * 4 * kSelThreads ? 8 : 16));
  // (four vectors: where not every thread maximum may be a group's of its own the direct way is the shorter one, 32 rows of 8000
  // with k_q = 1024 15.6 / 19.9; with k_q = 29 and no gather 5.7 / 5.3)
  if (p.E <= 4 * 4 * kSelThreads && plan.per < 4) plan.per = 0;
  return plan;
}

// Which rows: up to 8192 scores all (us per launch, clusters that exchange / this: 32 rows of 3963, k_q = 64, 10.0 / 5.2, k_q = 1024
// with as many sink and recent rows 24.6 / 13.2; 32 x 8184, k_q = 29, indices only, 9.6 / 5.3; 1024 x 8184, k_q = 240, 84 / 72).
// Up to 16384, where a CTA has its SM to itself (k_q = kept scores):
//  - those that clusters would need four CTAs or more for, all (512 rows x 16384, k_q = 600, 129 / 100);
//  - those for two CTAs, where this kernel copies the static rows along (128 rows x 16384, k_q = 400, 19.2 / 16.3; 512 rows, k_q = 512, 81.5 / 73.4).  With a
//    kernel of their own for these, which clusters with twice the warps may do without, a CTA's turn over 400 rows of K and V shows: 76 rows,
//    k_q = 512, 20.0 / 19.1, 128 22.7 / 23.8, 196, k_q = 400, 33.7 / 37.3; but 128 rows, k_q = 300, 17.1 / 16.8, with more static rows than kept ones,
//    k_q = 512, 25.8 / 24.4, and between one wave of these and two of such clusters, 152 rows, k_q = 400, 32.3 / 30.5 (where those need the kernel
//    too 33.6 / 35.3);
//  - those for one, two of which share an SM, up to one row per SM (k_q = 240: 32 rows 11.0 / 8.3, 128 16.8 / 15.1, 160 21.2 / 23.3, 256 25.7 /
//    32.0, 1024 82 / 107); without a gather longer (160 rows, k_q = 256, 12.8 / 12.4, 256 x 12500 13.5 / 12.8, 256 x 16384 13.4 / 14.1, 400 21.3 /
//    21.5, 1024 43.4 / 47.2);
//  - not behind very many static rows, for whose copies it leaves less room (96 rows, k_q = 256, 98328 of them 25.7 / 27.4; 64, 65552 19.7 / 19.3);
//  - with a histogram behind the rows, which saves a cluster its exchanges: 64 rows, k_q = 479, 15.2 / 13.1, but 128 21.6 / 24.6; 128 with
//    k_q = 128 13.2 / 12.5; 256 with k_q = 64 16.4 / 22.1.
// Longer ones, where a thread has 64 scores, up to two rows for three SMs, and where
// nothing has to be copied beside: 32 x 25236, k_q = 479, 12.2 / 11.2; 84 x 25236 19.5 / 16.3; but 128 x 25236 20.3 / 21.9, and with 2049
// static rows 32 x 25236, k_q = 512, 14.3 / 15.7.
constexpr int kShortManyStatic = 80000;   // static rows of a launch
static bool short_rows_apply(const SelectParams &p, int n_sm, bool sketch) {
  if (p.E <= 4 * 4 * kSelThreads) return true;
  if (p.E > kShortMaxE) return false;
  const int64_t rows = (int64_t)p.B * p.H_q;
  const ShortPlan plan = short_plan(p, n_sm);
  if (p.E > 8 * 4 * kSelThreads) return !sketch && 3 * rows <= 2 * (int64_t)n_sm && plan.per > 0 && !plan.beside;
  if (plan.beside && p.k_q <= kSelThreads && (int64_t)p.B * p.H_kv * (p.S + p.R + 1) > kShortManyStatic) return false;
  if (sketch) return 2 * rows <= n_sm || (rows <= n_sm && 4 * p.k_q <= kSelThreads);
  if (p.k_q > kSelThreads) return true;
  if (p.Kc == nullptr)
    return 2 * p.k_q > kSelThreads || (rows <= 3 * (int64_t)n_sm && !(2 * rows > 3 * (int64_t)n_sm && rows <= 2 * (int64_t)n_sm && p.E > 7 * 4 * kSelThreads));
  if (2 * p.k_q <= kSelThreads) return rows <= n_sm;
  if (!plan.beside) return true;
  if (rows <= n_sm) return 3 * rows <= 2 * (int64_t)n_sm || 4 * p.k_q <= 3 * kSelThreads || p.S + p.R >= p.k_q;
  return 10 * rows <= 13 * (int64_t)n_sm && p.S + p.R < kStaticPerWarp * p.G * 2 * kSelWarps;
}

static cudaError_t launch_select_short(const SelectParams &p, int n_sm, cudaStream_t stream) {
  const ShortPlan plan = short_plan(p, n_sm);
  const int n_rows = p.B * p.H_q;
  SelectParams pl = p;
  pl.pdl = 0;                                            // (these launches wait at their entry and release nothing early)
  if (plan.beside) {
    const cudaError_t e = launch_copy_static(pl, n_sm, stream, false);
    if (e != cudaSuccess) return e;
  }
  if (p.E <= 4 * kSelThreads) return launch_select_short_vec<1, false>(pl, n_rows, plan, stream);
  if (p.E <= 2 * 4 * kSelThreads) return launch_select_short_vec<2, false>(pl, n_rows, plan, stream);
  if (p.E <= 4 * 4 * kSelThreads)
    return plan.per > 0 ? launch_select_short_vec<4, true>(pl, n_rows, plan, stream) : launch_select_short_vec<4, false>(pl, n_rows, plan, stream);
  if (p.E <= 8 * 4 * kSelThreads) return launch_select_short_vec<8, true>(pl, n_rows, plan, stream);
  return launch_select_short_vec<16, true>(pl, n_rows, plan, stream);
}

}  // namespace sagekv
