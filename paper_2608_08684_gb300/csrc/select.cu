// Pooling of the prefix votes and exact top-k selection per unit (SnapKV's
// selection rule kept by RippleKV; retained set S_l of Eq. 4).
//
// Three kernels, one result (bit for bit): select_pool_kernel for prefixes of up
// to 131072 tokens, which also gathers the unit's kept K and V rows, and for
// longer ones select_cluster_kernel (keys in the shared memory of 8 CTAs) and
// select_kernel (keys in global scratch). The steps, for one unit (b, h):
//   1. pooled score of every prefix token (max or mean over the clipped
//      window), mapped to an order-preserving uint32 key;
//   2. radix select over the keys from the top bits finds the K-th largest key
//      tau and how many keys equal to tau are kept;
//   3. an ordered compaction writes every token with key > tau and the first
//      tokens with key == tau (lower index wins ties) in ascending order,
//      followed by the w window positions P..T-1.
// The result is bit-exact and deterministic for a given vote array.
#include <math.h>
#include <stddef.h>

#include "common.cuh"
#include "kernels.cuh"

namespace ripple {
namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kBins = 2048;
// Shared words after the histogram: scan scratch [0, 33), control [40, 48),
// per-warp exclusive counts [0, 32) and [48, 80) during the compaction.
constexpr int kCtrlWords = 128;

// Order-preserving map float -> uint32 (larger float, larger key); -0 folds to +0.
__device__ __forceinline__ uint32_t order_key(float x) {
  const uint32_t b = __float_as_uint(x + 0.0f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Exclusive block-wide prefix sum of one int per thread; *total gets the sum.
__device__ __forceinline__ int block_exclusive_scan(int x, int *warp_tot, int *total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    int t = warp_tot[lane];
    int ti = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, ti, o);
      if (lane >= o) ti += y;
    }
    warp_tot[lane] = ti - t;  // exclusive warp offsets
    if (lane == 31) warp_tot[32] = ti;
  }
  __syncthreads();
  const int res = warp_tot[wid] + incl - x;
  *total = warp_tot[32];
  __syncthreads();
  return res;
}

__global__ void __launch_bounds__(kThreads) select_kernel(LayerGeom g, const float *votes,
                                                          uint32_t *keys_global, int n_keep,
                                                          int32_t *idx, int32_t *status) {
  extern __shared__ uint32_t sm[];
  uint32_t *hist = sm;                              // [kBins]
  int *warp_tot = (int *)(sm + kBins);              // [33]
  int *ctrl = warp_tot + 40;                        // [8] control words
  uint32_t *keys = keys_global + (size_t)blockIdx.x * g.P;

  const int unit = blockIdx.x;
  const int P = g.P, K = n_keep - g.W;
  const float *v = votes + (size_t)unit * P;
  int32_t *out = idx + (size_t)unit * n_keep;
  const int tid = threadIdx.x;

  for (int j = tid; j < g.W; j += kThreads) out[K + j] = P + j;
  if (K <= 0) return;
  if (K >= P) {
    for (int t = tid; t < P; t += kThreads) out[t] = t;
    return;
  }

  // Pooling: each warp step loads 32 consecutive votes (coalesced) and the
  // lanes away from the edges take their window through shuffles.
  const int half = g.pool_kernel / 2;
  const int lane = tid & 31, wid = tid >> 5;
  const int step = 32 - 2 * half;
  for (int seg = wid * step; seg < P; seg += kWarps * step) {
    const int src = seg - half + lane;
    const bool in = src >= 0 && src < P;
    const float x = in ? v[src] : 0.f;
    float r;
    if (g.pool_type == RIPPLE_POOL_MAX) {
      r = in ? x : -INFINITY;
      const float own = r;
      for (int d = 1; d <= half; ++d) {
        r = fmaxf(r, __shfl_up_sync(0xffffffffu, own, d));
        r = fmaxf(r, __shfl_down_sync(0xffffffffu, own, d));
      }
    } else if (g.pool_type == RIPPLE_POOL_AVG) {
      // ascending positions from zero, like the definition's sum
      float s = 0.f;
      int cnt = 0;
      for (int d = -half; d <= half; ++d) {
        const float xv = d < 0 ? __shfl_up_sync(0xffffffffu, x, -d)
                               : __shfl_down_sync(0xffffffffu, x, d);
        const int pos = src + d;
        if (pos >= 0 && pos < P) {
          s = __fadd_rn(s, d == 0 ? x : xv);
          ++cnt;
        }
      }
      r = __fdiv_rn(s, (float)cnt);
    } else {
      r = x;
    }
    if (lane >= half && lane < 32 - half && src < P) keys[src] = order_key(r);
  }
  __syncthreads();

  // Radix select of the K-th largest key.
  uint32_t prefix = 0, mask = 0;
  int remaining = K;
  const int shifts[3] = {21, 10, 0};
  const int widths[3] = {11, 11, 10};
  for (int round = 0; round < 3; ++round) {
    const int shift = shifts[round];
    const uint32_t dmask = (1u << widths[round]) - 1u;
    for (int i = tid; i < kBins; i += kThreads) hist[i] = 0;
    __syncthreads();
    // Scores cluster in few bins: lanes with the same bin add once per warp.
    for (int base = 0; base < P; base += kThreads) {
      const int t = base + tid;
      const uint32_t u = t < P ? keys[t] : 0u;
      const bool hit = t < P && (u & mask) == prefix;
      const uint32_t bin = hit ? (u >> shift) & dmask : 0xffffffffu;
      const uint32_t peers = __match_any_sync(0xffffffffu, bin);
      if (hit && (threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&hist[bin], __popc(peers));
    }
    __syncthreads();
    // Thread j owns digits 2047-2j and 2046-2j (descending).
    const int d0 = kBins - 1 - 2 * tid, d1 = d0 - 1;
    const int c0 = (int)hist[d0], c1 = (int)hist[d1];
    int total;
    const int above0 = block_exclusive_scan(c0 + c1, warp_tot, &total);
    const int above1 = above0 + c0;
    if (above0 < remaining && remaining <= above0 + c0) {
      ctrl[0] = d0;
      ctrl[1] = remaining - above0;
    } else if (above1 < remaining && remaining <= above1 + c1) {
      ctrl[0] = d1;
      ctrl[1] = remaining - above1;
    }
    __syncthreads();
    prefix |= (uint32_t)ctrl[0] << shift;
    mask |= dmask << shift;
    remaining = ctrl[1];
    __syncthreads();
  }
  const uint32_t tau = prefix;
  const int take_eq = remaining;  // keys equal to tau that are kept (>= 1)

  // Ordered compaction: all keys > tau, plus the first take_eq keys == tau.
  // Each warp owns one contiguous index range: it counts, one block scan gives
  // every warp its output offsets, then it writes its range in order.
  const int per = ((P + kWarps - 1) / kWarps + 31) & ~31;
  const int r0 = min(P, wid * per), r1 = min(P, r0 + per);
  int cgt = 0, ceq = 0;
  for (int b = r0; b < r1; b += 32) {
    const int t = b + lane;
    const uint32_t u = t < r1 ? keys[t] : 0u;
    cgt += __popc(__ballot_sync(0xffffffffu, t < r1 && u > tau));
    ceq += __popc(__ballot_sync(0xffffffffu, t < r1 && u == tau));
  }
  int *wgt = warp_tot, *weq = warp_tot + 40 + 8;  // [32] each
  if (lane == 0) {
    wgt[wid] = cgt;
    weq[wid] = ceq;
  }
  __syncthreads();
  if (wid == 0) {
    int a = wgt[lane], e = weq[lane];
    int ia = a, ie = e;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int ya = __shfl_up_sync(0xffffffffu, ia, o), ye = __shfl_up_sync(0xffffffffu, ie, o);
      if (lane >= o) {
        ia += ya;
        ie += ye;
      }
    }
    wgt[lane] = ia - a;
    weq[lane] = ie - e;
  }
  __syncthreads();
  int gt_before = wgt[wid], eq_before = weq[wid];
  const uint32_t below = (1u << lane) - 1u;
  for (int b = r0; b < r1; b += 32) {
    const int t = b + lane;
    const uint32_t u = t < r1 ? keys[t] : 0u;
    const bool gt = t < r1 && u > tau, eq = t < r1 && u == tau;
    const uint32_t bg = __ballot_sync(0xffffffffu, gt), be = __ballot_sync(0xffffffffu, eq);
    const int g_rank = gt_before + __popc(bg & below);
    const int e_rank = eq_before + __popc(be & below);
    if (gt || (eq && e_rank < take_eq)) out[guard(g_rank + min(e_rank, take_eq), 1, K, status)] = t;
    gt_before += __popc(bg);
    eq_before += __popc(be);
  }
}

// ---------------------------------------------------------------------------
// The same selection spread over a cluster of kCluster CTAs per unit: CTA r
// pools and keeps keys [r S, (r + 1) S) in its shared memory; per radix round
// each CTA builds the histogram of its keys, and after a cluster barrier every
// CTA reads all the cluster's histograms through distributed shared memory and
// derives the same digit; the compaction offsets of a CTA are the counts of
// the lower-ranked CTAs. Same result as select_kernel, bit for bit.

constexpr int kCluster = 8;
constexpr int kCThreads = 512;
constexpr int kCWarps = kCThreads / 32;

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Shared::cluster address of the same shared-memory word in CTA `rank`.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, uint32_t rank) {
  uint32_t out;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(smem_u32(p)), "r"(rank));
  return out;
}
__device__ __forceinline__ uint4 ld_cluster_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ uint2 ld_cluster_v2(uint32_t addr) {
  uint2 v;
  asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_cluster_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Exclusive prefix sum of one int per thread over kCThreads threads.
__device__ __forceinline__ int cta_exclusive_scan(int x, int *warp_tot, int *total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    const int t = lane < kCWarps ? warp_tot[lane] : 0;
    int ti = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, ti, o);
      if (lane >= o) ti += y;
    }
    if (lane < kCWarps) warp_tot[lane] = ti - t;
    if (lane == 31) warp_tot[32] = ti;
  }
  __syncthreads();
  const int res = warp_tot[wid] + incl - x;
  *total = warp_tot[32];
  __syncthreads();
  return res;
}

// Layers of one launch: units per layer, and per layer the kept count and the
// index output [upl][n_keep].
struct SelTable {
  int upl;
  int n_keep[kCompressMaxLayers];
  int32_t *idx[kCompressMaxLayers];
  int32_t *status;
  // select_pool_kernel, which also copies each unit's kept rows (with gather):
  int row_bytes, gather;
  const uint8_t *k[kCompressMaxLayers];
  const uint8_t *v[kCompressMaxLayers];
  uint8_t *k_out[kCompressMaxLayers];
  uint8_t *v_out[kCompressMaxLayers];
  int cap[kCompressMaxLayers];
};

__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kCThreads)
    select_cluster_kernel(LayerGeom g, const float *votes, const __grid_constant__ SelTable tab) {
  extern __shared__ uint32_t sm[];
  uint32_t *hist2 = sm;                            // [2][kBins], one per round parity
  int *warp_tot = (int *)(sm + 2 * kBins);         // [33]
  int *ctrl = warp_tot + 40;                       // [8]
  int *cnt = ctrl + 8;                             // [2]: this CTA's (> tau, == tau) counts
  int *wgt = cnt + 8, *weq = wgt + 32;             // [32] each
  uint32_t *keys = sm + 2 * kBins + kCtrlWords;    // [S]

  const uint32_t rank = cluster_rank();
  const int unit = blockIdx.x / kCluster;  // over all layers of the launch
  const int layer = unit / tab.upl;
  const int n_keep = tab.n_keep[layer];
  const int P = g.P, K = n_keep - g.W;
  const int S = ((P + kCluster - 1) / kCluster + 31) & ~31;
  const int k0 = min(P, (int)rank * S), k1 = min(P, k0 + S);
  const float *v = votes + (size_t)unit * P;
  int32_t *out = tab.idx[layer] + (size_t)(unit % tab.upl) * n_keep;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;

  if (rank == 0)
    for (int j = tid; j < g.W; j += kCThreads) out[K + j] = P + j;
  if (K <= 0) return;
  if (K >= P) {
    for (int t = k0 + tid; t < k1; t += kCThreads) out[t] = t;
    return;
  }

  // This CTA's votes and the pooling halo, staged in shared memory with all
  // loads in flight at once (one memory latency instead of one per step).
  const int half = g.pool_kernel / 2;
  const int lo = max(0, k0 - half), hi = min(P, k1 + half);
  float *vs = reinterpret_cast<float *>(keys + S);  // [S + 2 * half]
  {
    constexpr int kU = 8;
    for (int b0 = lo; b0 < hi; b0 += kU * kCThreads) {
      float x[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int j = b0 + u * kCThreads + tid;
        x[u] = j < hi ? __ldcg(v + j) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int j = b0 + u * kCThreads + tid;
        if (j < hi) vs[j - lo] = x[u];
      }
    }
  }
  __syncthreads();
  // Pooled keys of this CTA's range (the window reads across range edges).
  const int step = 32 - 2 * half;
  for (int seg = k0 + wid * step; seg < k1; seg += kCWarps * step) {
    const int src = seg - half + lane;
    const bool in = src >= 0 && src < P;
    const float x = in ? vs[src - lo] : 0.f;
    float r;
    if (g.pool_type == RIPPLE_POOL_MAX) {
      r = in ? x : -INFINITY;
      const float own = r;
      for (int d = 1; d <= half; ++d) {
        r = fmaxf(r, __shfl_up_sync(0xffffffffu, own, d));
        r = fmaxf(r, __shfl_down_sync(0xffffffffu, own, d));
      }
    } else if (g.pool_type == RIPPLE_POOL_AVG) {
      float s = 0.f;
      int c = 0;
      for (int d = -half; d <= half; ++d) {
        const float xv = d < 0 ? __shfl_up_sync(0xffffffffu, x, -d)
                               : __shfl_down_sync(0xffffffffu, x, d);
        const int pos = src + d;
        if (pos >= 0 && pos < P) {
          s = __fadd_rn(s, d == 0 ? x : xv);
          ++c;
        }
      }
      r = __fdiv_rn(s, (float)c);
    } else {
      r = x;
    }
    if (lane >= half && lane < 32 - half && src >= k0 && src < k1)
      keys[src - k0] = order_key(r);
  }
  __syncthreads();

  // Radix select of the K-th largest key over the whole unit.
  uint32_t prefix = 0, mask = 0;
  int remaining = K;
  const int shifts[3] = {21, 10, 0};
  const int widths[3] = {11, 11, 10};
  const int n_local = k1 - k0;
  for (int round = 0; round < 3; ++round) {
    const int shift = shifts[round];
    const uint32_t dmask = (1u << widths[round]) - 1u;
    uint32_t *hist = hist2 + (round & 1) * kBins;
    for (int i = tid; i < kBins; i += kCThreads) hist[i] = 0;
    __syncthreads();
    for (int base = 0; base < n_local; base += kCThreads) {
      const int t = base + tid;
      const uint32_t u = t < n_local ? keys[t] : 0u;
      if (t < n_local && (u & mask) == prefix) atomicAdd(&hist[(u >> shift) & dmask], 1u);
    }
    cluster_sync_all();  // every CTA's histogram of this round is complete
    // Thread j sums digits 2047-4j .. 2044-4j (descending) over the cluster:
    // one 16-byte load from every CTA's histogram, all in flight together.
    int c[4] = {0, 0, 0, 0};
    const int d0 = kBins - 1 - 4 * tid;
    {
      uint4 h[kCluster];
#pragma unroll
      for (uint32_t r = 0; r < kCluster; ++r) h[r] = ld_cluster_v4(cluster_addr(hist + d0 - 3, r));
#pragma unroll
      for (uint32_t r = 0; r < kCluster; ++r) {
        c[0] += (int)h[r].w;
        c[1] += (int)h[r].z;
        c[2] += (int)h[r].y;
        c[3] += (int)h[r].x;
      }
    }
    int total;
    int above = cta_exclusive_scan(c[0] + c[1] + c[2] + c[3], warp_tot, &total);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (above < remaining && remaining <= above + c[q]) {
        ctrl[0] = d0 - q;
        ctrl[1] = remaining - above;
      }
      above += c[q];
    }
    __syncthreads();
    prefix |= (uint32_t)ctrl[0] << shift;
    mask |= dmask << shift;
    remaining = ctrl[1];
    __syncthreads();
  }
  const uint32_t tau = prefix;
  const int take_eq = remaining;

  // Ordered compaction over the cluster: counts per warp range, per CTA,
  // then offsets from the lower-ranked CTAs.
  const int per = ((n_local + kCWarps - 1) / kCWarps + 31) & ~31;
  const int r0 = min(n_local, wid * per), r1 = min(n_local, r0 + per);
  int cgt = 0, ceq = 0;
  for (int b = r0; b < r1; b += 32) {
    const int t = b + lane;
    const uint32_t u = t < r1 ? keys[t] : 0u;
    cgt += __popc(__ballot_sync(0xffffffffu, t < r1 && u > tau));
    ceq += __popc(__ballot_sync(0xffffffffu, t < r1 && u == tau));
  }
  if (lane == 0) {
    wgt[wid] = cgt;
    weq[wid] = ceq;
  }
  __syncthreads();
  if (wid == 0) {
    const int a = lane < kCWarps ? wgt[lane] : 0, e = lane < kCWarps ? weq[lane] : 0;
    int ia = a, ie = e;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int ya = __shfl_up_sync(0xffffffffu, ia, o), ye = __shfl_up_sync(0xffffffffu, ie, o);
      if (lane >= o) {
        ia += ya;
        ie += ye;
      }
    }
    if (lane < kCWarps) {
      wgt[lane] = ia - a;
      weq[lane] = ie - e;
    }
    if (lane == 31) {
      cnt[0] = ia;
      cnt[1] = ie;
    }
  }
  cluster_sync_all();  // every CTA's counts are published
  int gt_cta = 0, eq_cta = 0;
  for (uint32_t r = 0; r < rank; ++r) {
    const uint2 c = ld_cluster_v2(cluster_addr(cnt, r));
    gt_cta += (int)c.x;
    eq_cta += (int)c.y;
  }
  int gt_before = gt_cta + wgt[wid], eq_before = eq_cta + weq[wid];
  const uint32_t below = (1u << lane) - 1u;
  for (int b = r0; b < r1; b += 32) {
    const int t = b + lane;
    const uint32_t u = t < r1 ? keys[t] : 0u;
    const bool gt = t < r1 && u > tau, eq = t < r1 && u == tau;
    const uint32_t bg = __ballot_sync(0xffffffffu, gt), be = __ballot_sync(0xffffffffu, eq);
    const int g_rank = gt_before + __popc(bg & below);
    const int e_rank = eq_before + __popc(be & below);
    if (gt || (eq && e_rank < take_eq))
      out[guard(g_rank + min(e_rank, take_eq), 1, K, tab.status)] = k0 + t;
    gt_before += __popc(bg);
    eq_before += __popc(be);
  }
  cluster_sync_all();  // no CTA leaves while others may still read its memory
}

// ---------------------------------------------------------------------------
// Prefixes of up to kPoolMaxP tokens: pooling, selection and gather in one
// launch, a cluster of C CTAs (1 to 8) per unit.
//
// CTA r of a unit takes KPT consecutive tokens a thread, warp w of it KPT rows of
// 32 consecutive tokens, one token of a row per lane, so that votes are loaded
// coalesced straight into registers (a row more at either end is the pooling
// halo) and a neighbour d tokens away is one select and one shuffle. The K-th
// largest key is found by one radix round over all keys (2048 bins of a 32nd of a
// binade; only the first of a warp's run of equal digits, which pooling makes,
// adds to the histogram); the keys of its bucket, if at most kPoolCand, are then
// copied to every CTA of the unit, which finishes on them alone, without the
// cluster: up to kPoolRank of them by counting, more by two rounds of 9 bits.
// Larger buckets (many equal votes) take further rounds over all keys. Kept
// tokens go to a list in shared memory, from which the positions are written and
// the rows gathered (or the gather kernel copies them, gather_apart).
//
// Bound: latency (barriers, votes from L2) for few units, HBM of the gather for
// many. One layer of 32 units, 32736 tokens, 1024 kept, takes 16.7 us
// (17.8 with 8 bins a binade, where more atomics meet in a bin and its keys
// take two more rounds); three 11-bit rounds over 8-CTA clusters, every CTA
// reading all the histograms, and a gather kernel took 41 us, and 256 units of
// 5991 tokens 98 us against 35.
constexpr int kPoolThreads = 512;
constexpr int kPoolMaxCta = 8;                       // CTAs per unit, at most
constexpr int kPoolMaxP = kPoolMaxCta * kPoolThreads * 32;
constexpr int kPoolCand = 2048;
constexpr int kPoolRank = 192;                       // bucket keys ranked directly
constexpr int kPoolBin0 = (0x80000000u >> 18) + (72 << 5);  // key >> 18 of 2^-55: bin 0

struct PoolSmem {
  alignas(16) uint32_t hist[2][kBins];  // one per round parity; read 16 bytes at a time
  uint32_t cand[kPoolCand];     // this CTA's bucket keys
  uint32_t all[kPoolCand];      // the unit's bucket keys
  int n_cand;                   // this CTA's
  alignas(8) int cnt[2];        // this CTA's kept keys: above tau, equal to tau; read as a pair
  int wsum[2][32];
  int wgt[32], weq[32];
  int digit[2][3];              // per round parity: digit, remaining, bucket keys
  uint32_t tau[2];              // the threshold of a small bucket and its keys kept
};
static_assert(offsetof(PoolSmem, cnt) % 8 == 0 && offsetof(PoolSmem, hist) % 16 == 0 &&
                  sizeof(PoolSmem) % 16 == 0,
              "vector reads of shared memory");

// kCols bins of a histogram downwards from `top`, in CTA r of the cluster.
template <int kCols>
__device__ __forceinline__ void load_bins(const uint32_t *top, uint32_t r, int n_cta,
                                          int (&c)[kCols]) {
  const uint32_t *p = top - (kCols - 1);
  if constexpr (kCols == 4) {
    const uint4 h = n_cta > 1 ? ld_cluster_v4(cluster_addr(p, r))
                              : *reinterpret_cast<const uint4 *>(p);
    c[0] = (int)h.w;
    c[1] = (int)h.z;
    c[2] = (int)h.y;
    c[3] = (int)h.x;
  } else {
    static_assert(kCols == 2, "bins per thread");
    const uint2 h = n_cta > 1 ? ld_cluster_v2(cluster_addr(p, r))
                              : *reinterpret_cast<const uint2 *>(p);
    c[0] = (int)h.y;
    c[1] = (int)h.x;
  }
}

// The digit of the K-th largest (`remaining`-th) key from 2048 bin counts, kCols
// per thread in descending order (c[q]: bin 2047 - kCols tid - q). Two barriers.
template <int kCols>
__device__ __forceinline__ void find_digit(const int (&c)[kCols], int &remaining, int par,
                                           PoolSmem &s, int &digit, int &bucket) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int sum = 0;
#pragma unroll
  for (int q = 0; q < kCols; ++q) sum += c[q];
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s.wsum[par][wid] = incl;
  __syncthreads();
  int before = lane < wid ? s.wsum[par][lane] : 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
  int above = before + incl - sum;
#pragma unroll
  for (int q = 0; q < kCols; ++q) {
    if (above < remaining && remaining <= above + c[q]) {
      s.digit[par][0] = kBins - 1 - kCols * tid - q;
      s.digit[par][1] = remaining - above;
      s.digit[par][2] = c[q];
    }
    above += c[q];
  }
  __syncthreads();
  digit = s.digit[par][0];
  remaining = s.digit[par][1];
  bucket = s.digit[par][2];
}

// The value d tokens further on (d > 0) or back (d < 0) of a row `cur` between
// its neighbour rows; |d| <= 31.
__device__ __forceinline__ float ahead(float cur, float next, int d, int lane) {
  return __shfl_sync(0xffffffffu, lane < d ? next : cur, lane + d);
}
__device__ __forceinline__ float behind(float prev, float cur, int d, int lane) {
  return __shfl_sync(0xffffffffu, lane >= 32 - d ? prev : cur, lane - d);
}

template <int KPT, int kThr>
__global__ void __launch_bounds__(kThr, 1024 / kThr)
    select_pool_kernel(LayerGeom g, const float *votes, const __grid_constant__ SelTable tab,
                       int n_cta) {
  extern __shared__ __align__(16) uint8_t pool_sm[];
  PoolSmem &s = *reinterpret_cast<PoolSmem *>(pool_sm);
  int *list = reinterpret_cast<int *>(pool_sm + sizeof(PoolSmem));  // kept tokens of this CTA
  constexpr int kCols = kBins / kThr;  // histogram bins of a thread
  constexpr int kCtaTokens = kThr * KPT;
  const int rank = n_cta > 1 ? (int)cluster_rank() : 0;
  const int unit = blockIdx.x / n_cta;  // over all layers of the launch
  const int layer = unit / tab.upl;
  const int n_keep = tab.n_keep[layer];
  const int P = g.P, K = n_keep - g.W;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int t0 = rank * kCtaTokens;                 // this CTA's first token
  int first = 0, kept = 0;                          // its rows of the compact cache
  pdl_wait();  // the votes

  if (K <= 0 || K >= P) {
    // window only, or every token: this CTA's share of the tokens in order
    if (K > 0) {
      first = min(t0, P);
      kept = min(P, t0 + kCtaTokens) - first;
      for (int i = tid; i < kept; i += kThr) list[i] = first + i;
    }
  } else {
    // ---------------- pooled keys
    const int w0 = t0 + wid * (KPT * 32);           // this warp's first token
    const float *v = votes + (size_t)unit * P;
    const float fill = g.pool_type == RIPPLE_POOL_MAX ? -INFINITY : 0.f;
    float x[KPT + 2];  // rows -1 .. KPT
#pragma unroll
    for (int i = 0; i < KPT + 2; ++i) {
      const int j = w0 + (i - 1) * 32 + lane;
      x[i] = j >= 0 && j < P ? __ldcg(v + j) : fill;
    }
    for (int i = tid; i < kBins; i += kThr) s.hist[0][i] = 0;
    const int half = g.pool_kernel / 2;
    if (g.pool_type == RIPPLE_POOL_MAX && half > 0) {
      // x[j] = max of the width tokens from j on, width the largest power of
      // two within the window; the window is two of those runs
      int width = 1;
      for (; 2 * width <= g.pool_kernel; width *= 2) {
#pragma unroll
        for (int i = 0; i < KPT + 2; ++i)
          x[i] = fmaxf(x[i], ahead(x[i], i < KPT + 1 ? x[i + 1] : fill, width, lane));
      }
      const int b = width - 1 - half;
#pragma unroll
      for (int i = KPT; i >= 1; --i)
        x[i] = fmaxf(behind(x[i - 1], x[i], half, lane), behind(x[i - 1], x[i], b, lane));
    } else if (g.pool_type == RIPPLE_POOL_AVG) {
      // ascending positions from zero, like the definition's sum (positions
      // outside the prefix add nothing)
      float prev = x[0];
#pragma unroll
      for (int i = 1; i <= KPT; ++i) {
        const float cur = x[i];
        float sum = 0.f;
        for (int d = half; d > 0; --d) sum = __fadd_rn(sum, behind(prev, cur, d, lane));
        sum = __fadd_rn(sum, cur);
        for (int d = 1; d <= half; ++d) sum = __fadd_rn(sum, ahead(cur, x[i + 1], d, lane));
        const int j = w0 + (i - 1) * 32 + lane;
        const int n = max(1, min(P - 1, j + half) - max(0, j - half) + 1);
        x[i] = __fdiv_rn(sum, (float)n);
        prev = cur;
      }
    }
    uint32_t key[KPT];
#pragma unroll
    for (int i = 0; i < KPT; ++i) key[i] = order_key(x[i + 1]);
    const int live = P - w0 - lane;  // key[i] is a token's if 32 i < live

    // ---------------- the K-th largest key
    // First round: 64 binades of 32 bins, 2^-55 up to 2^9 (votes are sums of at
    // most 256 probabilities); further rounds over the 18 bits below. Keys
    // beyond (smaller, zero, negative or larger) count in the lowest and the
    // highest bin; if the threshold falls into one of those, the search starts
    // over on all 32 bits.
    uint32_t prefix = 0, mask = 0;
    int remaining = K;
    bool full = false;
    auto shift_of = [&](int level) { return level == 2 ? 0 : full ? (level == 0 ? 21 : 10) : 9; };
    auto dmask_of = [&](int level) { return !full ? 511u : level == 2 ? 1023u : 2047u; };
    __syncthreads();  // the first histogram is clear
    for (int it = 0, level = 0; level < 3; ++it, ++level) {
      uint32_t *hist = s.hist[it & 1];
      const bool first = level == 0 && !full;
      const int shift = first ? 18 : shift_of(level), bin0 = first ? kPoolBin0 : 0;
      const uint32_t dmask = first ? ~0u : dmask_of(level);
#pragma unroll
      for (int i = 0; i < KPT; ++i) {
        const bool in = 32 * i < live && (key[i] & mask) == prefix;
        uint32_t d = min(max((int)(key[i] >> shift & dmask) - bin0, 0), kBins - 1);
        // the first lane of a run of equal digits adds the run's length
        if (!in) d = 0xffffffffu;
        const uint32_t up = __shfl_up_sync(0xffffffffu, d, 1);
        const bool head = lane == 0 || up != d;
        const uint32_t heads = __ballot_sync(0xffffffffu, head);
        if (head && in) {
          const uint32_t later = lane == 31 ? 0u : heads >> (lane + 1);
          atomicAdd(&hist[d], (uint32_t)(later ? __ffs(later) : 32 - lane));
        }
      }
      const int d0 = kBins - 1 - kCols * tid;  // this thread's bins, down from d0
      int c[kCols] = {};
      if (n_cta > 1)
        cluster_sync_all();  // every CTA's histogram of this round is complete
      else
        __syncthreads();
      for (int r = 0; r < n_cta; ++r) {
        int h[kCols];
        load_bins(hist + d0, r, n_cta, h);
#pragma unroll
        for (int q = 0; q < kCols; ++q) c[q] += h[q];
      }
      // the other histogram, for the next round (its readers have passed this
      // round's barrier)
      for (int i = tid; i < kBins; i += kThr) s.hist[(it & 1) ^ 1][i] = 0;
      if (tid == 0) s.n_cand = 0;
      int digit, bucket;
      find_digit(c, remaining, it & 1, s, digit, bucket);
      if (first) {
        if (digit == 0 || digit == kBins - 1) {
          full = true;
          remaining = K;
          level = -1;
          continue;
        }
        prefix = (uint32_t)(digit + kPoolBin0) << 18;
        mask = ~0u << 18;
      } else {
        prefix |= (uint32_t)digit << shift_of(level);
        mask |= dmask_of(level) << shift_of(level);
      }
      if (level == 2 || bucket > kPoolCand) continue;
      // ---------------- the bucket's keys, to every CTA of the unit
#pragma unroll
      for (int i = 0; i < KPT; ++i) {
        const bool in = 32 * i < live && (key[i] & mask) == prefix;
        const uint32_t m = __ballot_sync(0xffffffffu, in);
        if (m == 0) continue;
        int at = 0;
        if (lane == 0) at = atomicAdd(&s.n_cand, __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
        if (in) s.cand[at] = key[i];
      }
      const uint32_t *all = s.cand;
      if (n_cta > 1) {
        cluster_sync_all();
        int off = 0;
        for (int r = 0; r < n_cta; ++r) {
          const int n = (int)ld_cluster_u32(cluster_addr(&s.n_cand, r));
          for (int i = tid; i < n; i += kThr)
            s.all[off + i] = ld_cluster_u32(cluster_addr(&s.cand[i], r));
          off += n;
        }
        all = s.all;
      }
      __syncthreads();
      if (bucket <= kPoolRank) {
        // few: each of them counts the keys above and equal to it, and the one
        // with remaining - 1 above and at least remaining above or equal is tau
        if (tid < bucket) {
          const uint32_t u = all[tid];
          int above = 0, same = 0;
          for (int i = 0; i < bucket; ++i) {
            const uint32_t y = all[i];
            above += y > u;
            same += y == u;
          }
          if (above < remaining && remaining <= above + same) {
            s.tau[0] = u;
            s.tau[1] = (uint32_t)(remaining - above);
          }
        }
        __syncthreads();
        prefix = s.tau[0];
        remaining = (int)s.tau[1];
        break;
      }
      // else the remaining rounds on those keys alone
      for (++it, ++level; level < 3; ++it, ++level) {
        uint32_t *h2 = s.hist[it & 1];
        const int sh = shift_of(level);
        const uint32_t dm = dmask_of(level);
        for (int i = tid; i < bucket; i += kThr) {
          const uint32_t u = all[i];
          if ((u & mask) == prefix) atomicAdd(&h2[u >> sh & dm], 1u);
        }
        __syncthreads();
        int cc[kCols];
        load_bins(h2 + d0, 0, 1, cc);
        for (int i = tid; i < kBins; i += kThr) s.hist[(it & 1) ^ 1][i] = 0;
        int n_eq;
        find_digit(cc, remaining, it & 1, s, digit, n_eq);
        prefix |= (uint32_t)digit << sh;
        mask |= dm << sh;
      }
    }
    const uint32_t tau = prefix;
    const int take_eq = remaining;  // keys equal to tau that are kept (>= 1)

    // ---------------- ordered compaction into the list
    int cgt = 0, ceq = 0;
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
      cgt += __popc(__ballot_sync(0xffffffffu, 32 * i < live && key[i] > tau));
      ceq += __popc(__ballot_sync(0xffffffffu, 32 * i < live && key[i] == tau));
    }
    if (lane == 0) {
      s.wgt[wid] = cgt;
      s.weq[wid] = ceq;
    }
    __syncthreads();
    int gt = lane < kThr / 32 ? s.wgt[lane] : 0, eq = lane < kThr / 32 ? s.weq[lane] : 0;
    int gt_w = lane < wid ? gt : 0, eq_w = lane < wid ? eq : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      gt += __shfl_xor_sync(0xffffffffu, gt, o);
      eq += __shfl_xor_sync(0xffffffffu, eq, o);
      gt_w += __shfl_xor_sync(0xffffffffu, gt_w, o);
      eq_w += __shfl_xor_sync(0xffffffffu, eq_w, o);
    }
    int gt_c = 0, eq_c = 0;  // of the lower-ranked CTAs
    if (n_cta > 1) {
      if (tid == 0) {
        s.cnt[0] = gt;
        s.cnt[1] = eq;
      }
      cluster_sync_all();  // every CTA's counts are published
      for (int r = 0; r < rank; ++r) {
        const uint2 c = ld_cluster_v2(cluster_addr(s.cnt, r));
        gt_c += (int)c.x;
        eq_c += (int)c.y;
      }
      cluster_arrive();  // this CTA reads no other's shared memory any more
    }
    first = gt_c + min(eq_c, take_eq);
    kept = gt_c + gt + min(eq_c + eq, take_eq) - first;
    int gt_before = gt_c + gt_w, eq_before = eq_c + eq_w;
    const uint32_t below = (1u << lane) - 1u;
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
      const bool is_gt = 32 * i < live && key[i] > tau, is_eq = 32 * i < live && key[i] == tau;
      const uint32_t bg = __ballot_sync(0xffffffffu, is_gt);
      const uint32_t be = __ballot_sync(0xffffffffu, is_eq);
      if ((bg | be) == 0) continue;
      const int g_rank = gt_before + __popc(bg & below), e_rank = eq_before + __popc(be & below);
      if (is_gt || (is_eq && e_rank < take_eq))
        list[guard(g_rank + min(e_rank, take_eq) - first, 1, kCtaTokens, tab.status)] =
            w0 + i * 32 + lane;
      gt_before += __popc(bg);
      eq_before += __popc(be);
    }
  }

  // ---------------- positions and rows; the last CTA has the window as well
  const int window = rank == n_cta - 1 ? g.W : 0;
  if (window > 0) {
    if (kept == 0) first = max(K, 0);
    for (int i = tid; i < window; i += kThr) list[kept + i] = P + i;
  }
  const int rows = kept + window;
  __syncthreads();
  const int local = unit % tab.upl;
  int32_t *out = tab.idx[layer] + (size_t)local * n_keep + first;
  for (int i = tid; i < rows; i += kThr) out[i] = list[i];
  if (tab.gather) {
    // row_bytes / 16 consecutive threads copy one row 16 bytes each, four rows a
    // thread in flight
    const int rb = tab.row_bytes, lpr = rb >> 4, rpp = kThr / lpr;
    const int r_in = tid / lpr, c16 = (tid % lpr) * 16;
    const uint8_t *kin = tab.k[layer] + (size_t)local * g.T * rb;
    const uint8_t *vin = tab.v[layer] + (size_t)local * g.T * rb;
    uint8_t *kout = tab.k_out[layer] + ((size_t)local * tab.cap[layer] + first) * rb;
    uint8_t *vout = tab.v_out[layer] + ((size_t)local * tab.cap[layer] + first) * rb;
    for (int r0 = 0; r0 < rows; r0 += 4 * rpp) {
      uint4 xk[4], xv[4];
  #pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = r0 + u * rpp + r_in;
        if (r < rows) {
          const long long t = guard(list[r], 1, g.T, tab.status);
          xk[u] = __ldcs(reinterpret_cast<const uint4 *>(kin + t * rb + c16));
          xv[u] = __ldcs(reinterpret_cast<const uint4 *>(vin + t * rb + c16));
        }
      }
  #pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = r0 + u * rpp + r_in;
        if (r < rows) {
          *reinterpret_cast<uint4 *>(kout + (size_t)r * rb + c16) = xk[u];
          *reinterpret_cast<uint4 *>(vout + (size_t)r * rb + c16) = xv[u];
        }
      }
    }
  }
  // no CTA leaves while others may still read its shared memory
  if (n_cta > 1 && K > 0 && K < P) cluster_wait();
}

}  // namespace

namespace {

// Prefixes beyond kPoolMaxP: 8-CTA clusters with their keys in shared memory, or
// one CTA per unit with its keys in global scratch.
cudaError_t select_long(const LayerGeom &g, int n_layers, const float *votes, const CompressWs &ws,
                        const int *n_keep, int32_t *const *idx, int32_t *status,
                        cudaStream_t st) {
  const int per_cta = ((g.P + kCluster - 1) / kCluster + 31) & ~31;
  if (g.P <= kSelectClusterMaxP) {
    SelTable tab;
    tab.upl = g.units;
    tab.status = status;
    for (int l = 0; l < n_layers; ++l) {
      tab.n_keep[l] = n_keep[l];
      tab.idx[l] = idx[l];
    }
    // histograms, control words, keys, staged votes (with the pooling halo)
    const size_t smem = sizeof(uint32_t) * (2 * kBins + kCtrlWords + 2 * per_cta + 32);
    cudaError_t e = cudaFuncSetAttribute(select_cluster_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    select_cluster_kernel<<<g.units * n_layers * kCluster, kCThreads, smem, st>>>(g, votes, tab);
    count_launches(1);
    return cudaGetLastError();
  }
  // Very long prefixes: one CTA per unit, layer by layer.
  const size_t smem = sizeof(uint32_t) * (kBins + kCtrlWords);
  for (int l = 0; l < n_layers; ++l) {
    select_kernel<<<g.units, kThreads, smem, st>>>(g, votes + (size_t)l * g.units * g.P, ws.keys,
                                                   n_keep[l], idx[l], status);
    count_launches(1);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// The CTAs of a unit: `threads` threads of `keys` keys each.
struct PoolShape {
  int keys, threads, n_cta;
};

// Shapes of the selecting CTAs. While 16 keys a thread make at most one wave of
// two CTAs per SM: 16, or 8 where they fill the CTA (P <= 4096) or where 16 leave
// three quarters of the SMs idle (one layer of 32 units and 32736 tokens, 8 / 16 /
// 32 keys: 21.6 / 16.6 / 23.6 us; 8 units of 8160 tokens, with scoring, 37.1 / 40.0 /
// 47.0). With more CTAs than that the waves count, and 32 keys a thread, in CTAs
// of 512 threads or one of 1024, make fewer of them; where many rows are kept,
// though, their copies count, which more and smaller CTAs overlap better. Keys
// and values a unit keeps, us with 16 x 512 / 32 x 512 / 32 x 1024 (one layer, bf16,
// d 128 or 64):
//   8968 tokens, 256 units    128 KB 35 / 27 / 46, 256 KB 43 / 37 / 60, 512 KB 65 / 69 / 87
//   16968 tokens, 256 units    64 KB 46 / 46 / 42, 256 KB 57 / 64 / 58, 512 KB 77 / 99 / 88
//   16968 tokens, 1024 units   64 KB 159 / 162 / 147, 256 KB 204 / 228 / 209
//   23968 tokens, 256 units   128 KB 50 / 50 / 47, 256 KB 58 / 64 / 62, 512 KB 77 / 92 / 88
//   32736 tokens, 128 units   256 KB 40 / 32 / 30, 512 KB 49 / 42 / 42
//   32736 tokens, 256 units   128 KB 60 / 50 / 49, 256 KB 70 / 70 / 68, 512 KB 85 / 91 / 90
//   32736 tokens, 1024 units (with scoring) 750 KB 2540 / 2491 / 2512
// Beyond 32768 tokens 32 x 512 is left; beyond 65536, where 16 x 512 are more than 8
// CTAs, 16 x 1024 while all units' clusters are resident, one CTA an SM: 4 units of
// 80000 tokens, 20000 kept, 19 us against 29 with 32 x 512 (16 units of 100000,
// whose 7-CTA clusters no longer fit at once, 34 against 28).
PoolShape pool_shape(const LayerGeom &g, int n_layers, const int *n_keep) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int P = g.P;
  auto ctas = [&](int tokens) { return P > tokens ? (P + tokens - 1) / tokens : 1; };
  auto shape = [&](int keys, int threads) {
    return PoolShape{keys, threads, ctas(keys * threads)};
  };
  const long long units = (long long)g.units * n_layers;
  const int c16 = ctas(16 * kPoolThreads);
  if (P <= 8 * kPoolThreads ||
      (ctas(8 * kPoolThreads) <= kPoolMaxCta && units * c16 * 4 <= sms))
    return shape(8, kPoolThreads);
  if (c16 > kPoolMaxCta)
    return units * ctas(32 * kPoolThreads) * 3 <= 2LL * sms ? shape(16, 2 * kPoolThreads)
                                                            : shape(32, kPoolThreads);
  if (P <= 16 * kPoolThreads || units * c16 <= 2LL * sms) return shape(16, kPoolThreads);
  long long rows = 0;
  for (int l = 0; l < n_layers; ++l) rows += n_keep[l];
  const long long kb =  // keys and values a unit keeps, on average
      rows * 2 * g.D * (g.dtype == RIPPLE_F32 ? 4 : 2) / n_layers >> 10;
  if (P > 64 * kPoolThreads) return shape(32, kPoolThreads);
  if (P <= 32 * kPoolThreads) return shape(kb < 384 ? 32 : 16, kPoolThreads);
  if (kb < 256 || (units <= sms && P > 48 * kPoolThreads && kb < 2048))
    return shape(32, 2 * kPoolThreads);
  return shape(P > 48 * kPoolThreads && (kb < 512 || units >= 512) ? 32 : 16, kPoolThreads);
}

// Whether the rows are copied by the gather kernel instead of the CTAs that
// selected them: where few CTAs would copy many rows each. A CTA copies about 64
// GB/s, and the launch costs 4 us, which pay at 256 KB of keys and values a CTA
// while few CTAs run; the more CTAs, the nearer they are to HBM's rate by
// themselves (where every token is kept a CTA does nothing else, and the line lies
// lower). Measured, rows copied by the selecting CTAs / by the gather kernel
// (bf16, d 128): 1 CTA of 256 KB 12.4 / 12.7 us, of 512 KB 18.0 / 13.7; 32 of 512
// KB 18.4 / 13.1 to 20.3 / 17.5; 64 of 512 KB 25.9 / 26.0, of 1 MB 39.9 / 36.7; 128
// of 1 MB 59.4 / 63.0, of 1.5 MB 144 / 102; 256 of 1 MB 98 / 101, of 2 MB 184 / 177;
// one unit of 100000 tokens, all kept, 176 / 25, 32 of 8192, all kept, 59.6 / 49.4.
bool gather_apart(const LayerGeom &g, int n_layers, const int *n_keep, const PoolShape &sh) {
  const int row_bytes = g.D * (g.dtype == RIPPLE_F32 ? 4 : 2);
  int most = 0;
  for (int l = 0; l < n_layers; ++l) most = n_keep[l] > most ? n_keep[l] : most;
  const long long ctas = (long long)g.units * n_layers * sh.n_cta;
  // of the rows of a unit, the share of a CTA that is full of tokens
  const int tokens = sh.keys * sh.threads < g.P ? sh.keys * sh.threads : g.P;
  const long long bytes = g.P > 0 ? 2LL * row_bytes * most * tokens / g.P : 0;
  const long long most_kb = most == g.T ? 960 : 1536;
  const long long line_kb = 256 + 8 * ctas < most_kb ? 256 + 8 * ctas : most_kb;
  return bytes >= line_kb * 1024;
}

template <int KPT, int kThr>
cudaError_t launch_pool(const LayerGeom &g, int n_units, const float *votes, const SelTable &tab,
                        int n_cta, cudaStream_t st) {
  const size_t smem = sizeof(PoolSmem) + sizeof(int) * (kThr * KPT + 64);
  cudaError_t e = cudaFuncSetAttribute(select_pool_kernel<KPT, kThr>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_units * n_cta);
  cfg.blockDim = dim3(kThr);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = n_cta;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  e = cudaLaunchKernelEx(&cfg, select_pool_kernel<KPT, kThr>, g, votes, tab, n_cta);
  count_launches(1);
  return e;
}

}  // namespace

cudaError_t launch_select(const LayerGeom &g, int n_layers, const float *votes,
                          const CompressWs &ws, const int *n_keep, int32_t *const *idx,
                          int32_t *status, cudaStream_t st, const GatherArgs &gather) {
  if (n_layers < 1 || n_layers > kCompressMaxLayers) return cudaErrorInvalidValue;
  const int n_units = g.units * n_layers;
  cudaError_t e;
  if (g.P <= kPoolMaxP) {
    SelTable tab;
    tab.upl = g.units;
    tab.status = status;
    tab.row_bytes = g.D * (g.dtype == RIPPLE_F32 ? 4 : 2);
    for (int l = 0; l < n_layers; ++l) {
      tab.n_keep[l] = n_keep[l];
      tab.idx[l] = idx[l];
      tab.k[l] = (const uint8_t *)gather.k[l];
      tab.v[l] = (const uint8_t *)gather.v[l];
      tab.k_out[l] = (uint8_t *)gather.k_out[l];
      tab.v_out[l] = (uint8_t *)gather.v_out[l];
      tab.cap[l] = gather.cap[l];
    }
    const PoolShape sh = pool_shape(g, n_layers, n_keep);
    tab.gather = !gather_apart(g, n_layers, n_keep, sh);
    e = sh.keys == 8    ? launch_pool<8, kPoolThreads>(g, n_units, votes, tab, sh.n_cta, st)
        : sh.keys == 16 && sh.threads == kPoolThreads
            ? launch_pool<16, kPoolThreads>(g, n_units, votes, tab, sh.n_cta, st)
        : sh.keys == 16 ? launch_pool<16, 2 * kPoolThreads>(g, n_units, votes, tab, sh.n_cta, st)
        : sh.threads == kPoolThreads
            ? launch_pool<32, kPoolThreads>(g, n_units, votes, tab, sh.n_cta, st)
            : launch_pool<32, 2 * kPoolThreads>(g, n_units, votes, tab, sh.n_cta, st);
    if (tab.gather) return e;
  } else {
    e = select_long(g, n_layers, votes, ws, n_keep, idx, status, st);
  }
  if (e != cudaSuccess) return e;
  return launch_gather(g, n_layers, gather.k, gather.v, (const int32_t *const *)idx, n_keep,
                       gather.k_out, gather.v_out, gather.cap, status, st);
}

}  // namespace ripple
