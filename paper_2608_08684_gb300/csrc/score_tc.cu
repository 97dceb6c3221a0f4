// Observation-window token scoring on the 5th-generation tensor cores
// (tcgen05, accumulators in TMEM), bf16 keys and queries, d = 64 or 128, 129 to
// 256 window rows G * w (padded to 256). SnapKV's rule as RippleKV keeps it (Sec. 4.4, last
// paragraph): logits x = scale * q.k of the window rows against every key,
// causal inside the window, softmax per row over all visible keys, vote of a
// prefix key = sum over rows of its probability.
//
// One launch for all the layers of a call (a unit is a (layer, b, h); each
// layer's keys and queries come through its own tensor maps and its votes go
// to its slot of the vote array), one persistent CTA per SM, co-resident
// (cooperative launch). A unit is cut into items of `tpi` key tiles; item i belongs
// to CTA i mod grid, so every unit is spread over many CTAs that work on it at
// the same time. Each CTA runs its items in the order
//     P1(a0) P1(a1) P2(a0) P1(a2) P2(a1) ...
//   pass 1 of an item: per window row, (max, sum of exp) over the item's key
//     tiles -> partial[unit][item][row] (the publisher warp combines the two
//     epilogue warpgroups' statistics); it counts the unit's finished items
//     and the last one merges them into
//     lognorm[unit][row] = max + log2(sum) and raises ready[unit];
//   pass 2 of an item: per prefix key, vote = sum over rows of
//     exp2(x * scale * log2e - lognorm[row]), once ready[unit] is up.
// An item's keys are read again one item later, so the second read is served
// from L2 (about two items per SM are in flight). A pass-2 wait only depends
// on first passes of strictly earlier units as long as a unit has at most
// twice as many items as there are CTAs, so with every CTA resident the
// schedule cannot deadlock.
//
// Warp roles (352 threads): warp 0 = TMA producers (keys, queries), warp 1 = MMA issuer and
// TMEM owner, warps 2-9 = two epilogue warpgroups taking alternate key tiles,
// warp 10 = publisher of pass-1 results. Pass 1 computes D[row][key]
// (A = window queries, B = key tile); pass 2 computes D[key][row] (A = key
// tile, B = window queries), so each epilogue thread owns one row (pass 1) or
// one key (pass 2) and every reduction is thread-local.
// Every wait is bounded: on timeout the CTA raises RIPPLE_ETIMEOUT, all roles
// leave their loops, and TMEM is released.
#include <cuda.h>
#include <math.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"
#include "tc_ptx.cuh"

namespace ripple {
namespace {

constexpr int kTile = 128;                      // keys per tile
constexpr int kHalfBytes = kTile * 64 * 2;      // 64 bf16 columns of 128 rows: 16 KB
constexpr int kThreads = 352;
constexpr int kPubSlots = 2;
// A unit is cut into items of 8 tiles (up to 64 tiles) or 16, but at most 16
// items: more partial statistics take the one publisher that merges them too
// long, and fewer items leave small calls on few SMs. A function of the layer's
// shape alone, so that one layer's call and a multi-layer call merge the same
// statistics. Measured with items of 4 / 8 / 16 / 32 / 64 tiles, us a call:
//   64 tiles, one layer of 8 units     40 /   46 /   63 /   96 /  161
//   64 tiles, 32 such layers          335 /  312 /  296 /  319 /  316
//   65 tiles, one layer of 8 units     40 /   48 /   58 /   75 /   97
//   65 tiles, 32 such layers          386 /  370 /  325 /  343 /  350
//   128 tiles, one layer of 8 units    54 /   48 /   63 /   96 /  162
//   128 tiles, 16 such layers         379 /  302 /  288 /  312 /  312
//   1024 tiles, 16 such layers             3546 / 2188 / 2024 / 2011
// Smaller items gain a single layer and cost many layers, which decide from 65
// tiles on.
// Prompts of more than 256 tiles can take other numbers where those fill the SMs
// better in a layer's units (items_per_unit).
constexpr int kTilesPerItem = 16, kTilesPerItemShort = 8;
constexpr int kShortTiles = 64;
constexpr int kMaxItems = 16;
constexpr int kTilesPerItemLong = 64;


// ------------------------------------------------------------ work list

struct TcParams {
  int units, upl, T, P, W, R;  // units of all scored layers, units per layer, window rows
  int n_tiles1, n_tiles2;  // key tiles of pass 1 (all keys) and pass 2 (prefix keys)
  int tpi, n_ch;           // key tiles per item, items per unit
  int total_items;
  float scale2;
  float2 *partial;  // [units][n_ch][R] (max, sum) per item and row, log2 domain
  float *lognorm;   // [units][R]
  float *votes;     // [n_layers][upl][P]: unit u's votes at layer_of[u / upl]
  int layer_of[kCompressMaxLayers];  // the layer (votes slot) of each scored layer
  int n_slots;                       // layers (votes slots) of the votes array
  int *ctrl;        // [u] items of unit u published; [units + u] row statistics ready
  int32_t *status;
  long long wait_cycles;  // bound of the in-kernel waits
};

struct ItemRef {
  int unit, chunk;
};

// The k-th item of this CTA.
__device__ __forceinline__ ItemRef item_of(const TcParams &p, int k) {
  const int i = (int)blockIdx.x + k * (int)gridDim.x;
  return {i / p.n_ch, i % p.n_ch};
}

__device__ __forceinline__ int items_of_cta(const TcParams &p) {
  const int b = (int)blockIdx.x;
  return b < p.total_items ? (p.total_items - 1 - b) / (int)gridDim.x + 1 : 0;
}

__device__ __forceinline__ void tiles_of(const TcParams &p, const ItemRef &it, int pass, int &t0,
                                         int &t1) {
  t0 = it.chunk * p.tpi;
  t1 = min(pass == 1 ? p.n_tiles1 : p.n_tiles2, t0 + p.tpi);
}

// ------------------------------------------------------------ shared memory

// 256 window rows (fewer are padded with zero rows, which count for nothing),
// in two halves of 128 for pass 1. D: head dims.
template <int D>
struct Cfg {
  static constexpr int NR = 2;                   // row halves
  static constexpr int R = 128 * NR;             // window rows
  static constexpr int TileBytes = D / 64 * kHalfBytes;  // one 128 x D bf16 tile
  static constexpr int KSteps = D / 16;          // MMAs per 128 x 128 product
  // Key-tile stages: 128 KB in flight hide the latency of HBM. The queries
  // have one buffer, loaded anew for every pass of an item; with two buffers
  // and half the stages the loads' latency bound the kernel.
  static constexpr int NK = D == 128 ? 4 : 8;
  // TMEM accumulators, one per row half of a tile, two tiles in flight. Each is
  // filled and released by itself: with whole tiles (2 x 256 columns) the MMAs
  // of a tile began only when its warpgroup had folded the first half of the
  // tile before and loaded the second, and tensor cores and exponentials took
  // turns (45% busy each).
  static constexpr int NA = 2 * NR;
  static constexpr int ACC_COLS = 128;
  static constexpr int QBYTES = NR * TileBytes;  // [D / 64][256 rows][64 dims]
  static constexpr int OFF_K = 0;
  static constexpr int OFF_Q = OFF_K + NK * TileBytes;
  static constexpr int OFF_MISC = OFF_Q + QBYTES;
};

struct Misc {
  uint64_t k_full[8], k_empty[8], q_full, q_empty, acc_full[4], acc_empty[4], mma_done;
  uint64_t pub_full[kPubSlots], pub_empty[kPubSlots];
  uint32_t tmem_base;
  int abort_flag;
  long long wait_cycles;  // bound of the waits of this launch
  alignas(16) float off[2][256];  // per-warpgroup row log-normalisers of a pass-2 item
  float2 pstat[kPubSlots][2][256];  // pass-1 row statistics per slot and warpgroup
};

static_assert(offsetof(Misc, off) % 16 == 0, "float4-read shared arrays are 16-byte aligned");

template <int D>
constexpr int smem_bytes() {
  return Cfg<D>::OFF_MISC + (int)sizeof(Misc) + 1024;  // + 1024-byte alignment slack
}

// Bounded mbarrier wait that also gives up as soon as another role aborted.
__device__ __forceinline__ bool wait_bar(uint64_t *bar, uint32_t parity, Misc *ms,
                                         int32_t *status) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*(volatile int *)&ms->abort_flag) return false;
    if (clock64() - t0 > ms->wait_cycles) {
      *(volatile int *)&ms->abort_flag = 1;
      report(status, RIPPLE_ETIMEOUT);
      return false;
    }
  }
}

// Warp-uniform variant: all lanes wait, the warp then agrees on the outcome
// (and is converged for the .sync.aligned TMEM loads that follow).
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, Misc *ms,
                                          int32_t *status) {
  const bool ok = wait_bar(bar, parity, ms, status);
  return __all_sync(0xffffffffu, ok);
}

__device__ __forceinline__ bool wait_ready(const int *flag, Misc *ms, int32_t *status) {
  if (ld_acquire(flag)) return true;
  const long long t0 = clock64();
  for (;;) {
    if (ld_acquire(flag)) return true;
    if (*(volatile int *)&ms->abort_flag) return false;
    if (clock64() - t0 > ms->wait_cycles) {
      *(volatile int *)&ms->abort_flag = 1;
      report(status, RIPPLE_ETIMEOUT);
      return false;
    }
    __nanosleep(64);
  }
}

__device__ __forceinline__ void combine(float &m, float &l, float m2, float l2) {
  const float mm = fmaxf(m, m2);
  if (mm == -INFINITY) return;
  l = l * fast_exp2(m - mm) + l2 * fast_exp2(m2 - mm);
  m = mm;
}

// ------------------------------------------------------------ kernel

// Kernel argument: the keys of every scored layer as 3-D tensor maps
// [unit][T][128], their window queries as 2-D maps [B * Hq * W][128], and the
// parameters.
struct TcLaunch {
  CUtensorMap kmap[kCompressMaxLayers];
  CUtensorMap qmap[kCompressMaxLayers];
  TcParams p;
};

// kPad: fewer than 256 window rows.
template <int D, bool kPad>
__global__ void __launch_bounds__(kThreads, 1)
    score_tc_kernel(const __grid_constant__ TcLaunch lp) {
  using C = Cfg<D>;
  constexpr int NR = C::NR;
  constexpr int kTileBytes = C::TileBytes;
  const TcParams &p = lp.p;
  // window rows, a constant without padding: with the count from the parameters
  // the loads of a merge were predicated one by one and overlapped less (5 to 15
  // us a call of one layer)
  const int R = kPad ? p.R : C::R;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t *ktiles = smem + C::OFF_K;
  uint8_t *qbufs = smem + C::OFF_Q;
  Misc *ms = (Misc *)(smem + C::OFF_MISC);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = items_of_cta(p);

  if (threadIdx.x == 0) {
    for (int i = 0; i < C::NK; ++i) {
      mbar_init(&ms->k_full[i], 1);
      mbar_init(&ms->k_empty[i], 1);
    }
    mbar_init(&ms->q_full, 1);
    mbar_init(&ms->q_empty, 1);
    for (int i = 0; i < C::NA; ++i) {
      mbar_init(&ms->acc_full[i], 1);
      mbar_init(&ms->acc_empty[i], 4);
    }
    for (int i = 0; i < kPubSlots; ++i) {
      mbar_init(&ms->pub_full[i], 8);
      mbar_init(&ms->pub_empty[i], 1);
    }
    mbar_init(&ms->mma_done, 1);
    ms->abort_flag = 0;
    ms->wait_cycles = p.wait_cycles;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&ms->tmem_base, 512);
    tmem_relinquish();
  }
  if constexpr (kPad) {
    // the padding rows of the query buffers (no copy writes them) hold zeros
    for (int i = threadIdx.x; i < C::QBYTES / 16; i += kThreads)
      reinterpret_cast<uint4 *>(qbufs)[i] = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ms->tmem_base;

  // Every role walks the same sequence: for k = 0..n, P1(item k) if k < n,
  // then P2(item k - 1) if k >= 1.
  if (warp == 0) {
    // ------------------------------------------------ TMA producers
    // Lane 0 streams key tiles through the ring; lane 1 loads each item's
    // window queries as soon as a query buffer is free, so that the key
    // stream never waits for a query load.
    if (lane == 0) {
      int kcount = 0;
      const uint64_t keep = policy_evict_last(), drop = policy_evict_first();
      bool ok = true;
      for (int k = 0; k <= n && ok; ++k) {
        for (int pass = 1; pass <= 2 && ok; ++pass) {
          if ((pass == 1 && k >= n) || (pass == 2 && k < 1)) continue;
          const ItemRef it = item_of(p, pass == 1 ? k : k - 1);
          int t0, t1;
          tiles_of(p, it, pass, t0, t1);
          for (int t = t0; t < t1; ++t) {
            const int ks = kcount % C::NK;
            if (!wait_bar(&ms->k_empty[ks], ((kcount / C::NK) & 1) ^ 1, ms, p.status)) {
              ok = false;
              break;
            }
            mbar_arrive_expect_tx(&ms->k_full[ks], kTileBytes);
            uint8_t *kb = ktiles + ks * kTileBytes;
            const uint64_t pol = pass == 1 ? keep : drop;
            const CUtensorMap *km = &lp.kmap[it.unit / p.upl];
            const int local = it.unit % p.upl;
#pragma unroll
            for (int half = 0; half < D / 64; ++half)
              tma_load_3d(kb + half * kHalfBytes, km, half * 64, t * kTile, local,
                          &ms->k_full[ks], pol);
            ++kcount;
          }
        }
      }
      // Let every issued copy land before the CTA can exit (matters only after
      // an abort; in normal operation every stage was already consumed).
      for (int j = max(0, kcount - C::NK); j < kcount; ++j)
        mbar_wait(&ms->k_full[j % C::NK], (j / C::NK) & 1, nullptr);
    } else if (lane == 1) {
      // in the order of the passes: P1(0) P1(1) P2(0) P1(2) P2(1) ..
      int qcount = 0;
      bool ok = true;
      for (int k = 0; k <= n && ok; ++k) {
        for (int pass = 1; pass <= 2 && ok; ++pass) {
          if ((pass == 1 && k >= n) || (pass == 2 && k < 1)) continue;
          const ItemRef it = item_of(p, pass == 1 ? k : k - 1);
          const int local = it.unit % p.upl;
          const CUtensorMap *qm = &lp.qmap[it.unit / p.upl];
          if (!wait_bar(&ms->q_empty, (qcount & 1) ^ 1, ms, p.status)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&ms->q_full, (uint32_t)(R * D * 2));
#pragma unroll
          for (int half = 0; half < D / 64; ++half)
            tma_load_2d(qbufs + half * (NR * kHalfBytes), qm, half * 64, local * R, &ms->q_full);
          ++qcount;
        }
      }
      if (qcount > 0) mbar_wait(&ms->q_full, (qcount - 1) & 1, nullptr);
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer (the whole warp
    // runs the loop and waits; one elected lane issues)
    {
      int kcount = 0, acount = 0, qcount = 0;
      constexpr uint32_t id = idesc_bf16(128, 128);
      const uint32_t kbase = smem_u32(ktiles), qbase = smem_u32(qbufs);
      bool ok = true;
      for (int k = 0; k <= n && ok; ++k) {
        for (int pass = 1; pass <= 2 && ok; ++pass) {
          if ((pass == 1 && k >= n) || (pass == 2 && k < 1)) continue;
          const ItemRef it = item_of(p, pass == 1 ? k : k - 1);
          if (!warp_wait(&ms->q_full, qcount & 1, ms, p.status)) {
            ok = false;
            break;
          }
          ++qcount;
          const uint32_t qa = qbase;
          int t0, t1;
          tiles_of(p, it, pass, t0, t1);
          for (int t = t0; t < t1; ++t) {
            const int ks = kcount % C::NK;
            if (!warp_wait(&ms->k_full[ks], (kcount / C::NK) & 1, ms, p.status)) {
              ok = false;
              break;
            }
            const uint64_t kd = sw128_desc(kbase + ks * kTileBytes);
#pragma unroll
            for (int nr = 0; nr < NR; ++nr) {
              const int as = acount % C::NA;
              if (!warp_wait(&ms->acc_empty[as], ((acount / C::NA) & 1) ^ 1, ms, p.status)) {
                ok = false;
                break;
              }
              tc_fence_after();
              const uint32_t d = tmem + as * C::ACC_COLS;
              // the first K step's descriptors; the others differ only in their
              // start-address field (16-byte units, no carry)
              const uint64_t qd = sw128_desc(qa + nr * kHalfBytes);
              if (elect_one()) {
#pragma unroll
              for (int kk = 0; kk < C::KSteps; ++kk) {
                const uint64_t ko = kd + (uint64_t)(((kk >> 2) * kHalfBytes + (kk & 3) * 32) >> 4);
                const uint64_t qo =
                    qd + (uint64_t)(((kk >> 2) * (NR * kHalfBytes) + (kk & 3) * 32) >> 4);
                mma_bf16(d, pass == 1 ? qo : ko, pass == 1 ? ko : qo, id, kk > 0);
              }
              mma_commit(&ms->acc_full[as]);
              if (nr == NR - 1) mma_commit(&ms->k_empty[ks]);
              }
              __syncwarp();
              ++acount;
            }
            if (!ok) break;
            ++kcount;
          }
          if (ok && elect_one()) mma_commit(&ms->q_empty);  // the pass is done with its queries
          __syncwarp();
        }
      }
      // All issued MMAs complete before TMEM is released.
      if (elect_one()) mma_commit(&ms->mma_done);
      __syncwarp();
      mbar_wait(&ms->mma_done, 0, nullptr);
    }
  } else if (warp == 10) {
    // ------------------------------------------------ publisher of pass-1 results
    constexpr int RJ = C::R / 32;   // rows per lane
    constexpr int CB = 32 / RJ;     // items merged per batch: 32 loads in flight per lane
    for (int k = 0; k < n; ++k) {
      const int slot = k % kPubSlots;
      if (!warp_wait(&ms->pub_full[slot], (k / kPubSlots) & 1, ms, p.status)) break;
      const ItemRef it = item_of(p, k);
      // One partial per item: the two warpgroups' statistics combined here.
      float2 *mine = p.partial + guard((long long)it.unit * p.n_ch + it.chunk, 1,
                                       (long long)p.units * p.n_ch, p.status) *
                                     R;
#pragma unroll
      for (int j = 0; j < RJ; ++j) {
        const int r = lane + 32 * j;
        float2 a = ms->pstat[slot][0][r];
        const float2 b = ms->pstat[slot][1][r];
        combine(a.x, a.y, b.x, b.y);
        if (r < R) mine[r] = a;
      }
      __syncwarp();  // all lanes' rows are written (and the slot read) before lane 0 goes on
      int last = 0;
      if (lane == 0) {
        mbar_arrive(&ms->pub_empty[slot]);
        __threadfence();  // the item's partial becomes visible GPU-wide before it is counted
        last = atomicAdd(&p.ctrl[guard(it.unit, 1, p.units, p.status)], 1) == p.n_ch - 1;
      }
      last = __shfl_sync(0xffffffffu, last, 0);
      if (last) {
        // Last item of the unit: merge its n_ch partials per row.
        __threadfence();
        const float2 *part =
            p.partial + guard((long long)it.unit * p.n_ch, p.n_ch, (long long)p.units * p.n_ch,
                              p.status) *
                            R;
        float mm[RJ], ll[RJ];
#pragma unroll
        for (int j = 0; j < RJ; ++j) {
          mm[j] = -INFINITY;
          ll[j] = 0.f;
        }
        for (int c0 = 0; c0 < p.n_ch; c0 += CB) {
          float2 q[CB][RJ];
#pragma unroll
          for (int c = 0; c < CB; ++c)
#pragma unroll
            for (int j = 0; j < RJ; ++j)
              q[c][j] = c0 + c < p.n_ch && lane + 32 * j < R
                            ? __ldcg(&part[(size_t)(c0 + c) * R + lane + 32 * j])
                            : make_float2(-INFINITY, 0.f);
#pragma unroll
          for (int c = 0; c < CB; ++c)
#pragma unroll
            for (int j = 0; j < RJ; ++j) combine(mm[j], ll[j], q[c][j].x, q[c][j].y);
        }
#pragma unroll
        for (int j = 0; j < RJ; ++j)
          if (lane + 32 * j < R)
            p.lognorm[guard(it.unit, 1, p.units, p.status) * R + lane + 32 * j] =
                mm[j] + __log2f(ll[j]);
        __threadfence();
        __syncwarp();
        if (lane == 0) st_release(&p.ctrl[guard(p.units + it.unit, 1, 2LL * p.units, p.status)], 1);
      }
    }
  } else {
    // ------------------------------------------------ epilogue warpgroups
    const int wg = (warp - 2) >> 2;
    const int quarter = warp & 3;              // TMEM lanes this warp may access
    const int lrow = quarter * 32 + lane;      // row (pass 1) or key (pass 2) in the tile
    const int wtid = threadIdx.x - 64 - wg * 128;  // 0..127 within the warpgroup
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    int tcount = 0;
    // Inside an item every warp follows the same control flow even if a wait
    // gives up (the tile is then skipped), so that the named barriers below
    // are always reached by all of their threads.
    for (int k = 0; k <= n; ++k) {
      if (k < n) {
        // ---------------- pass 1 of item k
        const ItemRef it = item_of(p, k);
        int t0, t1;
        tiles_of(p, it, 1, t0, t1);
        float m[NR], l[NR];
        int last_vis[NR];
#pragma unroll
        for (int nr = 0; nr < NR; ++nr) {
          m[nr] = -INFINITY;
          l[nr] = 0.f;
          last_vis[nr] = p.P + (lrow + nr * 128) % p.W;
        }
        for (int t = t0; t < t1; ++t, ++tcount) {
          if ((tcount & 1) != wg) continue;
          const bool masked = (t + 1) * kTile - 1 >= p.P;
#pragma unroll
          for (int nr = 0; nr < NR; ++nr) {
            const int at = tcount * NR + nr, as = at % C::NA;
            if (!warp_wait(&ms->acc_full[as], (at / C::NA) & 1, ms, p.status)) continue;
            tc_fence_after();
            uint32_t x[4][32];
            const uint32_t base = tmem + lane_addr + as * C::ACC_COLS;
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld32(base + c * 32, x[c]);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&ms->acc_empty[as]);
            if (masked) {  // keys this row cannot see (causal window, past T) -> -inf
#pragma unroll
              for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int j = 0; j < 32; ++j)
                  if (t * kTile + c * 32 + j > last_vis[nr]) x[c][j] = 0xff800000u;
            }
            // Eight independent chains keep the max and the sum off one long
            // dependency chain.
            float mx[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) mx[i] = -INFINITY;
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
              for (int j = 0; j < 32; ++j) mx[j & 7] = fmaxf(mx[j & 7], __uint_as_float(x[c][j]));
            const float tmax = fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])),
                                     fmaxf(fmaxf(mx[4], mx[5]), fmaxf(mx[6], mx[7])));
            if (tmax == -INFINITY) continue;
            const float mnew = fmaxf(m[nr], tmax * p.scale2);
            // fp32x2: logits scaled and shifted two at a time, sums in pairs
            float2 sv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) sv[i] = make_float2(0.f, 0.f);
            const float2 s2 = make_float2(p.scale2, p.scale2), mn2 = make_float2(-mnew, -mnew);
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
              for (int j = 0; j < 32; j += 2) {
                const float2 y = __ffma2_rn(
                    make_float2(__uint_as_float(x[c][j]), __uint_as_float(x[c][j + 1])), s2, mn2);
                sv[(j >> 1) & 3] =
                    __fadd2_rn(sv[(j >> 1) & 3], make_float2(fast_exp2(y.x), fast_exp2(y.y)));
              }
            const float s = ((sv[0].x + sv[0].y) + (sv[1].x + sv[1].y)) +
                            ((sv[2].x + sv[2].y) + (sv[3].x + sv[3].y));
            l[nr] = l[nr] * fast_exp2(m[nr] - mnew) + s;
            m[nr] = mnew;
          }
        }
        // This warpgroup's row statistics of the item go to the publisher warp
        // through a shared-memory slot.
        const int slot = k % kPubSlots;
        warp_wait(&ms->pub_empty[slot], ((k / kPubSlots) & 1) ^ 1, ms, p.status);
#pragma unroll
        for (int nr = 0; nr < NR; ++nr) ms->pstat[slot][wg][nr * 128 + lrow] = make_float2(m[nr], l[nr]);
        __syncwarp();  // every lane's rows are written before lane 0 arrives
        if (lane == 0) mbar_arrive(&ms->pub_full[slot]);
      }
      if (k >= 1) {
        // ---------------- pass 2 of item k - 1
        const ItemRef it = item_of(p, k - 1);
        int t0, t1;
        tiles_of(p, it, 2, t0, t1);
        if (t1 > t0) {
          if (wtid == 0)
            wait_ready(&p.ctrl[guard(p.units + it.unit, 1, 2LL * p.units, p.status)], ms, p.status);
          named_bar_sync(3 + wg, 128);
          for (int r = wtid; r < R; r += 128)
            ms->off[wg][r] = __ldcg(&p.lognorm[guard(it.unit, 1, p.units, p.status) * R + r]);
          named_bar_sync(3 + wg, 128);
        }
        const float4 *off4 = (const float4 *)ms->off[wg];
        // the unit's votes slot: its layer's in the vote array
        const int vunit = p.layer_of[it.unit / p.upl] * p.upl + it.unit % p.upl;
        for (int t = t0; t < t1; ++t, ++tcount) {
          if ((tcount & 1) != wg) continue;
          // fp32x2: logits scaled and shifted two at a time, sums in pairs
          float2 vs[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) vs[i] = make_float2(0.f, 0.f);
          const float2 s2 = make_float2(p.scale2, p.scale2);
          bool got = true;
#pragma unroll
          for (int c4 = 0; c4 < NR; ++c4) {
            const int at = tcount * NR + c4, as = at % C::NA;
            got = got && warp_wait(&ms->acc_full[as], (at / C::NA) & 1, ms, p.status);
            if (!got) continue;
            tc_fence_after();
            uint32_t x[4][32];
            const uint32_t base = tmem + lane_addr + as * C::ACC_COLS;
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld32(base + c * 32, x[c]);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&ms->acc_empty[as]);
            auto columns = [&](int c, auto some_padding) {
#pragma unroll
              for (int j = 0; j < 32; j += 4) {
                const float4 o = off4[(c4 * 128 + c * 32 + j) >> 2];
                const int h = (j >> 1) & 2;  // two pair chains per 4 columns: 4 in flight
                const float2 y0 = __ffma2_rn(
                    make_float2(__uint_as_float(x[c][j]), __uint_as_float(x[c][j + 1])), s2,
                    make_float2(-o.x, -o.y));
                const float2 y1 = __ffma2_rn(
                    make_float2(__uint_as_float(x[c][j + 2]), __uint_as_float(x[c][j + 3])), s2,
                    make_float2(-o.z, -o.w));
                float2 e0 = make_float2(fast_exp2(y0.x), fast_exp2(y0.y));
                float2 e1 = make_float2(fast_exp2(y1.x), fast_exp2(y1.y));
                if constexpr (decltype(some_padding)::value) {
                  const int left = R - (c4 * 128 + c * 32 + j);  // rows from this column on
                  if (left < 1) e0.x = 0.f;
                  if (left < 2) e0.y = 0.f;
                  if (left < 3) e1.x = 0.f;
                  if (left < 4) e1.y = 0.f;
                }
                vs[h] = __fadd2_rn(vs[h], e0);
                vs[h + 1] = __fadd2_rn(vs[h + 1], e1);
              }
            };
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const int first = c4 * 128 + c * 32;
              if (!kPad || first + 32 <= R)
                columns(c, std::false_type{});
              else if (first < R)
                columns(c, std::true_type{});
            }
          }
          const float vote = ((vs[0].x + vs[0].y) + (vs[1].x + vs[1].y)) +
                             ((vs[2].x + vs[2].y) + (vs[3].x + vs[3].y));
          const int key = t * kTile + lrow;
          if (got && key < p.P)
            p.votes[guard((long long)vunit * p.P + key, 1, (long long)p.n_slots * p.upl * p.P,
                          p.status)] = vote;
        }
      }
    }
  }

  tc_fence_before();
  __syncwarp();  // idle lanes of the single-thread roles wait for their lane 0 here
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ------------------------------------------------------------ host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (fn == nullptr) {
    void *ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)ptr;
  }
  return fn;
}

int sm_count() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

// Items a unit of n_tiles key tiles is cut into, in layers of `units` units: see
// kTilesPerItem. Of more than 256 tiles 16, or another number from an item per 64
// tiles on that takes less modelled time, the layer's waves of items times an
// item's tiles (4% less, or 12% for fewer items, as the waves of many layers even
// out): one unit of 4096 tiles 1049 us in 64 items, 1461
// in 16; 4 units of 1563 tiles 217 us in 25, 281 in 16; 8 of 4096 tiles 1348 us in
// 19, 1430 in 16, 1524 in 64; 16 of 1172 tiles 352 us in 19, 400 in 16; 32 of 547
// tiles 314 us in 9, 360 in 16. No more items than SMs (the schedule is free of
// deadlock up to twice as many).
int items_per_unit(int n_tiles, int units, int sms) {
  const int per = n_tiles <= kShortTiles ? kTilesPerItemShort : kTilesPerItem;
  const int items = (n_tiles + per - 1) / per;
  if (items <= kMaxItems) return std::min(items, sms);
  const int per_long = (n_tiles + kTilesPerItemLong - 1) / kTilesPerItemLong;
  const int most = std::min(std::max(per_long, kMaxItems), sms);
  int best = std::min(kMaxItems, sms);
  auto cost = [&](int n) {
    return ((long long)units * n + sms - 1) / sms * ((n_tiles + n - 1) / n);
  };
  for (int n = std::min(per_long, best); n <= most; ++n)
    if (cost(n) * 100 < cost(best) * (n < kMaxItems && best == kMaxItems ? 88 : 96)) best = n;
  return best;
}

template <int D>
cudaError_t launch_d(const LayerGeom &g, int n_slots, const int *slots, int n_scored,
                      const void *const *q_win, const void *const *k, const CompressWs &ws,
                      float *votes, int32_t *status, cudaStream_t st) {
  EncodeTiledFn enc = encode_fn();
  if (enc == nullptr) return cudaErrorNotSupported;
  if (n_scored < 1 || n_scored > kCompressMaxLayers || n_slots < 1) return cudaErrorInvalidValue;
  static TcLaunch lp;  // large: kept off the stack, filled under the lock
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  for (int l = 0; l < n_scored; ++l) {
    cuuint64_t dims[3] = {D, (cuuint64_t)g.T, (cuuint64_t)g.units};
    cuuint64_t strides[2] = {D * 2, (cuuint64_t)g.T * D * 2};
    cuuint32_t box[3] = {64, 128, 1};
    cuuint32_t es[3] = {1, 1, 1};
    if (enc(&lp.kmap[l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(k[l]), dims,
            strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
    cuuint64_t qdims[2] = {D, (cuuint64_t)g.units * g.R};
    cuuint64_t qstrides[1] = {D * 2};
    cuuint32_t qbox[2] = {64, (cuuint32_t)g.R};  // one unit's rows
    cuuint32_t qes[2] = {1, 1};
    if (enc(&lp.qmap[l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(q_win[l]), qdims,
            qstrides, qbox, qes, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  const int sms = sm_count();
  TcParams &p = lp.p;
  p.upl = g.units;
  p.units = g.units * n_scored;
  p.T = g.T;
  p.P = g.P;
  p.W = g.W;
  p.R = g.R;
  p.n_tiles1 = (g.T + kTile - 1) / kTile;
  p.n_tiles2 = (g.P + kTile - 1) / kTile;
  p.n_ch = items_per_unit(p.n_tiles1, g.units, sms);
  p.tpi = (p.n_tiles1 + p.n_ch - 1) / p.n_ch;
  p.n_ch = (p.n_tiles1 + p.tpi - 1) / p.tpi;
  p.total_items = p.units * p.n_ch;
  p.scale2 = g.scale2;
  p.partial = ws.row_partial;
  p.lognorm = ws.row_lognorm;
  p.votes = votes;
  for (int l = 0; l < n_scored; ++l) {
    if (slots[l] < 0 || slots[l] >= n_slots) return cudaErrorInvalidValue;
    p.layer_of[l] = slots[l];
  }
  p.n_slots = n_slots;
  p.ctrl = ws.counters;
  p.status = status;
  p.wait_cycles = wait_limit_cycles();
  cudaError_t e = cudaMemsetAsync(ws.counters, 0, sizeof(int) * 2 * p.units, st);
  if (e != cudaSuccess) return e;
  constexpr int smem = smem_bytes<D>();
  static_assert(smem <= 227 * 1024, "shared memory budget");
  const void *kernel = g.R == 256 ? (const void *)score_tc_kernel<D, false>
                                  : (const void *)score_tc_kernel<D, true>;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int grid = p.total_items < sms ? p.total_items : sms;
  // Cooperative launch: every CTA resident at once, which the cross-CTA waits
  // of the schedule rely on.
  void *args[] = {(void *)&lp};
  e = cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(kThreads), args, (size_t)smem, st);
  count_launches(1);
  return e;
}

}  // namespace

bool score_tc_supported(const LayerGeom &g) {
  return g.dtype == RIPPLE_BF16 && g.R > 128 && g.R <= 256 && g.P > 0;
}

cudaError_t launch_score_tc(const LayerGeom &g, int n_slots, const int *slots, int n_scored,
                            const void *const *q_win, const void *const *k, const CompressWs &ws,
                            float *votes, int32_t *status, cudaStream_t st) {
  if (g.D == 64)
    return launch_d<64>(g, n_slots, slots, n_scored, q_win, k, ws, votes, status, st);
  return launch_d<128>(g, n_slots, slots, n_scored, q_win, k, ws, votes, status, st);
}

}  // namespace ripple
