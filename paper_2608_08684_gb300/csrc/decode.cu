// GQA decode attention over the ragged compressed caches (Sec. 4.1: each new
// query attends to the cached states), with the append of the new token.
//
// One persistent launch per step covers every layer; one CTA per SM with 8
// compute warps and one producer warp. Work item = up to p.item_rows cache rows
// of one (layer, batch row, KV head) group; items are fetched with an atomic
// counter (one ahead), layers with the longest caches first. The producer
// stages each item's G query rows and then its sub-chunks of K and V rows in
// shared memory with bulk-async copies (TMA engine) through a ring of stages;
// the new token's key and value rows are copied into the stage behind the
// cached rows, and appended to the cache from there.
//
// Bound: HBM. One step over the 32 layers of the 32k workload (544 MB of cache
// rows) takes 83 us, 6.5 TB/s; 80 layers of the 70B shape (8 query heads per
// KV head, 677 MB) 112 us, 6.0 TB/s. On the CUDA cores, whose FMAs per cached
// byte grow with the heads, the same steps took 97 and 218 us.
//
// bf16 caches: warp-level matrix instructions, probabilities split into three
// bf16 parts so that nothing is lost against fp32 (consume_mma). mma.sync and
// not tcgen05, because a step is bound by its bytes, and its few rows (8 heads)
// would leave tcgen05's 128-row tiles empty.
//
// fp32 caches: CUDA cores (consume). Lane layout (the same for Q.K and P.V):
// the rows of a warp step are split over R row groups of S lanes; each lane
// owns DL head dims (its 16-byte pieces of the row) of every query head of the
// group: it reads those dims of the scaled fp32 queries from shared memory
// (converted once per item, in the order the lanes read them) and keeps those
// dims of the output accumulator in registers. Per row:
//   scores   fp32x2 FMAs over the lane's dims, then a reduce-scatter over the
//            S lanes of the row group (warp shuffles) that leaves each lane
//            with the full dot product of one head;
//   softmax  each (row group, head) keeps its own running max and sum (online
//            softmax; scores are in log2 units and the max is moved, and the
//            state rescaled, only when a score exceeds it by more than 8, a
//            probability factor of 2^8, so rescaling is rare);
//            the probability is computed once per head and all-gathered over
//            the row group (warp shuffles);
//   output   fp32x2 FMAs of the probabilities with the lane's value dims.
// At an item's end the row groups of a warp are merged by a shuffle butterfly.
//
// Both: the 8 warps' results of an item are merged through shared memory. An
// item covering its whole group writes the output; otherwise its unnormalised
// partial is stored and the group's last finishing item (atomic count)
// combines the partials in item order (deterministic).
//
// The step's counters live in the caller's workspace, whose contents are
// arbitrary: CTA 0 zeroes them at the start of every call and then raises an
// init flag tagged with the call's epoch; the other CTAs use no counter
// before they see it (their first item needs none). The last block advances the
// lengths once all have read them and seen the flag. Each launch is a
// programmatic dependent of the previous one on the stream: its CTAs take
// SMs as the previous step's CTAs leave and wait (griddepcontrol.wait) until
// that step has completed.
// CTA b's first item is item b, so that before that wait it can already
// prefetch its first sub-chunks into L2.
// Every wait is bounded; on timeout the CTA raises RIPPLE_ETIMEOUT and all
// roles leave their loops together.
#include <math.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "decode.cuh"
#include "kernels.cuh"

namespace ripple {
namespace {

constexpr int kWarps = 8;                     // compute warps
constexpr int kThreads = (kWarps + 1) * 32;   // + one producer warp
constexpr int kMaxStageBytes = 32768;         // K (or V) bytes of one sub-chunk, at most
constexpr int kRowsPerGroup = 4;              // rows per row group and sub-chunk (warp steps)
constexpr int kItemSlots = 4;
constexpr int kMaxStages = 6;
// Lazy rescaling: a running max (log2 units) is only moved when a score
// exceeds it by more than kRescaleLog2, so probabilities relative to a stale
// max stay <= 2^kRescaleLog2.
constexpr float kRescaleLog2 = 8.f;
constexpr int kSmemBudget = 226 * 1024;
constexpr int kMiscBytes = 4096;              // barriers, work list, merge statistics
constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxComb = 16;                  // partials of a group combined at a time, at most
constexpr int kPlanPerLane = RIPPLE_MAX_LAYERS / 32;  // layers per lane of the work list
constexpr uint32_t kSuspendNs = 1000000;      // of a poll of an mbarrier, at most

constexpr int cmax(int a, int b) { return a > b ? a : b; }
constexpr int cmin(int a, int b) { return a < b ? a : b; }

// fp32 caches (CUDA cores).
template <typename Tin, int D, int G>
struct DecCfg {
  static constexpr bool kMma = false;
  static constexpr int ROW_BYTES = D * (int)sizeof(Tin);
  static constexpr int NPIECE = ROW_BYTES / 16;             // 16-byte pieces per row
  static constexpr int PE = 16 / (int)sizeof(Tin);          // elements per piece
  // lanes per row: the queries and accumulators of a lane stay at 64
  // registers each, at least one lane per head, and a warp step's rows fit a
  // sub-chunk
  static constexpr int S = cmax(cmax(G * D / 64, G), cmax(ROW_BYTES / 128, 1));
  static constexpr int R = 32 / S;                          // row groups (rows per warp step)
  static constexpr int NIT =                                // warp steps per sub-chunk
      cmax(1, cmin(kRowsPerGroup, kMaxStageBytes / (kWarps * R * ROW_BYTES)));
  static constexpr int RPW = R * NIT;                       // rows per warp per sub-chunk
  static constexpr int CR = RPW * kWarps;                   // rows per sub-chunk
  static constexpr int STAGE_BYTES = CR * ROW_BYTES;
  // a sub-chunk is one run of rows in shared memory, consumed by all warps
  static constexpr int CHUNKS = 1, CHUNK_ROWS = CR, CHUNK_PITCH = STAGE_BYTES;
  static constexpr int QF = G * D;                          // converted queries, fp32
  static constexpr int RED_PITCH = D;                       // floats per head in red_o
  static constexpr int RED = kWarps;                        // merge buffers
  static constexpr int PPL = NPIECE / S;                    // pieces per lane
  static constexpr int DL = PPL * PE;                       // head dims per lane
  static constexpr int HL = S / G;                          // lanes per head after the reduce-scatter
  static constexpr int QBYTES = G * ROW_BYTES;              // one group's queries
  static constexpr int NH = PE / 4;                         // float4 per piece in fp32
  static constexpr int STAGES =
      cmin(kMaxStages, (kSmemBudget - kMiscBytes - kItemSlots * QBYTES - (kWarps + 2) * G * D * 4) /
                           (2 * STAGE_BYTES));
  static_assert(S <= 32 && S <= NPIECE && NPIECE % S == 0, "lanes per row");
  static_assert(STAGE_BYTES <= kMaxStageBytes, "stage size");
  static_assert(DL % 2 == 0 && PE % 2 == 0, "fp32x2 pairs");
  static_assert(STAGES >= 2, "shared memory budget");
};

// bf16 caches (mma.sync). A sub-chunk (32 KB of K and of V: 128 rows of 128
// dims, 256 of 64) lies in shared memory as 8 chunks of 4 KB, one pad piece of
// 16 bytes after each: row i of the 8 chunks is then one 8 x 8 matrix row set
// of ldmatrix without bank conflicts (rows of one run, 256 bytes apart, would
// conflict 8 ways). Warp w takes rows w * CHUNK_ROWS / 8 .. of every chunk, 16
// cache rows at a time. Chunks of 4 KB because the copy engine is bound by
// copies below that: 8 steps of the 32k workload took 832 us with 2 KB chunks
// (64-row sub-chunks), 680 us with 4 KB.
template <int D, int G>
struct DecCfg<__nv_bfloat16, D, G> {
  static constexpr bool kMma = true;
  static constexpr int ROW_BYTES = D * 2;
  static constexpr int NPIECE = ROW_BYTES / 16;
  static constexpr int CHUNKS = 8, CHUNK_ROWS = 4096 / ROW_BYTES;
  static constexpr int CHUNK_PITCH = CHUNK_ROWS * ROW_BYTES + 16;
  static constexpr int PAIRS = CHUNK_ROWS / 16;             // 16-row steps of a warp
  static constexpr int CR = CHUNKS * CHUNK_ROWS;
  static constexpr int STAGE_BYTES = CHUNKS * CHUNK_PITCH;
  static constexpr int QBYTES = G * ROW_BYTES;
  static constexpr int QF = 4;                              // queries go to registers as they are
  static constexpr int RED_PITCH = D + 8;  // the 8 rows of a merge store on different banks
  // merge buffers: with 8 heads of 128 dims the warps share four, so that a
  // third stage fits
  static constexpr int RED = G * D > 512 ? kWarps / 2 : kWarps;
  static constexpr int STAGES =
      cmin(kMaxStages,
           (kSmemBudget - kMiscBytes - kItemSlots * QBYTES - RED * G * RED_PITCH * 4) /
               (2 * STAGE_BYTES));
  static_assert(STAGES >= 3 && STAGE_BYTES % 16 == 0, "shared memory budget");
};

// Byte offset of row r of a sub-chunk in its K or V stage.
template <typename C>
__device__ __forceinline__ int stage_row(int r) {
  return r / C::CHUNK_ROWS * C::CHUNK_PITCH + r % C::CHUNK_ROWS * C::ROW_BYTES;
}

template <typename Tin, int D, int G>
struct DecSmem {
  using C = DecCfg<Tin, D, G>;
  alignas(128) uint8_t kv[C::STAGES][2][C::STAGE_BYTES];  // [stage][K, V]
  alignas(128) uint8_t qs[kItemSlots][C::QBYTES];      // each item's query rows
  alignas(16) float qf[2][C::QF];                      // scaled fp32 queries, lane-piece order
  alignas(16) float red_o[C::RED][G * C::RED_PITCH];              // per-warp outputs at an item's end
  float red_m[C::RED][G], red_l[C::RED][G];
  uint64_t full[C::STAGES], empty[C::STAGES], item_full[kItemSlots], item_empty[kItemSlots];
  int item_id[kItemSlots];
  int len[RIPPLE_MAX_LAYERS];    // by work-order position; -1 = full layer
  int nch[RIPPLE_MAX_LAYERS];    // items per group, by work-order position
  int base[RIPPLE_MAX_LAYERS + 1];
  int abort_flag;
  int last;
  int init_seen;  // this CTA's producer has seen the init flag
};

struct ItemInfo {
  int pos, layer, group, b, h, chunk, nch, len, r0, rows, full;
};

template <typename S>
__device__ __forceinline__ ItemInfo item_info(const DecParams &p, const S &s, int it) {
  int lo = 0, hi = p.L - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (s.base[mid] <= it) lo = mid; else hi = mid - 1;
  }
  ItemInfo f;
  f.pos = lo;
  f.layer = p.order[lo];
  f.nch = s.nch[lo];
  const int local = it - s.base[lo];
  const int unit = local / f.nch;
  f.chunk = local % f.nch;
  f.b = unit / p.Hkv;
  f.h = unit % p.Hkv;
  f.group = (f.layer * p.B + f.b) * p.Hkv + f.h;
  f.len = s.len[lo];
  f.full = f.len < 0;
  f.r0 = f.chunk * p.item_rows;
  // rows 0..len: the cached rows and the new token
  f.rows = f.full ? 0 : min(p.item_rows, f.len + 1 - f.r0);
  return f;
}

// Whether the phase has completed, after suspending the thread for at most about
// `ns` nanoseconds until it does.
__device__ __forceinline__ bool mbar_try_wait_for(uint64_t *bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n"
      " mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, %3;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(ns)
      : "memory");
  return ok != 0;
}

// Bounded wait on an mbarrier phase. Gives up when another role of the CTA
// has given up, or after p.wait_cycles (then raises the CTA's abort flag and
// reports RIPPLE_ETIMEOUT). A poll suspends the thread for p.suspend_ns at most,
// which is within the bound, so that short bounds are kept by the same path.
__device__ __forceinline__ bool wait_bar(uint64_t *bar, uint32_t parity, int *abort_flag,
                                         const DecParams &p) {
  if (mbar_try_wait_for(bar, parity, p.suspend_ns)) return true;
  const long long t0 = clock64();
  for (;;) {
    if (mbar_try_wait_for(bar, parity, p.suspend_ns)) return true;
    if (*(volatile int *)abort_flag) return false;
    if (clock64() - t0 > p.wait_cycles) {
      *(volatile int *)abort_flag = 1;
      report(p.status, RIPPLE_ETIMEOUT);
      return false;
    }
  }
}

// Waits until CTA 0 has zeroed this call's counters (the init flag holds the
// call's epoch). Bounded like wait_bar.
__device__ __forceinline__ bool wait_init(const DecParams &p, int *abort_flag) {
  if (ld_acquire(&p.ctrl[kCtrlFlag]) == p.epoch) return true;
  const long long t0 = clock64();
  for (;;) {
    if (ld_acquire(&p.ctrl[kCtrlFlag]) == p.epoch) return true;
    if (*(volatile int *)abort_flag) return false;
    if (clock64() - t0 > p.wait_cycles) {
      *(volatile int *)abort_flag = 1;
      report(p.status, RIPPLE_ETIMEOUT);
      return false;
    }
    __nanosleep(32);
  }
}

// Block-scope acquire load / release store of a flag in shared memory: what the
// storing thread has itself acquired (another block's writes included) is
// ordered before what the loading thread does next.
__device__ __forceinline__ int ld_acquire_cta(const int *p) {
  int v;
  asm volatile("ld.acquire.cta.shared::cta.b32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_cta(int *p, int v) {
  asm volatile("st.release.cta.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}

// Waits until this CTA's producer has seen the init flag. Release and acquire on
// the shared word hand on what the producer acquired with the flag: CTA 0's
// zeroing comes before this thread's counting on the counters.
__device__ __forceinline__ bool wait_seen(const DecParams &p, const int *seen, int *abort_flag) {
  const long long t0 = clock64();
  while (!ld_acquire_cta(seen)) {
    if (*(volatile int *)abort_flag) return false;
    if (clock64() - t0 > p.wait_cycles) {
      *(volatile int *)abort_flag = 1;
      report(p.status, RIPPLE_ETIMEOUT);
      return false;
    }
  }
  return true;
}

// Named barrier over the compute warps that also ORs a predicate over them.
__device__ __forceinline__ bool compute_bar_or(bool pred) {
  __syncwarp();
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n"
      " setp.ne.u32 p, %1, 0;\n"
      " barrier.red.or.pred q, 1, %2, p;\n"
      " selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)pred), "n"(kWarps * 32)
      : "memory");
  return r != 0;
}

// 2*NP consecutive fp32 values (one aligned 16-byte load) as pairs.
template <int NP>
__device__ __forceinline__ void load_pairs(const float *p, float2 (&o)[NP]) {
  static_assert(NP == 2, "one 16-byte piece");
  const float4 u = *reinterpret_cast<const float4 *>(p);
  o[0] = make_float2(u.x, u.y);
  o[1] = make_float2(u.z, u.w);
}

// Per-head values of a lane are kept in an order permuted by the lane's own
// head hq = (lane % S) / (S / G): entry j holds head j ^ hq. Then every step
// of the reduce-scatter and of the all-gather over the S lanes of a row group
// is a plain shuffle (the partner's entry that this lane needs sits at a fixed
// index), with no per-lane selects.
//
// Reduce-scatter of G per-lane partial sums: afterwards v[0] of every lane is
// the full sum of its head hq. At the step over lane bit o the partner's head
// differs from this lane's in the head bit being split, which is bit
// log2(nv / 2) of the entry index.
template <int S, int G>
__device__ __forceinline__ void reduce_scatter(float (&v)[G]) {
#pragma unroll
  for (int o = S / 2, nv = G; o >= 1; o >>= 1) {
    if (nv > 1) {
#pragma unroll
      for (int i = 0; i < G / 2; ++i)
        if (i < nv / 2) v[i] += __shfl_xor_sync(kFull, v[i + nv / 2], o);
      nv /= 2;
    } else {
      v[0] += __shfl_xor_sync(kFull, v[0], o);
    }
  }
}

// Inverse of the head split of reduce_scatter: from x (the value of head hq)
// every lane of the row group receives o[j] = the value of head j ^ hq.
template <int S, int G>
__device__ __forceinline__ void all_gather(float x, float (&o)[G]) {
  o[0] = x;
#pragma unroll
  for (int lev = 0; (1 << lev) < G; ++lev)
#pragma unroll
    for (int i = 0; i < (1 << lev); ++i)
      o[(1 << lev) + i] = __shfl_xor_sync(kFull, o[i], (S / G) << lev);
}

// ------------------------------------------------------------ producer
// Holds the producer until the bulk copies it has issued have landed (the
// last phase armed on each stage and item slot), so that no copy writes into
// shared memory after the CTA has left even when the consumers gave up early;
// when they did not, these phases have long completed. Fixed bound,
// independent of the launch's wait limit.
template <typename Tin, int D, int G>
__device__ __forceinline__ void drain(DecSmem<Tin, D, G> &s, uint32_t j,
                                      const int (&last_use)[kItemSlots]) {
  using C = DecCfg<Tin, D, G>;
  for (uint32_t jj = j > (uint32_t)C::STAGES ? j - C::STAGES : 0; jj < j; ++jj)
    mbar_wait(&s.full[jj % C::STAGES], (jj / C::STAGES) & 1, nullptr);
  for (int slot = 0; slot < kItemSlots; ++slot)
    if (last_use[slot] >= 0)
      mbar_wait(&s.item_full[slot], (last_use[slot] / kItemSlots) & 1, nullptr);
}

// The producer warp: every lane walks the same items and stages, lane 0 fetches
// items and arms the barriers, and lane i issues copy i of a stage (K or V of
// one chunk), since one lane's address arithmetic for all of a stage's copies
// took longer than their transfer (steps of the 32k workload, 2 KB copies: 128
// us with one issuing lane, 104 us with one lane per copy).
template <typename Tin, int D, int G>
__device__ __forceinline__ void produce(const DecParams &p, DecSmem<Tin, D, G> &s, int total,
                                        int lane) {
  using C = DecCfg<Tin, D, G>;
  const int units = p.B * p.Hkv;
  uint32_t j = 0;                                // sub-chunk stages armed
  int last_use[kItemSlots] = {-1, -1, -1, -1};   // last item count that armed each slot
  static_assert(kItemSlots == 4, "last_use initialiser");
  static_assert(2 * C::CHUNKS <= 32, "one copy per lane");
  const int kv = lane & 1, row0 = (lane >> 1) * C::CHUNK_ROWS;  // this lane's copy
  const bool copies = lane < 2 * C::CHUNKS;
  auto wait_all = [&](uint64_t *bar, uint32_t parity) {
    return __all_sync(kFull, wait_bar(bar, parity, &s.abort_flag, p)) != 0;
  };
  // The item after `cur`, asked for from the counter once CTA 0 has zeroed it
  // (lane 0's value; it arrives while the item's copies are issued).
  // Without a second item for any CTA there is nothing to ask for.
  bool init_seen = false;
  auto see_init = [&] {  // lane 0
    if (!init_seen && wait_init(p, &s.abort_flag)) init_seen = true;
    return init_seen;
  };
  auto ask_next = [&](int cur) {
    int n = total;
    if (lane == 0 && cur < total && total > (int)gridDim.x && see_init())
      n = atomicAdd(&p.ctrl[kCtrlItem], 1) + (int)gridDim.x;
    return n;
  };
  // This CTA has read the lengths and seen the init flag, which its consumers
  // wait for in shared memory: from here on it needs neither.
  auto arrive = [&] {  // lane 0, once, before the first item's end
    if (see_init()) {
      st_release_cta(&s.init_seen, 1);
      atomicAdd(&p.ctrl[kCtrlArrived], 1);
    }
  };
  bool arrived = false;
  // The first item of CTA b is item b; later ones come from the counter, one
  // item ahead (for the first item, once its first loads are issued).
  int it = min((int)blockIdx.x, total);
  for (int icount = 0;; ++icount) {
    const int slot = icount % kItemSlots;
    bool asked = icount > 0;
    int nxt = asked ? ask_next(it) : total;
    if (!wait_all(&s.item_empty[slot], ((icount / kItemSlots) & 1) ^ 1)) {
      drain(s, j, last_use);
      return;
    }
    const int cur = min(it, total);
    if (lane == 0) s.item_id[slot] = cur;
    last_use[slot] = icount;
    if (cur >= total) {
      if (lane == 0) {
        mbar_arrive(&s.item_full[slot]);
        if (!arrived) arrive();
      }
      drain(s, j, last_use);  // returns at once unless the consumers gave up
      return;
    }
    const ItemInfo f = item_info(p, s, cur);
    if (f.full) {
      if (lane == 0) mbar_arrive(&s.item_full[slot]);
    } else {
      if (lane == 0) {
        const size_t qrow = ((size_t)f.layer * p.B + f.b) * p.Hq + (size_t)f.h * G;
        mbar_arrive_expect_tx(&s.item_full[slot], C::QBYTES);
        const long long qr = guard((long long)qrow, G, (long long)p.L * p.B * p.Hq, p.status);
        bulk_g2s(s.qs[slot], (const uint8_t *)p.q + qr * C::ROW_BYTES, C::QBYTES,
                 &s.item_full[slot]);
      }
      const int nsub = (f.rows + C::CR - 1) / C::CR;
      const size_t gbase = (size_t)(f.b * p.Hkv + f.h) * p.cap[f.layer];
      const size_t nb = guard((long long)f.layer * units + f.b * p.Hkv + f.h, 1,
                              (long long)p.L * units, p.status) *
                        C::ROW_BYTES;
      const uint8_t *cache = (const uint8_t *)(kv ? p.vc[f.layer] : p.kc[f.layer]);
      const uint8_t *fresh = (const uint8_t *)(kv ? p.v_new : p.k_new) + nb;
      for (int sub = 0; sub < nsub; ++sub, ++j) {
        const int stage = j % C::STAGES;
        if (sub == 1 && !asked) {
          nxt = ask_next(it);
          asked = true;
        }
        if (!wait_all(&s.empty[stage], ((j / C::STAGES) & 1) ^ 1)) {
          drain(s, j, last_use);
          return;
        }
        const int rs = f.r0 + sub * C::CR;
        const int re = min(rs + C::CR, f.len);  // rows >= len are not in the cache yet
        const int nk = re > rs ? re - rs : 0;
        const bool has_new = f.len >= rs && f.len < rs + C::CR;
        if (lane == 0)
          mbar_arrive_expect_tx(&s.full[stage], 2u * (nk + (has_new ? 1 : 0)) * C::ROW_BYTES);
        __syncwarp();
        if (copies && row0 < nk) {
          const size_t off =
              guard((long long)(gbase + rs), nk, (long long)units * p.cap[f.layer], p.status) *
              C::ROW_BYTES;
          bulk_g2s(s.kv[stage][kv] + (lane >> 1) * C::CHUNK_PITCH,
                   cache + off + (size_t)row0 * C::ROW_BYTES,
                   (uint32_t)min(nk - row0, C::CHUNK_ROWS) * C::ROW_BYTES, &s.full[stage]);
        }
        if (has_new && lane < 2)
          bulk_g2s(s.kv[stage][kv] + stage_row<C>(f.len - rs), fresh, C::ROW_BYTES,
                   &s.full[stage]);
      }
    }
    if (!asked) nxt = ask_next(it);
    if (!arrived && lane == 0) arrive();
    arrived = true;
    it = __shfl_sync(kFull, nxt, 0);
  }
}

// ------------------------------------------------------------ compute warps
// The end of an item, all compute warps: merge their partial outputs (red_o,
// red_m, red_l), write the output of a group that is one item, or store the
// partial and, as the group's last item, combine the group's partials in item
// order.
template <typename Tin, int D, int G>
__device__ __forceinline__ void finish_item(const DecParams &p, DecSmem<Tin, D, G> &s,
                                            const ItemInfo &f, int tid) {
  using C = DecCfg<Tin, D, G>;
  const size_t qrow = ((size_t)f.layer * p.B + f.b) * p.Hq + (size_t)f.h * G;
  named_bar_sync(1, kWarps * 32);
  const bool single = f.nch == 1;
  const int item_base = s.base[f.pos] + (f.b * p.Hkv + f.h) * f.nch;
  const int item = item_base + f.chunk;
  for (int e = tid; e < G * D; e += kWarps * 32) {
    const int g = e / D;
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < C::RED; ++w) M = fmaxf(M, s.red_m[w][g]);
    const float M_sub = M == -INFINITY ? 0.f : M;  // -infinity: scores of that alone
    float num = 0.f, den = 0.f;
#pragma unroll
    for (int w = 0; w < C::RED; ++w) {
      const float wgt = fast_exp2(s.red_m[w][g] - M_sub);
      num += wgt * s.red_o[w][g * C::RED_PITCH + e % D];
      den += wgt * s.red_l[w][g];
    }
    if (single) {
      p.out[guard(qrow * D + e, 1, (long long)p.L * p.B * p.Hq * D, p.status)] = num / den;
    } else {
      const long long wi = guard(item, 1, p.ws_items, p.status);
      p.ws_o[wi * G * D + e] = num;
      if (e % D == 0) p.ws_ml[wi * G + g] = make_float2(M, den);
    }
  }
  if (!single) {
    __threadfence();
    named_bar_sync(1, kWarps * 32);
    if (tid == 0) {
      // without the counters (a wait gave up) no item combines the group
      s.last = wait_seen(p, &s.init_seen, &s.abort_flag) &&
               atomicAdd(&p.ctrl[guard(kCtrlGroup + f.group, 1, p.n_ctrl, p.status)], 1) ==
                   f.nch - 1;
    }
    named_bar_sync(1, kWarps * 32);
    if (s.last) {
      __threadfence();
      const long long ib = guard(item_base, f.nch, p.ws_items, p.status);
      // partials in item order, kComb at a time so that their loads overlap (as
      // few more than there are: 16 loads for 3 partials cost 0.6 us a step)
      auto combine = [&](auto comb) {
        constexpr int kComb = decltype(comb)::value;
        for (int e = tid; e < G * D; e += kWarps * 32) {
          const int g = e / D;
          float M = -INFINITY, num = 0.f, den = 0.f;
          for (int c0 = 0; c0 < f.nch; c0 += kComb) {
            float2 ml[kComb];
            float o[kComb];
#pragma unroll
            for (int c = 0; c < kComb; ++c) {
              const size_t i = ib + min(c0 + c, f.nch - 1);
              ml[c] = __ldcg(&p.ws_ml[i * G + g]);
              o[c] = __ldcg(&p.ws_o[i * G * D + e]);
              if (c0 + c >= f.nch) {  // no partial: nothing for its weight of 0 to scale
                ml[c] = make_float2(-INFINITY, 0.f);
                o[c] = 0.f;
              }
            }
            float Mn = M;
#pragma unroll
            for (int c = 0; c < kComb; ++c) Mn = fmaxf(Mn, ml[c].x);
            const float M_sub = Mn == -INFINITY ? 0.f : Mn;
            const float a = fast_exp2(M - M_sub);
            num *= a;
            den *= a;
            M = Mn;
#pragma unroll
            for (int c = 0; c < kComb; ++c) {
              const float wgt = fast_exp2(ml[c].x - M_sub);
              den += wgt * ml[c].y;
              num += wgt * o[c];
            }
          }
          p.out[guard(qrow * D + e, 1, (long long)p.L * p.B * p.Hq * D, p.status)] = num / den;
        }
      };
      if (f.nch <= 4)
        combine(std::integral_constant<int, 4>{});
      else if (f.nch <= 8)
        combine(std::integral_constant<int, 8>{});
      else
        combine(std::integral_constant<int, kMaxComb>{});
    }
  }
}

// The new token's rows, staged behind the cached rows of the item's last
// sub-chunk, go to the cache (one warp).
template <typename Tin, int D, int G>
__device__ __forceinline__ void append_new(const DecParams &p, DecSmem<Tin, D, G> &s,
                                           const ItemInfo &f, int sub, int stage, int lane) {
  using C = DecCfg<Tin, D, G>;
  const int rs = f.r0 + sub * C::CR;
  if (f.len < rs || f.len >= rs + C::CR) return;
  const size_t dst = guard((long long)(f.b * p.Hkv + f.h) * p.cap[f.layer] + f.len, 1,
                           (long long)p.B * p.Hkv * p.cap[f.layer], p.status) *
                     C::ROW_BYTES;
  for (int e = lane; e < 2 * C::NPIECE; e += 32) {
    const int kvsel = e >= C::NPIECE, pc = e % C::NPIECE;
    const uint4 val = reinterpret_cast<const uint4 *>(s.kv[stage][kvsel] +
                                                      stage_row<C>(f.len - rs))[pc];
    reinterpret_cast<uint4 *>((uint8_t *)(kvsel ? p.vc[f.layer] : p.kc[f.layer]) + dst)[pc] = val;
  }
}

template <typename Tin, int D, int G>
__device__ __forceinline__ void consume(const DecParams &p, DecSmem<Tin, D, G> &s, int total,
                                        int warp, int lane) {
  using C = DecCfg<Tin, D, G>;
  constexpr int S = C::S, R = C::R, NIT = C::NIT, PPL = C::PPL, PE = C::PE, DL = C::DL;
  const int tid = warp * 32 + lane;
  const int sl = lane % S;              // lane within its row group
  const int rg = lane / S;              // row group
  const int hq = sl / C::HL;            // head of this lane after the reduce-scatter;
                                        // per-head arrays hold head j ^ hq at entry j
  const int rw0 = warp * C::RPW;        // this warp's first row in a sub-chunk
  uint32_t j = 0;
  for (int icount = 0;; ++icount) {
    const int slot = icount % kItemSlots;
    bool ok = wait_bar(&s.item_full[slot], (icount / kItemSlots) & 1, &s.abort_flag, p);
    ok = __all_sync(kFull, ok);
    const int it = ok ? s.item_id[slot] : total;
    // Queries to fp32, scaled to log2 units, in the order the lanes read them:
    // [entry j][piece k][half h][lane sl][4], entry j of lane sl being head
    // j ^ hq(sl).
    float *qf = s.qf[icount & 1];
    if (it < total) {
      const Tin *qg = (const Tin *)s.qs[slot];
      for (int e = tid; e < G * D; e += kWarps * 32) {
        const int c = e % 4, l4 = (e / 4) % S, h = (e / (4 * S)) % C::NH;
        const int k = (e / (4 * S * C::NH)) % PPL, jj = e / (4 * S * C::NH * PPL);
        const int g = jj ^ (l4 / C::HL);
        qf[e] = to_f32(qg[g * D + (l4 + k * S) * PE + h * 4 + c]) * p.scale2;
      }
    }
    // All compute warps leave together (the item's merge has named barriers);
    // this barrier also frees the merge buffers of the previous item and
    // publishes the fp32 queries.
    if (compute_bar_or(it >= total || *(volatile int *)&s.abort_flag)) {
      if (lane == 0) mbar_arrive(&s.item_empty[slot]);
      break;
    }
    const ItemInfo f = item_info(p, s, it);
    const size_t qrow = ((size_t)f.layer * p.B + f.b) * p.Hq + (size_t)f.h * G;
    if (f.full) {
      if (lane == 0) mbar_arrive(&s.item_empty[slot]);
      for (int e = tid; e < G * D; e += kWarps * 32)
        p.out[guard(qrow * D + e, 1, (long long)p.L * p.B * p.Hq * D, p.status)] = 0.f;
      continue;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&s.item_empty[slot]);

    float2 acc[G][DL / 2];  // entry j: head j ^ hq, the lane's dims
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int e = 0; e < DL / 2; ++e) acc[g][e] = make_float2(0.f, 0.f);
    float m_run = -INFINITY, l_run = 0.f;  // of head hq over this row group's rows

    // One sub-chunk of this warp's rows; kMask: some rows are past nrows
    // (their index is clamped to a valid row; they count for nothing by their
    // place, not by that row's score).
    auto rows_step = [&](const Tin *ks, const Tin *vs, int nrows, auto mask_tag) {
      constexpr bool kMask = decltype(mask_tag)::value;
      float2 d2[NIT][G];
#pragma unroll
      for (int t = 0; t < NIT; ++t)
#pragma unroll
        for (int g = 0; g < G; ++g) d2[t][g] = make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < PPL; ++k) {
        float2 kp[NIT][PE / 2];
#pragma unroll
        for (int t = 0; t < NIT; ++t) {
          const int row = rw0 + t * R + rg;
          const int rr = kMask ? min(row, nrows - 1) : row;
          load_pairs<PE / 2>(ks + (size_t)rr * D + (sl + k * S) * PE, kp[t]);
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
          float2 qp[PE / 2];
#pragma unroll
          for (int h = 0; h < C::NH; ++h) {
            const float4 x =
                *reinterpret_cast<const float4 *>(&qf[(((g * PPL + k) * C::NH + h) * S + sl) * 4]);
            qp[2 * h] = make_float2(x.x, x.y);
            qp[2 * h + 1] = make_float2(x.z, x.w);
          }
#pragma unroll
          for (int t = 0; t < NIT; ++t)
#pragma unroll
            for (int e = 0; e < PE / 2; ++e) d2[t][g] = __ffma2_rn(qp[e], kp[t][e], d2[t][g]);
        }
      }
      float sc[NIT];
#pragma unroll
      for (int t = 0; t < NIT; ++t) {
        const int row = rw0 + t * R + rg;
        float v[G];
#pragma unroll
        for (int g = 0; g < G; ++g) v[g] = d2[t][g].x + d2[t][g].y;
        reduce_scatter<S, G>(v);
        sc[t] = (!kMask || row < nrows) ? v[0] : -INFINITY;
      }
      float mb = sc[0];
#pragma unroll
      for (int t = 1; t < NIT; ++t) mb = fmaxf(mb, sc[t]);
      const bool grow = mb > m_run + kRescaleLog2;  // true for the first rows (m_run = -inf)
      if (__any_sync(kFull, grow)) {
        const float mn = grow ? mb : m_run;
        const float a = grow ? fast_exp2(m_run - mn) : 1.f;
        l_run *= a;
        float ag[G];
        all_gather<S, G>(a, ag);
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
          for (int e = 0; e < DL / 2; ++e) acc[g][e] = __fmul2_rn(acc[g][e], make_float2(ag[g], ag[g]));
        m_run = mn;
      }
      const float m_sub = m_run == -INFINITY ? 0.f : m_run;  // scores of -infinity alone
#pragma unroll
      for (int t = 0; t < NIT; ++t) {
        const int row = rw0 + t * R + rg;
        const int rr = kMask ? min(row, nrows - 1) : row;
        const bool live = !kMask || row < nrows;
        const float pt = live ? fast_exp2(sc[t] - m_sub) : 0.f;
        l_run += pt;
        float pg[G];
        all_gather<S, G>(pt, pg);
#pragma unroll
        for (int k = 0; k < PPL; ++k) {
          float2 vp[PE / 2];
          load_pairs<PE / 2>(vs + (size_t)rr * D + (sl + k * S) * PE, vp);
          if (!live) {  // 0 times an infinite value of the row in its place is NaN
#pragma unroll
            for (int e = 0; e < PE / 2; ++e) vp[e] = make_float2(0.f, 0.f);
          }
#pragma unroll
          for (int g = 0; g < G; ++g)
#pragma unroll
            for (int e = 0; e < PE / 2; ++e)
              acc[g][k * PE / 2 + e] =
                  __ffma2_rn(make_float2(pg[g], pg[g]), vp[e], acc[g][k * PE / 2 + e]);
        }
      }
    };

    const int nsub = (f.rows + C::CR - 1) / C::CR;
    for (int sub = 0; sub < nsub; ++sub, ++j) {
      const int stage = j % C::STAGES;
      wait_bar(&s.full[stage], (j / C::STAGES) & 1, &s.abort_flag, p);
      __syncwarp();
      const int nrows = min(C::CR, f.rows - sub * C::CR);
      const Tin *ks = (const Tin *)s.kv[stage][0];
      const Tin *vs = (const Tin *)s.kv[stage][1];
      if (rw0 + C::RPW <= nrows)
        rows_step(ks, vs, nrows, std::false_type{});
      else if (rw0 < nrows)
        rows_step(ks, vs, nrows, std::true_type{});
      if (warp == 0) append_new<Tin, D, G>(p, s, f, sub, stage, lane);
      __syncwarp();
      if (lane == 0) mbar_arrive(&s.empty[stage]);
    }

    // Item end. (1) Merge the warp's row groups (butterfly over lanes with
    // the same position in their row group, hence the same head).
#pragma unroll
    for (int o = S; o < 32; o <<= 1) {
      const float mo = __shfl_xor_sync(kFull, m_run, o);
      const float lo = __shfl_xor_sync(kFull, l_run, o);
      const float M = fmaxf(m_run, mo);
      const float as = m_run == -INFINITY ? 0.f : fast_exp2(m_run - M);
      const float ao = mo == -INFINITY ? 0.f : fast_exp2(mo - M);
      l_run = l_run * as + lo * ao;
      m_run = M;
      float gs[G], go[G];
      all_gather<S, G>(as, gs);
      all_gather<S, G>(ao, go);
#pragma unroll
      for (int g = 0; g < G; ++g)
#pragma unroll
        for (int e = 0; e < DL / 2; ++e) {
          float2 other;
          other.x = __shfl_xor_sync(kFull, acc[g][e].x, o);
          other.y = __shfl_xor_sync(kFull, acc[g][e].y, o);
          acc[g][e] = __ffma2_rn(acc[g][e], make_float2(gs[g], gs[g]),
                                 __fmul2_rn(other, make_float2(go[g], go[g])));
        }
    }
    // (2) Merge the 8 warps through shared memory.
    if (rg == 0) {
#pragma unroll
      for (int g = 0; g < G; ++g)
#pragma unroll
        for (int k = 0; k < PPL; ++k)
#pragma unroll
          for (int e = 0; e < PE / 2; ++e)
            *reinterpret_cast<float2 *>(
                &s.red_o[warp][(g ^ hq) * C::RED_PITCH + (sl + k * S) * PE + 2 * e]) = acc[g][k * PE / 2 + e];
      if (sl % C::HL == 0) {
        s.red_m[warp][hq] = m_run;
        s.red_l[warp][hq] = l_run;
      }
    }
    finish_item<Tin, D, G>(p, s, f, tid);
  }
}

// ------------------------------------------------------------ compute warps, bf16
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
// C (16 x 8, fp32) += A (16 x 16) . B (16 x 8), bf16.
__device__ __forceinline__ void mma_16x8x16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                            uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// The high halves of two fp32 values: both cut to bf16.
__device__ __forceinline__ uint32_t high_halves(float x0, float x1) {
  return __byte_perm(__float_as_uint(x0), __float_as_uint(x1), 0x7632);
}
// x less its bf16 part, at least `least`.
__device__ __forceinline__ float below_bf16(float x, float least) {
  return fmaxf(x - __uint_as_float(__float_as_uint(x) & 0xffff0000u), least);
}
// A pair of fp32 values >= 0 as h + m + 2 l, bf16 pairs: 24 bits of each, so
// that products with bf16 values lose nothing against fp32. Each part is cut off,
// not rounded, and m and l are at least the smallest bf16 value, 2^-133: no part
// of a positive probability times an infinite value is a NaN or has the other
// sign (with rounded parts every output of a column with an infinite value was
// NaN), and a finite value v comes out at most 2^-131 |v| too large.
__device__ __forceinline__ void split3(float x0, float x1, uint32_t &h, uint32_t &m, uint32_t &l) {
  h = high_halves(x0, x1);
  const float r0 = below_bf16(x0, 0x1p-133f), r1 = below_bf16(x1, 0x1p-133f);
  m = high_halves(r0, r1);
  l = high_halves(0.5f * below_bf16(r0, 0x1p-132f), 0.5f * below_bf16(r1, 0x1p-132f));
}

// The compute warps of a bf16 step. Per 16 cache rows (two blocks of 8 keys):
//   scores   S[row][key] = Q . K^T, A = the queries (registers), B = keys
//            (ldmatrix); accumulator lane (g, t) holds row g, keys 2t, 2t + 1;
//   softmax  on those lanes, as in the fp32 kernel (lazy maximum per row);
//   output   O[row][dim] += P . V with the probabilities, as they lie, as the
//            A operand and V (ldmatrix.trans) as B. A probability is split
//            into three bf16 parts that fill the operand's 16 rows: 8 heads
//            take rows 0-7 (high parts), 8-15 (middle) and a second MMA (half
//            of the low part on all 16); up to 4 heads repeat in rows 4-7 and
//            take rows 0-3 (high), 4-7 (middle) and 8-15 (half of the low part,
//            twice) of one MMA. No row of a head holds a 0 for a positive
//            probability, which an infinite value would turn into a NaN.
// Matrix instructions cut their sums off rather than round them, so only short
// chains stay in their accumulators (32 dims of a score, 16 rows of an output)
// and the rest is added on the fp32 pipes.
template <int D, int G>
__device__ __forceinline__ void consume_mma(const DecParams &p,
                                            DecSmem<__nv_bfloat16, D, G> &s, int total, int warp,
                                            int lane) {
  using C = DecCfg<__nv_bfloat16, D, G>;
  constexpr bool kWide = G > 4;       // 8 heads: rows 0-7 are heads
  constexpr int NB = D / 8;           // output column blocks
  const int tid = warp * 32 + lane;
  const int g = lane >> 2, t = lane & 3;
  const int head = kWide ? g : g & 3;  // of this lane's rows g and g + 8
  const int row0 = warp * (C::CHUNK_ROWS / 8);  // this warp's first row in a chunk
  // this lane's ldmatrix row in a stage: keys, row row0 (+ block) of chunk
  // lane % 8, piece lane / 8; values, row row0 + (lane / 8) % 2, piece lane / 16
  const uint32_t k_off = (lane & 7) * C::CHUNK_PITCH + row0 * C::ROW_BYTES + (lane >> 3) * 16;
  const uint32_t v_off = (lane & 7) * C::CHUNK_PITCH +
                         (row0 + ((lane >> 3) & 1)) * C::ROW_BYTES + (lane >> 4) * 16;
  uint32_t j = 0;
  for (int icount = 0;; ++icount) {
    const int slot = icount % kItemSlots;
    bool ok = wait_bar(&s.item_full[slot], (icount / kItemSlots) & 1, &s.abort_flag, p);
    ok = __all_sync(kFull, ok);
    const int it = ok ? s.item_id[slot] : total;
    uint32_t qa[D / 16][2];  // A operand, rows g: dims 2t, 2t + 1 and 2t + 8, 2t + 9
#pragma unroll
    for (int k = 0; k < D / 16; ++k) qa[k][0] = qa[k][1] = 0;
    if (it < total && head < G) {
      const uint32_t *q32 = reinterpret_cast<const uint32_t *>(s.qs[slot]) + head * (D / 2) + t;
#pragma unroll
      for (int k = 0; k < D / 16; ++k) {
        qa[k][0] = q32[k * 8];
        qa[k][1] = q32[k * 8 + 4];
      }
    }
    // All compute warps leave together (the item's merge has named barriers);
    // this barrier also frees the merge buffers of the previous item.
    if (compute_bar_or(it >= total || *(volatile int *)&s.abort_flag)) {
      if (lane == 0) mbar_arrive(&s.item_empty[slot]);
      break;
    }
    const ItemInfo f = item_info(p, s, it);
    if (f.full) {
      const size_t qrow = ((size_t)f.layer * p.B + f.b) * p.Hq + (size_t)f.h * G;
      if (lane == 0) mbar_arrive(&s.item_empty[slot]);
      for (int e = tid; e < G * D; e += kWarps * 32)
        p.out[guard(qrow * D + e, 1, (long long)p.L * p.B * p.Hq * D, p.status)] = 0.f;
      continue;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&s.item_empty[slot]);

    // rows g and g + 8 together, dims 8 b + 2t, 8 b + 2t + 1
    float2 acc[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[b] = make_float2(0.f, 0.f);
    float m_run = -INFINITY, l_run = 0.f;  // of this lane's head; the sum over its own keys

    // 16 rows: rows r and r + 1 of every chunk; kMask: some are past nrows.
    auto rows_step = [&](uint32_t kbase, uint32_t vbase, int r, int nrows, auto mask_tag) {
      constexpr bool kMask = decltype(mask_tag)::value;
      float sc[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
      for (int k2 = 0; k2 < D / 32; ++k2) {
        uint32_t kb[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i) ldsm_x4(kbase + i * C::ROW_BYTES + k2 * 64, kb[i]);
        float part[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int e = 0; e < 4; ++e) part[i][e] = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int i = 0; i < 2; ++i)
            mma_16x8x16(part[i], qa[2 * k2 + h][0], 0u, qa[2 * k2 + h][1], 0u, kb[i][2 * h],
                        kb[i][2 * h + 1]);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          sc[i][0] += part[i][0];
          sc[i][1] += part[i][1];
        }
      }
      // this lane's keys: chunk 2t + e, row r + i
      float x[2][2];
      bool live[2][2];
      uint32_t vmask[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        vmask[i] = 0xffffffffu;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          live[i][e] = !kMask || (2 * t + e) * C::CHUNK_ROWS + r + i < nrows;
          x[i][e] = live[i][e] ? sc[i][e] * p.scale2 : -INFINITY;
          if (!live[i][e]) vmask[i] &= e ? 0x0000ffffu : 0xffff0000u;
        }
      }
      const float mb = fmaxf(fmaxf(x[0][0], x[0][1]), fmaxf(x[1][0], x[1][1]));
      if (__any_sync(kFull, mb > m_run + kRescaleLog2)) {
        float mr = fmaxf(mb, __shfl_xor_sync(kFull, mb, 1));
        mr = fmaxf(mr, __shfl_xor_sync(kFull, mr, 2));
        if (mr > m_run + kRescaleLog2) {
          const float a = fast_exp2(m_run - mr);
          l_run *= a;
#pragma unroll
          for (int b = 0; b < NB; ++b) acc[b] = __fmul2_rn(acc[b], make_float2(a, a));
          m_run = mr;
        }
        __syncwarp();
      }
      // a row past the cached ones counts for nothing by its place, not by its
      // score, so that a NaN score of a cached row reaches the output; scores of
      // -infinity alone leave no finite maximum; and the fused multiply-add, which
      // leaves out the rounding of the score, must not meet a maximum whose own
      // rounding is a large part of 1
      const float m_sub = m_run == -INFINITY ? 0.f : m_run;
      const bool rounded = fabsf(m_sub) >= 65536.f;
      uint32_t hi[2], mi[2], lo[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        float pt[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float y = rounded ? x[i][e] - m_sub : fmaf(sc[i][e], p.scale2, -m_sub);
          pt[e] = live[i][e] ? fast_exp2(y) : 0.f;
          l_run += pt[e];
        }
        split3(pt[0], pt[1], hi[i], mi[i], lo[i]);
      }
      uint32_t a0[2], a1[2];  // rows g and g + 8 of the first MMA, key block i
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        a0[i] = kWide || g < 4 ? hi[i] : mi[i];
        a1[i] = kWide ? mi[i] : lo[i];
      }
#pragma unroll
      for (int b2 = 0; b2 < NB / 2; ++b2) {
        uint32_t vb[4];  // key blocks 0, 1 of 8 dims, then of the next 8
        ldsm_x4_trans(vbase + b2 * 32, vb);
        if (kMask) {
#pragma unroll
          for (int e = 0; e < 4; ++e) vb[e] &= vmask[e & 1];
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float part[4] = {0.f, 0.f, 0.f, 0.f};
          if (kWide) mma_16x8x16(part, lo[0], lo[0], lo[1], lo[1], vb[2 * e], vb[2 * e + 1]);
          mma_16x8x16(part, a0[0], a1[0], a0[1], a1[1], vb[2 * e], vb[2 * e + 1]);
          acc[2 * b2 + e] =
              __fadd2_rn(acc[2 * b2 + e], make_float2(part[0] + part[2], part[1] + part[3]));
        }
      }
    };

    const int nsub = (f.rows + C::CR - 1) / C::CR;
    for (int sub = 0; sub < nsub; ++sub, ++j) {
      const int stage = j % C::STAGES;
      wait_bar(&s.full[stage], (j / C::STAGES) & 1, &s.abort_flag, p);
      __syncwarp();
      const int nrows = min(C::CR, f.rows - sub * C::CR);
      const uint32_t kbase = smem_u32(s.kv[stage][0]) + k_off;
      const uint32_t vbase = smem_u32(s.kv[stage][1]) + v_off;
#pragma unroll 1
      for (int pr = 0; pr < C::PAIRS; ++pr) {
        const uint32_t at = pr * 2 * C::ROW_BYTES;
        if (nrows == C::CR)
          rows_step(kbase + at, vbase + at, row0 + 2 * pr, nrows, std::false_type{});
        else if (row0 + 2 * pr < nrows)
          rows_step(kbase + at, vbase + at, row0 + 2 * pr, nrows, std::true_type{});
      }
      if (warp == 0) append_new<__nv_bfloat16, D, G>(p, s, f, sub, stage, lane);
      __syncwarp();
      if (lane == 0) mbar_arrive(&s.empty[stage]);
    }

    // Item end: the row's sum over its four lanes, the parts of each head's
    // output added up, and the warp's partial into the merge buffers.
    l_run += __shfl_xor_sync(kFull, l_run, 1);
    l_run += __shfl_xor_sync(kFull, l_run, 2);
    float2(&o)[NB] = acc;
    if (!kWide) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        o[b].x += __shfl_xor_sync(kFull, o[b].x, 16);
        o[b].y += __shfl_xor_sync(kFull, o[b].y, 16);
      }
    }
    const int buf = warp % C::RED;
    auto to_buffer = [&] {
      if (g < G) {
#pragma unroll
        for (int b = 0; b < NB; ++b)
          *reinterpret_cast<float2 *>(&s.red_o[buf][g * C::RED_PITCH + b * 8 + 2 * t]) = o[b];
        if (t == 0) {
          s.red_m[buf][g] = m_run;
          s.red_l[buf][g] = l_run;
        }
      }
    };
    if constexpr (C::RED < kWarps) {
      // the upper warps' partials first; the lower warps add them to theirs
      if (warp >= C::RED) to_buffer();
      named_bar_sync(1, kWarps * 32);
      if (warp < C::RED) {
        const float mo = s.red_m[buf][g], M = fmaxf(m_run, mo);
        const float as = m_run == -INFINITY ? 0.f : fast_exp2(m_run - M);
        const float ao = mo == -INFINITY ? 0.f : fast_exp2(mo - M);
        l_run = l_run * as + s.red_l[buf][g] * ao;
        m_run = M;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const float2 x =
              *reinterpret_cast<const float2 *>(&s.red_o[buf][g * C::RED_PITCH + b * 8 + 2 * t]);
          o[b].x = o[b].x * as + x.x * ao;
          o[b].y = o[b].y * as + x.y * ao;
        }
        __syncwarp();
        to_buffer();
      }
    } else {
      to_buffer();
    }
    finish_item<__nv_bfloat16, D, G>(p, s, f, tid);
  }
}

// This step's work list from the lengths as they read now, by one warp: lane i
// takes the layers at work-order positions i, i + 32, .. (one load latency for
// all of them; a loop over the layers in one thread paid one per layer).
struct LayerPlan {
  int len[kPlanPerLane];   // -1 = full layer
  int nch[kPlanPerLane];   // items per group
  int base[kPlanPerLane];  // items before this position
  int total;
};

__device__ __forceinline__ LayerPlan plan_layers(const DecParams &p, int lane) {
  LayerPlan w;
#pragma unroll
  for (int i = 0; i < kPlanPerLane; ++i) {
    const int t = i * 32 + lane;
    w.len[i] = t < p.L ? *(const volatile int32_t *)&p.lens[p.order[t]] : -1;
  }
  const int units = p.B * p.Hkv;
  int before = 0;
#pragma unroll
  for (int i = 0; i < kPlanPerLane; ++i) {
    const int t = i * 32 + lane;
    w.nch[i] = w.base[i] = 0;
    if (i * 32 >= p.L) continue;
    if (w.len[i] < 0 || (t < p.L && w.len[i] >= p.cap[p.order[t]])) w.len[i] = -1;
    w.nch[i] = t >= p.L ? 0 : w.len[i] < 0 ? 1 : (w.len[i] + p.item_rows) / p.item_rows;
    int incl = units * w.nch[i];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    w.base[i] = before + incl - units * w.nch[i];
    before += __shfl_sync(kFull, incl, 31);
  }
  w.total = before;
  return w;
}

// Before the previous step has completed: the first sub-chunks of this CTA's
// first item (item blockIdx.x) into L2, from the lengths as they read now
// (one less than this step's if the previous step has not yet advanced
// them; a prefetch is only a hint), so that this step's first loads do not
// start from DRAM after the previous step's tail. One warp.
template <typename Tin, int D, int G>
__device__ __forceinline__ void prefetch_first_item(const DecParams &p, int lane) {
  using C = DecCfg<Tin, D, G>;
  const int units = p.B * p.Hkv;
  const LayerPlan w = plan_layers(p, lane);
#pragma unroll
  for (int i = 0; i < kPlanPerLane; ++i) {
    const int rest = (int)blockIdx.x - w.base[i];
    if (rest < 0 || rest >= units * w.nch[i] || w.len[i] < 0) continue;
    const int l = p.order[i * 32 + lane];
    const int unit = rest / w.nch[i], chunk = rest % w.nch[i];
    const int r0 = chunk * p.item_rows, r1 = min(w.len[i], r0 + p.item_rows);
    const int rows = min(r1 - r0, C::STAGES * C::CR);
    if (rows <= 0) continue;
    const size_t off = guard((long long)unit * p.cap[l] + r0, rows, (long long)units * p.cap[l],
                             p.status) *
                       C::ROW_BYTES;
    bulk_prefetch_l2((const uint8_t *)p.kc[l] + off, (uint32_t)rows * C::ROW_BYTES);
    bulk_prefetch_l2((const uint8_t *)p.vc[l] + off, (uint32_t)rows * C::ROW_BYTES);
  }
}

template <typename Tin, int D, int G>
__global__ void __launch_bounds__(kThreads, 1) decode_kernel(const __grid_constant__ DecParams p) {
  using C = DecCfg<Tin, D, G>;
  extern __shared__ __align__(128) uint8_t smem_raw[];
  DecSmem<Tin, D, G> &s = *reinterpret_cast<DecSmem<Tin, D, G> *>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int units = p.B * p.Hkv;

  // Launched as a programmatic dependent of the previous step: let the next
  // step's CTAs take SMs as this grid's CTAs leave, and wait here until the
  // previous grid has completed and its writes (lengths, appended rows,
  // counters) are visible.
  pdl_launch_dependents();
  if (warp == 0) prefetch_first_item<Tin, D, G>(p, lane);
  if (tid == 32) {
    for (int i = 0; i < C::STAGES; ++i) {
      mbar_init(&s.full[i], 1);
      mbar_init(&s.empty[i], kWarps);
    }
    for (int i = 0; i < kItemSlots; ++i) {
      mbar_init(&s.item_full[i], 1);
      mbar_init(&s.item_empty[i], kWarps);
    }
    s.abort_flag = 0;
    s.init_seen = 0;
    fence_mbar_init();
  }
  pdl_wait();
  // CTA 0 zeroes this call's counters (the workspace may hold anything),
  // then raises the init flag; the other CTAs use no counter before they see
  // it (wait_init).
  const int n_ctrl = (kCtrlGroup - kCtrlItem) + p.L * units;
  if (blockIdx.x == 0)
    for (int i = tid; i < n_ctrl; i += kThreads) p.ctrl[kCtrlItem + i] = 0;
  // Work list of this step from the current lengths (read once, before the last
  // block can advance them: that happens once every CTA has counted itself as
  // arrived, which it does after this).
  if (warp == 0) {
    const LayerPlan w = plan_layers(p, lane);
#pragma unroll
    for (int i = 0; i < kPlanPerLane; ++i) {
      const int t = i * 32 + lane;
      if (t >= p.L) continue;
      s.len[t] = w.len[i];
      s.nch[t] = w.nch[i];
      s.base[t] = w.base[i];
      if (w.len[i] < 0 && blockIdx.x == 0) report(p.status, RIPPLE_EFULL);
    }
    if (lane == 0) s.base[p.L] = w.total;
  }
  __syncthreads();
  if (blockIdx.x == 0 && tid == 0) {
    __threadfence();
    st_release(&p.ctrl[kCtrlFlag], p.epoch);
  }
  const int total = s.base[p.L];

  if (warp == kWarps) {
    produce<Tin, D, G>(p, s, total, lane);
  } else {
    if constexpr (C::kMma)
      consume_mma<D, G>(p, s, total, warp, lane);
    else
      consume<Tin, D, G>(p, s, total, warp, lane);
  }

  // Once every CTA has read the lengths and seen the init flag, the last block
  // (idle, or the lightest, when the items fill one wave) advances the lengths
  // of the layers appended to and lowers the flag (a replay of this launch
  // starts from CTA 0's zeroing again). The others leave at once: an exit
  // counter cost every CTA a fence and an atomic at the end of its critical
  // path. A CTA that never saw the flag (its wait gave up) does not arrive; the
  // call has then reported RIPPLE_ETIMEOUT.
  __syncwarp();
  __syncthreads();
  if (blockIdx.x == gridDim.x - 1 && warp == 0) {
    int all = 0;
    if (lane == 0) {
      const long long t0 = clock64();
      while (!(all = ld_acquire(&p.ctrl[kCtrlFlag]) == p.epoch &&
                     ld_acquire(&p.ctrl[kCtrlArrived]) == (int)gridDim.x)) {
        if (clock64() - t0 > p.wait_cycles) {
          report(p.status, RIPPLE_ETIMEOUT);
          break;
        }
        __nanosleep(32);
      }
    }
    if (__shfl_sync(kFull, all, 0)) {
      for (int t = lane; t < p.L; t += 32)
        if (s.len[t] >= 0) p.lens[p.order[t]] = s.len[t] + 1;
      if (lane == 0) st_release(&p.ctrl[kCtrlFlag], 0);
    }
  }
}

// ------------------------------------------------------------ host side

constexpr int kMaxDevices = 64;

// Per-device caches of the SM count and of the kernels' shared-memory
// attribute; atomics, as several host threads may make their first calls at
// once (a repeated look-up or attribute set is harmless).
int sm_count(int dev) {
  static std::atomic<int> n[kMaxDevices];
  if (dev < 0 || dev >= kMaxDevices) return 1;
  int v = n[dev].load(std::memory_order_relaxed);
  if (v == 0) {
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    v = v > 0 ? v : 1;
    n[dev].store(v, std::memory_order_relaxed);
  }
  return v;
}

template <typename Tin, int D, int G>
cudaError_t launch_g(const DecParams &p, int dev, cudaStream_t st) {
  static std::atomic<bool> attr_set[kMaxDevices];
  const int smem = (int)sizeof(DecSmem<Tin, D, G>);
  static_assert(sizeof(DecSmem<Tin, D, G>) <= 227 * 1024, "shared memory per CTA");
  if (!attr_set[dev].load(std::memory_order_acquire)) {
    const cudaError_t e = cudaFuncSetAttribute(decode_kernel<Tin, D, G>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    attr_set[dev].store(true, std::memory_order_release);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(sm_count(dev));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, decode_kernel<Tin, D, G>, p);
  count_launches(1);
  return e;
}

template <typename Tin, int D>
cudaError_t launch_d(const DecParams &p, int dev, cudaStream_t st) {
  switch (p.G) {
    case 1: return launch_g<Tin, D, 1>(p, dev, st);
    case 2: return launch_g<Tin, D, 2>(p, dev, st);
    case 4: return launch_g<Tin, D, 4>(p, dev, st);
    case 8: return launch_g<Tin, D, 8>(p, dev, st);
    default: return cudaErrorInvalidValue;
  }
}

// Epoch of a call: a per-process sequence (never 0) that starts at a value
// taken from the clock, so that an init flag left in reused memory by an
// earlier call or process is unlikely to match.
int next_epoch() {
  static std::atomic<uint32_t> seq{(uint32_t)std::chrono::steady_clock::now()
                                       .time_since_epoch()
                                       .count() *
                                   2654435761u};
  uint32_t e;
  do {
    e = seq.fetch_add(1, std::memory_order_relaxed) + 1;
  } while (e == 0);
  return (int)e;
}

// Work items of these capacities cut into `rows` cache rows each.
long long items_of(const ripple_decode_desc *d, const int32_t *caps, int rows) {
  long long n = 0;
  for (int l = 0; l < d->n_layers; ++l)
    n += (long long)d->batch * d->n_kv_heads * ((caps[l] + rows - 1) / rows);
  return n;
}

// Cache rows per work item for these capacities: kMaxItemRows when that already
// gives at least one item per SM; otherwise (a single layer's step, short caches)
// items that fit one wave of one CTA per SM, so that no CTA takes two one after
// the other, cut so that the longest group takes the least modelled time: its
// item's bytes at kItemBytesPerNs, plus, when the group has several items, their
// hand-over and combination. Measured on graphs of 32 single-layer steps, 8 groups, 4 heads
// of 128 dims, per step: one item 4.75 us + 6.6 ns a row; items of 128 rows
// 7.5 us for 3 to 7 of them (320 rows: 210 us for the 32 layers as one item, 240
// as three; 576 rows 264 as one, 239 as five).
int item_rows(const ripple_decode_desc *d, const int32_t *caps) {
  int dev = 0;
  cudaGetDevice(&dev);
  const long long sms = sm_count(dev);
  auto items = [&](int rows) { return items_of(d, caps, rows); };
  if (items(kMaxItemRows) >= sms) return kMaxItemRows;
  // the fewest rows whose items fit one wave: items() only falls as they grow,
  // so bisect the steps
  int lo = 0, hi = (kMaxItemRows - kMinItemRows) / kItemRowStep;
  while (lo < hi) {
    const int mid = (lo + hi) / 2;
    if (items(kMinItemRows + mid * kItemRowStep) <= sms) hi = mid; else lo = mid + 1;
  }
  const int least = kMinItemRows + lo * kItemRowStep;
  int longest = 0;
  for (int l = 0; l < d->n_layers; ++l) longest = caps[l] > longest ? caps[l] : longest;
  const int row_bytes = 2 * d->head_dim * (d->dtype == RIPPLE_F32 ? 4 : 2);  // K and V
  int best = kMaxItemRows;
  long long best_ns = -1;
  for (int n = (longest + kMaxItemRows - 1) / kMaxItemRows; ; ++n) {
    int rows = (longest + n - 1) / n;
    rows = (rows + kItemRowStep - 1) / kItemRowStep * kItemRowStep;
    if (rows > kMaxItemRows) rows = kMaxItemRows;
    const bool end = rows <= least;
    if (end) rows = least;
    const int parts = (longest + rows - 1) / rows;
    const long long ns = (long long)rows * row_bytes / kItemBytesPerNs +
                         (parts > 1 ? 2000 + 50 * parts + (parts - 1) / kMaxComb * 900 : 0);
    if (best_ns < 0 || ns < best_ns) {
      best = rows;
      best_ns = ns;
    }
    if (end) break;
  }
  return best;
}

static size_t round_up(size_t x) { return (x + 255) & ~(size_t)255; }

// Workspace layout for these capacities: control block, partial (max, sum),
// partial outputs. Returns the total bytes; fills p's pointers if given. The
// partials are not counted by the items of item_rows, whose number falls where
// some more rows are cut differently (caches of 2048 rows take 16 items a group,
// of 2080 rows 13), but by a bound of them that grows with the layers, the batch
// and every capacity: a workspace made for a program's largest step has to
// serve all smaller ones. It bounds the kernel's items, since a step's lengths
// are at most its capacities.
size_t plan(const ripple_decode_desc *d, const int32_t *caps, void *ws, DecParams *p) {
  const int G = d->n_q_heads / d->n_kv_heads;
  int dev = 0;
  cudaGetDevice(&dev);
  // item_rows cuts into one wave at most, of items of at least kMinItemRows, or
  // into items of kMaxItemRows
  const long long wave = std::min<long long>(items_of(d, caps, kMinItemRows), sm_count(dev));
  const size_t items = (size_t)std::max<long long>(items_of(d, caps, kMaxItemRows), wave);
  const size_t groups = (size_t)d->n_layers * d->batch * d->n_kv_heads;
  const size_t ctrl = round_up(sizeof(int) * (kCtrlGroup + groups));
  const size_t ml = round_up(sizeof(float2) * items * G);
  const size_t o = round_up(sizeof(float) * items * G * d->head_dim);
  if (p != nullptr) {
    uint8_t *base = (uint8_t *)ws;
    p->item_rows = item_rows(d, caps);
    p->ws_items = (long long)items;
    p->n_ctrl = (int)(kCtrlGroup + groups);
    p->ctrl = (int *)base;
    p->ws_ml = (float2 *)(base + ctrl);
    p->ws_o = (float *)(base + ctrl + ml);
  }
  return ctrl + ml + o;
}

bool desc_ok(const ripple_decode_desc *d) {
  if (d == nullptr) return false;
  if (d->n_layers < 1 || d->n_layers > RIPPLE_MAX_LAYERS) return false;
  if (d->batch < 1 || d->n_kv_heads < 1 || d->n_q_heads < 1) return false;
  if (d->n_q_heads % d->n_kv_heads != 0) return false;
  const int G = d->n_q_heads / d->n_kv_heads;
  if (G != 1 && G != 2 && G != 4 && G != 8) return false;
  if (d->head_dim != 64 && d->head_dim != 128) return false;
  if (d->dtype != RIPPLE_F32 && d->dtype != RIPPLE_BF16) return false;
  if (!(d->scale >= 0.f) || isinf(d->scale)) return false;
  if ((int64_t)d->n_layers * d->batch * d->n_kv_heads > (1 << 24)) return false;
  return true;
}

// Shared argument checks and parameter set-up of both decode entry points.
ripple_status prepare(const ripple_decode_desc *desc, const void *q, const void *k_new,
                      const void *v_new, void *const *k_caches_host, void *const *v_caches_host,
                      const int32_t *caps_host, int32_t *lens, float *out, int32_t *dev_status,
                      DecParams *p) {
  if (!desc_ok(desc)) return RIPPLE_EINVAL;
  if (!q || !k_new || !v_new || !k_caches_host || !v_caches_host || !caps_host || !lens || !out)
    return RIPPLE_EINVAL;
  auto aligned = [](const void *ptr) { return ((uintptr_t)ptr & 15u) == 0; };
  if (!aligned(q) || !aligned(k_new) || !aligned(v_new) || !aligned(out)) return RIPPLE_EINVAL;
  const int L = desc->n_layers;
  for (int l = 0; l < L; ++l) {
    if (!k_caches_host[l] || !v_caches_host[l] || caps_host[l] < 1) return RIPPLE_EINVAL;
    if (!aligned(k_caches_host[l]) || !aligned(v_caches_host[l])) return RIPPLE_EINVAL;
    p->kc[l] = k_caches_host[l];
    p->vc[l] = v_caches_host[l];
    p->cap[l] = caps_host[l];
    p->order[l] = l;
  }
  // longest caches first (stable insertion sort, L <= 128)
  for (int i = 1; i < L; ++i) {
    const int v = p->order[i];
    int k = i - 1;
    while (k >= 0 && p->cap[p->order[k]] < p->cap[v]) {
      p->order[k + 1] = p->order[k];
      --k;
    }
    p->order[k + 1] = v;
  }
  p->L = L;
  p->B = desc->batch;
  p->Hq = desc->n_q_heads;
  p->Hkv = desc->n_kv_heads;
  p->G = p->Hq / p->Hkv;
  const float scale = desc->scale > 0.f ? desc->scale : 1.0f / sqrtf((float)desc->head_dim);
  p->scale2 = scale * kLog2e;
  p->q = q;
  p->k_new = k_new;
  p->v_new = v_new;
  p->lens = lens;
  p->out = out;
  p->status = dev_status;
  return RIPPLE_OK;
}

ripple_status run(const ripple_decode_desc *desc, DecParams &p, void *stream) {
  p.epoch = next_epoch();
  p.wait_cycles = wait_limit_cycles();
  // a quarter of the bound's cycles, at 2 GHz half of its time
  p.suspend_ns = (uint32_t)std::min<long long>(p.wait_cycles / 4, kSuspendNs);
  cudaStream_t st = (cudaStream_t)stream;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return RIPPLE_ECUDA;
  cudaError_t e;
  if (desc->dtype == RIPPLE_F32)
    e = desc->head_dim == 64 ? launch_d<float, 64>(p, dev, st) : launch_d<float, 128>(p, dev, st);
  else
    e = desc->head_dim == 64 ? launch_d<__nv_bfloat16, 64>(p, dev, st)
                             : launch_d<__nv_bfloat16, 128>(p, dev, st);
  return e == cudaSuccess ? RIPPLE_OK : RIPPLE_ECUDA;
}

}  // namespace
}  // namespace ripple

using namespace ripple;

extern "C" ripple_status ripple_decode_workspace_bytes(const ripple_decode_desc *desc,
                                                       const int32_t *caps_host,
                                                       size_t *bytes_host) {
  if (!desc_ok(desc) || caps_host == nullptr || bytes_host == nullptr) return RIPPLE_EINVAL;
  for (int l = 0; l < desc->n_layers; ++l)
    if (caps_host[l] < 1) return RIPPLE_EINVAL;
  *bytes_host = plan(desc, caps_host, nullptr, nullptr);
  return RIPPLE_OK;
}

extern "C" ripple_status ripple_decode_attn(const ripple_decode_desc *desc, const void *q,
                                            const void *k_new, const void *v_new,
                                            void *const *k_caches_host,
                                            void *const *v_caches_host,
                                            const int32_t *caps_host, int32_t *lens, float *out,
                                            void *workspace, size_t workspace_bytes,
                                            int32_t *dev_status, void *stream) {
  DecParams p;
  const ripple_status s = prepare(desc, q, k_new, v_new, k_caches_host, v_caches_host,
                                  caps_host, lens, out, dev_status, &p);
  if (s != RIPPLE_OK) return s;
  if (workspace == nullptr || ((uintptr_t)workspace & 255u)) return RIPPLE_EINVAL;
  if (workspace_bytes < plan(desc, caps_host, workspace, &p)) return RIPPLE_EWORKSPACE;
  return run(desc, p, stream);
}

// ---------------------------------------------------------------------------
// Decode for callers that cannot allocate device memory (no paper counterpart).
//
// A plugin inside a host program that owns all device memory through its own
// pool, or a fixed-footprint server that reserves every byte at start-up, may
// have no way to hand this library a scratch buffer. For those callers the
// step's control counters and split-K partials live in the file-scope device
// array below instead of a caller workspace. Every GPU that loads the library
// keeps it until the process exits; all calls on a device share it. Every
// call zeroes the counters it uses before using them, and every partial a call
// reads it has written itself, so no state carries over from the previous call
// (not even from one that ended with RIPPLE_ETIMEOUT). Calls that overlap on
// the GPU race on it.

static __device__ __align__(256) float
    g_decode_scratch[RIPPLE_DECODE_NOALLOC_SCRATCH_BYTES / sizeof(float)];

namespace {

std::mutex g_scratch_mutex;
float *g_scratch_addr[kMaxDevices] = {};

// Device address of g_decode_scratch on the current device. In host code the
// array's name is only a host-side handle, so the address is looked up once
// per device (with that device current) and cached.
ripple_status scratch_on_current_device(float **out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return RIPPLE_ECUDA;
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (g_scratch_addr[dev] == nullptr) {
    void *ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_decode_scratch) != cudaSuccess || ptr == nullptr)
      return RIPPLE_ECUDA;
    g_scratch_addr[dev] = (float *)ptr;
  }
  *out = g_scratch_addr[dev];
  return RIPPLE_OK;
}

}  // namespace

extern "C" ripple_status ripple_decode_attn_noalloc(const ripple_decode_desc *desc, const void *q,
                                                    const void *k_new, const void *v_new,
                                                    void *const *k_caches_host,
                                                    void *const *v_caches_host,
                                                    const int32_t *caps_host, int32_t *lens,
                                                    float *out, int32_t *dev_status,
                                                    void *stream) {
  DecParams p;
  const ripple_status s = prepare(desc, q, k_new, v_new, k_caches_host, v_caches_host,
                                  caps_host, lens, out, dev_status, &p);
  if (s != RIPPLE_OK) return s;
  if (plan(desc, caps_host, nullptr, nullptr) > RIPPLE_DECODE_NOALLOC_SCRATCH_BYTES)
    return RIPPLE_EWORKSPACE;
  float *scratch = nullptr;
  const ripple_status a = scratch_on_current_device(&scratch);
  if (a != RIPPLE_OK) return a;
  plan(desc, caps_host, scratch, &p);
  return run(desc, p, stream);
}
