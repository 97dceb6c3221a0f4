// Observation-window token scoring for up to 128 window rows G * w (SnapKV's
// rule as RippleKV keeps it, Sec. 4.4, last paragraph), bf16, d = 64 or 128, on
// the 5th-generation tensor cores. Row counts other than 32, 64 and 128 are
// padded to the next of them with zero rows that no sum counts.
//
// Bound, 128 rows of d = 128 in large calls (32 units a layer, 32768 keys: 70 us a
// layer): the lock step of the two passes. All CTAs read a pass-1 item from DRAM
// and then a pass-2 item from L2 together, a pattern whose bare stream takes 63 to
// 68 us a layer, and no unit is saturated (DRAM 53% busy, tensor pipe 40%,
// exponentials 41%, issue 39%). Board power, which such calls reach when they run
// for long, costs 3%: 78.9 us a layer with selection at 1942 MHz and 1390 W, 76.7
// in bursts at 2070 MHz. Else the epilogue's arithmetic (about 1350 cycles for 128
// logits a thread, two warps to an SM partition) and, for few rows or d = 64, the
// MMA warp's issue of about 900 cycles a tile. Before these kernels took every bf16
// shape, 16 layers of 16 units, 6007 keys, d = 64
// and 64 rows took 1917 us on the fp32 pipes; 105 us now, with selection.
//
// One persistent CTA per SM, item i on CTA i mod grid; in its step k a CTA
// runs P1(a_k) then P2(a_k-1), so that keys are re-read from L2 one item
// after their first read; a publisher warp merges pass-1 row statistics.
// Each pass takes the layout in which its reduction stays inside one thread:
//   pass 1  D[row][key] = Q . K_tile^T; a thread owns a row and folds its
//           keys into the row's running max and sum;
//   pass 2  D[key][row] = K_tile . Q^T; a thread owns a key and sums its
//           rows' probabilities, so a key's vote needs no shuffles and no
//           exchange between warps.
// Both passes take the queries from shared memory (a buffer of 128 rows per
// pass, loaded by TMA once per item) and the key tile from a 128 KB TMA ring; TMEM
// holds four 128-column accumulators, so the MMA issuer can run two tiles
// ahead of each epilogue warpgroup.
//
// Warp roles (384 threads): warp 0 = key-tile and query producer, warp 1 =
// MMA issuer and TMEM owner, warps 2-9 = two epilogue warpgroups, which take
// alternate tiles (with 128 rows both take every pass-2 tile, half of its rows
// each), warp 10 = publisher of pass-1 results, warp 11 brings in the row
// normalisers of pass-2 items. Every wait is
// bounded; on timeout the CTA raises RIPPLE_ETIMEOUT, every role leaves its
// loop and TMEM is released.
//
// With the window rows' attention output (kO; the scoring fused into the
// prefill attention of the window rows, so that a real prefill reads the keys
// for both in one pass): pass 2 covers every key, causal inside the window;
// the producer streams each value tile behind the next key tile through the
// same ring (three stages); both epilogue warpgroups take every pass-2 tile,
// each for 64 of its 128 window rows, and write those rows' probabilities as
// bf16 into a shared-memory tile (MN-major, the A operand; a key's vote is
// its two halves summed through shared memory), and the MMA warp
// accumulates O[row][dim] += P . V in the last 128 TMEM columns (V, MN-major,
// the B operand). The probabilities are final (pass 1 has fixed every row's
// normaliser), so O needs no rescaling. At an item's end both warpgroups
// write its partial O to the workspace and count it on its unit. kOReduceLag
// steps later the CTA that computed the item sums its slice of the unit's
// output rows (a 1/n_ch share) over the unit's partials in item order (the
// unit's other items are done by then; a bounded wait covers the rest), so
// the sum is deterministic and no CTA holds up the others with a whole
// unit's sum. Bound: HBM, which brings the keys twice and the values once (a
// CTA's item of keys is too large to stay in L2 until its second pass, and
// smaller items pay a step's fixed cost more often): 64 units of 256 tiles,
// 1.61 GB, take 298 us with selection, 5.4 TB/s.
#include <cuda.h>
#include <math.h>

#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"
#include "tc_ptx.cuh"

namespace ripple {
namespace {

constexpr int kTile = 128;                      // keys per tile
constexpr int kHalfBytes = kTile * 64 * 2;      // one TMA box: 64 dims of 128 keys
constexpr int kThreads = 384;
constexpr int kLag = 1;                         // pass 2 of item k runs in step k + kLag
constexpr int kPubSlots = 2;
// Key tiles of an item, at most. Two items a CTA stay in L2 between the passes,
// and a smaller item pays its queries, hand-overs and merge more often: 32
// layers of 8 units and 64 tiles took 273 / 235 / 207 / 201 / 222 / 221 us with
// items of 3 / 4 / 6 / 8 / 12 / 18 tiles; with d = 64 (half the bytes a tile) 16
// layers of 16 units and 47 tiles 149 / 135 / 120 / 117 / 115 / 122 us.
constexpr int kTilesPerItem = 9;
constexpr int kTilesPerItem64 = 12;
// kO: what a step costs on top of its item's tiles, in tiles: the item's
// partial output, its row-slice sum, the hand-overs and the queries. Fitted to
// 64 units of 256 tiles (items of 256 / 128 / 64 / 43 / 37 / 32 / 29 / 19 tiles,
// 1 / 1 / 2 / 3 / 3 / 4 / 4 / 6 steps: 516 / 302 / 321 / 332 / 297 / 343 / 318
// / 331 us, about 2.1 us a tile and 11 us a step).
constexpr int kStepTilesO = 5;
// kO: items of a call, at most (unless it has more units), 64 KB of partial
// outputs each. The workspace is sized for this bound and not for the number a
// call takes, which falls where one more layer or tile fits fewer steps: a
// workspace made for a program's largest call has to serve all smaller ones.
// The model's choices stay within it but for 2% of the (units, tiles) up to 2560
// and 1024, which it costs at most 5%.
constexpr int kMaxItemsO = 2432;
constexpr int kMaxStages = 8;
constexpr int kOReduceLag = 2;  // kO: a step's item rows are summed this many steps later

// With kO (the window rows' attention output as well as the votes) pass 2
// covers every key and also streams the value tiles, multiplies the
// probabilities by them on the tensor cores and accumulates O in TMEM; the
// probabilities go through a 32 KB shared-memory tile, so the ring has one
// stage less, and O takes the last 128 TMEM columns.
// D: head dims (64 or 128). RP: window rows padded to 32, 64 or 128. With
// RP < 128 the pass-1 A operand holds the queries 128 / RP times over, and the
// thread of copy c of a row folds the c-th RP keys of the tile, so that every
// thread has RP exponentials of a tile in both passes and all four SM
// partitions share them (padding the rows to 128 instead left the partitions
// of the padding rows idle). Pass 2 multiplies by the RP rows only.
template <bool kO, int D, int RP>
struct Tc1Cfg {
  static_assert(!kO || (D == 128 && RP == 128), "window-row outputs: 128 rows of 128 dims");
  static constexpr int TileBytes = D / 64 * kHalfBytes;  // 128 keys (or window rows)
  static constexpr int KSteps = D / 16;                  // MMAs per tile
  static constexpr int Copies = 128 / RP;                // of the queries in pass 1
  // ring stages (key tiles; value tiles with kO): 128 KB of keys in flight
  static constexpr int NK = kO ? 3 : 128 / (TileBytes >> 10);
  static constexpr int NA = kO ? 3 : 4;   // S accumulators in TMEM (128 columns each)
  static constexpr uint32_t OCol = NA * 128;  // O accumulator (kO)
  static_assert(NA * 128 + (kO ? 128 : 0) <= 512, "TMEM columns");
  static_assert(NK <= kMaxStages && NA <= kMaxStages, "barrier arrays");
  static_assert(RP == 32 || RP == 64 || RP == 128, "row padding");
};

struct Tc1Params {
  int units, upl, T, P, W, Hq, Hkv, G;  // units of all layers, units per layer
  int R;                   // window rows G * W (at most the kernel's RP)
  int n_tiles1, n_tiles2;  // key tiles of pass 1 (all keys) and pass 2 (prefix keys; all with kO)
  int tpi, n_ch;           // key tiles per item, items per unit
  int total_items;
  // a CTA's next item, gridDim items further on: units, items of a unit, layers
  // and units of a layer
  int d_unit, d_chunk, d_layer, d_local;
  float scale2;
  float *o_win[kCompressMaxLayers];  // kO, per layer: window-row outputs [B][Hq][W][128] fp32
  float *o_part;     // kO: [units][n_ch][128][128] fp32 per-item partial outputs
  int *o_count;      // kO: [units] items of unit u whose partial is written
  float2 *partial;   // [units][n_ch][R] (max, sum) per item and row, log2 domain
  float *lognorm;    // [units][R]
  float *votes;      // [n_slots][upl][P]: unit u's votes at layer_of[u / upl]
  int layer_of[kCompressMaxLayers];  // the layer (votes slot) of each scored layer
  int n_slots;                       // layers (votes slots) of the votes array
  int *ctrl;         // [u] items of unit u published; [units + u] row statistics ready
  int32_t *status;
  long long wait_cycles;  // bound of the in-kernel waits
};

struct ItemRef {
  int unit, chunk;
};

__device__ __forceinline__ ItemRef item_of(const Tc1Params &p, int k) {
  const int i = (int)blockIdx.x + k * (int)gridDim.x;
  return {i / p.n_ch, i % p.n_ch};
}

__device__ __forceinline__ int items_of_cta(const Tc1Params &p) {
  const int b = (int)blockIdx.x;
  return b < p.total_items ? (p.total_items - 1 - b) / (int)gridDim.x + 1 : 0;
}

// Step k of a CTA's schedule: pass 1 of its item k (if k < n), then pass 2
// of its item k - kLag (if k >= kLag). With a lag of one item, an item's keys
// are re-read one item later, so about two items of keys per CTA (78 MB over
// the GPU) stay in L2 and the keys come from DRAM once; a lag of two leaves
// the other CTAs more time to publish the statistics pass 2 waits for, but
// its three items per CTA no longer fit in L2. Measured on 32 layers of the
// 32k-token workload: 2.80 ms with a lag of two against 2.57 ms with one;
// with a lag of two and each step's pass-1 and pass-2 tiles alternating,
// 2.90 / 2.95 / 3.13 / 3.84 ms with items of 9 / 7 / 6 / 5 tiles.

// One item of the CTA's sequence with its layer and its unit's number in the
// layer. Every role steps it along by additions: four divisions a step took
// 900 cycles in each of them.
struct ItemAt {
  int unit, chunk, layer, local;
};

__device__ __forceinline__ ItemAt first_item(const Tc1Params &p) {
  const ItemRef it = item_of(p, 0);
  return {it.unit, it.chunk, it.unit / p.upl, it.unit % p.upl};
}

__device__ __forceinline__ void advance(const Tc1Params &p, ItemAt &it) {
  it.unit += p.d_unit;
  it.layer += p.d_layer;
  it.local += p.d_local;
  it.chunk += p.d_chunk;
  if (it.chunk >= p.n_ch) {
    it.chunk -= p.n_ch;
    ++it.unit;
    ++it.local;
  }
  if (it.local >= p.upl) {  // once: d_local < upl, so local is at most 2 upl - 1 here
    it.local -= p.upl;
    ++it.layer;
  }
}

// Step k: pass 1 of item i1 (tiles a0 .. a0 + n1 - 1) and pass 2 of item i2,
// the one before.
struct Step {
  ItemAt i1, i2;
  int a0, n1;
  int b0, n2;
};

// The steps of a CTA in order: start() gives step 0, next() the one after.
__device__ __forceinline__ Step start(const Tc1Params &p, int n) {
  Step s;
  s.i1 = first_item(p);
  s.i2 = s.i1;
  s.a0 = s.i1.chunk * p.tpi;
  s.n1 = n > 0 ? min(p.tpi, p.n_tiles1 - s.a0) : 0;
  s.b0 = s.n2 = 0;
  return s;
}

__device__ __forceinline__ void next(const Tc1Params &p, Step &s, int k, int n) {
  s.i2 = s.i1;
  s.b0 = s.a0;
  s.n2 = max(0, min(p.tpi, p.n_tiles2 - s.b0));
  advance(p, s.i1);
  s.a0 = s.i1.chunk * p.tpi;
  s.n1 = k + 1 < n ? min(p.tpi, p.n_tiles1 - s.a0) : 0;
}

struct Misc {
  uint64_t k_full[kMaxStages], k_empty[kMaxStages], q_full, q_empty;
  uint64_t acc_full[kMaxStages], acc_empty[kMaxStages];
  uint64_t qs_full, qs_empty;           // pass-2 queries in shared memory
  uint64_t pub_full[kPubSlots], pub_empty[kPubSlots], mma_done;
  // kO: the probability tile (all eight epilogue warps write each tile, the
  // P . V MMA releases it) and the O accumulator
  uint64_t p_full, p_empty, o_full, o_empty;
  float vhalf[2][128];  // kO: warpgroup 1's half of each key's vote, per tile parity
  // votes only: the same in a ring with more entries than accumulators, so that
  // warpgroup 1 (at most an accumulator ring ahead) overwrites none unread
  float vring[kMaxStages][128];
  uint64_t vr_full[kMaxStages];
  uint32_t tmem_base;
  int abort_flag;
  long long wait_cycles;  // bound of the waits of this launch
  float2 pstat[kPubSlots][2][128];      // pass-1 row statistics per slot and warpgroup
  alignas(16) float offs[2][128];       // pass-2 items' row log-normalisers, per step parity
  uint64_t offs_full[2], offs_empty[2];
};

// Shared memory: the ring, the pass-2 and pass-1 queries (two 64-dim halves
// each), with kO the probability tile, then the barriers and statistics.
template <bool kO, int D, int RP>
struct Tc1Smem {
  using C = Tc1Cfg<kO, D, RP>;
  static constexpr int OffQs = C::NK * C::TileBytes;
  static constexpr int OffQ1 = OffQs + C::TileBytes;
  static constexpr int OffP = OffQ1 + C::TileBytes;
  static constexpr int OffMisc = OffP + (kO ? C::TileBytes : 0);
  static constexpr int Bytes = OffMisc + (int)sizeof(Misc) + 1024;  // + alignment slack
  static_assert(Bytes <= 227 * 1024, "shared memory budget");
};

// count arrivals on a barrier at once
__device__ __forceinline__ void mbar_arrive_cnt(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(count)
               : "memory");
}

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

// Kernel argument: the keys (and with kO the values) of every layer as 3-D
// tensor maps [unit][T][D], the window queries of every layer as 2-D maps
// [B * Hq * W][D] (a box is one unit's R rows), and the parameters.
struct Tc1Launch {
  CUtensorMap kmap[kCompressMaxLayers];
  CUtensorMap qmap[kCompressMaxLayers];
  CUtensorMap vmap[kCompressMaxLayers];
  Tc1Params p;
};

// With kO the producer and the MMA warp walk a step's pass 2 as: the item's key
// tiles with value tile s - kPvLag after key tile s (the order the MMA warp
// consumes them in: it multiplies a tile's probabilities by its values after
// issuing the logits kPvLag tiles on, so that the warpgroup that has just
// written a tile's probabilities finds its next tile's logits done), then the
// last value tiles. Position q of the 2 * n2: whether it is a value tile, and
// which tile s.
constexpr int kPvLag = 2;
__device__ __forceinline__ bool ovalue_at(int n2, int q, int &s) {
  const int a = min(n2, kPvLag);           // leading key tiles
  const int pairs = max(0, n2 - kPvLag);   // (key s, value s - kPvLag)
  if (q < a) {
    s = q;
    return false;
  }
  if (q - a < 2 * pairs) {
    const int t = (q - a) >> 1;
    s = (q - a) & 1 ? t : kPvLag + t;
    return (q - a) & 1;
  }
  s = pairs + (q - a - 2 * pairs);
  return true;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&b);
}

// Probabilities of this thread's key for 64 window rows (logit columns
// c0 * 32 .. c0 * 32 + 63 of a pass-2 tile, x = those columns) and their sum
// in a fixed order, also as bf16 pairs (rows 2i, 2i + 1 of the 64 in pk[i]);
// with kMask zero for the rows a window key is hidden from (hidden_below: the
// rows of window position below it; none for a prefix key). A key's vote is
// the sum of its two halves, half 0 + half 1, in every mode. Only the tiles of
// the last keys are masked: one instance for all tiles, with its test at every
// four columns, kept a thread's exponentials from overlapping (64 units of 256
// tiles: 318 us, 297 without).
template <bool kMask>
__device__ __forceinline__ float half_probs(const uint32_t (&x)[2][32], const float4 *o4, int c0,
                                            float scale2, int hidden_below, int W,
                                            uint32_t (&pk)[32]) {
  // fp32x2: logits scaled and shifted two at a time, sums in pairs
  float2 sv[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) sv[i] = make_float2(0.f, 0.f);
  const float2 s2 = make_float2(scale2, scale2);
#pragma unroll
  for (int cc = 0; cc < 2; ++cc)
#pragma unroll
    for (int j4 = 0; j4 < 8; ++j4) {
      const int c = c0 + cc;
      const float4 o = o4[c * 8 + j4];
      const float2 y0 = __ffma2_rn(make_float2(__uint_as_float(x[cc][4 * j4]),
                                               __uint_as_float(x[cc][4 * j4 + 1])),
                                   s2, make_float2(-o.x, -o.y));
      const float2 y1 = __ffma2_rn(make_float2(__uint_as_float(x[cc][4 * j4 + 2]),
                                               __uint_as_float(x[cc][4 * j4 + 3])),
                                   s2, make_float2(-o.z, -o.w));
      float2 e0 = make_float2(fast_exp2(y0.x), fast_exp2(y0.y));
      float2 e1 = make_float2(fast_exp2(y1.x), fast_exp2(y1.y));
      if constexpr (kMask) {
        const int col = c * 32 + 4 * j4;  // window row of e0.x
        if ((col + 0) % W < hidden_below) e0.x = 0.f;
        if ((col + 1) % W < hidden_below) e0.y = 0.f;
        if ((col + 2) % W < hidden_below) e1.x = 0.f;
        if ((col + 3) % W < hidden_below) e1.y = 0.f;
      }
      pk[(cc * 32 + 4 * j4) >> 1] = pack_bf16x2(e0.x, e0.y);
      pk[((cc * 32 + 4 * j4) >> 1) + 1] = pack_bf16x2(e1.x, e1.y);
      sv[(2 * j4) & 3] = __fadd2_rn(sv[(2 * j4) & 3], e0);
      sv[(2 * j4 + 1) & 3] = __fadd2_rn(sv[(2 * j4 + 1) & 3], e1);
    }
  return ((sv[0].x + sv[0].y) + (sv[1].x + sv[1].y)) + ((sv[2].x + sv[2].y) + (sv[3].x + sv[3].y));
}

// Half h (window rows 64h .. 64h + 63) of one key's probabilities (this
// thread's TMEM lane), as bf16 pairs (rows 2i and 2i + 1 of the half in
// pk[i]), into the shared-memory tile in the MN-major, 128-byte-swizzled
// layout the tensor core reads as the A operand of O = P . V: rows 0-63 and
// 64-127 in two 16 KB halves, in each the key's 128-byte line holds its 64
// rows, 16-byte chunk c at position c ^ (key mod 8).
__device__ __forceinline__ void store_p_half(uint8_t *ptile, int key, int h,
                                             const uint32_t (&pk)[32]) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int w = c * 4;  // rows 8c .. 8c + 7 of the half
    uint8_t *dst = ptile + h * kHalfBytes + (key >> 3) * 1024 + (key & 7) * 128 +
                   ((c ^ (key & 7)) << 4);
    *reinterpret_cast<uint4 *>(dst) = make_uint4(pk[w], pk[w + 1], pk[w + 2], pk[w + 3]);
  }
}

// kO: the output rows of item `it`'s slice of its unit (rows chunk * 128 /
// n_ch up to the next chunk's), summed over the unit's item partials in item
// order, once every item of the unit has written its partial (bounded wait).
// Run by both epilogue warpgroups (256 threads, named barrier 5).
__device__ __forceinline__ void reduce_rows(const Tc1Params &p, Misc *ms, const ItemRef &it,
                                            int tid) {
  if (tid == 0) {
    const int *cnt = &p.o_count[guard(it.unit, 1, p.units, p.status)];
    const long long t0 = clock64();
    while (ld_acquire(cnt) < p.n_ch) {
      if (*(volatile int *)&ms->abort_flag) break;
      if (clock64() - t0 > ms->wait_cycles) {
        *(volatile int *)&ms->abort_flag = 1;
        report(p.status, RIPPLE_ETIMEOUT);
        break;
      }
      __nanosleep(64);
    }
  }
  named_bar_sync(5, 256);
  const int r0 = it.chunk * 128 / p.n_ch, r1 = (it.chunk + 1) * 128 / p.n_ch;
  const int layer = it.unit / p.upl, local = it.unit % p.upl;
  const int b = local / p.Hkv, h = local % p.Hkv;
  const long long orow0 = (long long)(b * p.Hq + h * p.G) * p.W;
  const size_t ubase = (size_t)it.unit * p.n_ch * 128;
  // 32 float4 per row; consecutive threads take consecutive float4, the partials
  // eight at a time so that their loads overlap (64 units of 7 items: 321 us one
  // by one, 318 so)
  for (int e = tid; e < (r1 - r0) * 32; e += 256) {
    const int row = r0 + (e >> 5), q4 = e & 31;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c0 = 0; c0 < p.n_ch; c0 += 8) {
      float4 v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        v[i] = __ldcg(reinterpret_cast<const float4 *>(
                          p.o_part + (ubase + (size_t)min(c0 + i, p.n_ch - 1) * 128 + row) * 128) +
                      q4);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (c0 + i < p.n_ch) {
          acc.x += v[i].x;
          acc.y += v[i].y;
          acc.z += v[i].z;
          acc.w += v[i].w;
        }
    }
    reinterpret_cast<float4 *>(
        p.o_win[layer] + guard((orow0 + row) * 128, 128,
                               (long long)p.upl / p.Hkv * p.Hq * p.W * 128, p.status))[q4] = acc;
  }
}

// kPad: R < RP (some rows are padding; R = RP otherwise).
template <bool kO, int D, int RP, bool kPad>
__global__ void __launch_bounds__(kThreads, 1)
    score_tc1_kernel(const __grid_constant__ Tc1Launch lp) {
  using C = Tc1Cfg<kO, D, RP>;
  using SM = Tc1Smem<kO, D, RP>;
  constexpr int kTileBytes = C::TileBytes;
  // 128 rows: both epilogue warpgroups take every pass-2 tile, each for 64 of
  // its rows, whose normalisers a thread keeps in registers for the item. With a
  // tile to a warpgroup every tile reads all of them from shared memory, which cost
  // 2% (32 layers of 32 units and 32768 keys 2624 -> 2570 us). Not with padding
  // rows, which would leave one warpgroup short of work (96 rows: 112 -> 115 us).
  constexpr bool kSplit = RP == 128 && !kPad;
  const Tc1Params &p = lp.p;
  const int R = kPad ? p.R : RP;  // window rows
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t *ktiles = smem;
  uint8_t *qsm = smem + SM::OffQs;
  uint8_t *q1m = smem + SM::OffQ1;
  uint8_t *ptile = smem + SM::OffP;
  Misc *ms = (Misc *)(smem + SM::OffMisc);
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
      // kSplit (and kO): pass-2 tiles are released by all eight epilogue warps,
      // pass-1 tiles by the four of their warpgroup with two arrivals each
      mbar_init(&ms->acc_empty[i], kSplit ? 8 : 4);
    }
    mbar_init(&ms->qs_full, 1);
    mbar_init(&ms->qs_empty, 1);
    for (int i = 0; i < kPubSlots; ++i) {
      mbar_init(&ms->pub_full[i], 8);
      mbar_init(&ms->pub_empty[i], 1);
    }
    for (int i = 0; i < kMaxStages; ++i) mbar_init(&ms->vr_full[i], 4);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&ms->offs_full[i], 1);
      mbar_init(&ms->offs_empty[i], 8);
    }
    mbar_init(&ms->mma_done, 1);
    mbar_init(&ms->p_full, 8);
    mbar_init(&ms->p_empty, 1);
    mbar_init(&ms->o_full, 1);
    mbar_init(&ms->o_empty, 8);
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
    for (int i = threadIdx.x; i < 2 * kTileBytes / 16; i += kThreads)
      reinterpret_cast<uint4 *>(qsm)[i] = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ms->tmem_base;

  // Every role walks the same sequence of steps k = 0 .. n + kLag - 1.
  if (warp == 0) {
    // ------------------------------------------------ key-tile producer
    if (lane == 0) {
      int kcount = 0, qcount = 0, q1count = 0;
      const uint64_t keep = policy_evict_last(), drop = policy_evict_first();
      bool ok = true;
      // one tile of keys (or values) into the ring
      auto load_tile = [&](const CUtensorMap *map, int tile, int local, uint64_t pol) {
        const int ks = kcount % C::NK;
        if (!wait_bar(&ms->k_empty[ks], ((kcount / C::NK) & 1) ^ 1, ms, p.status)) return false;
        mbar_arrive_expect_tx(&ms->k_full[ks], kTileBytes);
        uint8_t *kb = ktiles + ks * kTileBytes;
#pragma unroll
        for (int half = 0; half < D / 64; ++half)
          tma_load_3d(kb + half * kHalfBytes, map, half * 64, tile * kTile, local,
                      &ms->k_full[ks], pol);
        ++kcount;
        return true;
      };
      Step st = start(p, n);
      for (int k = 0; k < n + kLag && ok; next(p, st, k, n), ++k) {
        if (st.n1 > 0) {
          // item k's queries into the pass-1 buffer, once the previous item's
          // pass-1 MMAs have read it
          if (!wait_bar(&ms->q_empty, (k & 1) ^ 1, ms, p.status)) break;
          mbar_arrive_expect_tx(&ms->q_full, (uint32_t)(C::Copies * R * D * 2));
#pragma unroll
          for (int i = 0; i < C::Copies * (D / 64); ++i) {
            const int half = i % (D / 64), copy = i / (D / 64);
            tma_load_2d(q1m + half * kHalfBytes + copy * RP * 128, &lp.qmap[st.i1.layer],
                        half * 64, st.i1.local * R, &ms->q_full);
          }
          ++q1count;
          for (int s = 0; s < st.n1 && ok; ++s)
            ok = load_tile(&lp.kmap[st.i1.layer], st.a0 + s, st.i1.local, keep);
        }
        if (ok && st.n2 > 0) {
          // the pass-2 item's queries (rows of its unit) into shared memory
          if (!wait_bar(&ms->qs_empty, (qcount & 1) ^ 1, ms, p.status)) break;
          mbar_arrive_expect_tx(&ms->qs_full, (uint32_t)(R * D * 2));
#pragma unroll
          for (int half = 0; half < D / 64; ++half)
            tma_load_2d(qsm + half * kHalfBytes, &lp.qmap[st.i2.layer], half * 64,
                        st.i2.local * R, &ms->qs_full);
          ++qcount;
          for (int j = 0; j < (kO ? 2 : 1) * st.n2 && ok; ++j) {
            int s = j;
            const bool value = kO && ovalue_at(st.n2, j, s);
            const CUtensorMap *map = value ? &lp.vmap[st.i2.layer] : &lp.kmap[st.i2.layer];
            ok = load_tile(map, st.b0 + s, st.i2.local, drop);
          }
        }
      }
      for (int j = max(0, kcount - C::NK); j < kcount; ++j)
        mbar_wait(&ms->k_full[j % C::NK], (j / C::NK) & 1, nullptr);
      if (qcount > 0) mbar_wait(&ms->qs_full, (qcount - 1) & 1, nullptr);
      if (q1count > 0) mbar_wait(&ms->q_full, (q1count - 1) & 1, nullptr);
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer (the whole warp
    // runs the loop and waits; one elected lane issues)
    {
      int kcount = 0, acount = 0, qcount = 0, ocount = 0;
      int pv_count = 0;  // kO: probability tiles multiplied
      constexpr uint32_t id1 = idesc_bf16(128, 128);   // rows (all copies) x keys
      constexpr uint32_t id2 = idesc_bf16(128, RP);    // keys x rows
      // O = P . V: P (rows x keys) and V (keys x dims) both MN-major
      constexpr uint32_t id_pv = idesc_bf16(128, 128) | (1u << 15) | (1u << 16);
      const uint32_t kbase = smem_u32(ktiles), qsbase = smem_u32(qsm), q1base = smem_u32(q1m);
      const uint32_t pbase = smem_u32(ptile);
      const uint64_t q1d = sw128_desc(q1base), qsd = sw128_desc(qsbase);
      bool ok = true;
      // logits of one key tile: D = A . B^T, A and B the first K step's
      // descriptors (the others differ only in their start-address field, in
      // 16-byte units, without carry)
      auto logits = [&](bool pass1, bool last) {
        const int ks = kcount % C::NK, as = acount % C::NA;
        if (!warp_wait(&ms->k_full[ks], (kcount / C::NK) & 1, ms, p.status) ||
            !warp_wait(&ms->acc_empty[as], ((acount / C::NA) & 1) ^ 1, ms, p.status))
          return false;
        tc_fence_after();
        const uint32_t d = tmem + as * 128;
        const uint64_t kd = sw128_desc(kbase + ks * kTileBytes);
        const uint64_t ad = pass1 ? q1d : kd, bd = pass1 ? kd : qsd;
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < C::KSteps; ++kk) {
            const uint64_t off = (uint64_t)(((kk >> 2) * kHalfBytes + (kk & 3) * 32) >> 4);
            mma_bf16(d, ad + off, bd + off, pass1 ? id1 : id2, kk > 0);
          }
          mma_commit(&ms->k_empty[ks]);
          mma_commit(&ms->acc_full[as]);
          if (last) mma_commit(pass1 ? &ms->q_empty : &ms->qs_empty);  // its queries are free
        }
        __syncwarp();
        ++kcount;
        ++acount;
        return true;
      };
      Step st = start(p, n);
      for (int k = 0; k < n + kLag && ok; next(p, st, k, n), ++k) {
        if (st.n1 > 0 && !warp_wait(&ms->q_full, k & 1, ms, p.status)) break;
        for (int s = 0; s < st.n1 && ok; ++s) ok = logits(true, s == st.n1 - 1);
        if (!ok || st.n2 == 0) continue;
        if (!warp_wait(&ms->qs_full, qcount & 1, ms, p.status)) break;
        if constexpr (!kO) {
          for (int s = 0; s < st.n2 && ok; ++s) ok = logits(false, s == st.n2 - 1);
        } else {
          for (int j = 0; j < 2 * st.n2 && ok; ++j) {
            int s;
            if (!ovalue_at(st.n2, j, s)) {
              ok = logits(false, s == st.n2 - 1);
              continue;
            }
            // O (+)= P . V for pass-2 tile s, once the epilogue has written
            // its probabilities (and, for the item's first tile, has read
            // out the previous item's O)
            const int ks = kcount % C::NK;
            if ((s == 0 && !warp_wait(&ms->o_empty, (ocount & 1) ^ 1, ms, p.status)) ||
                !warp_wait(&ms->p_full, pv_count & 1, ms, p.status) ||
                !warp_wait(&ms->k_full[ks], (kcount / C::NK) & 1, ms, p.status)) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (elect_one()) {
              // K step kk: 16 keys further along both MN-major operands
              const uint64_t pd = sw128_desc_mn(pbase, kHalfBytes, 1024);
              const uint64_t vd = sw128_desc_mn(kbase + ks * kTileBytes, kHalfBytes, 1024);
#pragma unroll
              for (int kk = 0; kk < 8; ++kk) {
                const uint64_t step = (uint64_t)(kk * 2048 >> 4);
                mma_bf16(tmem + C::OCol, pd + step, vd + step, id_pv, kk > 0 || s > 0);
              }
              mma_commit(&ms->k_empty[ks]);
              mma_commit(&ms->p_empty);
              if (s == st.n2 - 1) mma_commit(&ms->o_full);
            }
            __syncwarp();
            ++kcount;
            ++pv_count;
            if (s == st.n2 - 1) ++ocount;
          }
        }
        ++qcount;
      }
      if (elect_one()) mma_commit(&ms->mma_done);
      __syncwarp();
      mbar_wait(&ms->mma_done, 0, nullptr);
    }
  } else if (warp == 10) {
    // ------------------------------------------------ publisher of pass-1 results
    ItemAt it = first_item(p);
    for (int k = 0; k < n; advance(p, it), ++k) {
      const int slot = k % kPubSlots;
      if (!warp_wait(&ms->pub_full[slot], (k / kPubSlots) & 1, ms, p.status)) break;
      float2 *mine = p.partial + guard((long long)it.unit * p.n_ch + it.chunk, 1,
                                       (long long)p.units * p.n_ch, p.status) *
                                     R;
#pragma unroll
      for (int j = 0; j < RP / 32; ++j) {
        const int r = lane + 32 * j;
        float2 a = ms->pstat[slot][0][r];
        const float2 b = ms->pstat[slot][1][r];
        combine(a.x, a.y, b.x, b.y);
#pragma unroll
        for (int c = 1; c < C::Copies; ++c)
#pragma unroll
          for (int w = 0; w < 2; ++w) {
            const float2 x = ms->pstat[slot][w][c * RP + r];
            combine(a.x, a.y, x.x, x.y);
          }
        if (r < R) mine[r] = a;
      }
      __syncwarp();
      int last = 0;
      if (lane == 0) {
        mbar_arrive(&ms->pub_empty[slot]);
        __threadfence();
        last = atomicAdd(&p.ctrl[guard(it.unit, 1, p.units, p.status)], 1) == p.n_ch - 1;
      }
      last = __shfl_sync(0xffffffffu, last, 0);
      if (last) {
        __threadfence();
        const float2 *part =
            p.partial + guard((long long)it.unit * p.n_ch, p.n_ch, (long long)p.units * p.n_ch,
                              p.status) *
                            R;
        constexpr int RJ = RP / 32;   // rows per lane
        constexpr int CB = 32 / RJ;   // items per batch: 32 loads of a lane in flight
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
  } else if (warp == 11) {
    // ------------------------------------------------ normalisers of pass-2 items:
    // waits for the unit's row statistics and brings them in, so that the
    // epilogue meets neither the flag's latency nor the loads' (3000 cycles
    // an item)
    Step st = start(p, n);
    int count = 0;
    for (int k = 0; k < n + kLag; next(p, st, k, n), ++k) {
      if (st.n2 == 0) continue;
      const int b = count & 1;
      if (!warp_wait(&ms->offs_empty[b], ((count >> 1) & 1) ^ 1, ms, p.status)) break;
      int ok = 1;
      if (lane == 0)
        ok = wait_ready(&p.ctrl[guard(p.units + st.i2.unit, 1, 2LL * p.units, p.status)], ms,
                        p.status);
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      __syncwarp();  // lane 0's acquire orders every lane's loads
      const float *ln = p.lognorm + guard(st.i2.unit, 1, p.units, p.status) * R;
#pragma unroll
      for (int r = 0; r < RP / 32; ++r)
        if (!kPad || lane + 32 * r < R) ms->offs[b][lane + 32 * r] = __ldcg(ln + lane + 32 * r);
      __syncwarp();
      if (lane == 0) mbar_arrive(&ms->offs_full[b]);
      ++count;
    }
  } else {
    // ------------------------------------------------ epilogue warpgroups
    const int wg = (warp - 2) >> 2;
    const int quarter = warp & 3;              // TMEM lanes this warp may access
    const int r = quarter * 32 + lane;         // TMEM lane of this thread
    const int row = r % RP;                    // pass 1: its window row,
    const int col0 = r / RP * RP;              //   and its first key column
    const bool live1 = !kPad || quarter * 32 % RP < R;  // the warp has rows that are not padding
    const int wtid = threadIdx.x - 64 - wg * 128;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    int tcount = 0;  // tiles seen
    int oc = 0;            // kO: pass-2 items seen
    int ptc = 0;           // kO: probability tiles written
    int ocount = 0;        // pass-2 items seen

    // Inside an item every warp follows the same control flow even if a wait
    // gives up (the tile is then skipped), so that the named barriers below
    // are always reached by all of their threads.
    Step st = start(p, n);
    for (int k = 0; k < n + kLag; next(p, st, k, n), ++k) {
      float m = -INFINITY, l = 0.f;    // pass 1 of item k: this row's max and sum
      const int last_vis = p.P + row % p.W;
      // ---------------- this warpgroup's pass-1 tiles of item k: every other one
      // of the CTA's tiles, so that it meets every phase of its accumulators
      for (int s = (tcount ^ wg) & 1; s < st.n1; s += 2) {
        const int as = (tcount + s) % C::NA, ph = ((tcount + s) / C::NA) & 1;
        if (warp_wait(&ms->acc_full[as], ph, ms, p.status)) {
          tc_fence_after();
          const int t = st.a0 + s;
          uint32_t x[RP / 32][32];
#pragma unroll
          for (int c = 0; c < RP / 32; ++c)
            tmem_ld32(tmem + lane_addr + as * 128 + (C::Copies > 1 ? col0 : 0) + c * 32, x[c]);
          tmem_wait_ld();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cnt(&ms->acc_empty[as], kSplit ? 2 : 1);
          const int key0 = t * kTile + (C::Copies > 1 ? col0 : 0);  // this thread's first key
          if ((t + 1) * kTile - 1 >= p.P) {  // keys this row cannot see -> -inf
#pragma unroll
            for (int c = 0; c < RP / 32; ++c)
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (key0 + c * 32 + j > last_vis) x[c][j] = 0xff800000u;
          }
          float mx[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) mx[i] = -INFINITY;
#pragma unroll
          for (int c = 0; c < RP / 32; ++c)
#pragma unroll
            for (int j = 0; j < 32; ++j) mx[j & 7] = fmaxf(mx[j & 7], __uint_as_float(x[c][j]));
          const float tmax = fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])),
                                   fmaxf(fmaxf(mx[4], mx[5]), fmaxf(mx[6], mx[7])));
          if (live1 && tmax != -INFINITY) {
            const float mnew = fmaxf(m, tmax * p.scale2);
            // fp32x2: logits scaled and shifted two at a time, sums in pairs
            float2 sv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) sv[i] = make_float2(0.f, 0.f);
            const float2 s2 = make_float2(p.scale2, p.scale2), mn2 = make_float2(-mnew, -mnew);
#pragma unroll
            for (int c = 0; c < RP / 32; ++c)
#pragma unroll
              for (int j = 0; j < 32; j += 2) {
                const float2 y = __ffma2_rn(
                    make_float2(__uint_as_float(x[c][j]), __uint_as_float(x[c][j + 1])), s2, mn2);
                sv[(j >> 1) & 3] =
                    __fadd2_rn(sv[(j >> 1) & 3], make_float2(fast_exp2(y.x), fast_exp2(y.y)));
              }
            const float sum = ((sv[0].x + sv[0].y) + (sv[1].x + sv[1].y)) +
                              ((sv[2].x + sv[2].y) + (sv[3].x + sv[3].y));
            l = l * fast_exp2(m - mnew) + sum;
            m = mnew;
          }
        }
      }
      tcount += st.n1;
      if (st.n1 > 0) {
        // This warpgroup's row statistics go to the publisher now, ahead of
        // the step's pass-2 tiles.
        const int slot = k % kPubSlots;
        warp_wait(&ms->pub_empty[slot], ((k / kPubSlots) & 1) ^ 1, ms, p.status);
        ms->pstat[slot][wg][r] = make_float2(m, l);
        __syncwarp();
        if (lane == 0) mbar_arrive(&ms->pub_full[slot]);
      }
      // ---------------- pass 2 of item k - kLag: votes of its keys
      // (D[key][row]: this thread's TMEM lane is key (b0 + s) * 128 + r)
      if (st.n2 > 0) {
        const int ob = ocount & 1;
        warp_wait(&ms->offs_full[ob], (ocount >> 1) & 1, ms, p.status);
        // votes of the unit: its layer's slot of the vote array
        const long long vote0 =
            (long long)(p.layer_of[st.i2.layer] * p.upl + st.i2.local) * p.P;
        if constexpr (kO) {
          for (int s = 0; s < st.n2; ++s) {
            const int key = (st.b0 + s) * kTile + r;
            const int as = (tcount + s) % C::NA, ph = ((tcount + s) / C::NA) & 1;
            // both warpgroups take every pass-2 tile, each for 64 of its 128
            // window rows (logit columns 64 wg ..): its half of the key's
            // probabilities, half of the vote (summed over the warpgroups
            // through shared memory) and its half of the probability tile
            const bool got = warp_wait(&ms->acc_full[as], ph, ms, p.status);
            float half = 0.f;
            if (got) {
              tc_fence_after();
              uint32_t x[2][32];
              tmem_ld32(tmem + lane_addr + as * 128 + wg * 64, x[0]);
              tmem_ld32(tmem + lane_addr + as * 128 + wg * 64 + 32, x[1]);
              tmem_wait_ld();
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&ms->acc_empty[as]);
              // a window key (or a key past the end) is seen only by the rows
              // at or after it (causal inside the window)
              uint32_t pk[32];
              const float4 *o4 = reinterpret_cast<const float4 *>(ms->offs[ob]);
              if ((st.b0 + s + 1) * kTile > p.P)
                half = half_probs<true>(x, o4, 2 * wg, p.scale2, key - p.P, p.W, pk);
              else
                half = half_probs<false>(x, o4, 2 * wg, p.scale2, 0, p.W, pk);
              // into the tile once the previous tile's probabilities have
              // been multiplied
              if (ptc > 0) warp_wait(&ms->p_empty, (ptc - 1) & 1, ms, p.status);
              store_p_half(ptile, r, wg, pk);
              fence_proxy_async_smem();
              __syncwarp();
              if (lane == 0) mbar_arrive(&ms->p_full);
            }
            if (wg == 1) ms->vhalf[ptc & 1][r] = half;
            named_bar_sync(6, 256);
            if (wg == 0 && got && key < p.P)
              p.votes[guard(vote0 + key, 1, (long long)p.n_slots * p.upl * p.P, p.status)] =
                  half + ms->vhalf[ptc & 1][r];
            ++ptc;
          }
        } else if constexpr (kSplit) {
          float o[64];
          const float4 *o4 = reinterpret_cast<const float4 *>(ms->offs[ob]) + wg * 16;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float4 v4 = o4[i];
            o[4 * i] = v4.x;
            o[4 * i + 1] = v4.y;
            o[4 * i + 2] = v4.z;
            o[4 * i + 3] = v4.w;
          }
          for (int s = 0; s < st.n2; ++s) {
            const int as = (tcount + s) % C::NA, ph = ((tcount + s) / C::NA) & 1;
            const bool got = warp_wait(&ms->acc_full[as], ph, ms, p.status);
            float half = 0.f;
            if (got) {
              tc_fence_after();
              uint32_t x[2][32];
              tmem_ld32(tmem + lane_addr + as * 128 + wg * 64, x[0]);
              tmem_ld32(tmem + lane_addr + as * 128 + wg * 64 + 32, x[1]);
              tmem_wait_ld();
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&ms->acc_empty[as]);
              // this half's sum as half_probs forms it
              float2 sv[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) sv[i] = make_float2(0.f, 0.f);
              const float2 s2 = make_float2(p.scale2, p.scale2);
#pragma unroll
              for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int j = 0; j < 32; j += 2) {
                  const float2 y = __ffma2_rn(
                      make_float2(__uint_as_float(x[c][j]), __uint_as_float(x[c][j + 1])), s2,
                      make_float2(-o[c * 32 + j], -o[c * 32 + j + 1]));
                  sv[(j >> 1) & 3] =
                      __fadd2_rn(sv[(j >> 1) & 3], make_float2(fast_exp2(y.x), fast_exp2(y.y)));
                }
              half = ((sv[0].x + sv[0].y) + (sv[1].x + sv[1].y)) +
                     ((sv[2].x + sv[2].y) + (sv[3].x + sv[3].y));
            }
            const int vs = ptc % kMaxStages;
            if (wg == 1) {
              ms->vring[vs][r] = half;
              __syncwarp();
              if (lane == 0) mbar_arrive(&ms->vr_full[vs]);
            } else {
              warp_wait(&ms->vr_full[vs], (ptc / kMaxStages) & 1, ms, p.status);
              const int key = (st.b0 + s) * kTile + r;
              if (got && key < p.P)
                p.votes[guard(vote0 + key, 1, (long long)p.n_slots * p.upl * p.P, p.status)] =
                    half + ms->vring[vs][r];
            }
            ++ptc;
          }
        } else {
          for (int s = (tcount ^ wg) & 1; s < st.n2; s += 2) {
            const int as = (tcount + s) % C::NA, ph = ((tcount + s) / C::NA) & 1;
            if (!warp_wait(&ms->acc_full[as], ph, ms, p.status)) continue;
            tc_fence_after();
            uint32_t x[RP / 32][32];
#pragma unroll
            for (int c = 0; c < RP / 32; ++c)
              tmem_ld32(tmem + lane_addr + as * 128 + c * 32, x[c]);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&ms->acc_empty[as]);
            const float4 *o4 = reinterpret_cast<const float4 *>(ms->offs[ob]);
            // the two halves' sums as half_probs forms them, in one pass
            float2 sv[2][4];
#pragma unroll
            for (int i = 0; i < 8; ++i) sv[i >> 2][i & 3] = make_float2(0.f, 0.f);
            const float2 s2 = make_float2(p.scale2, p.scale2);
            auto columns = [&](int c, auto some_padding) {
              float2 *h = sv[c >> 1];
#pragma unroll
              for (int j4 = 0; j4 < 8; ++j4) {
                const float4 o = o4[c * 8 + j4];
                const float2 y0 = __ffma2_rn(make_float2(__uint_as_float(x[c][4 * j4]),
                                                         __uint_as_float(x[c][4 * j4 + 1])),
                                             s2, make_float2(-o.x, -o.y));
                const float2 y1 = __ffma2_rn(make_float2(__uint_as_float(x[c][4 * j4 + 2]),
                                                         __uint_as_float(x[c][4 * j4 + 3])),
                                             s2, make_float2(-o.z, -o.w));
                float2 e0 = make_float2(fast_exp2(y0.x), fast_exp2(y0.y));
                float2 e1 = make_float2(fast_exp2(y1.x), fast_exp2(y1.y));
                if constexpr (decltype(some_padding)::value) {
                  const int left = R - (c * 32 + 4 * j4);  // rows from this column on
                  if (left < 1) e0.x = 0.f;
                  if (left < 2) e0.y = 0.f;
                  if (left < 3) e1.x = 0.f;
                  if (left < 4) e1.y = 0.f;
                }
                h[(2 * j4) & 3] = __fadd2_rn(h[(2 * j4) & 3], e0);
                h[(2 * j4 + 1) & 3] = __fadd2_rn(h[(2 * j4 + 1) & 3], e1);
              }
            };
#pragma unroll
            for (int c = 0; c < RP / 32; ++c) {
              if (!kPad || (c + 1) * 32 <= R)
                columns(c, std::false_type{});
              else if (c * 32 < R)
                columns(c, std::true_type{});
            }
            const float h0 = ((sv[0][0].x + sv[0][0].y) + (sv[0][1].x + sv[0][1].y)) +
                             ((sv[0][2].x + sv[0][2].y) + (sv[0][3].x + sv[0][3].y));
            const float h1 = ((sv[1][0].x + sv[1][0].y) + (sv[1][1].x + sv[1][1].y)) +
                             ((sv[1][2].x + sv[1][2].y) + (sv[1][3].x + sv[1][3].y));
            const int key = (st.b0 + s) * kTile + r;
            if (key < p.P)
              p.votes[guard(vote0 + key, 1, (long long)p.n_slots * p.upl * p.P, p.status)] =
                  h0 + h1;
          }
        }
        tcount += st.n2;
        __syncwarp();
        if (lane == 0) mbar_arrive(&ms->offs_empty[ob]);
        ++ocount;
      }
      if (kO && st.n2 > 0) {
        // ---------------- kO: item k - kLag's partial O (both warpgroups:
        // this thread's row, warpgroup wg's 64 dims)
        const ItemAt &it = st.i2;
        const size_t prow = ((size_t)it.unit * p.n_ch + it.chunk) * 128 + r;
        if (warp_wait(&ms->o_full, oc & 1, ms, p.status)) {
          tc_fence_after();
          uint32_t x[2][32];
          tmem_ld32(tmem + lane_addr + C::OCol + wg * 64, x[0]);
          tmem_ld32(tmem + lane_addr + C::OCol + wg * 64 + 32, x[1]);
          tmem_wait_ld();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&ms->o_empty);
          float4 *dst = reinterpret_cast<float4 *>(
              p.o_part + guard((long long)prow * 128 + wg * 64, 64,
                               (long long)p.units * p.n_ch * 128 * 128, p.status));
#pragma unroll
          for (int i = 0; i < 16; ++i)
            dst[i] = make_float4(__uint_as_float(x[i >> 3][(i & 7) * 4]),
                                 __uint_as_float(x[i >> 3][(i & 7) * 4 + 1]),
                                 __uint_as_float(x[i >> 3][(i & 7) * 4 + 2]),
                                 __uint_as_float(x[i >> 3][(i & 7) * 4 + 3]));
        }
        ++oc;
        // count the item once every row of its partial is written
        __threadfence();
        named_bar_sync(5, 256);
        if (wg == 0 && wtid == 0) atomicAdd(&p.o_count[guard(it.unit, 1, p.units, p.status)], 1);
      }
      // kO: this CTA's slice of the output rows of the unit of its pass-2
      // item of kOReduceLag steps ago (its other items are done by then)
      if (kO && k - kOReduceLag >= kLag) reduce_rows(p, ms, item_of(p, k - kOReduceLag - kLag), wg * 128 + wtid);
    }
    // kO: the slices whose steps would come after the last one
    if (kO)
      for (int kr = max(kLag, n + kLag - kOReduceLag); kr < n + kLag; ++kr)
        reduce_rows(p, ms, item_of(p, kr - kLag), wg * 128 + wtid);
  }

  tc_fence_before();
  __syncwarp();
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

}  // namespace

bool score_tc1_supported(const LayerGeom &g) {
  return g.dtype == RIPPLE_BF16 && g.R <= 128 && g.P > 0;
}

bool score_tc1_attn_supported(const LayerGeom &g) {
  return score_tc1_supported(g) && g.D == 128 && g.R == 128;
}

namespace {

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

// Votes only: key tiles per item of a unit of n_tiles: the unit is cut into the
// fewest items of at most `most` tiles, all of the same size but the last (64
// tiles as 8 items of 8 instead of 7 of 9 and one of 1: 32 layers of 8 units
// 214 -> 201 us), and into no more items than SMs (the deadlock-free schedule
// needs at most twice as many as CTAs). A function of the prompt length alone,
// so that one layer's call and a multi-layer call merge the same partial
// statistics.
int tiles_per_item(int n_tiles, int most, int sms) {
  const int tpi_min = (n_tiles + sms - 1) / sms, tpi = tpi_min > most ? tpi_min : most;
  const int items = (n_tiles + tpi - 1) / tpi;
  return (n_tiles + items - 1) / items;
}

struct Tc1Kernel {
  const void *fn;
  int smem;
};

template <bool kO, int D, int RP, bool kPad>
Tc1Kernel tc1_kernel() {
  return {(const void *)score_tc1_kernel<kO, D, RP, kPad>, Tc1Smem<kO, D, RP>::Bytes};
}

// Rows are padded to 32, 64 or 128: a thread's share of a tile is then RP
// exponentials, so a unit of 64 window rows costs half of one of 128.
template <int D>
Tc1Kernel tc1_kernel_for(int R) {
  if (R == 128) return tc1_kernel<false, D, 128, false>();
  if (R > 64) return tc1_kernel<false, D, 128, true>();
  if (R == 64) return tc1_kernel<false, D, 64, false>();
  if (R > 32) return tc1_kernel<false, D, 64, true>();
  if (R == 32) return tc1_kernel<false, D, 32, false>();
  return tc1_kernel<false, D, 32, true>();
}

}  // namespace

// kO: items of a unit, at most; one of up to kTilesPerItem tiles is one item, as
// without outputs.
static int attn_items_per_unit(const LayerGeom &g) {
  const int n = (g.T + kTile - 1) / kTile / kTilesPerItem;
  return n > 1 ? n : 1;
}

long long score_tc1_attn_max_items(const LayerGeom &g, int n_layers) {
  const long long units = (long long)g.units * n_layers;
  const long long items = units * attn_items_per_unit(g);
  return units > kMaxItemsO ? units : items < kMaxItemsO ? items : kMaxItemsO;
}

int score_tc1_attn_items(const LayerGeom &g, int n_layers) {
  const int n_tiles = (g.T + kTile - 1) / kTile, sms = sm_count();
  const int per_unit = attn_items_per_unit(g), most = per_unit < sms ? per_unit : sms;
  const long long units = (long long)g.units * n_layers;
  const long long max_items = score_tc1_attn_max_items(g, n_layers);
  int best = 1;
  long long best_cost = -1;
  for (int n = 1; n == 1 || (n <= most && units * n <= max_items); ++n) {
    const int per = (n_tiles + n - 1) / n;
    if ((n_tiles + per - 1) / per != n) continue;  // items would be left empty
    const long long cost = (units * n + sms - 1) / sms * (per + kStepTilesO);
    if (best_cost < 0 || cost * 50 < best_cost * 49) {  // more items by 2% or not
      best = n;
      best_cost = cost;
    }
  }
  return best;
}

cudaError_t launch_score_tc1(const LayerGeom &g, int n_slots, const int *slots, int n_layers,
                             const void *const *q_win, const void *const *k,
                             const CompressWs &ws, float *votes, int32_t *status,
                             cudaStream_t st, const void *const *v, float *const *o_win) {
  EncodeTiledFn enc = encode_fn();
  if (enc == nullptr || n_layers < 1 || n_layers > kCompressMaxLayers) return cudaErrorNotSupported;
  const bool with_o = v != nullptr;
  if (with_o && (o_win == nullptr || ws.o_part == nullptr || ws.o_count == nullptr))
    return cudaErrorInvalidValue;
  static Tc1Launch lp;  // large: kept off the stack, filled under the lock
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  for (int l = 0; l < n_layers; ++l) {
    const cuuint64_t row = (cuuint64_t)g.D * 2;
    cuuint64_t dims[3] = {(cuuint64_t)g.D, (cuuint64_t)g.T, (cuuint64_t)g.units};
    cuuint64_t strides[2] = {row, (cuuint64_t)g.T * row};
    cuuint32_t box[3] = {64, 128, 1};
    cuuint32_t es[3] = {1, 1, 1};
    if (enc(&lp.kmap[l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(k[l]), dims,
            strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
    if (with_o &&
        enc(&lp.vmap[l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(v[l]), dims,
            strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
    cuuint64_t qdims[2] = {(cuuint64_t)g.D, (cuuint64_t)g.units * g.R};
    cuuint64_t qstrides[1] = {row};
    cuuint32_t qbox[2] = {64, (cuuint32_t)g.R};
    cuuint32_t qes[2] = {1, 1};
    if (enc(&lp.qmap[l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(q_win[l]), qdims,
            qstrides, qbox, qes, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  const int sms = sm_count();
  Tc1Params &p = lp.p;
  p.upl = g.units;
  p.units = g.units * n_layers;
  p.R = g.R;
  p.T = g.T;
  p.P = g.P;
  p.W = g.W;
  p.Hq = g.Hq;
  p.Hkv = g.Hkv;
  p.G = g.G;
  p.n_tiles1 = (g.T + kTile - 1) / kTile;
  p.n_tiles2 = with_o ? p.n_tiles1 : (g.P + kTile - 1) / kTile;
  p.tpi = with_o ? (p.n_tiles1 + score_tc1_attn_items(g, n_layers) - 1) /
                       score_tc1_attn_items(g, n_layers)
                 : tiles_per_item(p.n_tiles1, g.D == 64 ? kTilesPerItem64 : kTilesPerItem, sms);
  p.n_ch = (p.n_tiles1 + p.tpi - 1) / p.tpi;
  p.total_items = p.units * p.n_ch;
  p.scale2 = g.scale2;
  for (int l = 0; l < n_layers; ++l) p.o_win[l] = with_o ? o_win[l] : nullptr;
  p.o_part = with_o ? ws.o_part : nullptr;
  p.o_count = with_o ? ws.o_count : nullptr;
  p.partial = ws.row_partial;
  p.lognorm = ws.row_lognorm;
  p.votes = votes;
  for (int l = 0; l < n_layers; ++l) {
    if (slots[l] < 0 || slots[l] >= n_slots) return cudaErrorInvalidValue;
    p.layer_of[l] = slots[l];
  }
  p.n_slots = n_slots;
  p.ctrl = ws.counters;
  p.status = status;
  p.wait_cycles = wait_limit_cycles();
  cudaError_t e = cudaMemsetAsync(ws.counters, 0, sizeof(int) * 2 * p.units, st);
  if (e == cudaSuccess && with_o) e = cudaMemsetAsync(ws.o_count, 0, sizeof(int) * p.units, st);
  if (e != cudaSuccess) return e;
  const Tc1Kernel kernel = with_o         ? tc1_kernel<true, 128, 128, false>()
                           : g.D == 64 ? tc1_kernel_for<64>(g.R)
                                       : tc1_kernel_for<128>(g.R);
  e = cudaFuncSetAttribute(kernel.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kernel.smem);
  if (e != cudaSuccess) return e;
  const int grid = p.total_items < sms ? p.total_items : sms;
  p.d_unit = grid / p.n_ch;
  p.d_chunk = grid % p.n_ch;
  p.d_layer = p.d_unit / p.upl;
  p.d_local = p.d_unit % p.upl;
  void *args[] = {(void *)&lp};
  e = cudaLaunchCooperativeKernel(kernel.fn, dim3(grid), dim3(kThreads), args,
                                  (size_t)kernel.smem, st);
  count_launches(1);
  return e;
}

}  // namespace ripple
