// Observation-window token scoring on the fp32 pipes (SnapKV rule kept by
// RippleKV, Sec. 4.4 last paragraph), for fp32 caches, where running the
// contraction on tf32 tensor cores would spend the score tolerance.
//
// All layers of a call in two or three launches; a CTA takes kScoreChunk keys of
// one unit and all of its window rows, in both passes:
//   pass 1: per window row, (max, sum of exp) over the chunk's visible keys;
//   merge : per row, combine the chunk partials into max + log2(sum) (inside
//           pass 2 while a unit has few chunks, else a launch of its own);
//   pass 2: per prefix key, sum over rows of exp2(x - lognorm_row).
// All arithmetic in the log2 domain: x = scale * log2(e) * q.k.
//
// Keys and window rows lie in shared memory dim by dim, and a thread has 4 rows
// x 8 keys of a 64 x 128 block in registers: three 16-byte shared loads for 16
// packed FMAs. Bound: shared memory (83% of its rate, the FMA pipe 45%): 16 layers
// of 8 units, 1192 tokens, 128 rows of d = 128 take 323 us with selection, 31
// TFLOP/s over the two passes; 32 layers of 8 units and 8192 tokens 38. One row x
// 16 keys a thread with a scalar load per FMA, three launches a layer, took the
// first 1610 us. Few CTAs, as in a 512-token prompt, are bound by latency: four
// layers 24.6 us with selection, against 152 us with three launches each.
#include <math.h>

#include "common.cuh"
#include "kernels.cuh"

namespace ripple {
namespace {

constexpr int kThreads = 256;
constexpr int kRows = 64;             // window rows of a register block
constexpr int kRT = 4, kKT = 8;       // rows and keys per thread
constexpr int kKeyLanes = kScoreChunk / kKT;
constexpr int kRowLanes = kRows / kRT;
constexpr int kFuseMerge = 16;        // chunks up to which pass 2 merges by itself
static_assert(kKeyLanes * kRowLanes == kThreads && kKeyLanes == 16, "thread layout");

// Layers of one launch: units per layer, the scored layers' inputs and votes
// slots.
struct SimtTable {
  const float *q[kCompressMaxLayers];  // [B][Hq][w][D]
  const float *k[kCompressMaxLayers];  // [upl][T][D]
  int slot[kCompressMaxLayers];
  float2 *partial;                     // [units][n_chunks][R]
  float *lognorm;                      // [units][R]
  float *votes;                        // [n_slots][upl][P]
  int n_units, n_slots, n_chunks;
  int32_t *status;
};

template <int D>
struct SimtSmem {
  // [dim][key] and [dim][row]; the pad keeps 16-byte rows and spreads the
  // transposing stores over the banks
  float k[D][kScoreChunk + 4];
  float q[D][kRows + 4];
};

// n rows of D floats (zeros past n_live) into dst[dim][row].
template <int D, int N>
__device__ __forceinline__ void load_transposed(const float *src, int n_live, float (*dst)[N + 4]) {
  // consecutive lanes take consecutive rows, so that the stores of a dim go to
  // consecutive words
  for (int e = threadIdx.x; e < N * (D / 4); e += kThreads) {
    const int row = e % N, c = e / N * 4;
    const float4 x = row < n_live ? *reinterpret_cast<const float4 *>(src + (size_t)row * D + c)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
    dst[c][row] = x.x;
    dst[c + 1][row] = x.y;
    dst[c + 2][row] = x.z;
    dst[c + 3][row] = x.w;
  }
}

// acc[i][j] = q_{4 tr + i} . k_{4 tk + (j < 4 ? j : 60 + j)}, summed in dim order.
template <int D>
__device__ __forceinline__ void dot_block(const SimtSmem<D> &s, int tr, int tk,
                                          float2 (&acc)[kRT][kKT / 2]) {
#pragma unroll
  for (int i = 0; i < kRT; ++i)
#pragma unroll
    for (int j = 0; j < kKT / 2; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 8
  for (int c = 0; c < D; ++c) {
    const float4 a = *reinterpret_cast<const float4 *>(&s.k[c][tk * 4]);
    const float4 b = *reinterpret_cast<const float4 *>(&s.k[c][tk * 4 + kScoreChunk / 2]);
    const float4 q = *reinterpret_cast<const float4 *>(&s.q[c][tr * 4]);
    const float2 kk[4] = {make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(b.x, b.y),
                          make_float2(b.z, b.w)};
    const float qq[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < kRT; ++i)
#pragma unroll
      for (int j = 0; j < kKT / 2; ++j)
        acc[i][j] = __ffma2_rn(make_float2(qq[i], qq[i]), kk[j], acc[i][j]);
  }
}

// Key of entry (j, e) of a thread's accumulators within the chunk.
__device__ __forceinline__ int key_of(int tk, int j, int e) {
  return tk * 4 + (j & 1) * 2 + e + (j >> 1) * (kScoreChunk / 2);
}

__device__ __forceinline__ void combine(float &m, float &l, float m2, float l2) {
  const float mm = fmaxf(m, m2);
  if (mm == -INFINITY) return;
  l = l * exp2f(m - mm) + l2 * exp2f(m2 - mm);
  m = mm;
}

// max + log2(sum) of row r of a unit from its chunks' partials.
__device__ __forceinline__ float merged_row(const SimtTable &t, int R, int unit, int r) {
  float m = -INFINITY, l = 0.f;
  const float2 *part = t.partial + guard((long long)unit * t.n_chunks, t.n_chunks,
                                         (long long)t.n_units * t.n_chunks, t.status) *
                                       R;
  for (int c0 = 0; c0 < t.n_chunks; c0 += 8) {
    float2 p[8];
#pragma unroll
    for (int c = 0; c < 8; ++c)
      p[c] = c0 + c < t.n_chunks ? __ldcg(&part[(size_t)(c0 + c) * R + r])
                                 : make_float2(-INFINITY, 0.f);
#pragma unroll
    for (int c = 0; c < 8; ++c) combine(m, l, p[c].x, p[c].y);
  }
  return m + log2f(l);
}

template <int D>
__global__ void __launch_bounds__(kThreads) score_pass1_simt(LayerGeom g,
                                                             const __grid_constant__ SimtTable t) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  SimtSmem<D> &s = *reinterpret_cast<SimtSmem<D> *>(smem_raw);
  pdl_launch_dependents();
  const int unit = blockIdx.y, chunk = blockIdx.x;
  const int layer = unit / g.units, local = unit % g.units;
  const int key0 = chunk * kScoreChunk;
  load_transposed<D, kScoreChunk>(t.k[layer] + ((size_t)local * g.T + key0) * D, g.T - key0, s.k);
  const float *q_unit = t.q[layer] + (size_t)local * g.R * D;
  const int tr = threadIdx.x / kKeyLanes, tk = threadIdx.x % kKeyLanes;
  for (int row0 = 0; row0 < g.R; row0 += kRows) {
    if (row0 > 0) __syncthreads();
    load_transposed<D, kRows>(q_unit + (size_t)row0 * D, g.R - row0, s.q);
    __syncthreads();
    float2 acc[kRT][kKT / 2];
    dot_block<D>(s, tr, tk, acc);
#pragma unroll
    for (int i = 0; i < kRT; ++i) {
      const int r = row0 + tr * kRT + i;
      const int last_visible = g.P + (r % g.W);  // causal inside the window (< T)
      float x[kKT], m = -INFINITY;
#pragma unroll
      for (int j = 0; j < kKT; ++j) {
        const float v = j & 1 ? acc[i][j >> 1].y : acc[i][j >> 1].x;
        x[j] = key0 + key_of(tk, j >> 1, j & 1) <= last_visible ? v * g.scale2 : -INFINITY;
        m = fmaxf(m, x[j]);
      }
      float l = 0.f;
      if (m != -INFINITY) {
#pragma unroll
        for (int j = 0; j < kKT; ++j) l += exp2f(x[j] - m);
      }
#pragma unroll
      for (int o = 1; o < kKeyLanes; o <<= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
        const float l2 = __shfl_xor_sync(0xffffffffu, l, o);
        combine(m, l, m2, l2);
      }
      if (tk == 0 && r < g.R)
        t.partial[guard(((long long)unit * t.n_chunks + chunk) * g.R + r, 1,
                        (long long)t.n_units * t.n_chunks * g.R, t.status)] = make_float2(m, l);
    }
  }
}

__global__ void merge_row_stats(LayerGeom g, const __grid_constant__ SimtTable t) {
  const int unit = blockIdx.x;
  for (int r = threadIdx.x; r < g.R; r += blockDim.x)
    t.lognorm[guard((long long)unit * g.R + r, 1, (long long)t.n_units * g.R, t.status)] =
        merged_row(t, g.R, unit, r);
}

template <int D>
__global__ void __launch_bounds__(kThreads) score_pass2_simt(LayerGeom g,
                                                             const __grid_constant__ SimtTable t,
                                                             int fused_merge) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  SimtSmem<D> &s = *reinterpret_cast<SimtSmem<D> *>(smem_raw);
  __shared__ float ln[256];                          // the unit's row normalisers
  __shared__ float red[kRowLanes][kScoreChunk + 4];  // a key's votes per row group
  const int unit = blockIdx.y, chunk = blockIdx.x;
  const int layer = unit / g.units, local = unit % g.units;
  const int key0 = chunk * kScoreChunk;
  load_transposed<D, kScoreChunk>(t.k[layer] + ((size_t)local * g.T + key0) * D, g.T - key0, s.k);
  const float *q_unit = t.q[layer] + (size_t)local * g.R * D;
  load_transposed<D, kRows>(q_unit, g.R, s.q);
  // the inputs were there before pass 1 began; its results from here on
  pdl_wait();
  for (int r = threadIdx.x; r < 256; r += kThreads)
    ln[r] = r >= g.R ? INFINITY  // rows past the last count for nothing
            : fused_merge ? merged_row(t, g.R, unit, r)
                          : __ldcg(&t.lognorm[(size_t)unit * g.R + r]);
  const int tr = threadIdx.x / kKeyLanes, tk = threadIdx.x % kKeyLanes;
  float vote[kKT];
#pragma unroll
  for (int j = 0; j < kKT; ++j) vote[j] = 0.f;
  for (int row0 = 0; row0 < g.R; row0 += kRows) {
    if (row0 > 0) {
      __syncthreads();
      load_transposed<D, kRows>(q_unit + (size_t)row0 * D, g.R - row0, s.q);
    }
    __syncthreads();
    float2 acc[kRT][kKT / 2];
    dot_block<D>(s, tr, tk, acc);
#pragma unroll
    for (int i = 0; i < kRT; ++i) {
      const int r = row0 + tr * kRT + i;
      if (r >= g.R) break;
      const float off = ln[r];
#pragma unroll
      for (int j = 0; j < kKT; ++j) {
        const float v = j & 1 ? acc[i][j >> 1].y : acc[i][j >> 1].x;
        vote[j] += exp2f(fmaf(v, g.scale2, -off));
      }
    }
  }
  // Sum over the row groups of each key in a fixed order.
#pragma unroll
  for (int j = 0; j < kKT; ++j) red[tr][key_of(tk, j >> 1, j & 1)] = vote[j];
  __syncthreads();
  if (threadIdx.x < kScoreChunk) {
    const int key = key0 + threadIdx.x;
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < kRowLanes; ++i) sum += red[i][threadIdx.x];
    if (key < g.P)
      t.votes[guard((long long)(t.slot[layer] * g.units + local) * g.P + key, 1,
                    (long long)t.n_slots * g.units * g.P, t.status)] = sum;
  }
}

template <int D>
cudaError_t launch_d(const LayerGeom &g, const SimtTable &t, cudaStream_t st) {
  const int smem = (int)sizeof(SimtSmem<D>);
  cudaError_t e = cudaFuncSetAttribute(score_pass1_simt<D>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(score_pass2_simt<D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem);
  if (e != cudaSuccess) return e;
  score_pass1_simt<D><<<dim3(t.n_chunks, t.n_units), kThreads, smem, st>>>(g, t);
  const int fused = t.n_chunks <= kFuseMerge;
  if (!fused) merge_row_stats<<<t.n_units, 256, 0, st>>>(g, t);
  // pass 2 starts while pass 1 (or the merge) ends and loads its inputs
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((g.P + kScoreChunk - 1) / kScoreChunk, t.n_units);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, score_pass2_simt<D>, g, t, fused);
  count_launches(fused ? 2 : 3);
  return e;
}

}  // namespace

cudaError_t launch_score_simt(const LayerGeom &g, int n_slots, const int *slots, int n_scored,
                              const void *const *q_win, const void *const *k,
                              const CompressWs &ws, float *votes, int32_t *status,
                              cudaStream_t st) {
  if (g.dtype != RIPPLE_F32 || n_scored < 1 || n_scored > kCompressMaxLayers || g.P < 1)
    return cudaErrorInvalidValue;
  SimtTable t;
  for (int l = 0; l < n_scored; ++l) {
    t.q[l] = (const float *)q_win[l];
    t.k[l] = (const float *)k[l];
    t.slot[l] = slots[l];
  }
  t.partial = ws.row_partial;
  t.lognorm = ws.row_lognorm;
  t.votes = votes;
  t.n_units = g.units * n_scored;
  t.n_slots = n_slots;
  t.n_chunks = (g.T + kScoreChunk - 1) / kScoreChunk;
  t.status = status;
  return g.D == 64 ? launch_d<64>(g, t, st) : launch_d<128>(g, t, st);
}

}  // namespace ripple
