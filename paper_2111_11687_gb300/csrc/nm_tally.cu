// Tally statistics (§2.1 dose and uncertainty maps, Eq. 1-3).
//
// For each batch b of n_b histories the fold moves the int64 batch tally T_b into
// the exact cumulative tally and accumulates, in FP64, S2 = sum_b T_b^2 / n_b
// per voxel and the organ sums O_b = sum over the organ's voxels of the batch
// dose.  With N = sum n_b histories and K batches the per-decay mean of a
// voxel is x = Tsum / N and the batch estimate of its variance is
//   var(x) = (S2 - Tsum^2 / N) / ((K - 1) N),
// the n_b-weighted form of the batch-means estimator.  Every reduction has a
// fixed tree (columns of a tile, then fixed warp trees, then tiles in index
// order), so the statistics are the same on every run.
#include <algorithm>

#include "nm_internal.cuh"

namespace nm {
namespace {

__device__ __forceinline__ double warp_sum_d(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Sums per label keep one order, whatever kernel forms them, since the variance
// of an organ's mean cancels and turns their last bits into leading ones of a
// small sigma: a tile is kFoldTile voxels; column t of a label sums, in voxel
// order, those of its voxels t, t + 128, ... of the tile; the tile's partial is
// columns 0 .. 127 (column_sum), and the label's sum is the partials of all
// tiles (tile_sum).  Partials: [quantity or slot][label][tile].
constexpr int kColumn = kFoldTile / kFoldThreads;          // voxels of a column
constexpr int kSub = 2048;                                 // voxels a CTA of 128 threads has in flight
constexpr int kSubs = kFoldTile / kSub;
constexpr int kPerThread = kSub / kFoldThreads;

__device__ __forceinline__ double column_sum(const double* col, int lane) {
  double sum = 0.0;
#pragma unroll
  for (int j = 0; j < kFoldThreads / 32; ++j) sum += col[lane + 32 * j];
  return warp_sum_d(sum);
}

__device__ __forceinline__ double tile_sum(const double* __restrict__ part, int n_tiles, int lane) {
  double s = 0.0;
#pragma unroll 8
  for (int i = lane; i < n_tiles; i += 32) s += part[i];
  return warp_sum_d(s);
}

// The tile's labels into shared memory, and the set of them that each warp met
// in each sub-tile.  Ends with a barrier.
template <int THREADS>
__device__ __forceinline__ void tile_labels(const uint8_t* __restrict__ labels, int64_t v0, int64_t V, uint8_t* s_lab,
                                            uint32_t (*s_mask)[THREADS / 32]) {
#pragma unroll 1
  for (int s = 0; s < kSubs; ++s) {
    uint32_t mask = 0;
#pragma unroll
    for (int i = 0; i < kSub / THREADS; ++i) {
      const int k = s * kSub + i * THREADS + threadIdx.x;
      const uint32_t l = v0 + k < V ? labels[v0 + k] : 0u;
      s_lab[k] = (uint8_t)l;
      if (v0 + k < V) mask |= 1u << l;
    }
    mask = __reduce_or_sync(0xffffffffu, mask);
    if ((threadIdx.x & 31) == 0) s_mask[s][threadIdx.x >> 5] = mask;
  }
  __syncthreads();
}
template <int THREADS>
__device__ __forceinline__ uint32_t label_set(const uint32_t (*s_mask)[THREADS / 32], int s) {
  uint32_t mask = 0;
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) mask |= s_mask[s][w];
  return mask;
}

// Fold of a launch's NS (or fewer) batches in one pass over the voxels: per
// voxel the slots' tallies are read together and added in batch order, so the
// cumulative tally and S2 are read and written once for all of them, and they
// are the bits of a fold per batch.
//
// Bound by DRAM (8 B per slot and voxel read; written, with the 37 B of
// statistics, only where something was deposited) and, in densely hit volumes,
// by FP64 (four operations per deposit-holding voxel and slot; this GPU does
// about two per SM and clock).  A thread therefore loads NS x K tallies before
// it uses any, and lone voxels of other batches cost nothing.  256 x 253 x 300
// voxels, 6e6 decays in ten batches: 0.50 ms (ten folds 1.3).
//
// With labels a CTA takes a whole tile, for the order of its organ sums, in
// columns for fold_columns(NS) labels at a time; a tile with more labels is
// gone through again, sub-tiles without any of the next ones left out.
__host__ __device__ constexpr int fold_columns(int ns) { return ns == 1 ? 32 : ns == 2 ? 16 : ns <= 5 ? 8 : 4; }

template <int NS, bool LABELS>
__global__ void __launch_bounds__(kFoldThreads) fold_kernel(const FoldParams p, int subs) {
  constexpr int K = NS <= 2 ? 8 : 4;       // voxels of a thread in flight
  constexpr int C = fold_columns(NS);
  extern __shared__ double acc[];                         // [NS][C][kFoldThreads]
  __shared__ uint8_t s_lab[LABELS ? kFoldTile : 1];
  __shared__ uint32_t s_mask[kSubs][kFoldThreads / 32];
  __shared__ ull dep_w[kFoldThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t first = (int64_t)blockIdx.x * subs * kSub;
  ull dep = 0;
  const float gy = (float)p.gy_per_unit_vol;
  uint32_t labels_left = 1u;                              // of the tile; one pass without labels
  if (LABELS) {
    tile_labels<kFoldThreads>(p.labels, first, p.V, s_lab, s_mask);
    labels_left = 0;
    for (int s = 0; s < kSubs; ++s) labels_left |= label_set<kFoldThreads>(s_mask, s);
    for (int i = tid; i < p.n_slots * kLabelSlots; i += kFoldThreads)
      if (!(labels_left >> (i % kLabelSlots) & 1u)) p.organ_partial[(size_t)i * gridDim.x + blockIdx.x] = 0.0;
  }
  while (labels_left) {
    // the next labels, lowest first
    uint32_t group = labels_left;
    if (LABELS) {
      for (int i = 0; i < C; ++i) labels_left &= labels_left - 1;
      group &= ~labels_left;
      for (int i = 0; i < p.n_slots; ++i)
        for (int l = 0; l < __popc(group); ++l) acc[(i * C + l) * kFoldThreads + tid] = 0.0;
    } else {
      labels_left = 0;
    }
    for (int s = 0; s < subs; ++s) {
      const int64_t v0 = first + (int64_t)s * kSub;
      if (v0 >= p.V) break;
      const int64_t v1 = v0 + kSub < p.V ? v0 + kSub : p.V;
      bool fresh = true, last = true;                     // first and last time at these voxels
      if (LABELS) {
        const uint32_t here = label_set<kFoldThreads>(s_mask, s);
        if (!(here & group)) continue;
        fresh = (here & ((group & -group) - 1u)) == 0;
        last = (here & labels_left) == 0;
      }
#pragma unroll 1
      for (int c = 0; c < kPerThread; c += K) {
        ull t[NS][K];
        ull any[K];
#pragma unroll
        for (int b = 0; b < NS; ++b)
#pragma unroll
          for (int j = 0; j < K; ++j) {
            const int64_t v = v0 + tid + (int64_t)(c + j) * kFoldThreads;
            t[b][j] = b < p.n_slots && v < v1 ? p.tb[(int64_t)b * p.V + v] : 0ull;
          }
        ull ts[K];
        double s2v[K];
        float rho[K];
#pragma unroll
        for (int j = 0; j < K; ++j) {
          any[j] = 0;
#pragma unroll
          for (int b = 0; b < NS; ++b) any[j] |= t[b][j];
          ts[j] = 0; s2v[j] = 0.0; rho[j] = 1.0f;
          if (any[j]) {
            const int64_t v = v0 + tid + (int64_t)(c + j) * kFoldThreads;
            if (fresh) {
              ts[j] = p.tsum[v];
              s2v[j] = p.s2[v];
            }
            if (LABELS) rho[j] = p.density[v];
          }
        }
#pragma unroll
        for (int j = 0; j < K; ++j) {
          if (!any[j]) continue;
          const int64_t v = v0 + tid + (int64_t)(c + j) * kFoldThreads;
          // Gy per unit in FP32 (GB300's FP64 divide is slow); the sum stays FP64
          const double g = LABELS ? (double)__fdiv_rn(gy, rho[j]) : 0.0;
          int la = -1;                                    // the voxel's column, if one of this pass
          if (LABELS) {
            const uint32_t l = s_lab[s * kSub + tid + (c + j) * kFoldThreads];
            if (group >> l & 1u) la = __popc(group & ((1u << l) - 1u));
          }
#pragma unroll
          for (int b = 0; b < NS; ++b) {
            if (!t[b][j]) continue;
            const double x = (double)t[b][j];
            if (fresh) {
              ts[j] += t[b][j];
              s2v[j] = s2v[j] + x * x * p.inv_nb[b];
              dep += t[b][j];
            }
            if (LABELS && la >= 0) {
              double* const a = acc + (b * C + la) * kFoldThreads + tid;
              *a = fma(x, g, *a);
            }
            if (last) p.tb[(int64_t)b * p.V + v] = 0;
          }
          if (fresh) {
            p.tsum[v] = ts[j];
            p.s2[v] = s2v[j];
          }
        }
      }
    }
    if (LABELS) {
      const int n = __popc(group);
      __syncthreads();
      for (int i = wid; i < p.n_slots * n; i += kFoldThreads / 32) {
        const int b = i / n, l = i % n;
        const double sum = column_sum(acc + (b * C + l) * kFoldThreads, lane);
        if (lane == 0)
          p.organ_partial[((size_t)b * kLabelSlots + __fns(group, 0, l + 1)) * gridDim.x + blockIdx.x] = sum;
      }
      __syncthreads();
    }
  }
  // deposited-energy counter (integer, so the order of the adds does not matter)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dep += __shfl_xor_sync(0xffffffffu, dep, o);
  if (lane == 0) dep_w[wid] = dep;
  __syncthreads();
  if (tid == 0) {
    ull sum = 0;
    for (int w = 0; w < kFoldThreads / 32; ++w) sum += dep_w[w];
    if (sum) atomicAdd(p.deposited, sum);
  }
}

// The organ sums of a launch's batches alone, a CTA per tile and slot, ahead of
// a fold without labels: where the tiles are too few for the chip.
__global__ void __launch_bounds__(kFoldThreads) fold_slot_organs_kernel(const FoldParams p) {
  constexpr int K = 16;
  __shared__ double acc[kLabelSlots * kFoldThreads];
  __shared__ uint8_t s_lab[kFoldTile];
  __shared__ uint32_t s_mask[kSubs][kFoldThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, b = blockIdx.y;
  const int64_t v0 = (int64_t)blockIdx.x * kFoldTile;
  const ull* const tb = p.tb + (int64_t)b * p.V;
  const float gy = (float)p.gy_per_unit_vol;
  tile_labels<kFoldThreads>(p.labels, v0, p.V, s_lab, s_mask);
  uint32_t set = 0;
  for (int s = 0; s < kSubs; ++s) set |= label_set<kFoldThreads>(s_mask, s);
  const int n = __popc(set);
  for (int l = 0; l < n; ++l) acc[l * kFoldThreads + tid] = 0.0;
#pragma unroll 1
  for (int c = 0; c < kColumn; c += K) {
    ull t[K];
    float rho[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const int64_t v = v0 + tid + (int64_t)(c + j) * kFoldThreads;
      t[j] = v < p.V ? tb[v] : 0ull;
    }
#pragma unroll
    for (int j = 0; j < K; ++j)
      rho[j] = t[j] ? p.density[v0 + tid + (int64_t)(c + j) * kFoldThreads] : 1.0f;
#pragma unroll
    for (int j = 0; j < K; ++j) {
      if (!t[j]) continue;
      const uint32_t l = s_lab[tid + (c + j) * kFoldThreads];
      double* const a = acc + __popc(set & ((1u << l) - 1u)) * kFoldThreads + tid;
      *a = fma((double)t[j], (double)__fdiv_rn(gy, rho[j]), *a);
    }
  }
  __syncthreads();
  for (int l = wid; l < kLabelSlots; l += kFoldThreads / 32) {
    double sum = 0.0;
    if (set >> l & 1u) sum = column_sum(acc + __popc(set & ((1u << l) - 1u)) * kFoldThreads, lane);
    if (lane == 0) p.organ_partial[((size_t)b * kLabelSlots + l) * gridDim.x + blockIdx.x] = sum;
  }
}

// One CTA per label, one warp per slot; the slots are then added in batch order.
__global__ void fold_organs_kernel(const FoldParams p, int n_tiles) {
  __shared__ double sum[kMaxSlots];
  const int lane = threadIdx.x & 31, b = threadIdx.x >> 5, l = blockIdx.x;
  const double s = tile_sum(p.organ_partial + ((size_t)b * kLabelSlots + l) * n_tiles, n_tiles, lane);
  if (lane == 0) sum[b] = s;
  __syncthreads();
  if (threadIdx.x != 0) return;
  double s1 = p.org_s1[l], s2 = p.org_s2[l];
  for (int i = 0; i < p.n_slots; ++i) {
    if (!(p.n_b[i] > 0.0)) continue;
    s1 += sum[i];
    s2 += sum[i] * sum[i] / p.n_b[i];
  }
  p.org_s1[l] = s1;
  p.org_s2[l] = s2;
}

// Eq. 1 of a voxel with tally t > 0: FP64 where cancellation needs it (the
// mean and the variance, S2 - Tsum^2/N), the rest in FP32, whose precision the
// FP32 outputs have anyway.
__device__ __forceinline__ void voxel_dose(ull t, double s2, float rho, double inv_n, double inv_k1n, float gy_a,
                                           float& d, float& sg) {
  const double x = (double)t;
  const double mean = x * inv_n;                       // units per decay
  const double var = fma(-x, mean, s2) * inv_k1n;      // rounding may leave it below 0
  const float conv = __fdiv_rn(gy_a, rho);
  d = (float)mean * conv;                              // Eq. 1, Gy/s
  sg = sqrtf(fmaxf((float)var, 0.0f)) * conv;
}

// Eq. 1 per voxel: dose and sigma, either may be NULL.
//
// Bound by DRAM (25 B per voxel) and FP64.  Voxels without a deposit cost no
// FP64; eight voxels' loads go out together.  Whole body (157 M voxels): 3.3 ms
// -> 0.54 ms.
__global__ void __launch_bounds__(kFoldThreads) finalize_maps_kernel(const FinalizeParams p, int subs) {
  constexpr int K = 8;
  const double inv_n = 1.0 / p.n_total;
  const double inv_k1n = 1.0 / ((p.n_batches - 1.0) * p.n_total);
  const float gy_a = (float)(p.gy_per_unit_vol * p.activity_bq);
  for (int s = 0; s < subs; ++s) {
    const int64_t v0 = ((int64_t)blockIdx.x * subs + s) * kSub + threadIdx.x;
#pragma unroll 1
    for (int c = 0; c < kPerThread; c += K) {
      ull t[K];
      double s2v[K];
      float rho[K];
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const int64_t v = v0 + (int64_t)(c + j) * kFoldThreads;
        t[j] = v < p.V ? p.tsum[v] : 0ull;
      }
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const int64_t v = v0 + (int64_t)(c + j) * kFoldThreads;
        s2v[j] = t[j] ? p.s2[v] : 0.0;
        rho[j] = t[j] ? p.density[v] : 1.0f;
      }
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const int64_t v = v0 + (int64_t)(c + j) * kFoldThreads;
        if (v >= p.V) continue;
        float d = 0.0f, sg = 0.0f;
        if (t[j]) voxel_dose(t[j], s2v[j], rho[j], inv_n, inv_k1n, gy_a, d, sg);
        if (p.dose) p.dose[v] = d;
        if (p.sigma) p.sigma[v] = sg;
      }
    }
  }
}

// x as FP64, without the FP64 pipe where x is normal.
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x);
  if (((u >> 23) & 255u) - 1u >= 254u) return (double)x;
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}

// a + 1 rounded to nearest even, without the FP64 pipe from 1 to 2^40 and at 0:
// the mantissa plus one unit and, past the binade, half of that with the bit
// that drops out.
__device__ __forceinline__ double add_one(double a) {
  const ull b = (ull)__double_as_longlong(a), one = 1023ull << 52;
  if (b == 0) return 1.0;
  if (b - one >= 40ull << 52) return a + 1.0;
  const uint32_t ex = (uint32_t)(b >> 52);
  const ull m = ((b & ((1ull << 52) - 1)) | 1ull << 52) + (1ull << (52 + 1023 - ex));
  const ull h = m >> 1;
  const ull r = m >> 53 ? h + (m & h & 1ull) + ((ull)ex << 52) : m + ((ull)(ex - 1) << 52);
  return __longlong_as_double((long long)r);
}

// Partials of the NQ quantities staged in s_val (dose; then epsilon^2) for every
// label of the tile, by 512 threads: thread t of a group of 128 goes through
// column t's voxels once for one quantity and every WIDE-th label, the label
// at hand in a register, the others in `col`.  Zero doses add nothing.
constexpr int kOrganThreads = 512;
constexpr int kOrganColumns = 32;
struct OrganColumns {
  double col[kOrganColumns][kFoldThreads];
};
template <int NQ, int WIDE>
__device__ __forceinline__ void tile_partials(const float (*s_val)[kFoldTile], const uint8_t* s_lab, uint32_t set,
                                              OrganColumns& s, double* __restrict__ part) {
  constexpr int kMine = kOrganColumns / (NQ * WIDE), kRound = WIDE * kMine;   // columns of a group; labels of a round
  static_assert(NQ * WIDE <= kOrganThreads / kFoldThreads, "a group each");
  const int t = threadIdx.x & (kFoldThreads - 1), r = threadIdx.x >> 7, q = r % NQ, mine = r / NQ;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, n = __popc(set);
  if (threadIdx.x < NQ * kLabelSlots && !(set >> (threadIdx.x % kLabelSlots) & 1u))
    part[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = 0.0;
  for (int k0 = 0; k0 < n; k0 += kRound) {
    double(*const col)[kFoldThreads] = s.col + r * kMine;
    if (r < NQ * WIDE) {
      for (int c = 0; c < kMine && k0 + c * WIDE + mine < n; ++c) col[c][t] = 0.0;
      double a = 0.0;                                    // of column `at`
      int at = 0;
#pragma unroll 1
      for (int i0 = 0; i0 < kColumn; i0 += 16) {
        float x[16];
        int rank[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          x[i] = s_val[q][t + (i0 + i) * kFoldThreads];
          rank[i] = __popc(set & ((1u << s_lab[t + (i0 + i) * kFoldThreads]) - 1u)) - k0;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          if (x[i] == 0.0f || (unsigned)rank[i] % WIDE != mine || (unsigned)rank[i] >= (unsigned)kRound) continue;
          if (rank[i] / WIDE != at) {
            col[at][t] = a;
            at = rank[i] / WIDE;
            a = col[at][t];
          }
          if (q == 1 && x[i] == 1.0f) a = add_one(a);
          else a += widen(x[i]);
        }
      }
      col[at][t] = a;
    }
    __syncthreads();
    for (int i = wid; i < NQ * min(kRound, n - k0); i += kOrganThreads / 32) {
      const int qi = i % NQ, k = i / NQ;
      const double sum = column_sum(s.col[(k % WIDE * NQ + qi) * kMine + k / WIDE], lane);
      if (lane == 0) part[((size_t)qi * kLabelSlots + __fns(set, 0, k0 + k + 1)) * gridDim.x + blockIdx.x] = sum;
    }
    __syncthreads();
  }
}

// Eq. 1 maps (MAPS) and the sums behind Eq. 2 and Eq. 3 per label.  A CTA takes
// a tile: 512 threads form dose and epsilon^2 of its voxels in any order, eight
// voxels' loads of each in flight, and then the columns from shared memory.
// Bound by FP64 (six operations per voxel with a deposit, and two of the sums).
// Microseconds a call of Eq. 2 and 3, host and copies with it: 256 x 253 x 300
// voxels 505 -> 229, 64 x 61 x 75 84 -> 55.
template <int NQ>
struct OrganStage {
  OrganColumns c;
  float val[NQ][kFoldTile];
  uint8_t lab[kFoldTile];
};
template <bool MAPS>
__global__ void __launch_bounds__(kOrganThreads, 2) finalize_organ_tiles_kernel(const FinalizeParams p) {
  constexpr int K = 8;
  extern __shared__ __align__(16) unsigned char s_dyn[];
  OrganStage<2>& st = *reinterpret_cast<OrganStage<2>*>(s_dyn);
  __shared__ uint32_t s_mask[kSubs][kOrganThreads / 32];
  const double inv_n = 1.0 / p.n_total;
  const double inv_k1n = 1.0 / ((p.n_batches - 1.0) * p.n_total);
  const float gy_a = (float)(p.gy_per_unit_vol * p.activity_bq);
  const int64_t v0 = (int64_t)blockIdx.x * kFoldTile;
#pragma unroll 1
  for (int c = 0; c < kFoldTile / kOrganThreads; c += K) {
    ull t[K];
    double s2v[K];
    float rho[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const int64_t v = v0 + threadIdx.x + (c + j) * kOrganThreads;
      t[j] = v < p.V ? p.tsum[v] : 0ull;
    }
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const int64_t v = v0 + threadIdx.x + (c + j) * kOrganThreads;
      s2v[j] = t[j] ? p.s2[v] : 0.0;
      rho[j] = t[j] ? p.density[v] : 1.0f;
    }
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const int k = threadIdx.x + (c + j) * kOrganThreads;
      const int64_t v = v0 + k;
      float d = 0.0f, sg = 0.0f;
      if (t[j]) voxel_dose(t[j], s2v[j], rho[j], inv_n, inv_k1n, gy_a, d, sg);
      const float eps = d > 0.0f ? __fdiv_rn(sg, d) : 1.0f;
      st.val[0][k] = d;
      st.val[1][k] = v < p.V ? eps * eps : 0.0f;
      if (MAPS && v < p.V) {
        if (p.dose) p.dose[v] = d;
        if (p.sigma) p.sigma[v] = sg;
      }
    }
  }
  tile_labels<kOrganThreads>(p.labels, v0, p.V, st.lab, s_mask);
  uint32_t set = 0;
  for (int s = 0; s < kSubs; ++s) set |= label_set<kOrganThreads>(s_mask, s);
  tile_partials<2, 1>(st.val, st.lab, set, st.c, p.organ_partial);
}

__global__ void finalize_organs_kernel(const FinalizeParams p, int n_tiles) {
  const int lane = threadIdx.x & 31;
  const int l = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (l >= kLabelSlots) return;
  const double sd = tile_sum(p.organ_partial + (size_t)l * n_tiles, n_tiles, lane);
  const double se = tile_sum(p.organ_partial + (size_t)(kLabelSlots + l) * n_tiles, n_tiles, lane);
  if (lane != 0) return;
  const double cnt = (double)p.organ_count[l];
  double mean = 0.0, eps = 0.0, sig = 0.0;
  if (cnt > 0.0) {
    mean = sd / cnt;                                          // Eq. 2
    eps = sqrt(se / cnt);                                     // Eq. 3
    // Batch sigma of the organ mean: m_b = O_b / (n_b cnt) per decay.
    const double N = p.n_total;
    const double mbar = p.org_s1[l] / (N * cnt);
    const double sum_nm2 = p.org_s2[l] / (cnt * cnt);
    const double var = fmax(sum_nm2 - N * mbar * mbar, 0.0) / ((p.n_batches - 1.0) * N);
    sig = sqrt(var) * p.activity_bq;
  }
  p.organ_out[l] = mean;
  p.organ_out[kLabelSlots + l] = eps;
  p.organ_out[2 * kLabelSlots + l] = sig;
  p.organ_out[3 * kLabelSlots + l] = cnt;
}

// Eq. 2 over an arbitrary dose map: partials per label and tile.  256 x 253 x
// 300 voxels 165 -> 118 us a call.
__global__ void __launch_bounds__(kOrganThreads) map_organ_kernel(const float* __restrict__ dose,
                                                                  const uint8_t* __restrict__ labels, int64_t V,
                                                                  double* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  OrganStage<1>& st = *reinterpret_cast<OrganStage<1>*>(s_dyn);
  __shared__ uint32_t s_mask[kSubs][kOrganThreads / 32];
  const int64_t v0 = (int64_t)blockIdx.x * kFoldTile;
#pragma unroll
  for (int i = 0; i < kFoldTile / kOrganThreads; ++i) {
    const int k = threadIdx.x + i * kOrganThreads;
    st.val[0][k] = v0 + k < V ? dose[v0 + k] : 0.0f;
  }
  tile_labels<kOrganThreads>(labels, v0, V, st.lab, s_mask);
  uint32_t set = 0;
  for (int s = 0; s < kSubs; ++s) set |= label_set<kOrganThreads>(s_mask, s);
  tile_partials<1, 4>(st.val, st.lab, set, st.c, part);
}

__global__ void map_organ_final_kernel(const double* __restrict__ part, int n_tiles,
                                       const long long* __restrict__ count, double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int l = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (l >= kLabelSlots) return;
  const double s = tile_sum(part + (size_t)l * n_tiles, n_tiles, lane);
  if (lane == 0) out[l] = count[l] > 0 ? s / (double)count[l] : 0.0;
}

// lo + 2^64 hi += q_lo + 2^32 q_hi, and q_lo = q_hi = 0.
__global__ void fold_history_kernel(ull* __restrict__ q_lo, ull* __restrict__ q_hi, ull* __restrict__ lo,
                                    ull* __restrict__ hi, int64_t V) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
    const ull a = q_lo[v], b = q_hi[v];
    if (!(a | b)) continue;
    const ull l0 = lo[v], l1 = l0 + a, l2 = l1 + (b << 32);
    lo[v] = l2;
    hi[v] += (b >> 32) + (l1 < l0 ? 1ull : 0ull) + (l2 < l1 ? 1ull : 0ull);
    q_lo[v] = 0;
    q_hi[v] = 0;
  }
}

__global__ void history_sigma_kernel(const ull* __restrict__ tsum, const ull* __restrict__ lo,
                                     const ull* __restrict__ hi, const float* __restrict__ density, int64_t V,
                                     double n, float gy_a, float* __restrict__ sigma) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
    const ull t = tsum[v];
    float sg = 0.0f;
    if (t) {
      const double s2 = (double)hi[v] * 18446744073709551616.0 + (double)lo[v];
      const double mean = (double)t / n;                   // units per history
      const double var = fmax(s2 / n - mean * mean, 0.0) / (n - 1.0);   // of the mean
      sg = sqrtf((float)var) * __fdiv_rn(gy_a, density[v]);
    }
    sigma[v] = sg;
  }
}

}  // namespace

int organ_tiles(int64_t V) { return (int)((V + kFoldTile - 1) / kFoldTile); }

// Sub-tiles of a CTA of the passes without labels: one each while that leaves
// about 16 CTAs an SM.
static int pass_subs(int64_t V, int sms) {
  const int64_t subs = (V + kSub - 1) / kSub;
  return (int)std::max<int64_t>(1, (subs + 16 * sms - 1) / (16 * sms));
}
static int pass_blocks(int64_t V, int subs) { return (int)((V + (int64_t)subs * kSub - 1) / ((int64_t)subs * kSub)); }

cudaError_t launch_fold_history(ull* q_lo, ull* q_hi, ull* lo, ull* hi, int64_t V, cudaStream_t s) {
  const int64_t g = (V + 255) / 256;
  fold_history_kernel<<<(unsigned)(g < 8192 ? g : 8192), 256, 0, s>>>(q_lo, q_hi, lo, hi, V);
  return cudaGetLastError();
}

cudaError_t launch_history_sigma(const ull* tsum, const ull* s2h_lo, const ull* s2h_hi, const float* density,
                                 int64_t V, double n_total, double gy_a, float* sigma, cudaStream_t s) {
  const int64_t g = (V + 255) / 256;
  history_sigma_kernel<<<(unsigned)(g < 8192 ? g : 8192), 256, 0, s>>>(tsum, s2h_lo, s2h_hi, density, V, n_total,
                                                                       (float)gy_a, sigma);
  return cudaGetLastError();
}

cudaError_t launch_map_organ_means(const float* dose, const uint8_t* labels, int64_t V, double* part,
                                   const long long* count, double* out, cudaStream_t s) {
  const int n = organ_tiles(V);
  const cudaError_t e =
      cudaFuncSetAttribute(map_organ_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(OrganStage<1>));
  if (e != cudaSuccess) return e;
  map_organ_kernel<<<n, kOrganThreads, sizeof(OrganStage<1>), s>>>(dose, labels, V, part);
  map_organ_final_kernel<<<(kLabelSlots + 3) / 4, 128, 0, s>>>(part, n, count, out);
  return cudaGetLastError();
}

namespace {

// Statistics of two shards of one run (disjoint history ids): the exact
// tallies and counters add as integers, the 128-bit sums of squared history
// totals add with a carry, and the FP64 batch sums add because the batches of
// both shards are batches of the combined run.
__global__ void merge_stats_kernel(const MergeParams m) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < m.V; v += stride) {
    m.tsum[v] += m.o_tsum[v];
    m.s2[v] += m.o_s2[v];
    if (m.s2h_lo) {
      const ull lo = m.s2h_lo[v] + m.o_lo[v];
      m.s2h_hi[v] += m.o_hi[v] + (lo < m.o_lo[v] ? 1ull : 0ull);
      m.s2h_lo[v] = lo;
    }
  }
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i < kLabelSlots; i += blockDim.x) {
      m.org_s1[i] += m.o_org_s1[i];
      m.org_s2[i] += m.o_org_s2[i];
    }
    for (int i = threadIdx.x; i < kCtrCount; i += blockDim.x) m.counters[i] += m.o_counters[i];
  }
}

}  // namespace

cudaError_t launch_merge_stats(const MergeParams& m, int sms, cudaStream_t s) {
  const int64_t want = (m.V + 255) / 256;
  const int grid = (int)(want < 8LL * sms ? (want > 0 ? want : 1) : 8LL * sms);
  merge_stats_kernel<<<grid, 256, 0, s>>>(m);
  return cudaGetLastError();
}

namespace {

// Eq. 1 alone (no uncertainty, no organ sums): the dose rate the finalize
// pass writes, bit for bit (same FP64 mean, same FP32 conversion), streaming
// 16 bytes per voxel.
__global__ void dose_only_kernel(const ull* __restrict__ tsum, const float* __restrict__ density, int64_t V,
                                 double inv_n, float gy_a, float* __restrict__ dose) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += stride) {
    const ull ti = tsum[v];
    float d = 0.0f;
    if (ti) {
      const double mean = (double)ti * inv_n;
      d = (float)mean * __fdiv_rn(gy_a, density[v]);
    }
    dose[v] = d;
  }
}

}  // namespace

cudaError_t launch_dose_only(const FinalizeParams& p, int sms, cudaStream_t s) {
  const int64_t want = (p.V + 255) / 256;
  const int grid = (int)(want < 8LL * sms ? (want > 0 ? want : 1) : 8LL * sms);
  dose_only_kernel<<<grid, 256, 0, s>>>(p.tsum, p.density, p.V, 1.0 / p.n_total,
                                        (float)(p.gy_per_unit_vol * p.activity_bq), p.dose);
  return cudaGetLastError();
}

// Tiles per SM from which the fold takes whole tiles (fold_kernel); below, the
// organ sums go by tile and slot, and the rest by sub-tile.  Microseconds by
// slot and whole: one slot, 38 tiles 27 and 29, 300 tiles 39 and 35; ten slots,
// 300 tiles 150 and 220, 1200 tiles 441 and 349.
constexpr int split_tiles(int ns) { return ns <= 2 ? 1 : 4; }

template <int NS>
static cudaError_t launch_fold_t(const FoldParams& p, cudaStream_t s) {
  const int tiles = organ_tiles(p.V), subs = pass_subs(p.V, p.sms);
  if (!p.labels || tiles < split_tiles(NS) * p.sms) {
    if (p.labels) fold_slot_organs_kernel<<<dim3(tiles, p.n_slots), kFoldThreads, 0, s>>>(p);
    fold_kernel<NS, false><<<pass_blocks(p.V, subs), kFoldThreads, 0, s>>>(p, subs);
  } else {
    const size_t smem = (size_t)NS * fold_columns(NS) * kFoldThreads * sizeof(double);
    // per call: cheap, and correct for every device and calling thread
    const cudaError_t e =
        cudaFuncSetAttribute(fold_kernel<NS, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    fold_kernel<NS, true><<<tiles, kFoldThreads, smem, s>>>(p, kSubs);
  }
  if (p.labels) fold_organs_kernel<<<kLabelSlots, 32 * p.n_slots, 0, s>>>(p, tiles);
  return cudaGetLastError();
}

cudaError_t launch_fold(const FoldParams& p, cudaStream_t s) {
  // the smallest variant that holds the slots (registers grow with it)
  if (p.n_slots < 1 || p.n_slots > kMaxSlots) return cudaErrorInvalidValue;
  if (p.n_slots == 1) return launch_fold_t<1>(p, s);
  if (p.n_slots == 2) return launch_fold_t<2>(p, s);
  if (p.n_slots <= 5) return launch_fold_t<5>(p, s);
  if (p.n_slots <= 10) return launch_fold_t<10>(p, s);
  return launch_fold_t<kMaxSlots>(p, s);
}

template <bool MAPS>
static cudaError_t launch_organ_tiles(const FinalizeParams& p, cudaStream_t s) {
  const int tiles = organ_tiles(p.V);
  const cudaError_t e = cudaFuncSetAttribute(finalize_organ_tiles_kernel<MAPS>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(OrganStage<2>));
  if (e != cudaSuccess) return e;
  finalize_organ_tiles_kernel<MAPS><<<tiles, kOrganThreads, sizeof(OrganStage<2>), s>>>(p);
  finalize_organs_kernel<<<(kLabelSlots + 3) / 4, 128, 0, s>>>(p, tiles);
  return cudaGetLastError();
}

cudaError_t launch_finalize(const FinalizeParams& p, bool organs, int sms, cudaStream_t s) {
  const bool maps = p.dose || p.sigma;
  if (organs) return maps ? launch_organ_tiles<true>(p, s) : launch_organ_tiles<false>(p, s);
  const int subs = pass_subs(p.V, sms);
  if (maps) finalize_maps_kernel<<<pass_blocks(p.V, subs), kFoldThreads, 0, s>>>(p, subs);
  return cudaGetLastError();
}

}  // namespace nm

// ---------------------------------------------------------------------------
// Multi-time-point dosimetry: time-integrated activity per voxel.
// ---------------------------------------------------------------------------
namespace nm {
namespace {

constexpr int kMaxTimePoints = 16;

struct TimeIntegralArgs {
  const float* act[kMaxTimePoints];   // activity maps (Bq per voxel)
  double t[kMaxTimePoints];           // their times, seconds
  int n;
};

// Per voxel, in FP64: A_0 t_0 / 2 (linear uptake from zero), the trapezoids
// between time points, and A_n / lambda after the last one (physical decay,
// tail_s = 1 / lambda); the FP64 sum of a CTA's results goes to
// block_sums[block] (fixed tree).  A negative or non-finite activity sets
// NM_DEV_BAD_ACTIVITY.
__global__ void __launch_bounds__(256) time_integral_kernel(const TimeIntegralArgs a, int64_t V, double tail_s,
                                                            float* __restrict__ out, double* __restrict__ block_sums,
                                                            uint32_t* __restrict__ status) {
  __shared__ double red[256];
  double acc = 0.0;
  bool bad = false;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
    double prev = (double)a.act[0][v];
    bad |= !(prev >= 0.0) || isinf(prev);
    double s = 0.5 * prev * a.t[0];
    for (int k = 1; k < a.n; ++k) {
      const double cur = (double)a.act[k][v];
      bad |= !(cur >= 0.0) || isinf(cur);
      s += 0.5 * (prev + cur) * (a.t[k] - a.t[k - 1]);
      prev = cur;
    }
    s += prev * tail_s;
    out[v] = (float)s;
    acc += s;
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) block_sums[blockIdx.x] = red[0];
  if (bad) atomicOr(status, (uint32_t)NM_DEV_BAD_ACTIVITY);
}

}  // namespace

cudaError_t launch_time_integral(const float* const* act, const double* t_s, int n, int64_t V, double tail_s,
                                 float* out, double* block_sums, int blocks, cudaStream_t s) {
  if (n < 1 || n > kMaxTimePoints || blocks < 1) return cudaErrorInvalidValue;
  TimeIntegralArgs a;
  for (int k = 0; k < kMaxTimePoints; ++k) {
    a.act[k] = k < n ? act[k] : nullptr;
    a.t[k] = k < n ? t_s[k] : 0.0;
  }
  a.n = n;
  // the status word follows the block sums
  time_integral_kernel<<<blocks, 256, 0, s>>>(a, V, tail_s, out, block_sums,
                                              reinterpret_cast<uint32_t*>(block_sums + blocks));
  return cudaGetLastError();
}

}  // namespace nm
