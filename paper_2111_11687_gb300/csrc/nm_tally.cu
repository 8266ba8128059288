// Tally statistics (§2.1 dose and uncertainty maps, Eq. 1-3).
//
// For each batch b of n_b histories the fold moves the int64 batch tally T_b into
// the exact cumulative tally and accumulates, in FP64, S2 = sum_b T_b^2 / n_b
// per voxel and the organ sums O_b = sum over the organ's voxels of the batch
// dose.  With N = sum n_b histories and K batches the per-decay mean of a
// voxel is x = Tsum / N and the batch estimate of its variance is
//   var(x) = (S2 - Tsum^2 / N) / ((K - 1) N),
// the n_b-weighted form of the batch-means estimator.  Every reduction has a
// fixed tree (per-thread columns in shared memory, then fixed warp trees, then
// blocks in index order), so the statistics are the same on every run.
#include <algorithm>

#include "nm_internal.cuh"

namespace nm {
namespace {

__device__ __forceinline__ double warp_sum_d(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Sums per label.  A tile of kFoldTile voxels holds few labels, so each thread
// keeps FP64 sums for kAccLabels of them in columns of shared memory (one per
// quantity and label); a tile with more labels is read again for the next
// ones.  The columns, and then the tiles and blocks, are added in a fixed order.
constexpr int kAccLabels = 4;
constexpr int kPerThread = kFoldTile / kFoldThreads;       // voxels of a thread per tile

// Labels of this thread's voxels v0 + tid + i kFoldThreads, a byte each (0 past
// v1); returns the set of labels in the tile.
__device__ __forceinline__ uint32_t tile_labels(const uint8_t* __restrict__ labels, int64_t v0, int64_t v1,
                                                uint32_t (&lab)[kPerThread / 4], uint32_t* s_mask) {
  uint32_t mask = 0;
#pragma unroll
  for (int i = 0; i < kPerThread / 4; ++i) lab[i] = 0;
#pragma unroll
  for (int i = 0; i < kPerThread; ++i) {
    const int64_t v = v0 + threadIdx.x + (int64_t)i * kFoldThreads;
    const uint32_t l = v < v1 ? labels[v] : 0u;
    lab[i / 4] |= l << (8 * (i % 4));
    if (v < v1) mask |= 1u << l;
  }
  mask = __reduce_or_sync(0xffffffffu, mask);
  if ((threadIdx.x & 31) == 0) s_mask[threadIdx.x >> 5] = mask;
  __syncthreads();
  mask = 0;
#pragma unroll
  for (int w = 0; w < kFoldThreads / 32; ++w) mask |= s_mask[w];
  return mask;
}

// Column of the thread's i-th voxel among those for labels l0, l0 + 1, ... of
// the tile's set, or -1.
__device__ __forceinline__ int label_column(const uint32_t (&lab)[kPerThread / 4], int i, uint32_t mask, int l0) {
  const uint32_t l = (lab[i / 4] >> (8 * (i % 4))) & 255u;
  const int c = __popc(mask & ((1u << l) - 1u)) - l0;
  return c < kAccLabels ? c : -1;
}

// out[q][label] += the sum of the columns acc[q][0 .. n_acc) (labels l0, ... of
// the set) for q < n_q; one warp per column.  Ends with the columns free again.
__device__ __forceinline__ void add_columns(const double* acc, int n_q, int n_acc, uint32_t mask, int l0,
                                            double (*out)[kLabelSlots]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  for (int i = wid; i < n_q * n_acc; i += kFoldThreads / 32) {
    const int q = i / n_acc, l = i % n_acc;
    const double* col = acc + (q * kAccLabels + l) * kFoldThreads;
    double sum = 0.0;
#pragma unroll
    for (int j = 0; j < kFoldThreads / 32; ++j) sum += col[lane + 32 * j];
    sum = warp_sum_d(sum);
    if (lane == 0) out[q][__fns(mask, 0, l0 + l + 1)] += sum;
  }
  __syncthreads();
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
// it uses any, and lone voxels of other batches cost nothing.
//
// Benchmark phantom, ten batches: 10 x 0.18 ms as a fold each, 1.15 ms together.
template <int NS, bool LABELS>
__global__ void __launch_bounds__(kFoldThreads) fold_kernel(const FoldParams p, int tiles_per_block) {
  constexpr int K = NS <= 2 ? 8 : 4;       // voxels of a thread in flight
  extern __shared__ double acc[];                         // [NS][kAccLabels][kFoldThreads]
  __shared__ double out[LABELS ? NS : 1][kLabelSlots];
  __shared__ uint32_t s_mask[kFoldThreads / 32];
  __shared__ ull dep_w[kFoldThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (LABELS)
    for (int i = tid; i < NS * kLabelSlots; i += kFoldThreads) out[i / kLabelSlots][i % kLabelSlots] = 0.0;
  ull dep = 0;
  const float gy = (float)p.gy_per_unit_vol;
  const int64_t first = (int64_t)blockIdx.x * tiles_per_block * kFoldTile;
  for (int ti = 0; ti < tiles_per_block; ++ti) {
    const int64_t v0 = first + (int64_t)ti * kFoldTile;
    if (v0 >= p.V) break;
    const int64_t v1 = v0 + kFoldTile < p.V ? v0 + kFoldTile : p.V;
    uint32_t lab[kPerThread / 4];
    const uint32_t mask = LABELS ? tile_labels(p.labels, v0, v1, lab, s_mask) : 0u;
    const int n_lab = LABELS ? __popc(mask) : 1;
    for (int l0 = 0; l0 < n_lab; l0 += kAccLabels) {
      const int n_acc = min(kAccLabels, n_lab - l0);
      const bool last = l0 + kAccLabels >= n_lab;
      if (LABELS)
        for (int i = 0; i < p.n_slots; ++i)
          for (int l = 0; l < n_acc; ++l) acc[(i * kAccLabels + l) * kFoldThreads + tid] = 0.0;
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
            if (l0 == 0) {
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
          if (LABELS) la = label_column(lab, c + j, mask, l0);
#pragma unroll
          for (int b = 0; b < NS; ++b) {
            if (!t[b][j]) continue;
            const double x = (double)t[b][j];
            if (l0 == 0) {
              ts[j] += t[b][j];
              s2v[j] = s2v[j] + x * x * p.inv_nb[b];
              dep += t[b][j];
            }
            if (LABELS && la >= 0) acc[(b * kAccLabels + la) * kFoldThreads + tid] += x * g;
            if (last) p.tb[(int64_t)b * p.V + v] = 0;
          }
          if (l0 == 0) {
            p.tsum[v] = ts[j];
            p.s2[v] = s2v[j];
          }
        }
      }
      if (LABELS) add_columns(acc, p.n_slots, n_acc, mask, l0, out);
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
  if (LABELS)
    for (int i = tid; i < p.n_slots * kLabelSlots; i += kFoldThreads)
      p.organ_partial[((size_t)(i / kLabelSlots) * gridDim.x + blockIdx.x) * kLabelSlots + i % kLabelSlots] =
          out[i / kLabelSlots][i % kLabelSlots];
}

// One CTA per label, one warp per slot: blocks lane-strided, then a fixed tree;
// the slots are then added in batch order.
__global__ void fold_organs_kernel(const FoldParams p, int n_blocks) {
  __shared__ double sum[kMaxSlots];
  const int lane = threadIdx.x & 31, b = threadIdx.x >> 5, l = blockIdx.x;
  double s = 0.0;
  for (int i = lane; i < n_blocks; i += 32) s += p.organ_partial[((size_t)b * n_blocks + i) * kLabelSlots + l];
  s = warp_sum_d(s);
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

// Eq. 1 per voxel (MAPS: dose and sigma, either may be NULL) and the sums behind
// Eq. 2 and Eq. 3 per label (ORGANS).
//
// Bound by DRAM (25 B per voxel for the maps) and FP64, which therefore does
// only what needs it: the mean, the variance (S2 - Tsum^2/N cancels) and the
// organ sums; the rest is FP32, whose precision the FP32 outputs have anyway.
// Voxels without a deposit cost no FP64: their dose adds nothing and their
// epsilon of 1 is counted in integers.  Eight voxels' loads go out together.
// Whole body (157 M voxels): 3.3 ms for either -> 0.54 ms (maps), 1.02 ms (organs).
template <bool MAPS, bool ORGANS>
__global__ void __launch_bounds__(kFoldThreads) finalize_kernel(const FinalizeParams p, int tiles_per_block) {
  constexpr int K = 8;
  __shared__ double acc[ORGANS ? 2 * kAccLabels * kFoldThreads : 1];   // dose, epsilon^2
  __shared__ int zeros[ORGANS ? kAccLabels : 1][kFoldThreads];         // voxels without a deposit
  __shared__ double out[ORGANS ? 2 : 1][kLabelSlots];
  __shared__ uint32_t s_mask[kFoldThreads / 32];
  const int tid = threadIdx.x;
  if (ORGANS && tid < 2 * kLabelSlots) out[tid / kLabelSlots][tid % kLabelSlots] = 0.0;
  const double inv_n = 1.0 / p.n_total;
  const double inv_k1n = 1.0 / ((p.n_batches - 1.0) * p.n_total);
  const float gy_a = (float)(p.gy_per_unit_vol * p.activity_bq);
  const int64_t first = (int64_t)blockIdx.x * tiles_per_block * kFoldTile;
  for (int ti = 0; ti < tiles_per_block; ++ti) {
    const int64_t v0 = first + (int64_t)ti * kFoldTile;
    if (v0 >= p.V) break;
    const int64_t v1 = v0 + kFoldTile < p.V ? v0 + kFoldTile : p.V;
    uint32_t lab[kPerThread / 4];
    const uint32_t mask = ORGANS ? tile_labels(p.labels, v0, v1, lab, s_mask) : 0u;
    const int n_lab = ORGANS ? __popc(mask) : 1;
    for (int l0 = 0; l0 < n_lab; l0 += kAccLabels) {
      const int n_acc = min(kAccLabels, n_lab - l0);
      if (ORGANS)
        for (int l = 0; l < n_acc; ++l) {
          acc[l * kFoldThreads + tid] = acc[(kAccLabels + l) * kFoldThreads + tid] = 0.0;
          zeros[l][tid] = 0;
        }
#pragma unroll 1
      for (int c = 0; c < kPerThread; c += K) {
        ull t[K];
        double s2v[K];
        float rho[K];
#pragma unroll
        for (int j = 0; j < K; ++j) {
          const int64_t v = v0 + tid + (int64_t)(c + j) * kFoldThreads;
          t[j] = v < v1 ? p.tsum[v] : 0ull;
        }
#pragma unroll
        for (int j = 0; j < K; ++j) {
          const int64_t v = v0 + tid + (int64_t)(c + j) * kFoldThreads;
          s2v[j] = 0.0; rho[j] = 1.0f;
          if (t[j]) {
            s2v[j] = p.s2[v];
            rho[j] = p.density[v];
          }
        }
#pragma unroll
        for (int j = 0; j < K; ++j) {
          const int64_t v = v0 + tid + (int64_t)(c + j) * kFoldThreads;
          if (v >= v1) continue;
          float d = 0.0f, sg = 0.0f;
          if (t[j]) {
            const double x = (double)t[j];
            const double mean = x * inv_n;                       // units per decay
            const double var = fma(-x, mean, s2v[j]) * inv_k1n;  // rounding may leave it below 0
            const float conv = __fdiv_rn(gy_a, rho[j]);
            d = (float)mean * conv;                              // Eq. 1, Gy/s
            sg = sqrtf(fmaxf((float)var, 0.0f)) * conv;
          }
          if (MAPS) {
            if (p.dose) p.dose[v] = d;
            if (p.sigma) p.sigma[v] = sg;
          }
          if (ORGANS) {
            const int la = label_column(lab, c + j, mask, l0);
            if (la >= 0) {
              if (d > 0.0f) {
                const float eps = __fdiv_rn(sg, d);
                acc[la * kFoldThreads + tid] += (double)d;
                acc[(kAccLabels + la) * kFoldThreads + tid] += (double)(eps * eps);
              } else {
                zeros[la][tid] += 1;
              }
            }
          }
        }
      }
      if (ORGANS) {
        for (int l = 0; l < n_acc; ++l)
          if (zeros[l][tid]) acc[(kAccLabels + l) * kFoldThreads + tid] += (double)zeros[l][tid];
        add_columns(acc, 2, n_acc, mask, l0, out);
      }
    }
  }
  if (ORGANS && tid < 2 * kLabelSlots)
    p.organ_partial[(size_t)blockIdx.x * 2 * kLabelSlots + tid] = out[tid / kLabelSlots][tid % kLabelSlots];
}

__global__ void finalize_organs_kernel(const FinalizeParams p, int n_blocks) {
  const int lane = threadIdx.x & 31;
  const int l = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (l >= kLabelSlots) return;
  double sd = 0.0, se = 0.0;
  for (int b = lane; b < n_blocks; b += 32) {
    sd += p.organ_partial[(size_t)b * 2 * kLabelSlots + l];
    se += p.organ_partial[(size_t)b * 2 * kLabelSlots + kLabelSlots + l];
  }
  sd = warp_sum_d(sd);
  se = warp_sum_d(se);
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

// Eq. 2 over an arbitrary dose map: per-CTA per-label partial sums (fixed
// tree).  Zeros add nothing and cost no FP64 (benchmark phantom: 134 -> 96 us).
__global__ void __launch_bounds__(kFoldThreads) map_organ_kernel(const float* __restrict__ dose,
                                                                 const uint8_t* __restrict__ labels, int64_t V,
                                                                 int tiles_per_block, double* __restrict__ part) {
  __shared__ double acc[kAccLabels * kFoldThreads];
  __shared__ double out[1][kLabelSlots];
  __shared__ uint32_t s_mask[kFoldThreads / 32];
  const int tid = threadIdx.x;
  if (tid < kLabelSlots) out[0][tid] = 0.0;
  const int64_t first = (int64_t)blockIdx.x * tiles_per_block * kFoldTile;
  for (int ti = 0; ti < tiles_per_block; ++ti) {
    const int64_t v0 = first + (int64_t)ti * kFoldTile;
    if (v0 >= V) break;
    const int64_t v1 = v0 + kFoldTile < V ? v0 + kFoldTile : V;
    float d[kPerThread];
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
      const int64_t v = v0 + tid + (int64_t)i * kFoldThreads;
      d[i] = v < v1 ? dose[v] : 0.0f;
    }
    uint32_t lab[kPerThread / 4];
    const uint32_t mask = tile_labels(labels, v0, v1, lab, s_mask);
    const int n_lab = __popc(mask);
    for (int l0 = 0; l0 < n_lab; l0 += kAccLabels) {
      const int n_acc = min(kAccLabels, n_lab - l0);
      for (int l = 0; l < n_acc; ++l) acc[l * kFoldThreads + tid] = 0.0;
#pragma unroll
      for (int i = 0; i < kPerThread; ++i) {
        const int la = label_column(lab, i, mask, l0);
        if (d[i] != 0.0f && la >= 0) acc[la * kFoldThreads + tid] += (double)d[i];
      }
      add_columns(acc, 1, n_acc, mask, l0, out);
    }
  }
  if (tid < kLabelSlots) part[(size_t)blockIdx.x * kLabelSlots + tid] = out[0][tid];
}

__global__ void map_organ_final_kernel(const double* __restrict__ part, int n_blocks,
                                       const long long* __restrict__ count, double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int l = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (l >= kLabelSlots) return;
  double s = 0.0;
  for (int b = lane; b < n_blocks; b += 32) s += part[(size_t)b * kLabelSlots + l];
  s = warp_sum_d(s);
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

// Tiles of a CTA of the passes over the voxels: few enough CTAs for a small pass over their
// label sums, one tile each while that leaves every SM with work.
static int fold_tiles(int64_t V) {
  const int64_t tiles = (V + kFoldTile - 1) / kFoldTile;
  return (int)std::max<int64_t>(1, (tiles + 16 * 152 - 1) / (16 * 152));
}
int fold_blocks(int64_t V) {
  const int64_t per = (int64_t)fold_tiles(V) * kFoldTile;
  return (int)((V + per - 1) / per);
}

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
  const int nb = fold_blocks(V);
  map_organ_kernel<<<nb, kFoldThreads, 0, s>>>(dose, labels, V, fold_tiles(V), part);
  map_organ_final_kernel<<<(kLabelSlots + 3) / 4, 128, 0, s>>>(part, nb, count, out);
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

template <int NS>
static cudaError_t launch_fold_t(const FoldParams& p, cudaStream_t s) {
  const int nb = fold_blocks(p.V), tiles = fold_tiles(p.V);
  if (!p.labels) {
    fold_kernel<NS, false><<<nb, kFoldThreads, 0, s>>>(p, tiles);
    return cudaGetLastError();
  }
  const size_t smem = (size_t)NS * kAccLabels * kFoldThreads * sizeof(double);
  // per call: cheap, and correct for every device and calling thread
  const cudaError_t e =
      cudaFuncSetAttribute(fold_kernel<NS, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  fold_kernel<NS, true><<<nb, kFoldThreads, smem, s>>>(p, tiles);
  fold_organs_kernel<<<kLabelSlots, 32 * p.n_slots, 0, s>>>(p, nb);
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

cudaError_t launch_finalize(const FinalizeParams& p, bool organs, cudaStream_t s) {
  const int nb = fold_blocks(p.V), tiles = fold_tiles(p.V);
  const bool maps = p.dose || p.sigma;
  if (!organs) {
    if (maps) finalize_kernel<true, false><<<nb, kFoldThreads, 0, s>>>(p, tiles);
    return cudaGetLastError();
  }
  if (maps) finalize_kernel<true, true><<<nb, kFoldThreads, 0, s>>>(p, tiles);
  else finalize_kernel<false, true><<<nb, kFoldThreads, 0, s>>>(p, tiles);
  finalize_organs_kernel<<<(kLabelSlots + 3) / 4, 128, 0, s>>>(p, nb);
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
