// Weight gradient of a 3x3x3 convolution, one x-row of voxels per MMA:
//   dW[co][tap][ci] = sum over voxels v of dY[v][co] * X[v + off_tap][ci].
//
// A GEMM over voxels (K) whose MMAs are bound by how many are issued and how
// much shared memory each reads, not by tensor math (M = 64, K = 16).  So N is
// as wide as the layout allows: X rows are staged as [z][y][input chunk][x], 16
// channels (32 bytes) a voxel and 16 voxels a row, in which the rows of the
// three y-taps and G chunks of one voxel row follow each other at one stride
// (16 rows of 32 bytes): one MMA of N = 48 G covers them all.  A row is 14
// voxels of the tile and the halo voxel on each side, exactly the K = 16 of an
// MMA.  The x-taps shift dY instead of X: the M = 64 operand is four 16-channel
// atoms one voxel row (32 bytes) apart, so atom q reads dY shifted by q - 1
// voxels (tap dx = 1 - q; the fourth atom's rows of D are never read); dY is
// zero at its halo columns, which belong to other tiles, so that the shift
// runs over a row's ends.  The z-taps are the planes of X.  Per tile of 14 x 8
// x 2 voxels 16 K-steps of (COUT / 16) x (z-taps of the pass) MMAs:
// for 48 -> 16 channels 48 MMAs of N = 144, where one 16-channel chunk, or one
// chunk's y-taps, per MMA takes 351 of N = 48 for 512 voxels.
//
// Passes run over groups of G input chunks and ND z-taps (accumulators ND x
// COUT / 16 x 48 G columns of TMEM); the grid is (tiles, passes), so that few
// tiles still fill the chip.  The accumulators are added to the CTA's partial
// dW in FP32 after at most kChain tiles: the tensor core's running sum loses
// more the longer it is.  Against 64 bits, 4 x 64^3 voxels, 48 -> 16 channels:
// 6.1e-6 in one sum of 34 tiles (and in the shifted-window kernel), 2.9e-6 in
// sums of 17, 1.0e-6 of 7, 0.5e-6 of 4, at 129, 141, 155 and 179 us a call.
// The network's own training step does not come here: it keeps the summation
// order of the kernels that its saved weights and optimiser moments come from,
// since a last bit of dW that differs turns, over rounding the weights to BF16
// and Adam's step at gradients near zero, into another trajectory.
//   What bounds it is the MMA rate: MMAs of 48 to 144 columns run at about 90
// cycles each, the operands' shared-memory reads and the issue.  2 x 50 x 37 x
// 61 voxels, 96 -> 32 channels: 105 us (351 in the shifted-window kernel), the
// call 157 (522); 2 x 40 x 60 x 60, 128 -> 64: 390 us, the call 440 (1318 with
// the gather kernel).
//   warp 0    TMA producer: dY atoms and X planes of each tile into a stage ring;
//   warp 1    MMA issuer;
//   warps 2-5 zero dY's halo columns of each landed stage, and at the end of a
//             pass write the CTA's partial dW.
// Partials are summed over CTAs in a fixed order (deterministic).  Every wait
// is bounded; a time-out sets NM_DEV_TIMEOUT and drains what is in flight.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdlib>
#include <mutex>

#include "nm_internal.cuh"
#include "nm_tc.cuh"
#include "nm_wgrad.cuh"

namespace nm {
namespace {

typedef __nv_bfloat16 bf16;

constexpr int RX = 16, TX = 14, TY = 8, TZ = 2;  // padded row, tile
constexpr int PY = TY + 2;
constexpr int kSteps = TY * TZ;                  // K-steps of a tile
constexpr uint32_t kRow = RX * 32;               // one x-row of 16 channels, bytes
constexpr uint32_t kPad = 256;                   // zero rows before and after dY (the x-taps' shift)
constexpr uint32_t kYBytes = kSteps * kRow + 2 * kPad;
constexpr int kThreads = 192;
constexpr long long kWaitCycles = 4ll << 30;
constexpr int kChain = 10;                       // tiles summed in TMEM before they are added to the partial, at most

template <int COUT, int G, int ND>
struct RLayout {
  static constexpr int kYAtoms = COUT / 16;
  static constexpr int kN = 48 * G;                       // accumulator columns per z-tap and output atom
  static constexpr int kPlanes = TZ + ND - 1;             // X planes of a stage
  static constexpr uint32_t kPlane = PY * G * kRow;
  static constexpr uint32_t kTx = kYAtoms * kSteps * kRow + kPlanes * kPlane;   // bytes that land per stage
  static constexpr uint32_t kStage = (kYAtoms * kYBytes + kPlanes * kPlane + 1023) / 1024 * 1024;
  static constexpr int kStages = 4 * kStage <= 220 * 1024 ? 4 : 3 * kStage <= 220 * 1024 ? 3 : 2;
  static constexpr size_t kSmem = (size_t)kStages * kStage;
  static_assert(ND * kYAtoms * kN <= 512, "accumulators fit the tensor memory");
  static_assert(kSmem <= 227 * 1024, "shared memory");
  static_assert(kN <= 256, "one MMA");
};

struct RGrid {
  int n, d, h, w, tiles_x, tiles_y, tiles_z, cin, kpad, chain;
  long long tiles;
  __device__ void coords(long long t, int& b, int& x0, int& y0, int& z0) const {
    x0 = (int)(t % tiles_x) * TX; t /= tiles_x;
    y0 = (int)(t % tiles_y) * TY; t /= tiles_y;
    z0 = (int)(t % tiles_z) * TZ;
    b = (int)(t / tiles_z);
  }
};

// MN-major operand, 32-byte swizzle: lbo = stride between 16-element atoms
// along M/N, 256 = stride between groups of 8 K rows.
__device__ __forceinline__ uint64_t desc_mn_sw32(uint32_t saddr, uint32_t lbo) {
  return tc::smem_desc(saddr, lbo, 256) | ((uint64_t)6 << 61);
}

template <int COUT, int G, int ND>
__global__ void __launch_bounds__(kThreads, 1) wgrad_rows_kernel(const __grid_constant__ CUtensorMap tmx,
                                                                 const __grid_constant__ CUtensorMap tmy,
                                                                 const RGrid g, float* __restrict__ part,
                                                                 uint32_t* status) {
  typedef RLayout<COUT, G, ND> L;
  constexpr int S = L::kStages, kDz = 3 / ND;            // passes per chunk group
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t full[S], ready[S], empty[S], acc_full, acc_empty;
  __shared__ uint32_t s_tmem;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nchunks = (g.cin + 15) / 16;
  const long long my_tiles = g.tiles > blockIdx.x ? (g.tiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;
  const int passes = (nchunks + G - 1) / G * kDz;
  // tiles per read-out of the accumulators: equal shares of at most `chain`
  const long long reads = (my_tiles + g.chain - 1) / g.chain, seg = reads > 0 ? (my_tiles + reads - 1) / reads : 1;

  if (warp == 0) tc::tmem_alloc(&s_tmem, 512);
  // the rows before and after each dY atom stay zero
  for (int i = threadIdx.x; i < S * L::kYAtoms * 32; i += blockDim.x) {
    const int o = i % 32, a = i / 32 % L::kYAtoms, s = i / 32 / L::kYAtoms;
    const uint32_t at = o < 16 ? o * 16 : kYBytes - kPad + (o - 16) * 16;
    *reinterpret_cast<uint4*>(smem + s * L::kStage + a * kYBytes + at) = make_uint4(0, 0, 0, 0);
  }
  if (threadIdx.x == 32) {
    for (int i = 0; i < S; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&ready[i], 128);
      tc::mbar_init(&empty[i], 1);
    }
    tc::mbar_init(&acc_full, 1);
    tc::mbar_init(&acc_empty, 96);
    tc::mbar_fence_init();
  }
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = s_tmem;
  const uint32_t base = tc::smem_u32(smem);
  bool timeout = false;

  if (warp == 0) {
    // ---- producer ----------------------------------------------------------------
    if (lane == 0) {
      long long it = 0;
      for (int ps = blockIdx.y; ps < passes && !timeout; ps += gridDim.y) {
        const int c0 = ps / kDz * G, dz0 = ps % kDz * ND;
        for (long long k = 0; k < my_tiles; ++k, ++it) {
          const int s = (int)(it % S);
          if (it >= S && !tc::mbar_wait_bounded(&empty[s], (uint32_t)(((it / S) - 1) & 1), kWaitCycles)) {
            timeout = true;
            break;
          }
          int b, x0, y0, z0;
          g.coords(blockIdx.x + k * gridDim.x, b, x0, y0, z0);
          const uint32_t sy = base + s * L::kStage, sx = sy + L::kYAtoms * kYBytes;
          tc::mbar_arrive_expect_tx(&full[s], L::kTx);
          for (int q = 0; q < L::kYAtoms; ++q)
            tc::tma_load_5d(sy + q * kYBytes + kPad, &tmy, &full[s], q * 16, x0 - 1, y0, z0, b);
          for (int p = 0; p < L::kPlanes; ++p) {
            // planes of all batch items follow each other; one outside the
            // item's volume is read past the end of the tensor, as zeros
            const int z = z0 - 1 + dz0 + p;
            const int zn = z >= 0 && z < g.d ? b * g.d + z : g.n * g.d;
            tc::tma_load_5d(sx + p * L::kPlane, &tmx, &full[s], 0, x0 - 1, c0, y0 - 1, zn);
          }
        }
      }
      for (long long j = it > S ? it - S : 0; j < it; ++j)
        if (!tc::mbar_wait_bounded(&full[j % S], (uint32_t)((j / S) & 1), kWaitCycles)) timeout = true;
    }
  } else if (warp == 1) {
    // ---- MMA issuer ----------------------------------------------------------------
    if (lane == 0) {
      constexpr uint32_t idesc = tc::idesc_bf16_f32(64, L::kN, true, true);
      long long it = 0;
      int done = 0;                                      // read-outs
      for (int ps = blockIdx.y; ps < passes && !timeout; ps += gridDim.y) {
        for (long long k = 0; k < my_tiles; ++k, ++it) {
          // the previous segment's accumulators have been read out
          if (k % seg == 0 && done > 0 &&
              !tc::mbar_wait_bounded(&acc_empty, (uint32_t)((done - 1) & 1), kWaitCycles)) {
            timeout = true;
            break;
          }
          const int s = (int)(it % S);
          if (!tc::mbar_wait_bounded(&ready[s], (uint32_t)((it / S) & 1), kWaitCycles)) {
            timeout = true;
            break;
          }
          tc::fence_after_sync();
          const uint32_t sy = base + s * L::kStage, sx = sy + L::kYAtoms * kYBytes;
          // descriptors differ only in the start address (16-byte units)
          const uint64_t a0 = desc_mn_sw32(sy + kPad - 32, 32), b0 = desc_mn_sw32(sx, kRow);
          const uint32_t first = k % seg == 0 ? 0u : 1u;
#pragma unroll 4
          for (int ks = 0; ks < kSteps; ++ks) {
#pragma unroll
            for (int z = 0; z < ND; ++z) {
              const uint64_t bdesc = b0 + (uint64_t)((((ks / TY + z) * PY + ks % TY) * G * kRow) >> 4);
#pragma unroll
              for (int h = 0; h < L::kYAtoms; ++h)
                tc::mma_bf16(tmem + (z * L::kYAtoms + h) * L::kN, a0 + (uint64_t)((h * kYBytes + ks * kRow) >> 4),
                             bdesc, idesc, ks == 0 ? first : 1u);
            }
          }
          tc::mma_commit(&empty[s]);
          if (k % seg == seg - 1 || k == my_tiles - 1) {
            tc::mma_commit(&acc_full);
            ++done;
          }
        }
      }
      if (it > 0 && !tc::mbar_wait_bounded(&empty[(it - 1) % S], (uint32_t)(((it - 1) / S) & 1), kWaitCycles))
        timeout = true;
    }
  } else {
    // ---- halo columns, and the partial dW at the end of each segment ----------------
    const int t = threadIdx.x - 64;                      // 0..127
    // with M = 64, D row i sits in TMEM lane (i % 16) + 32 (i / 16), so atom q
    // (tap dx = 1 - q) is lanes 0-15 of quarter q, read by the warp of that
    // quarter; quarter 3 holds the unused fourth atom
    const int q = warp & 3;
    float* const dst = part + (size_t)blockIdx.x * g.kpad * COUT;
    long long it = 0;
    int done = 0;
    for (int ps = blockIdx.y; ps < passes && !timeout; ps += gridDim.y) {
      const int c0 = ps / kDz * G, dz0 = ps % kDz * ND;
      for (long long k = 0; k < my_tiles; ++k, ++it) {
        const int s = (int)(it % S);
        bool got = tc::mbar_wait_bounded(&full[s], (uint32_t)((it / S) & 1), kWaitCycles);
        if (!__all_sync(0xffffffffu, got)) {
          timeout = true;
          break;
        }
        // the first and last voxel of every dY row, both 16-byte halves
        for (int i = t; i < L::kYAtoms * kSteps * 4; i += 128) {
          const int half = i & 1, end = (i >> 1) & 1, r = (i >> 2) % kSteps, a = (i >> 2) / kSteps;
          *reinterpret_cast<uint4*>(smem + s * L::kStage + a * kYBytes + kPad + r * kRow + end * (kRow - 32) + half * 16) =
              make_uint4(0, 0, 0, 0);
        }
        tc::fence_async_smem();
        tc::mbar_arrive(&ready[s]);
        if (k % seg != seg - 1 && k != my_tiles - 1) continue;
        if (q != 3) {
          got = tc::mbar_wait_bounded(&acc_full, (uint32_t)(done & 1), kWaitCycles);
          if (!__all_sync(0xffffffffu, got)) {
            timeout = true;
            break;
          }
          tc::fence_after_sync();
          const bool add = k >= seg;
          for (int z = 0; z < ND; ++z)
            for (int h = 0; h < L::kYAtoms; ++h)
              for (int a = 0; a < 3 * G; ++a) {
                // column atom a: tap dy = a / G - 1, input chunk c0 + a % G
                const int tap = (dz0 + z) * 9 + a / G * 3 + (2 - q), ci = (c0 + a % G) * 16;
                float v[16];
                tc::tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (z * L::kYAtoms + h) * L::kN + a * 16, v);
                float4* const e = reinterpret_cast<float4*>(dst + (size_t)(h * 16 + lane) * g.kpad + tap * g.cin + ci);
                // 64 contiguous bytes of dW's own layout a thread; one thread
                // owns an element, so its sums come in a fixed order
                if (lane < 16)
#pragma unroll
                  for (int j = 0; j < 4; ++j)
                    if (ci + 4 * j < g.cin) {
                      const float4 u = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                      if (add) atomicAdd(e + j, u);
                      else e[j] = u;
                    }
              }
          tc::fence_before_sync();
          tc::mbar_arrive(&acc_empty);
        }
        ++done;
      }
    }
  }
  if (timeout) atomicOr(status, NM_DEV_TIMEOUT);
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// dW = the CTAs' partials, in dW's own layout, summed in a fixed order: per
// element eight warps each add a contiguous run of CTAs, then the runs are
// added in order.  n4: float4 of dW, a multiple of 32.  10.5 us for 152 partials
// of 96 x 32 channels; by (k, output), which writes a float a sector, 16.
__global__ void __launch_bounds__(256) wgrad_rows_reduce(const float4* __restrict__ part, int splits, int n4, int kpad,
                                                         int kreal, float4* __restrict__ dw, uint32_t* status) {
  __shared__ float4 red[8][32];
  const int lane = threadIdx.x & 31, run = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane, per = (splits + 7) / 8;
  const int t1 = min(splits, (run + 1) * per);
  const bool real = e * 4 % kpad < kreal;                // kreal is a multiple of 4
  float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (real)
#pragma unroll 4
    for (int t = run * per; t < t1; ++t) {
      const float4 p = __ldg(part + (size_t)t * n4 + e);
      v.x += p.x, v.y += p.y, v.z += p.z, v.w += p.w;
    }
  red[run][lane] = v;
  __syncthreads();
  if (run != 0) return;
#pragma unroll
  for (int q = 1; q < 8; ++q) {
    const float4 p = red[q][lane];
    v.x += p.x, v.y += p.y, v.z += p.z, v.w += p.w;
  }
  if (!isfinite(v.x) || !isfinite(v.y) || !isfinite(v.z) || !isfinite(v.w)) atomicOr(status, kWgradNonFinite);
  dw[e] = v;
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static std::once_flag once;
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    else
      cudaGetLastError();
  });
  return fn;
}

int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 1;
  return n;
}

long long row_tiles(const nm_conv3d_desc& d) {
  return (long long)((d.w + TX - 1) / TX) * ((d.h + TY - 1) / TY) * ((d.d + TZ - 1) / TZ) * d.n;
}

// Input chunks and z-taps of a pass: the widest MMAs whose groups divide the
// chunks (a group's missing chunks are zeros) and whose accumulators fit.
struct RForm {
  int g, nd;
};
RForm row_form(const nm_conv3d_desc& d) {
  const int c = (d.c0 + 15) / 16;
  if (d.cout <= 32) return {c % 3 ? 2 : 3, d.cout == 16 ? 3 : 1};
  return {d.cout == 64 && c > 1 ? 2 : 1, 1};
}

// The grid: x over tiles (each x writes partials), y over passes.  With up to 32
// outputs as many partials as SMs.  With more, dW is large and its partials
// would cost more to write and add than the MMAs (128 x 128 channels: 1.8 MB
// each): as many as the gather kernel makes, the SMs shared among the passes.
// Two tiles per CTA at least (four with many inputs) once all SMs have work,
// for the same reason.
dim3 row_grid(const nm_conv3d_desc& d) {
  const RForm f = row_form(d);
  const int passes = ((d.c0 + 15) / 16 + f.g - 1) / f.g * (3 / f.nd), sms = sm_count();
  int gy = 1;
  if (d.cout > 32)
    for (int k = 2; k <= std::min(passes, sms / std::max(1, 4 * 152 / (conv_kpad(d.c0) / 128))); ++k)
      if (passes % k == 0) gy = k;
  const int per = d.cout <= 32 ? 1 : d.c0 > 64 ? 4 : 2;
  const long long tiles = row_tiles(d);
  const int gx = (int)std::max<long long>(
      1, std::min<long long>(sms / gy, std::max<long long>((tiles + per - 1) / per, std::min<long long>(tiles, sms / passes))));
  return dim3(gx, std::max(gy, std::min(passes, sms / gx)));
}

// Tiles summed in tensor memory at a time.  With 64 and 128 outputs no more
// steps of 16 voxels than in the gather kernel's sums, which the row kernel takes
// the place of there, so that its error is no larger: 4 x 16^3 voxels, 64 -> 64
// channels 3.4e-7 in sums of three tiles (48 steps), 2.4e-7 in the gather
// kernel's of 24.
int row_chain(const nm_conv3d_desc& d) {
  if (d.cout <= 32) return kChain;
  const long long m = (long long)d.n * d.d * d.h * d.w, splits = conv_wgrad_splits(d);
  const long long theirs = ((m + splits - 1) / splits + 63) / 64 * 4;
  const long long rows = (long long)d.n * d.d * d.h * ((d.w + TX - 1) / TX);   // steps in all, without empty ones
  return (int)std::min<long long>(kChain, theirs * row_tiles(d) / std::max(rows, 1ll));
}

bool encode_tensor(CUtensorMap* map, const void* t, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                   const cuuint32_t* box) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  return enc && enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(t), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int COUT, int G, int ND>
cudaError_t launch_rows(const nm_conv3d_desc& d, const void* x, const void* dy, float* dw, float* db,
                        void* workspace, uint32_t* status, cudaStream_t s) {
  typedef RLayout<COUT, G, ND> L;
  const cuuint64_t c = (cuuint64_t)d.c0, w = (cuuint64_t)d.w, h = (cuuint64_t)d.h, dd = (cuuint64_t)d.d,
                   n = (cuuint64_t)d.n, co = COUT;
  const int nchunks = (d.c0 + 15) / 16;
  CUtensorMap mx, my;
  // X as (channel of the chunk, x, chunk, y, plane of all batch items)
  const cuuint64_t xd[5] = {std::min<cuuint64_t>(c, 16), w, (cuuint64_t)nchunks, h, dd * n};
  const cuuint64_t xs[4] = {c * 2, 32, w * c * 2, h * w * c * 2};
  const cuuint32_t xb[5] = {16, RX, (cuuint32_t)G, PY, 1};
  const cuuint64_t yd[5] = {co, w, h, dd, n};
  const cuuint64_t ys[4] = {co * 2, w * co * 2, h * w * co * 2, dd * h * w * co * 2};
  const cuuint32_t yb[5] = {16, RX, TY, TZ, 1};
  if (!encode_tensor(&mx, x, 5, xd, xs, xb) || !encode_tensor(&my, dy, 5, yd, ys, yb)) return cudaErrorInvalidValue;
  RGrid g;
  g.n = d.n; g.d = d.d; g.h = d.h; g.w = d.w;
  g.tiles_x = (d.w + TX - 1) / TX;
  g.tiles_y = (d.h + TY - 1) / TY;
  g.tiles_z = (d.d + TZ - 1) / TZ;
  g.tiles = row_tiles(d);
  g.cin = d.c0;
  g.kpad = conv_kpad(d.c0);
  g.chain = row_chain(d);
  const dim3 grid = row_grid(d);
  const cudaError_t e = cudaFuncSetAttribute(wgrad_rows_kernel<COUT, G, ND>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::kSmem);
  if (e != cudaSuccess) return e;
  wgrad_rows_kernel<COUT, G, ND><<<grid, kThreads, L::kSmem, s>>>(mx, my, g, (float*)workspace, status);
  float* const part = (float*)workspace;
  const int len = g.kpad * COUT;
  wgrad_rows_reduce<<<len / 128, 256, 0, s>>>((const float4*)part, grid.x, len / 4, g.kpad, 27 * d.c0, (float4*)dw,
                                           status);
  if (db) bias_grad(d, dy, part + (size_t)grid.x * len, db, s);
  return cudaGetLastError();
}

}  // namespace

bool conv_wgrad_rows_ok(const nm_conv3d_desc& d) {
  // NM_CONV_GATHER=1 and NM_WGRAD_TILE_UNPACKED=1 force the other kernels (all forms are tested)
  const char* gather = getenv("NM_CONV_GATHER");
  const char* tile = getenv("NM_WGRAD_TILE_UNPACKED");
  if ((gather && gather[0] == '1') || (tile && tile[0] == '1')) return false;
  if (d.c1 || d.src0_coarse || (d.c0 != 8 && d.c0 % 16)) return false;
  // Up to 32 outputs and one chunk: the shifted-window kernel's MMAs have N = 48
  // as well (4 x 64^3 voxels, 16 -> 16 channels: 116 us a call there, 125 here).
  // Two chunks: 636 there, 240 here (32 -> 32); three: 283 and 150 (48 -> 16).
  if (d.cout == 16 || d.cout == 32) return d.c0 > 16;
  // 64 and 128 outputs: where the gather kernel's sums are short, this kernel's
  // would be longer than they (row_chain), and a layer that small gains little
  // here: from two tiles a sum on.  With 128 outputs the read-out of 27 x inputs
  // x outputs counts too.  Microseconds a call with the gather and here, below
  // and above each line.  64 outputs: 4 x 16^3 voxels of 64 inputs 77, 84; 2 x 20
  // x 33 x 33 of 32 89, 81; 2 x 40 x 60 x 60 of 128 1307, 443.  128 outputs: 4 x
  // 24^3 of 64 178, 202; 4 x 30 x 26 x 26 of 64 298, 260, of 128 567, 464.
  if (row_chain(d) < 2) return false;
  const long long work = (long long)d.n * d.d * d.h * d.w * d.c0;
  return d.cout == 64 || (d.cout == 128 && work >= 1 << 22);
}

size_t conv_wgrad_rows_workspace(const nm_conv3d_desc& d) {
  return ((size_t)row_grid(d).x * conv_kpad(d.c0) + kBiasBlocks) * d.cout * sizeof(float);
}

cudaError_t conv3d_wgrad_rows(const nm_conv3d_desc& d, const void* x, const void* dy, float* dw, float* db,
                              void* workspace, uint32_t* status, cudaStream_t s) {
  const RForm f = row_form(d);
  switch (d.cout * 100 + f.g * 10 + f.nd) {
    case 1623: return launch_rows<16, 2, 3>(d, x, dy, dw, db, workspace, status, s);
    case 1633: return launch_rows<16, 3, 3>(d, x, dy, dw, db, workspace, status, s);
    case 3221: return launch_rows<32, 2, 1>(d, x, dy, dw, db, workspace, status, s);
    case 3231: return launch_rows<32, 3, 1>(d, x, dy, dw, db, workspace, status, s);
    case 6411: return launch_rows<64, 1, 1>(d, x, dy, dw, db, workspace, status, s);
    case 6421: return launch_rows<64, 2, 1>(d, x, dy, dw, db, workspace, status, s);
    case 12811: return launch_rows<128, 1, 1>(d, x, dy, dw, db, workspace, status, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace nm
