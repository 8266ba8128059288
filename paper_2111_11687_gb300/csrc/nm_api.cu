// C ABI of libnmdose (include/nm_dose.h): argument checks, device memory,
// the batch loop of nm_dose_run, and the read-out calls.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <deque>
#include <functional>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "nm_internal.cuh"
#include "nm_scratch.cuh"
#include "nm_trace.h"

using namespace nm;

namespace {

thread_local std::string g_err;

nm_status fail(nm_status st, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  g_err = buf;
  return st;
}

nm_status cuda_fail(cudaError_t e, const char* what) {
  if (e == cudaErrorMemoryAllocation)
    return fail(NM_ERR_OOM, "%s: %s", what, cudaGetErrorString(e));
  return fail(NM_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define NM_CUDA(call, what)                         \
  do {                                              \
    cudaError_t e_ = (call);                        \
    if (e_ != cudaSuccess) return cuda_fail(e_, what); \
  } while (0)

bool is_device_ptr(const void* p) {
  if (!p) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Klein-Nishina total cross section per electron (cm^2), FP64, with ln(1 + 2k)
// taken by log1p so that the low-energy end keeps its digits.
double sigma_kn(double e_mev) {
  const double k = e_mev / kElectronMassMeV;
  const double a = 1.0 + 2.0 * k;
  const double l = std::log1p(2.0 * k);
  const double t1 = (1.0 + k) / (k * k) * (2.0 * (1.0 + k) / a - l / k);
  const double t2 = l / (2.0 * k);
  const double t3 = (1.0 + 3.0 * k) / (a * a);
  return 2.0 * M_PI * kClassicalRadiusCm * kClassicalRadiusCm * (t1 + t2 - t3);
}

// Inverse CDF of the allowed beta+ spectrum, in FP64: with T the kinetic
// energy, E = T + m c^2 and p c = sqrt(T (T + 2 m c^2)),
//   N(T) = F p E (T_max - T)^2,  F = 2 pi eta / (1 - exp(-2 pi eta)),
//   eta = -Z alpha E / (p c)  (the non-relativistic Fermi function, positron),
// integrated by the trapezoid rule on 2^16 panels; node i of the table is the
// energy below which a fraction i / kBetaTable of the positrons lie (linear in
// the cumulative sum between panel edges).
// Several branches (endpoint T_b, fraction I_b of the decays) make the
// mixture sum_b I_b N_b(T) / integral(N_b); for an electron (sign -1) eta
// changes sign (attraction: F > 1).
// Every branch's density is evaluated once per panel edge (it was four times:
// 5.1 ms of host time per branch and handle before, 1.5 now).
std::vector<float> build_beta_inverse_cdf(const double* t_maxs, const double* inten, int n, int z, int sign) {
  constexpr double kAlpha = 7.2973525693e-3;
  auto density = [&](double t, double t_max) {
    if (!(t > 0.0) || !(t < t_max)) return 0.0;
    const double e = t + kElectronMassMeV;
    const double pc = std::sqrt(t * (t + 2.0 * kElectronMassMeV));
    double f = 1.0;
    if (z > 0) {
      const double x = -2.0 * M_PI * sign * z * kAlpha * e / pc;
      f = x / -std::expm1(-x);
    }
    return f * pc * e * (t_max - t) * (t_max - t);
  };
  double t_max = 0.0, itot = 0.0;
  for (int b = 0; b < n; ++b) {
    t_max = std::max(t_max, t_maxs[b]);
    itot += inten[b];
  }
  constexpr int kPanels = 1 << 16;
  const double h = t_max / kPanels;
  std::vector<double> mix(kPanels + 1, 0.0), den(kPanels + 1);   // mixture and branch at the panel edges
  for (int b = 0; b < n; ++b) {
    for (int i = 0; i <= kPanels; ++i) den[i] = density(i * h, t_maxs[b]);
    double norm = 0.0;
    for (int i = 0; i < kPanels; ++i) norm += 0.5 * h * (den[i] + den[i + 1]);
    const double weight = norm > 0.0 ? inten[b] / itot / norm : 0.0;
    for (int i = 0; i <= kPanels; ++i) mix[i] += weight * den[i];
  }
  std::vector<double> cum(kPanels + 1, 0.0);
  for (int i = 0; i < kPanels; ++i) cum[i + 1] = cum[i] + 0.5 * h * (mix[i] + mix[i + 1]);
  std::vector<float> tab(kBetaTable + 1);
  tab[0] = 0.0f;
  tab[kBetaTable] = (float)t_max;
  int j = 0;
  for (int i = 1; i < kBetaTable; ++i) {
    const double target = cum[kPanels] * i / kBetaTable;
    while (cum[j + 1] < target) ++j;
    const double w = (target - cum[j]) / (cum[j + 1] - cum[j]);
    tab[i] = (float)((j + w) * h);
  }
  return tab;
}

// The table is a function of the decay data alone: the last few radionuclides'
// tables are kept (by value, oldest out first; 4 KB each), as the
// Klein-Nishina tables are, so that a handle of a radionuclide in use costs no
// host integration.
std::vector<float> beta_inverse_cdf(const double* t_maxs, const double* inten, int n, int z, int sign) {
  constexpr size_t kKept = 16;
  static std::mutex mu;
  static std::deque<std::pair<std::vector<double>, std::vector<float>>> kept;
  std::vector<double> key{(double)z, (double)sign};
  key.insert(key.end(), t_maxs, t_maxs + n);
  key.insert(key.end(), inten, inten + n);
  {
    std::lock_guard<std::mutex> lock(mu);
    for (auto& k : kept)
      if (k.first == key) return k.second;
  }
  // integrated outside the lock: other threads' handles do not wait for it
  std::vector<float> tab = build_beta_inverse_cdf(t_maxs, inten, n, z, sign);
  std::lock_guard<std::mutex> lock(mu);
  for (auto& k : kept)
    if (k.first == key) return tab;
  if (kept.size() == kKept) kept.pop_front();
  kept.emplace_back(std::move(key), tab);
  return tab;
}

std::vector<float> beta_inverse_cdf(double t_max, int z) {
  const double one = 1.0;
  return beta_inverse_cdf(&t_max, &one, 1, z, 1);
}

// Fault injection for the tests: the n-th device allocation from now (through
// dalloc) fails as if the device were out of memory, the n-th step of a run
// (enqueue_run) fails instead of going to the device (0 = off).
std::atomic<int> g_fail_alloc{0}, g_fail_enqueue{0};

bool fail_now(std::atomic<int>& left) {
  int k = left.load();
  while (k > 0 && !left.compare_exchange_weak(k, k - 1)) {
  }
  return k == 1;
}

// Device buffers of handles and of per-call temporaries are recycled: dfree
// keeps a buffer (once nothing on the device can still use it) for the next
// dalloc of the same size on the same device, so that a handle created after
// one of the same grid is destroyed maps no new memory.  At most kCacheBytes
// stay cached; a failed cudaMalloc releases the cache and retries;
// nm_release_cached_memory releases it on request.
constexpr size_t kCacheBytes = 8ull << 30;
struct BufferCache {
  std::mutex mu;
  std::map<void*, std::pair<int, size_t>> live;          // dalloc'd: device, bytes
  std::multimap<std::pair<int, size_t>, void*> free;     // kept for reuse
  size_t cached = 0;
};
BufferCache& buffer_cache() {
  static BufferCache* c = new BufferCache();   // never destroyed: outlives every handle
  return *c;
}

// Memory for the batch tallies of runs under way, beyond the one that a handle
// keeps: all zero, since a fold leaves its tallies so, and taken by a run for as
// long as it lasts, so that handles share it however many they are and a new
// handle's first run finds it cleared.  Idle buffers are kept up to kIdleTallies,
// or what the live handles' runs ask for (`wants`) in a share of the device, and given back to the
// device by a failed allocation and nm_release_cached_memory.
constexpr uint64_t kIdleTallies = 8ull << 30;
constexpr uint64_t kSlotShare = 8;             // part of a device's memory for tallies beyond a handle's own
struct TallyPool {
  std::mutex mu;                                         // taken after BufferCache::mu, never before
  struct Dev {
    uint64_t total = 0;                                  // bytes of the device, once asked
    uint64_t busy = 0, idle = 0, wants = 0;
    uint64_t keep() const { return std::max(kIdleTallies, std::min(wants, total / kSlotShare)); }
    std::deque<std::pair<ull*, uint64_t>> free;          // idle buffers and their bytes, latest first
    // Takes the oldest idle buffers out until `most` bytes stay; to be freed after mu.
    void trim(uint64_t most, std::vector<ull*>& out) {
      while (idle > most) {
        out.push_back(free.back().first);
        idle -= free.back().second;
        free.pop_back();
      }
    }
  };
  std::map<int, Dev> dev;
};
TallyPool& tally_pool() {
  static TallyPool* p = new TallyPool();       // never destroyed, as the buffer cache
  return *p;
}

void release_cache_locked(BufferCache& c) {
  for (auto& kv : c.free) cudaFree(kv.second);
  c.free.clear();
  c.cached = 0;
  std::vector<ull*> out;
  {
    std::lock_guard<std::mutex> lock(tally_pool().mu);
    for (auto& kv : tally_pool().dev) kv.second.trim(0, out);
  }
  for (ull* p : out) {
    c.live.erase(p);
    cudaFree(p);
  }
}

template <class T>
cudaError_t dalloc(T** p, size_t n) {
  if (fail_now(g_fail_alloc)) {
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  const size_t bytes = n * sizeof(T) > 0 ? n * sizeof(T) : 1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  BufferCache& c = buffer_cache();
  std::lock_guard<std::mutex> lock(c.mu);
  auto it = c.free.find(std::make_pair(dev, bytes));
  if (it != c.free.end()) {
    *p = (T*)it->second;
    c.free.erase(it);
    c.cached -= bytes;
  } else {
    e = cudaMalloc((void**)p, bytes);
    if (e == cudaErrorMemoryAllocation) {
      cudaGetLastError();
      release_cache_locked(c);
      e = cudaMalloc((void**)p, bytes);
    }
    if (e != cudaSuccess) return e;
  }
  c.live[(void*)*p] = std::make_pair(dev, bytes);
  return cudaSuccess;
}

// Memory pools of stream_alloc, one per device, made at its first use there.
struct StreamPools {
  std::mutex mu;
  std::map<int, cudaMemPool_t> pool;
};
StreamPools& stream_pools() {
  static StreamPools* p = new StreamPools();   // never destroyed, as the buffer cache
  return *p;
}

// Returns a dalloc'd buffer; the caller guarantees that no device work still
// uses it (its stream was synchronised).  Other pointers are cudaFree'd.
void dfree(void* p) {
  if (!p) return;
  BufferCache& c = buffer_cache();
  std::lock_guard<std::mutex> lock(c.mu);
  auto it = c.live.find(p);
  if (it == c.live.end()) {
    cudaFree(p);
    return;
  }
  const std::pair<int, size_t> key = it->second;
  c.live.erase(it);
  if (c.cached + key.second > kCacheBytes) {
    cudaFree(p);
    return;
  }
  c.free.emplace(key, p);
  c.cached += key.second;
}

// Frees a dalloc'd buffer at once (cudaFree, with its synchronisation),
// bypassing the cache: for per-call temporaries of the check entry points.
void dfree_now(void* p) {
  if (!p) return;
  {
    BufferCache& c = buffer_cache();
    std::lock_guard<std::mutex> lock(c.mu);
    c.live.erase(p);
  }
  cudaFree(p);
}

}  // namespace

// Inverse CDF of the Klein-Nishina distribution of x = 1 - cos(theta) (per
// unit x proportional to P^2 (P + 1/P - x (2 - x)), P = 1 / (1 + k x),
// k = E / m c^2) at kKnInvE energies log spaced over [e_lo, e_hi]: node j of
// row i is the x below which a fraction j / kKnInvU of the scatters at energy
// i lie.  Trapezoid rule on 2^12 panels in FP64 (CDF error ~1e-7), linear
// between panel edges.
static std::vector<float> build_kn_inverse_cdf(double e_lo, double e_hi) {
  constexpr int kPanels = 1 << 12;
  std::vector<float> tab((size_t)kKnInvE * (kKnInvU + 1));
  std::vector<double> cum(kPanels + 1);
  const double dln = (std::log(e_hi) - std::log(e_lo)) / (kKnInvE - 1);
  const double h = 2.0 / kPanels;
  for (int i = 0; i < kKnInvE; ++i) {
    const double k = std::exp(std::log(e_lo) + i * dln) / kElectronMassMeV;
    auto f = [k](double x) {
      const double P = 1.0 / (1.0 + k * x);
      return P * P * (P + 1.0 / P - x * (2.0 - x));
    };
    cum[0] = 0.0;
    double prev = f(0.0);
    for (int q = 0; q < kPanels; ++q) {
      const double next = f((q + 1) * h);
      cum[q + 1] = cum[q] + 0.5 * h * (prev + next);
      prev = next;
    }
    float* row = &tab[(size_t)i * (kKnInvU + 1)];
    row[0] = 0.0f;
    row[kKnInvU] = 2.0f;
    int q = 0;
    for (int j = 1; j < kKnInvU; ++j) {
      const double target = cum[kPanels] * j / kKnInvU;
      while (cum[q + 1] < target) ++q;
      row[j] = (float)((q + (target - cum[q]) / (cum[q + 1] - cum[q])) * h);
    }
  }
  return tab;
}

// The table depends only on (cutoff, source energy): built once per pair and
// kept, so that creating a handle costs no host integration after the first.
const std::vector<float>& nm::kn_inverse_cdf(double e_lo, double e_hi) {
  static std::mutex mu;
  static std::map<std::pair<double, double>, std::vector<float>> cache;
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find({e_lo, e_hi});
  if (it == cache.end()) it = cache.emplace(std::make_pair(e_lo, e_hi), build_kn_inverse_cdf(e_lo, e_hi)).first;
  return it->second;
}

struct nm_dose {
  int nx = 0, ny = 0, nz = 0;
  float dx = 0, dy = 0, dz = 0;
  int64_t V = 0;
  nm_options opt{};
  int n_mat = 0;
  MaterialCoef mat[NM_MAX_MATERIALS]{};
  int rayleigh = 0;
  float cut = 0.01f;
  float e0 = 0.511f;
  int32_t q_e0 = 0, q_pos = 0;
  float ln_e_lo = 0, inv_dln = 0;
  cudaStream_t stream = nullptr;
  int device = 0, sms = 0;
  // device memory
  uint32_t* vox = nullptr;
  float* density = nullptr;
  uint8_t* labels = nullptr;
  unsigned long long* label_bad = nullptr;   // create-time label check: lowest offending voxel
  uint4* alias = nullptr;
  int64_t n_active = 0;
  ull* tb = nullptr;
  ull* tsum = nullptr;
  double* s2 = nullptr;
  float* kn = nullptr;
  float* minv = nullptr;
  float* minv_out = nullptr;
  float* beta_tab = nullptr;   // beta+ spectrum inverse CDF (kBetaTable + 1), or NULL
  float* kn_inv = nullptr;     // Klein-Nishina inverse CDF [kKnInvE][kKnInvU + 1]
  float kn_inv_lo = 0, kn_inv_idln = 0;
  int32_t q_beta_max = 0;      // q_units(beta endpoint): bound of one positron's energy
  // another radionuclide: annihilation pair on/off, gamma lines; `nuclide`
  // selects the transport variant that handles them (and the beta track)
  int annihilate = 1;
  int n_gamma = 0;
  float gamma_e[kMaxGammaLines] = {};
  int32_t gamma_q[kMaxGammaLines] = {};
  float gamma_y[kMaxGammaLines] = {};
  uint64_t q_gamma_sum = 0;
  bool nuclide = false;
  ull* s2h_lo = nullptr;       // history statistics (history_sigma): 128-bit sums of squares
  ull* s2h_hi = nullptr;
  ull* q_lo = nullptr;         // a launch's sums of their low and high 32 bits, zero between runs unless `broken`
  ull* q_hi = nullptr;
  // Counters, kCtrCount and a zero; the same before the launch under way, and
  // in the place of the zero the launch's work counter: one copy before a launch
  // sets both.
  ull* counters = nullptr;
  ull* kept = nullptr;
  unsigned* work = nullptr;    // in kept
  // tb: a batch tally [V], all zero between runs unless `broken`, for runs that
  // take no others (take_tallies).
  uint64_t want_bytes = 0;     // of the tallies that this handle's last run asked for, in TallyPool's `wants`
  int part_slots = 2;          // batches that organ_partial holds
  // A run ended in the middle of a fold: the statistics are not those of the
  // histories counted, and runs and read-outs are refused until reset or restore.
  bool broken = false;
  uint32_t* status = nullptr;
  uint32_t* rho_max_bits = nullptr;
  double* org_s1 = nullptr;
  double* org_s2 = nullptr;
  long long* organ_count = nullptr;
  double* organ_partial = nullptr;
  double* organ_out = nullptr;
  float* out_dose = nullptr;
  float* out_sigma = nullptr;
  // host state
  uint64_t hist_next = 0;         // histories simulated (the N of Eq. 1)
  uint64_t id_next = 0;           // id of the next history (RNG key with the seed)
  uint64_t n_batches = 0;
  uint32_t status_seen = 0;
  double transport_ms = 0, fold_ms = 0;
  int block = 256, chunk = 256, warp_agg = 0, regroup = 0, regroup_lanes = 12, grid = 0;
  std::vector<cudaEvent_t> ev;
  float blo[3] = {0, 0, 0}, bhi[3] = {0, 0, 0};  // tracking box, voxel units
  bool tuned = false;             // launch shape chosen by the autotuner

  ~nm_dose() {
    // nothing on the device may still use a buffer that is recycled
    cudaStreamSynchronize(stream);
    void* ptrs[] = {vox, density, labels, label_bad, alias, tb, tsum, s2, kn, minv, minv_out, beta_tab, kn_inv, s2h_lo, s2h_hi, q_lo, q_hi, counters, kept, status,
                    rho_max_bits, org_s1, org_s2, organ_count, organ_partial, organ_out,
                    out_dose, out_sigma};
    for (void* p : ptrs) dfree(p);
    for (auto e : ev) cudaEventDestroy(e);
    if (want_bytes) {
      std::vector<ull*> out;
      {
        std::lock_guard<std::mutex> lock(tally_pool().mu);
        TallyPool::Dev& d = tally_pool().dev[device];
        d.wants -= want_bytes;
        d.trim(d.keep(), out);
      }
      for (ull* p : out) dfree_now(p);
    }
  }

  int kind() const {
    return nuclide_kind(opt.source_mode == NM_SOURCE_DECAY, beta_tab != nullptr, annihilate != 0, n_gamma);
  }

  PatientGeom geom(uint64_t first, uint64_t n) const {
    PatientGeom g;
    memset(&g, 0, sizeof g);
    g.vox = vox;
    g.alias = alias;
    g.tally = tb;
    g.slot_stride = (uint32_t)V;
    g.split.slots = 1;
    g.counters = counters;
    g.work = work;
    g.n_active = (uint64_t)n_active;
    g.hist_begin = first;
    g.n_hist = n;
    g.nx = nx; g.ny = ny; g.nz = nz;
    g.fnx = (float)nx; g.fny = (float)ny; g.fnz = (float)nz;
    g.inv_dx = 1.0f / dx; g.inv_dy = 1.0f / dy; g.inv_dz = 1.0f / dz;
    g.source_mode = opt.source_mode;
    g.px = opt.point[0] / dx; g.py = opt.point[1] / dy; g.pz = opt.point[2] / dz;
    g.q_positron = beta_tab ? 0 : q_pos;
    g.beta_tab = beta_tab;
    for (int a = 0; a < 3; ++a) {
      g.blo[a] = blo[a];
      g.bhi[a] = bhi[a];
    }
    return g;
  }

  TransportParams params(uint64_t first, uint64_t n, uint64_t seed) const {
    TransportParams p;
    memset(&p, 0, sizeof p);
    p.g = geom(first, n);
    p.status = status;
    p.kn = kn;
    p.minv = minv;
    p.minv_out = minv_out;
    p.kn_inv = opt.kn_sampler == 0 ? kn_inv : nullptr;
    p.kn_inv_lo = kn_inv_lo;
    p.kn_inv_idln = kn_inv_idln;
    p.s2h_lo = q_lo;
    p.s2h_hi = q_hi;
    p.key = philox_key((uint32_t)seed, (uint32_t)(seed >> 32));
    p.e0 = e0;
    p.q_e0 = q_e0;
    p.cut = cut;
    p.n_mat = n_mat;
    for (int m = 0; m < NM_MAX_MATERIALS; ++m) p.mat[m] = mat[m];
    p.ln_e_lo = ln_e_lo;
    p.inv_dln_e = inv_dln;
    p.chunk = chunk;
    p.max_steps = opt.max_steps;
    p.regroup_compton = regroup_lanes;
    p.regroup_refill = regroup_lanes;
    p.annihilate = annihilate;
    p.n_gamma = n_gamma;
    for (int j = 0; j < kMaxGammaLines; ++j) {
      p.gamma_e[j] = gamma_e[j];
      p.gamma_q[j] = gamma_q[j];
      p.gamma_y[j] = gamma_y[j];
    }
    return p;
  }

  double gy_per_unit_vol() const {
    // one tally unit = 2^-6 eV; mass = rho [g/cm^3] * volume [cm^3] * 1e-3 kg/g
    return kJoulePerEv / 64.0 / (1e-3 * (double)dx * (double)dy * (double)dz);
  }
  // Upper bound of one history's energy (the exact value with a constant positron).
  uint64_t units_per_history() const {
    return opt.source_mode == NM_SOURCE_DECAY
               ? (annihilate ? 2ull * (uint64_t)q_e0 : 0ull) + (uint64_t)(beta_tab ? q_beta_max : q_pos) + q_gamma_sum
               : (uint64_t)q_e0;
  }
  // Energy emitted by the histories so far, from the counters of the
  // sampled parts (beta particles, gamma lines).
  int64_t emitted(const ull* v) const {
    if (opt.source_mode != NM_SOURCE_DECAY) return (int64_t)(hist_next * (uint64_t)q_e0);
    return (int64_t)(hist_next * (annihilate ? 2ull * (uint64_t)q_e0 : 0ull) +
                     (beta_tab ? v[kCtrPositronUnits] : hist_next * (uint64_t)q_pos) + v[kCtrGammaUnits]);
  }
};

extern "C" {

void nm_options_default(nm_options* o) {
  if (!o) return;
  memset(o, 0, sizeof *o);
  o->source_mode = NM_SOURCE_DECAY;
  o->photon_mev = 0.511;
  o->positron_mev = 0.25;
  o->batches = 10;
  o->activity_bq = 8.0e-3 * 3.7e10 * std::pow(2.0, -60.0 / 109.77);
  o->n_labels = 0;
  o->block_threads = 0;
  o->chunk = 0;
  o->warp_aggregate = -1;
  o->regroup = -1;
  o->max_steps = 100000;
  o->stream = nullptr;
  o->beta_max_mev = 0.0;
  o->beta_z = 8;
  o->kn_sampler = 0;
  o->no_annihilation = 0;
  o->beta_electron = 0;
  o->n_beta = 0;
  o->n_gamma = 0;
}

const char* nm_last_error(void) { return g_err.c_str(); }

}  // extern "C"

void nm::set_error_message(const char* msg) { g_err = msg; }

cudaError_t nm::stream_alloc(void** p, size_t bytes, cudaStream_t s) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e) return e;
  StreamPools& sp = stream_pools();
  std::lock_guard<std::mutex> lock(sp.mu);
  auto it = sp.pool.find(dev);
  if (it == sp.pool.end()) {
    cudaMemPoolProps props;
    memset(&props, 0, sizeof props);
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    uint64_t keep = kPoolKeep;
    if ((e = cudaMemPoolCreate(&pool, &props))) return e;
    if ((e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep))) {
      cudaMemPoolDestroy(pool);
      return e;
    }
    it = sp.pool.emplace(dev, pool).first;
  }
  return cudaMallocFromPoolAsync(p, bytes, it->second, s);
}

cudaError_t nm::stream_free(void* p, cudaStream_t s) { return cudaFreeAsync(p, s); }

// Checks shared by every entry point that takes a phantom: grid sizes and
// spacing, material constants, energies and options.  The positron energy is
// checked before anything derives fixed-point units from it, so a negative or
// NaN value never reaches q_units() or the overflow bound.
nm_status nm::check_problem(const nm_grid* g, const nm_materials* mt, const nm_options& o, const float* activity) {
  if (!g || !mt) return fail(NM_ERR_ARG, "grid or materials is NULL");
  if (g->nx <= 0 || g->ny <= 0 || g->nz <= 0) return fail(NM_ERR_ARG, "grid dimensions must be > 0");
  const int64_t V = (int64_t)g->nx * g->ny * g->nz;
  if (V >= (int64_t)1 << 31) return fail(NM_ERR_ARG, "grid has %lld voxels; the limit is 2^31 - 1", (long long)V);
  if (!(g->dx > 0 && g->dy > 0 && g->dz > 0) || !std::isfinite(g->dx) || !std::isfinite(g->dy) ||
      !std::isfinite(g->dz))
    return fail(NM_ERR_ARG, "voxel sizes must be finite and > 0");
  if (!g->density || !g->material) return fail(NM_ERR_ARG, "density or material is NULL");
  if (mt->n < 1 || mt->n > NM_MAX_MATERIALS || !mt->z_over_a || !mt->zeff)
    return fail(NM_ERR_ARG, "materials: need 1..%d materials with z_over_a and zeff", NM_MAX_MATERIALS);
  if (o.source_mode != NM_SOURCE_DECAY && o.source_mode != NM_SOURCE_POINT)
    return fail(NM_ERR_ARG, "unknown source_mode %d", o.source_mode);
  if (o.source_mode == NM_SOURCE_DECAY && !activity)
    return fail(NM_ERR_ARG, "decay mode needs an activity map");
  if (!(o.photon_mev > mt->photon_cut_mev) || !(mt->photon_cut_mev > 0) || !(o.photon_mev <= 1.0))
    return fail(NM_ERR_ARG, "need 0 < photon cutoff < photon energy <= 1 MeV");
  if (!(o.positron_mev >= 0) || o.positron_mev > 1.0) return fail(NM_ERR_ARG, "positron energy must be in [0, 1] MeV");
  if (!(o.activity_bq >= 0) || !std::isfinite(o.activity_bq)) return fail(NM_ERR_ARG, "activity_bq must be finite and >= 0");
  if (o.max_steps <= 0) return fail(NM_ERR_ARG, "max_steps must be > 0");
  if (o.kn_sampler != 0 && o.kn_sampler != 1) return fail(NM_ERR_ARG, "kn_sampler must be 0 (table) or 1 (Kahn)");
  if (!(o.beta_max_mev >= 0.0 && o.beta_max_mev < 20.0) || o.beta_z < 0 || o.beta_z > 100)
    return fail(NM_ERR_ARG, "beta_max_mev must be in [0, 20) MeV and beta_z in 0..100");
  if ((o.no_annihilation != 0 && o.no_annihilation != 1) || (o.beta_electron != 0 && o.beta_electron != 1))
    return fail(NM_ERR_ARG, "no_annihilation and beta_electron must be 0 or 1");
  if (o.n_beta < 0 || o.n_beta > kMaxBetaBranches || (o.n_beta > 0 && (!o.beta_endpoint_mev || !o.beta_intensity)))
    return fail(NM_ERR_ARG, "n_beta must be 0..%d with endpoint and intensity arrays", kMaxBetaBranches);
  if (o.n_beta > 0) {
    double sum = 0.0;
    for (int b = 0; b < o.n_beta; ++b) {
      if (!(o.beta_endpoint_mev[b] > 0.0 && o.beta_endpoint_mev[b] < 20.0) || !(o.beta_intensity[b] >= 0.0) ||
          !std::isfinite(o.beta_intensity[b]))
        return fail(NM_ERR_ARG, "beta branch %d: endpoint in (0, 20) MeV and intensity finite and >= 0", b);
      sum += o.beta_intensity[b];
    }
    if (!(sum > 0.0)) return fail(NM_ERR_ARG, "beta branch intensities sum to zero");
  }
  if (o.n_gamma < 0 || o.n_gamma > kMaxGammaLines || (o.n_gamma > 0 && (!o.gamma_mev || !o.gamma_yield)))
    return fail(NM_ERR_ARG, "n_gamma must be 0..%d with energy and yield arrays", kMaxGammaLines);
  for (int j = 0; j < o.n_gamma; ++j)
    if (!(o.gamma_mev[j] > mt->photon_cut_mev && o.gamma_mev[j] <= 1.0) ||
        !(o.gamma_yield[j] >= 0.0 && o.gamma_yield[j] <= 1.0))
      return fail(NM_ERR_ARG, "gamma line %d: energy in (photon cutoff, 1] MeV and yield in [0, 1]", j);
  for (int m = 0; m < mt->n; ++m)
    if (!(mt->z_over_a[m] >= 0) || !(mt->zeff[m] >= 0) || !std::isfinite(mt->z_over_a[m]) ||
        !std::isfinite(mt->zeff[m]))
      return fail(NM_ERR_ARG, "material %d: constants must be finite and >= 0", m);
  if (!(mt->pe_coeff >= 0) || !std::isfinite(mt->pe_coeff) || !std::isfinite(mt->pe_exp) ||
      !(mt->rayleigh_coeff >= 0) || !std::isfinite(mt->rayleigh_coeff))
    return fail(NM_ERR_ARG, "photoelectric and Rayleigh constants must be finite and >= 0");
  if (o.source_mode == NM_SOURCE_POINT) {
    const float L[3] = {g->nx * g->dx, g->ny * g->dy, g->nz * g->dz};
    for (int a = 0; a < 3; ++a)
      if (!(o.point[a] >= 0.0f && o.point[a] < L[a])) return fail(NM_ERR_ARG, "point source outside the grid");
  }
  return NM_OK;
}

extern "C" {

nm_status nm_ct_to_phantom(const int16_t* hu, int64_t n, float* density, uint8_t* material,
                           void* stream) {
  if (n < 0 || (n > 0 && (!hu || !density || !material)))
    return fail(NM_ERR_ARG, "nm_ct_to_phantom: bad arguments");
  if (n == 0) return NM_OK;
  cudaStream_t s = (cudaStream_t)stream;
  const bool din = is_device_ptr(hu), dd = is_device_ptr(density), dm = is_device_ptr(material);
  int16_t* h = nullptr;
  float* d = nullptr;
  uint8_t* m = nullptr;
  nm_status st = NM_OK;
  cudaError_t e = cudaSuccess;
  if (!din) e = dalloc(&h, n);
  if (!e && !dd) e = dalloc(&d, n);
  if (!e && !dm) e = dalloc(&m, n);
  if (!e && !din) e = cudaMemcpyAsync(h, hu, n * sizeof(int16_t), cudaMemcpyHostToDevice, s);
  if (!e) e = launch_ct_to_phantom(din ? hu : h, n, dd ? density : d, dm ? material : m, s);
  if (!e && !dd) e = cudaMemcpyAsync(density, d, n * sizeof(float), cudaMemcpyDeviceToHost, s);
  if (!e && !dm) e = cudaMemcpyAsync(material, m, n, cudaMemcpyDeviceToHost, s);
  if (!e) e = cudaStreamSynchronize(s);
  else cudaStreamSynchronize(s);
  if (e) st = cuda_fail(e, "nm_ct_to_phantom");
  dfree(h);
  dfree(d);
  dfree(m);
  return st;
}

// ---------------------------------------------------------------------------
// Launch shape: explicit options win; every knob left on "auto" is chosen by
// timed trial launches on the handle's own phantom (coordinate descent over
// Compton/new-history regrouping, CTA size and work-chunk size, then warp
// aggregation), cached per (device, grid, source mode, Rayleigh).  Trials use
// history ids above 2^62, which runs never reach, and their tallies and
// counters are cleared afterwards; any shape gives bit-identical results.
// ---------------------------------------------------------------------------
struct Shape {
  int block, chunk, warp_agg, regroup, lanes;
  bool operator<(const Shape& o) const {
    return std::tie(block, chunk, warp_agg, regroup, lanes) <
           std::tie(o.block, o.chunk, o.warp_agg, o.regroup, o.lanes);
  }
};

// (device, grid, source mode, Rayleigh, free-parameter bits + variant bits,
//  the fixed values of the parameters that are not tuned)
typedef std::tuple<int, int, int, int, int, int, int, int, int, int, int, int> TuneKey;
static std::mutex g_tune_mu;
static std::map<TuneKey, Shape> g_tune_cache;

static int grid_for_shape(const nm_dose* h, const Shape& sh) {
  return h->sms * transport_max_blocks_per_sm(sh.block, sh.warp_agg, h->rayleigh, h->opt.kn_sampler != 0,
                                              sh.regroup, h->opt.history_sigma != 0, h->kind());
}

// Histories per work grab of a launch of n: the handle's chunk, but where it is
// tuned (on 2^25 decays) at most half of a warp's share, in warps' widths.  A
// launch of 1e5 in chunks of 256 keeps 391 of 4864 warps busy (point source in
// water, 1e6 histories in ten batches: 0.85 ms in chunks of 256, 0.50 in chunks
// of 32, 0.59 in chunks of 16).
static int launch_chunk(int chunk, uint64_t warps, uint64_t n) {
  const uint64_t share = n / (2 * warps) / 32 * 32;
  return (int)std::min<uint64_t>(chunk, std::max<uint64_t>(share, 32));
}

static void apply_shape(nm_dose* h, const Shape& sh) {
  h->block = sh.block;
  h->chunk = sh.chunk;
  h->warp_agg = sh.warp_agg;
  h->regroup = sh.regroup;
  h->regroup_lanes = sh.lanes;
  h->grid = grid_for_shape(h, sh);
}

static nm_status autotune(nm_dose* h, Shape sh, bool free_block, bool free_chunk, bool free_agg,
                          bool free_regroup, bool free_lanes) {
  const TuneKey key{h->device, h->nx, h->ny, h->nz, h->opt.source_mode, h->rayleigh,
                    (free_block ? 1 : 0) | (free_chunk ? 2 : 0) | (free_agg ? 4 : 0) |
                        (free_regroup ? 8 : 0) | (free_lanes ? 16 : 0) | (h->opt.history_sigma ? 32 : 0) |
                        ((h->kind() + 1) << 6) | (h->opt.kn_sampler ? 256 : 0),
                    free_block ? 0 : sh.block, free_chunk ? 0 : sh.chunk, free_agg ? 0 : sh.warp_agg,
                    free_regroup ? 0 : sh.regroup, free_lanes ? 0 : sh.lanes};
  {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    auto it = g_tune_cache.find(key);
    if (it != g_tune_cache.end()) {
      apply_shape(h, it->second);
      h->tuned = true;
      return NM_OK;
    }
  }
  cudaStream_t s = h->stream;
  cudaEvent_t e0, e1;
  NM_CUDA(cudaEventCreate(&e0), "cudaEventCreate");
  NM_CUDA(cudaEventCreate(&e1), "cudaEventCreate");
  // 2^25 decays (several ms) per trial: shorter trials, dominated by the
  // launch's tail, ranked shapes 1 % apart differently from run to run
  const uint64_t n_trial = 1ull << 25;
  const uint64_t first = 1ull << 62;
  std::map<Shape, float> seen;
  auto trial = [&](const Shape& t, float* ms) -> nm_status {
    auto it = seen.find(t);
    if (it != seen.end()) { *ms = it->second; return NM_OK; }
    apply_shape(h, t);
    if (h->grid <= 0) { *ms = 1e30f; return NM_OK; }
    TransportParams p = h->params(first, n_trial, 0x7475u);
    NM_CUDA(cudaMemsetAsync(h->work, 0, sizeof(unsigned), s), "autotune");
    NM_CUDA(cudaEventRecord(e0, s), "autotune");
    NM_CUDA(launch_transport(p, h->grid, h->block, h->warp_agg, h->rayleigh, h->regroup, s, h->opt.history_sigma != 0),
            "autotune");
    NM_CUDA(cudaEventRecord(e1, s), "autotune");
    NM_CUDA(cudaEventSynchronize(e1), "autotune");
    NM_CUDA(cudaEventElapsedTime(ms, e0, e1), "autotune");
    seen[t] = *ms;
    return NM_OK;
  };
  float ms = 0;
  nm_status st = trial(sh, &ms);  // warm-up (module load, caches)
  seen.clear();
  if (st == NM_OK) st = trial(sh, &ms);
  float best = ms;
  auto consider = [&](Shape t) -> nm_status {
    float m = 0;
    nm_status r = trial(t, &m);
    if (r == NM_OK && m < best) { best = m; sh = t; }
    return r;
  };
  // The ring kernel regroups by itself, 32 photons at a time, so it has no lane
  // count to choose, and regrouping off (the lane kernel) is never faster.
  const bool ring = !h->opt.history_sigma && h->kind() >= 0 && sh.regroup;
  for (int pass = 0; pass < 2 && st == NM_OK; ++pass) {
    if ((free_regroup || free_lanes) && !ring) {
      const int lanes[] = {8, 12, 16};
      for (int l : lanes) {
        if (!free_lanes && l != sh.lanes) continue;
        Shape t = sh; t.regroup = 1; t.lanes = l;
        if ((st = consider(t)) != NM_OK) break;
      }
      if (free_regroup && st == NM_OK) { Shape t = sh; t.regroup = 0; st = consider(t); }
    }
    if (free_block && st == NM_OK)
      for (int b : {128, 256, 512}) { Shape t = sh; t.block = b; if ((st = consider(t)) != NM_OK) break; }
    if (free_chunk && st == NM_OK)
      for (int c : {64, 256, 1024}) { Shape t = sh; t.chunk = c; if ((st = consider(t)) != NM_OK) break; }
    if (free_agg && st == NM_OK)
      for (int a : {0, 1}) { Shape t = sh; t.warp_agg = a; if ((st = consider(t)) != NM_OK) break; }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st != NM_OK) return st;
  apply_shape(h, sh);
  h->tuned = true;
  // Trials tallied into the batch tally and counters: clear them.
  NM_CUDA(cudaMemsetAsync(h->tb, 0, h->V * sizeof(ull), s), "autotune");
  NM_CUDA(cudaMemsetAsync(h->counters, 0, kCtrCount * sizeof(ull), s), "autotune");
  NM_CUDA(cudaMemsetAsync(h->status, 0, sizeof(uint32_t), s), "autotune");
  if (h->s2h_lo) {
    NM_CUDA(cudaMemsetAsync(h->q_lo, 0, h->V * sizeof(ull), s), "autotune");
    NM_CUDA(cudaMemsetAsync(h->q_hi, 0, h->V * sizeof(ull), s), "autotune");
  }
  NM_CUDA(cudaStreamSynchronize(s), "autotune");
  std::lock_guard<std::mutex> lock(g_tune_mu);
  g_tune_cache[key] = sh;
  return NM_OK;
}

static nm_status choose_shape(nm_dose* h) {
  const nm_options& o = h->opt;
  if (o.block_threads > 0 && (o.block_threads % 32 || o.block_threads > 512))
    return fail(NM_ERR_ARG, "block_threads must be a multiple of 32, <= 512");
  if (o.chunk > 0 && o.chunk < 32) return fail(NM_ERR_ARG, "chunk must be >= 32");
  if (o.regroup_lanes > 32) return fail(NM_ERR_ARG, "regroup_lanes must be 1..32");
  Shape sh;
  sh.block = o.block_threads > 0 ? o.block_threads : 256;
  sh.chunk = o.chunk > 0 ? o.chunk : 256;
  // A point source concentrates deposits near the source, where lanes of a
  // warp often hit the same voxel; a spread-out source rarely does.
  sh.warp_agg = o.warp_aggregate >= 0 ? (o.warp_aggregate != 0) : (o.source_mode == NM_SOURCE_POINT);
  if (o.history_sigma || h->nuclide) {
    // per-history totals and positron tracks deposit lane by lane
    if (o.warp_aggregate > 0) return fail(NM_ERR_ARG, "history_sigma and the beta+ spectrum need warp_aggregate = 0");
    sh.warp_agg = 0;
  }
  sh.regroup = o.regroup >= 0 ? (o.regroup != 0) : 1;
  sh.lanes = o.regroup_lanes > 0 ? o.regroup_lanes : 12;
  apply_shape(h, sh);
  if (h->grid <= 0) return fail(NM_ERR_ARG, "transport kernel cannot launch with %d threads", h->block);
  const bool fb = o.block_threads <= 0, fc = o.chunk <= 0, fa = o.warp_aggregate < 0 && !o.history_sigma && !h->nuclide,
             fr = o.regroup < 0, fl = o.regroup_lanes <= 0 && sh.regroup;
  if (fb || fc || fa || fr || fl) return autotune(h, sh, fb, fc, fa, fr, fl);
  return NM_OK;
}

nm_status nm_dose_create(nm_dose** out, const nm_grid* g, const nm_materials* mt,
                         const float* activity, const uint8_t* labels, const nm_options* opts) {
  NvtxRange range("nm_dose_create");
  if (!out) return fail(NM_ERR_ARG, "out is NULL");
  *out = nullptr;
  nm_options o;
  if (opts) o = *opts; else nm_options_default(&o);
  const nm_status cp = check_problem(g, mt, o, activity);
  if (cp != NM_OK) return cp;
  // one batch per call is allowed: the uncertainty needs two batches in total
  if (o.batches < 1) return fail(NM_ERR_ARG, "batches must be >= 1");
  if (o.n_labels < 0 || o.n_labels > NM_MAX_LABELS) return fail(NM_ERR_ARG, "n_labels must be 0..%d", NM_MAX_LABELS);
  const int64_t V = (int64_t)g->nx * g->ny * g->nz;

  nm_dose* h = new nm_dose();
  h->nx = g->nx; h->ny = g->ny; h->nz = g->nz;
  h->dx = g->dx; h->dy = g->dy; h->dz = g->dz;
  h->V = V;
  h->opt = o;
  h->stream = (cudaStream_t)o.stream;
  h->n_mat = mt->n;
  h->rayleigh = mt->rayleigh != 0;
  h->cut = (float)mt->photon_cut_mev;
  h->e0 = (float)o.photon_mev;
  h->q_e0 = q_units(h->e0);
  h->q_pos = o.source_mode == NM_SOURCE_DECAY ? q_units((float)o.positron_mev) : 0;
  // The tables span the highest photon energy: the annihilation photons' or
  // a gamma line's.
  double e_top = o.photon_mev;
  if (o.source_mode == NM_SOURCE_DECAY) {
    h->annihilate = o.no_annihilation ? 0 : 1;
    h->n_gamma = o.n_gamma;
    for (int j = 0; j < o.n_gamma; ++j) {
      h->gamma_e[j] = (float)o.gamma_mev[j];
      h->gamma_q[j] = q_units(h->gamma_e[j]);
      h->gamma_y[j] = (float)o.gamma_yield[j];
      h->q_gamma_sum += (uint64_t)h->gamma_q[j];
      e_top = std::max(e_top, o.gamma_mev[j]);
    }
    h->nuclide = o.beta_max_mev > 0.0 || o.n_beta > 0 || o.n_gamma > 0 || o.no_annihilation;
  }
  auto bail = [&](nm_status st) { delete h; return st; };

  cudaError_t e;
  if ((e = cudaGetDevice(&h->device))) return bail(cuda_fail(e, "cudaGetDevice"));
  if ((e = cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, h->device)))
    return bail(cuda_fail(e, "cudaDeviceGetAttribute"));
  cudaStream_t s = h->stream;

  // Physics tables: N_A sigma_KN(E) on a log-energy grid (FP64 -> FP32).
  const double e_lo = 0.5 * mt->photon_cut_mev, e_hi = 1.05 * e_top;
  const double dln = (std::log(e_hi) - std::log(e_lo)) / (kKnTable - 1);
  h->ln_e_lo = (float)std::log(e_lo);
  h->inv_dln = (float)(1.0 / dln);
  std::vector<float> kn(kKnTable);
  for (int i = 0; i < kKnTable; ++i)
    kn[i] = (float)(kAvogadro * sigma_kn(std::exp(std::log(e_lo) + i * dln)));
  for (int m = 0; m < mt->n; ++m) {
    h->mat[m].za = (float)mt->z_over_a[m];
    h->mat[m].zp = (float)(mt->pe_coeff * std::pow(mt->zeff[m], mt->pe_exp));
    h->mat[m].zr = h->rayleigh ? (float)(mt->rayleigh_coeff * mt->zeff[m] * mt->zeff[m]) : 0.0f;
  }

  if ((e = dalloc(&h->vox, V)) || (e = dalloc(&h->density, V)) || (e = dalloc(&h->tb, V)) ||
      (e = dalloc(&h->tsum, V)) || (e = dalloc(&h->s2, V)) || (e = dalloc(&h->kn, kKnTable)) ||
      (e = dalloc(&h->minv, kKnTable)) || (e = dalloc(&h->minv_out, kKnTable)) ||
      (e = dalloc(&h->counters, kCtrCount + 1)) || (e = dalloc(&h->kept, kCtrCount + 1)) ||
      (e = dalloc(&h->status, 1)) || (e = dalloc(&h->rho_max_bits, NM_MAX_MATERIALS)) ||
      (e = dalloc(&h->org_s1, kLabelSlots)) || (e = dalloc(&h->org_s2, kLabelSlots)) ||
      (e = dalloc(&h->organ_count, kLabelSlots)) ||
      (e = dalloc(&h->organ_partial, (size_t)organ_tiles(V) * 2 * kLabelSlots)) ||
      (e = dalloc(&h->organ_out, 4 * kLabelSlots)))
    return bail(cuda_fail(e, "device allocation"));
  h->work = reinterpret_cast<unsigned*>(h->kept + kCtrCount);
  if (labels && ((e = dalloc(&h->labels, V)) || (e = dalloc(&h->label_bad, 1))))
    return bail(cuda_fail(e, "device allocation"));
  {
    const std::vector<float>& kt = kn_inverse_cdf(mt->photon_cut_mev, e_top);
    h->kn_inv_lo = (float)std::log(mt->photon_cut_mev);
    h->kn_inv_idln = (float)((kKnInvE - 1) / (std::log(e_top) - std::log(mt->photon_cut_mev)));
    if ((e = dalloc(&h->kn_inv, kt.size())) ||
        (e = cudaMemcpyAsync(h->kn_inv, kt.data(), kt.size() * sizeof(float), cudaMemcpyHostToDevice, s)) ||
        (e = cudaStreamSynchronize(s)))
      return bail(cuda_fail(e, "Klein-Nishina table"));
  }
  std::vector<float> beta;
  if (o.source_mode == NM_SOURCE_DECAY && (o.beta_max_mev > 0.0 || o.n_beta > 0)) {
    const double one = 1.0;
    const int sign = o.beta_electron ? -1 : 1;
    if (o.n_beta > 0) {
      beta = beta_inverse_cdf(o.beta_endpoint_mev, o.beta_intensity, o.n_beta, o.beta_z, sign);
      double tm = 0.0;
      for (int b = 0; b < o.n_beta; ++b) tm = std::max(tm, o.beta_endpoint_mev[b]);
      h->q_beta_max = q_units((float)tm);
    } else {
      beta = beta_inverse_cdf(&o.beta_max_mev, &one, 1, o.beta_z, sign);
      h->q_beta_max = q_units((float)o.beta_max_mev);
    }
    if ((e = dalloc(&h->beta_tab, kBetaTable + 1)) ||
        (e = cudaMemcpyAsync(h->beta_tab, beta.data(), (kBetaTable + 1) * sizeof(float), cudaMemcpyHostToDevice, s)))
      return bail(cuda_fail(e, "beta table"));
  }
  if (o.history_sigma) {
    if ((e = dalloc(&h->s2h_lo, V)) || (e = dalloc(&h->s2h_hi, V)) || (e = dalloc(&h->q_lo, V)) ||
        (e = dalloc(&h->q_hi, V)) || (e = cudaMemsetAsync(h->q_lo, 0, V * sizeof(ull), s)) ||
        (e = cudaMemsetAsync(h->q_hi, 0, V * sizeof(ull), s)) ||
        (e = cudaMemsetAsync(h->s2h_lo, 0, V * sizeof(ull), s)) || (e = cudaMemsetAsync(h->s2h_hi, 0, V * sizeof(ull), s)))
      return bail(cuda_fail(e, "device allocation"));
  }

  uint8_t* mat_dev = nullptr;
  if ((e = dalloc(&mat_dev, V))) return bail(cuda_fail(e, "device allocation"));
  e = cudaMemcpyAsync(h->density, g->density, V * sizeof(float), cudaMemcpyDefault, s);
  if (!e) e = cudaMemcpyAsync(mat_dev, g->material, V, cudaMemcpyDefault, s);
  if (!e && labels) e = cudaMemcpyAsync(h->labels, labels, V, cudaMemcpyDefault, s);
  if (!e) e = cudaMemcpyAsync(h->kn, kn.data(), kKnTable * sizeof(float), cudaMemcpyHostToDevice, s);
  if (!e) e = cudaMemsetAsync(h->status, 0, sizeof(uint32_t), s);
  if (!e) e = cudaMemsetAsync(h->rho_max_bits, 0, NM_MAX_MATERIALS * sizeof(uint32_t), s);
  if (!e) e = launch_pack_voxels(h->density, mat_dev, V, h->n_mat, h->vox, h->rho_max_bits, h->status, s);
  uint32_t rho_bits[NM_MAX_MATERIALS] = {0};
  uint32_t st = 0;
  if (!e) e = cudaMemcpyAsync(rho_bits, h->rho_max_bits, sizeof rho_bits, cudaMemcpyDeviceToHost, s);
  if (!e) e = cudaMemcpyAsync(&st, h->status, 4, cudaMemcpyDeviceToHost, s);
  if (!e) e = cudaStreamSynchronize(s);
  else cudaStreamSynchronize(s);
  dfree(mat_dev);
  if (e) return bail(cuda_fail(e, "nm_dose_create: upload"));
  if (st & NM_DEV_BAD_VOXEL)
    return bail(fail(NM_ERR_ARG, "density must be finite and > 0 and material < %d in every voxel", h->n_mat));
  for (int m = 0; m < NM_MAX_MATERIALS; ++m) {
    float r;
    memcpy(&r, &rho_bits[m], 4);
    h->mat[m].rho_max = m < h->n_mat ? r : 0.0f;
  }
  // Woodcock majorants per table bin: over the whole grid, and outside the
  // tracking box around the body.
  float rho_max[NM_MAX_MATERIALS], rho_out[NM_MAX_MATERIALS];
  for (int m = 0; m < NM_MAX_MATERIALS; ++m) rho_max[m] = h->mat[m].rho_max;
  {
    int* box_dev = nullptr;
    if ((e = dalloc(&box_dev, 16))) return bail(cuda_fail(e, "device allocation"));
    e = woodcock_regions(h->vox, h->nx, h->ny, h->nz, box_dev, (uint32_t*)(box_dev + 8), h->blo, h->bhi, rho_out, s);
    if (e) cudaStreamSynchronize(s);   // on success it has synchronised: nothing uses the buffer
    dfree(box_dev);
    if (e) return bail(cuda_fail(e, "tracking regions"));
  }
  std::vector<float> minv(kKnTable), minv_out(kKnTable);
  majorant_table(h->mat, h->n_mat, rho_max, kn.data(), e_lo, dln, minv.data());
  majorant_table(h->mat, h->n_mat, rho_out, kn.data(), e_lo, dln, minv_out.data());
  if ((e = cudaMemcpy(h->minv, minv.data(), kKnTable * sizeof(float), cudaMemcpyHostToDevice)) ||
      (e = cudaMemcpy(h->minv_out, minv_out.data(), kKnTable * sizeof(float), cudaMemcpyHostToDevice)))
    return bail(cuda_fail(e, "majorant table"));

  // Decay sampler: alias table over the active voxels, FP64 on the device.
  if (o.source_mode == NM_SOURCE_DECAY) {
    float* act = nullptr;
    uint8_t* scratch = nullptr;
    if ((e = dalloc(&act, V)) || (e = dalloc(&scratch, AliasScratch::bytes(V)))) {
      dfree(act);
      return bail(cuda_fail(e, "alias scratch"));
    }
    e = cudaMemcpyAsync(act, activity, V * sizeof(float), cudaMemcpyDefault, s);
    if (!e) e = dalloc(&h->alias, V);
    if (!e) e = build_alias_table(act, V, AliasScratch{scratch}, h->alias, &h->n_active, h->status, s);
    if (!e) e = cudaMemcpyAsync(&st, h->status, 4, cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaStreamSynchronize(s);
    else cudaStreamSynchronize(s);
    dfree(act);
    dfree(scratch);
    if (e) return bail(cuda_fail(e, "alias table"));
    if (st & NM_DEV_BAD_ACTIVITY) return bail(fail(NM_ERR_ARG, "activity must be finite and >= 0"));
    if (h->n_active == 0) return bail(fail(NM_ERR_ARG, "activity map sums to zero"));
  }

  e = cudaMemsetAsync(h->tb, 0, V * sizeof(ull), s);
  if (!e) e = cudaMemsetAsync(h->tsum, 0, V * sizeof(ull), s);
  if (!e) e = cudaMemsetAsync(h->s2, 0, V * sizeof(double), s);
  if (!e) e = cudaMemsetAsync(h->counters, 0, (kCtrCount + 1) * sizeof(ull), s);
  if (!e) e = cudaMemsetAsync(h->org_s1, 0, kLabelSlots * sizeof(double), s);
  if (!e) e = cudaMemsetAsync(h->org_s2, 0, kLabelSlots * sizeof(double), s);
  if (!e) e = cudaMemsetAsync(h->organ_count, 0, kLabelSlots * sizeof(long long), s);
  // labels must be <= n_labels: the lowest offending voxel, found with the counts
  unsigned long long first_bad = ~0ull;
  if (!e && h->labels) e = cudaMemsetAsync(h->label_bad, 0xff, sizeof(unsigned long long), s);
  if (!e && h->labels)
    e = launch_label_count(h->labels, V, o.n_labels, h->organ_count, h->label_bad, s);
  if (!e && h->labels)
    e = cudaMemcpyAsync(&first_bad, h->label_bad, sizeof first_bad, cudaMemcpyDeviceToHost, s);
  if (!e) e = cudaStreamSynchronize(s);
  if (e) return bail(cuda_fail(e, "nm_dose_create: init"));
  if (first_bad != ~0ull) {
    uint8_t l = 0;
    if ((e = cudaMemcpy(&l, h->labels + first_bad, 1, cudaMemcpyDeviceToHost))) return bail(cuda_fail(e, "labels"));
    return bail(fail(NM_ERR_ARG, "label %d at voxel %lld exceeds n_labels", l, (long long)first_bad));
  }
  nm_status cs = choose_shape(h);
  if (cs != NM_OK) return bail(cs);
  *out = h;
  return NM_OK;
}

// Memory of one run's batch tallies, at most; of all runs' under way beyond the
// first of each, at most this part of the device's, and of what is free when it
// is allocated, which leaves the rest to other handles and programs.
static constexpr uint64_t kSlotBytes = 16ull << 30;
static constexpr uint64_t kFreeShare = 4;

// Batch tallies for n histories in B batches on V voxels: as many as a launch
// can use (launch_batches; slot x voxel stays below 2^32) and memory allows, in
// near-equal launches; at least the one a handle is made with.
static int batch_slots(int64_t V, uint64_t n, int B, uint64_t free, uint64_t total, uint64_t held) {
  if (n / B < kMinSplit) return 1;
  const uint64_t each = (uint64_t)V * sizeof(ull), big = n / B + (n % B ? 1 : 0);
  const uint64_t share = total / kSlotShare > held ? total / kSlotShare - held : 0;
  const int most = (int)std::max<uint64_t>(
      1, std::min<uint64_t>({(uint64_t)kMaxSlots, (1ull << 31) / big, kSlotBytes / each,
                             ((1ull << 32) - 1) / (uint64_t)V, 1 + std::min(share, free / kFreeShare) / each}));
  const int launches = (B + most - 1) / most;
  return (B + launches - 1) / launches;
}

// One handle's part of a run or batched run, and the tallies it runs with:
// `slots` of them at `tb`, the handle's own one or more in a buffer of the pool.
struct RunPart {
  nm_dose* h;
  uint64_t n;
  int B;
  ull* tb;
  int slots;
};

// A buffer of the pool that parts in one stream share, one after the other.
struct TallyLoan {
  int device = 0;
  ull* p = nullptr;
  uint64_t bytes = 0;
};

// Ends a loan, after the device has: `zero` if the tallies are.
static void return_tallies(TallyLoan* loan, bool zero) {
  if (!loan->p) return;
  std::vector<ull*> out;
  {
    TallyPool& pool = tally_pool();
    std::lock_guard<std::mutex> lock(pool.mu);
    TallyPool::Dev& d = pool.dev[loan->device];
    d.busy -= loan->bytes;
    if (zero) {
      d.free.emplace_front(loan->p, loan->bytes);
      d.idle += loan->bytes;
      d.trim(d.keep(), out);
    } else {
      out.push_back(loan->p);
    }
  }
  for (ull* p : out) dfree_now(p);
  loan->p = nullptr;
}

// Tallies for parts that run one after the other on one stream, cleared on
// stream s if they are new; on one device.  Parts that get no more than one
// tally keep their handle's.
static nm_status take_tallies(RunPart* part, int n_parts, cudaStream_t s, TallyLoan* loan) {
  TallyPool& pool = tally_pool();
  loan->device = part[0].h->device;
  uint64_t need = 0;
  std::vector<ull*> out;
  auto most_bytes = [&](uint64_t free, uint64_t total, uint64_t held) {
    uint64_t bytes = 0;
    for (int i = 0; i < n_parts; ++i) {
      const RunPart& r = part[i];
      const int k = batch_slots(r.h->V, r.n, r.B, free, total, held);
      if (k > 1) bytes = std::max(bytes, (uint64_t)r.h->V * sizeof(ull) * k);
    }
    return bytes;
  };
  for (int i = 0; i < n_parts; ++i) {
    part[i].tb = part[i].h->tb;
    part[i].slots = 1;
  }
  if (most_bytes(UINT64_MAX, UINT64_MAX, 0) == 0) return NM_OK;
  size_t free = 0, total = 0;
  uint64_t busy = 0;
  {
    std::lock_guard<std::mutex> lock(pool.mu);
    TallyPool::Dev& d = pool.dev[loan->device];
    if (!d.total) {
      NM_CUDA(cudaMemGetInfo(&free, &total), "batch tallies");
      d.total = total;
    }
    total = d.total;
    busy = d.busy;
    need = most_bytes(UINT64_MAX, total, busy);
    for (int i = 0; i < n_parts; ++i) {
      nm_dose* h = part[i].h;
      const int k = batch_slots(h->V, part[i].n, part[i].B, UINT64_MAX, total, busy);
      const uint64_t want = k > 1 ? (uint64_t)h->V * sizeof(ull) * k : 0;
      d.wants += want - h->want_bytes;
      h->want_bytes = want;
    }
    if (need == 0) return NM_OK;
    auto best = d.free.end();                            // the smallest that holds it
    for (auto it = d.free.begin(); it != d.free.end(); ++it)
      if (it->second >= need && (best == d.free.end() || it->second < best->second)) best = it;
    if (best != d.free.end()) {
      loan->p = best->first;
      loan->bytes = best->second;
      d.idle -= loan->bytes;
      d.busy += loan->bytes;
      d.free.erase(best);
    } else {
      // a new one in the place of idle ones, where all are too many
      const uint64_t room = total / kSlotShare > busy + need ? total / kSlotShare - busy - need : 0;
      d.trim(room, out);
    }
  }
  for (ull* p : out) dfree_now(p);
  if (!loan->p) {
    NM_CUDA(cudaMemGetInfo(&free, &total), "batch tallies");
    if ((need = most_bytes(free, total, busy)) == 0) return NM_OK;
    const cudaError_t e = dalloc(&loan->p, need / sizeof(ull));
    if (e == cudaErrorMemoryAllocation) {
      cudaGetLastError();               // one batch per launch then
      return NM_OK;
    }
    if (e) return cuda_fail(e, "batch tallies");
    loan->bytes = need;
    {
      std::lock_guard<std::mutex> lock(pool.mu);
      pool.dev[loan->device].busy += need;
    }
    if (cudaError_t m = cudaMemsetAsync(loan->p, 0, need, s)) {
      return_tallies(loan, false);
      return cuda_fail(m, "batch tallies");
    }
  }
  for (int i = 0; i < n_parts; ++i) {
    RunPart& r = part[i];
    const uint64_t each = (uint64_t)r.h->V * sizeof(ull);
    int k = std::min<int>(batch_slots(r.h->V, r.n, r.B, UINT64_MAX, UINT64_MAX, 0),
                          (int)std::min<uint64_t>(loan->bytes / each, kMaxSlots));
    if (k < 2) continue;
    const int launches = (r.B + k - 1) / k;
    k = (r.B + launches - 1) / launches;                 // near-equal ones
    if (k < 2) continue;
    if (k > r.h->part_slots) {
      double* p = nullptr;
      const cudaError_t e = dalloc(&p, (size_t)organ_tiles(r.h->V) * k * kLabelSlots);
      if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        continue;
      }
      if (e) return cuda_fail(e, "organ partial sums");
      dfree(r.h->organ_partial);
      r.h->organ_partial = p;
      r.h->part_slots = k;
    }
    r.tb = loan->p;
    r.slots = k;
  }
  return NM_OK;
}

// Clears batch tallies and the launch's sums of squares.
static cudaError_t clear_tallies(nm_dose* h, ull* tb, int slots, cudaStream_t s) {
  const size_t V8 = 8 * (size_t)h->V;
  cudaError_t e = cudaMemsetAsync(tb, 0, V8 * slots, s);
  if (!e && h->q_lo) e = cudaMemsetAsync(h->q_lo, 0, V8, s);
  if (!e && h->q_hi) e = cudaMemsetAsync(h->q_hi, 0, V8, s);
  return e;
}

// Takes back a group of batches whose launch is on stream s and whose fold is not.
static cudaError_t undo_launch(const RunPart& r, cudaStream_t s) {
  nm_dose* h = r.h;
  uint32_t st = 0;
  cudaError_t e = cudaMemcpyAsync(h->counters, h->kept, kCtrCount * sizeof(ull), cudaMemcpyDeviceToDevice, s);
  if (!e) e = clear_tallies(h, r.tb, r.slots, s);
  if (!e) e = cudaMemcpyAsync(&st, h->status, 4, cudaMemcpyDeviceToHost, s);
  if (!e) e = cudaStreamSynchronize(s);
  if (!e) e = cudaMemsetAsync(h->status, 0, 4, s);
  h->status_seen |= st;
  return e;
}

static nm_status check_whole(const nm_dose* h) {
  return h->broken ? fail(NM_ERR_STATE, "a run of this handle ended half-way: nm_dose_reset or nm_dose_restore first")
                   : NM_OK;
}

static FoldParams fold_params(const RunPart& r) {
  const nm_dose* h = r.h;
  FoldParams fp;
  memset(&fp, 0, sizeof fp);
  fp.tb = r.tb; fp.tsum = h->tsum; fp.s2 = h->s2; fp.density = h->density;
  fp.labels = h->labels; fp.V = h->V; fp.sms = h->sms; fp.gy_per_unit_vol = h->gy_per_unit_vol();
  fp.organ_partial = h->organ_partial; fp.org_s1 = h->org_s1; fp.org_s2 = h->org_s2;
  fp.deposited = h->counters + kCtrDepositedUnits;
  return fp;
}

// Batches of n histories in B near-equal batches that one launch takes from
// batch b0 on: as many as there are tallies and 2^31 histories (the launch's
// work counter) allow; 1 for a batch above that, which takes several launches,
// and for batches of a few histories.
static int launch_batches(uint64_t n, int B, int b0, int slots) {
  if (n / B < kMinSplit) return 1;
  uint64_t sum = 0;
  int k = 0;
  while (k < slots && b0 + k < B) {
    sum += n / B + ((uint64_t)(b0 + k) < n % B ? 1 : 0);
    if (sum > (1ull << 31)) break;
    ++k;
  }
  return std::max(k, 1);
}

// Enqueues a part's histories in its batches on stream s with the launch shape of
// `like`: per group of batches one launch that tallies each batch in its own
// slot, then one fold of the slots in batch order, after which the group counts
// among the handle's histories.  mark() is called before a launch, after it
// and after its fold.  On an error the groups before the one at hand stay, and that one's
// launch is taken back; where that fails, or its fold had begun, the handle is
// `broken`.
static cudaError_t enqueue_run(const RunPart& run, uint64_t seed, const nm_dose* like, cudaStream_t s,
                               const std::function<cudaError_t()>& mark) {
  nm_dose* const h = run.h;
  const uint64_t n = run.n;
  const int B = run.B;
  const uint64_t q = n / B, r = n % B;
  cudaError_t e = cudaSuccess;
  auto step = [&e](auto&& f) {
    if (!e) e = fail_now(g_fail_enqueue) ? cudaErrorUnknown : f();
  };
  for (int b0 = 0; b0 < B && !e;) {
    NvtxRange batch_range("batches");
    const int k = launch_batches(n, B, b0, run.slots);
    const uint32_t big = (uint32_t)std::min<uint64_t>(r > (uint64_t)b0 ? r - b0 : 0, (uint64_t)k);
    const uint64_t total = q * k + big;
    FoldParams fp = fold_params(run);
    fp.n_slots = k;
    for (int b = 0; b < k; ++b) fp.set_batch(b, q + ((uint32_t)b < big ? 1 : 0));
    bool launched = false, folding = false;
    // a launch's squares fit their two sums; of several launches they go first
    auto fold_squares = [&] {
      folding = true;
      return launch_fold_history(h->q_lo, h->q_hi, h->s2h_lo, h->s2h_hi, h->V, s);
    };
    step(mark);
    for (uint64_t done = 0; done < total && !e;) {
      const uint64_t part = std::min<uint64_t>(total - done, 1ull << 31);
      TransportParams p = h->params(h->id_next + done, part, seed);
      p.g.tally = run.tb;
      if (k > 1) p.g.split = batch_split((uint32_t)k, big, (uint32_t)q);
      const int warps = like->block / 32;
      p.chunk = like->opt.chunk > 0 ? like->chunk : launch_chunk(like->chunk, (uint64_t)like->grid * warps, part);
      p.regroup_compton = p.regroup_refill = like->regroup_lanes;
      // no more CTAs than have a chunk to take
      const uint64_t want = (part + (uint64_t)p.chunk * warps - 1) / ((uint64_t)p.chunk * warps);
      if (done == 0)
        step([&] {
          return cudaMemcpyAsync(h->kept, h->counters, (kCtrCount + 1) * sizeof(ull), cudaMemcpyDeviceToDevice, s);
        });
      else
        step([&] { return cudaMemsetAsync(h->work, 0, sizeof(unsigned), s); });
      launched |= !e;
      step([&] {
        return launch_transport(p, (int)std::min<uint64_t>((uint64_t)like->grid, want), like->block, like->warp_agg,
                                h->rayleigh, like->regroup, s, h->opt.history_sigma != 0);
      });
      if (h->q_lo && part < total) step(fold_squares);
      done += part;
    }
    step(mark);
    step([&] {
      folding = true;
      return launch_fold(fp, s);
    });
    if (h->q_lo && total <= (1ull << 31)) step(fold_squares);
    if (e) {
      h->broken = folding || (launched && undo_launch(run, s) != cudaSuccess);
      break;
    }
    h->hist_next += total;
    h->id_next += total;
    h->n_batches += (uint64_t)k;
    step(mark);
    b0 += k;
  }
  return e;
}

nm_status nm_dose_run(nm_dose* h, uint64_t n, uint64_t seed) {
  NvtxRange range("nm_dose_run");
  if (!h) return fail(NM_ERR_ARG, "handle is NULL");
  if (n == 0) return NM_OK;
  nm_status ws = check_whole(h);
  if (ws != NM_OK) return ws;
  const uint64_t per = h->units_per_history();
  const uint64_t lim = (uint64_t)INT64_MAX / (per ? per : 1);
  if (h->hist_next > lim || n > lim - h->hist_next)
    return fail(NM_ERR_OVERFLOW, "%llu more histories could overflow the int64 tally",
                (unsigned long long)n);
  if (h->id_next + n < h->id_next || h->id_next + n > (1ull << 62))
    return fail(NM_ERR_OVERFLOW, "history ids exhausted");
  const int B = (uint64_t)h->opt.batches < n ? h->opt.batches : (int)n;
  cudaStream_t s = h->stream;
  RunPart part{h, n, B, nullptr, 0};
  TallyLoan loan;
  if ((ws = take_tallies(&part, 1, s, &loan)) != NM_OK) {
    return_tallies(&loan, cudaStreamSynchronize(s) == cudaSuccess);
    return ws;
  }
  // per launch: transport start and end, fold end
  size_t used = 0;
  const cudaError_t e = enqueue_run(part, seed, h, s, [&]() -> cudaError_t {
    if (used == h->ev.size()) {
      cudaEvent_t ev;
      if (cudaError_t c = cudaEventCreate(&ev)) return c;
      h->ev.push_back(ev);
    }
    return cudaEventRecord(h->ev[used++], s);
  });
  uint32_t st = 0;
  cudaError_t end = e ? cudaSuccess : cudaMemcpyAsync(&st, h->status, 4, cudaMemcpyDeviceToHost, s);
  if (!end) end = cudaStreamSynchronize(s);
  if (end) h->broken = true;            // the device did not get to the end of it
  return_tallies(&loan, !h->broken);
  if (e || end) return cuda_fail(e ? e : end, "nm_dose_run");
  for (size_t g = 0; g < used; g += 3) {
    float ms = 0;
    if (cudaEventElapsedTime(&ms, h->ev[g], h->ev[g + 1]) == cudaSuccess) h->transport_ms += ms;
    if (cudaEventElapsedTime(&ms, h->ev[g + 1], h->ev[g + 2]) == cudaSuccess) h->fold_ms += ms;
  }
  h->status_seen |= st;
  if (st) {
    NM_CUDA(cudaMemsetAsync(h->status, 0, 4, s), "status reset");
    return fail(NM_ERR_DEVICE, "device check fired (flags 0x%x: %s%s%s)", st,
                (st & NM_DEV_STEP_LIMIT) ? "photon step limit " : "",
                (st & NM_DEV_KAHN_LIMIT) ? "Kahn trial limit " : "",
                (st & NM_DEV_RAYLEIGH_LIMIT) ? "Rayleigh trial limit" : "");
  }
  return NM_OK;
}

// ---------------------------------------------------------------------------
// Many patients in one call: each patient's launches and folds go to one of a
// few streams, so that a patient's transport fills the SMs that others' last
// photons and folds leave, and small patients run side by side.  (One launch
// over all patients' queues, whose lanes carried their patient, took 23.3 ms
// for eight patients of 1e7; the patients' own launches take 14.5 ms, folds included.)
// ---------------------------------------------------------------------------
static bool same_physics(const nm_dose* a, const nm_dose* b) {
  if (a->n_mat != b->n_mat || a->rayleigh != b->rayleigh || a->e0 != b->e0 || a->cut != b->cut ||
      a->ln_e_lo != b->ln_e_lo || a->inv_dln != b->inv_dln || a->device != b->device ||
      a->opt.batches != b->opt.batches || a->opt.max_steps != b->opt.max_steps ||
      a->opt.kn_sampler != b->opt.kn_sampler)
    return false;
  for (int m = 0; m < a->n_mat; ++m)
    if (a->mat[m].za != b->mat[m].za || a->mat[m].zp != b->mat[m].zp || a->mat[m].zr != b->mat[m].zr)
      return false;
  return true;
}

constexpr int kBatchStreams = 4;

extern "C" nm_status nm_dose_run_batch(nm_dose* const* hs, int32_t n, const uint64_t* n_decays,
                                       uint64_t seed) {
  NvtxRange range("nm_dose_run_batch");
  if (!hs || !n_decays || n < 1 || n > kMaxBatchPatients)
    return fail(NM_ERR_ARG, "need 1..%d handles and their decay counts", kMaxBatchPatients);
  for (int i = 0; i < n; ++i) {
    if (!hs[i]) return fail(NM_ERR_ARG, "handle %d is NULL", i);
    const nm_status ws = check_whole(hs[i]);
    if (ws != NM_OK) return ws;
    for (int j = 0; j < i; ++j)
      if (hs[j] == hs[i]) return fail(NM_ERR_ARG, "handle %d appears twice", i);
    if (hs[i]->opt.history_sigma || hs[i]->nuclide)
      return fail(NM_ERR_ARG, "handle %d: history_sigma and beta+ spectrum handles run with nm_dose_run, not in batches",
                  i);
    if (!same_physics(hs[0], hs[i]))
      return fail(NM_ERR_ARG, "handle %d: all patients of a batch need the same materials, energies, batches and device", i);
    const uint64_t per = hs[i]->units_per_history();
    const uint64_t lim = (uint64_t)INT64_MAX / (per ? per : 1);
    if (hs[i]->hist_next > lim || n_decays[i] > lim - hs[i]->hist_next ||
        hs[i]->id_next + n_decays[i] > (1ull << 62))
      return fail(NM_ERR_OVERFLOW, "handle %d: too many histories", i);
  }
  nm_dose* h0 = hs[0];
  cudaStream_t s = h0->stream;
  const int B = h0->opt.batches;
  uint64_t total = 0;
  for (int i = 0; i < n; ++i) total += n_decays[i];
  if (total == 0) return NM_OK;

  for (int i = 0; i < n; ++i)
    if (n_decays[i] / B + (n_decays[i] % B ? 1 : 0) >= (1ull << 31))
      return fail(NM_ERR_ARG, "handle %d: batches above 2^31 histories", i);
  // parts by stream, which share the stream's tallies
  const int n_streams = std::min(n, kBatchStreams);
  std::vector<RunPart> parts[kBatchStreams];
  TallyLoan loans[kBatchStreams];
  for (int i = 0; i < n; ++i)
    if (n_decays[i])
      parts[i % n_streams].push_back({hs[i], n_decays[i], (int)std::min<uint64_t>(B, n_decays[i]), nullptr, 0});
  auto return_loans = [&] {
    for (int j = 0; j < n_streams; ++j) {
      bool zero = true;
      for (const RunPart& r : parts[j]) zero = zero && !r.h->broken;
      return_tallies(&loans[j], zero);
    }
  };
  for (int j = 0; j < n_streams; ++j) {
    if (parts[j].empty()) continue;
    const nm_status ts = take_tallies(parts[j].data(), (int)parts[j].size(), s, &loans[j]);
    if (ts != NM_OK) {
      cudaStreamSynchronize(s);
      return_loans();
      return ts;
    }
  }
  cudaStream_t st[kBatchStreams] = {};
  cudaEvent_t e0 = nullptr, e1 = nullptr, join = nullptr;
  auto cleanup = [&]() {
    for (cudaStream_t& c : st)
      if (c) {
        cudaStreamSynchronize(c);
        cudaStreamDestroy(c);
      }
    cudaStreamSynchronize(s);
    for (cudaEvent_t c : {e0, e1, join})
      if (c) cudaEventDestroy(c);
    return_loans();
  };
  cudaError_t e = cudaEventCreate(&e0);
  if (!e) e = cudaEventCreate(&e1);
  if (!e) e = cudaEventCreateWithFlags(&join, cudaEventDisableTiming);
  if (!e) e = cudaEventRecord(e0, s);
  for (int j = 0; j < n_streams && !e; ++j) {
    e = cudaStreamCreateWithFlags(&st[j], cudaStreamNonBlocking);
    if (!e) e = cudaStreamWaitEvent(st[j], e0, 0);
  }
  // the launch shape is the first handle's, the majorants each its own
  for (int i = 0; i < n && !e; ++i) {
    const std::vector<RunPart>& mine = parts[i % n_streams];
    for (size_t k = 0; k < mine.size() && !e; ++k)
      if (mine[k].h == hs[i]) e = enqueue_run(mine[k], seed, h0, st[i % n_streams], [] { return cudaSuccess; });
  }
  if (e) {
    cleanup();                          // the patients and batches before the failed one stay
    return cuda_fail(e, "nm_dose_run_batch");
  }
  for (int i = 0; i < n; ++i) hs[i]->broken = n_decays[i] != 0;   // unless the device gets to the end of it
  for (int j = 0; j < n_streams && !e; ++j) {
    e = cudaEventRecord(join, st[j]);
    if (!e) e = cudaStreamWaitEvent(s, join, 0);
  }
  float ms = 0;
  std::vector<uint32_t> flag(n, 0);
  if (!e) e = cudaEventRecord(e1, s);
  for (int i = 0; i < n && !e; ++i) e = cudaMemcpyAsync(&flag[i], hs[i]->status, 4, cudaMemcpyDeviceToHost, s);
  if (!e) e = cudaStreamSynchronize(s);
  if (!e) e = cudaEventElapsedTime(&ms, e0, e1);
  uint32_t flags = 0;
  std::string flagged;                  // handles whose own checks fired
  for (int i = 0; i < n && !e; ++i)
    if (flag[i]) {
      flags |= flag[i];
      flagged += " " + std::to_string(i);
      e = cudaMemsetAsync(hs[i]->status, 0, 4, s);
    }
  if (e) {
    cleanup();
    return cuda_fail(e, "nm_dose_run_batch");
  }
  for (int i = 0; i < n; ++i) {
    if (n_decays[i] == 0) continue;
    hs[i]->broken = false;
    hs[i]->transport_ms += ms * (double)n_decays[i] / (double)total;  // the call's device time, shared by decays
    hs[i]->status_seen |= flag[i];
  }
  cleanup();
  if (flags) return fail(NM_ERR_DEVICE, "device check fired (flags 0x%x, handles%s)", flags, flagged.c_str());
  return NM_OK;
}

static nm_status finalize(nm_dose* h, float* dose, float* sigma, bool organs) {
  const nm_status ws = check_whole(h);
  if (ws != NM_OK) return ws;
  if (h->hist_next == 0) return fail(NM_ERR_STATE, "no histories simulated yet");
  if (h->n_batches < 2) return fail(NM_ERR_STATE, "need at least 2 batches for the uncertainty");
  cudaStream_t s = h->stream;
  FinalizeParams p;
  p.tsum = h->tsum; p.s2 = h->s2; p.density = h->density; p.labels = h->labels; p.V = h->V;
  p.n_total = (double)h->hist_next;
  p.n_batches = (double)h->n_batches;
  p.gy_per_unit_vol = h->gy_per_unit_vol();
  p.activity_bq = h->opt.activity_bq;
  p.dose = dose;
  p.sigma = sigma;
  p.organ_partial = h->organ_partial;
  p.org_s1 = h->org_s1; p.org_s2 = h->org_s2;
  p.organ_count = h->organ_count;
  p.organ_out = h->organ_out;
  NM_CUDA(launch_finalize(p, organs && h->labels, h->sms, s), "finalize launch");
  return NM_OK;
}

nm_status nm_dose_get(nm_dose* h, float* dose, float* sigma, double* organ_dose) {
  NvtxRange range("nm_dose_get");
  if (!h) return fail(NM_ERR_ARG, "handle is NULL");
  const nm_status ws = check_whole(h);
  if (ws != NM_OK) return ws;
  cudaStream_t s = h->stream;
  const bool dd = is_device_ptr(dose), ds = is_device_ptr(sigma);
  if ((dose && !dd) || (sigma && !ds)) {
    if (!h->out_dose) NM_CUDA(dalloc(&h->out_dose, h->V), "output buffer");
    if (!h->out_sigma) NM_CUDA(dalloc(&h->out_sigma, h->V), "output buffer");
  }
  float* d_out = dose ? (dd ? dose : h->out_dose) : nullptr;
  float* s_out = sigma ? (ds ? sigma : h->out_sigma) : nullptr;
  if (dose && !sigma && !organ_dose) {
    // the dose map alone: one streaming pass, no uncertainty or organ sums
    if (h->hist_next == 0) return fail(NM_ERR_STATE, "no histories simulated yet");
    FinalizeParams p;
    memset(&p, 0, sizeof p);
    p.tsum = h->tsum; p.density = h->density; p.V = h->V; p.n_total = (double)h->hist_next;
    p.gy_per_unit_vol = h->gy_per_unit_vol(); p.activity_bq = h->opt.activity_bq; p.dose = d_out;
    NM_CUDA(launch_dose_only(p, h->sms, s), "dose launch");
  } else {
    nm_status st = finalize(h, d_out, s_out, organ_dose != nullptr);
    if (st != NM_OK) return st;
  }
  if (dose && !dd) NM_CUDA(cudaMemcpyAsync(dose, d_out, h->V * sizeof(float), cudaMemcpyDeviceToHost, s), "dose copy");
  if (sigma && !ds) NM_CUDA(cudaMemcpyAsync(sigma, s_out, h->V * sizeof(float), cudaMemcpyDeviceToHost, s), "sigma copy");
  if (organ_dose)
    NM_CUDA(cudaMemcpyAsync(organ_dose, h->organ_out, (h->opt.n_labels + 1) * sizeof(double),
                            cudaMemcpyDefault, s), "organ copy");
  NM_CUDA(cudaStreamSynchronize(s), "nm_dose_get");
  return NM_OK;
}

nm_status nm_dose_get_organs(nm_dose* h, double* mean, double* eps_rms, double* sigma_mean,
                             int64_t* voxels) {
  NvtxRange range("nm_dose_get_organs");
  if (!h) return fail(NM_ERR_ARG, "handle is NULL");
  const nm_status ws = check_whole(h);
  if (ws != NM_OK) return ws;
  if (!eps_rms && h->labels) {
    // Eq. 2 and the batch sigma from the per-organ batch sums of the fold, no
    // pass over the voxels: mean = A sum_b O_b / (N cnt) with O_b the batch's
    // summed voxel doses (the same FP32 voxel doses the full pass sums)
    if (h->hist_next == 0) return fail(NM_ERR_STATE, "no histories simulated yet");
    if (sigma_mean && h->n_batches < 2) return fail(NM_ERR_STATE, "need at least 2 batches for the uncertainty");
    std::vector<double> s1(kLabelSlots), s2(kLabelSlots);
    std::vector<long long> cnt(kLabelSlots);
    cudaStream_t s = h->stream;
    NM_CUDA(cudaMemcpyAsync(s1.data(), h->org_s1, kLabelSlots * sizeof(double), cudaMemcpyDeviceToHost, s), "organ sums");
    NM_CUDA(cudaMemcpyAsync(s2.data(), h->org_s2, kLabelSlots * sizeof(double), cudaMemcpyDeviceToHost, s), "organ sums");
    NM_CUDA(cudaMemcpyAsync(cnt.data(), h->organ_count, kLabelSlots * sizeof(long long), cudaMemcpyDeviceToHost, s),
            "organ counts");
    NM_CUDA(cudaStreamSynchronize(s), "nm_dose_get_organs");
    const double N = (double)h->hist_next, A = h->opt.activity_bq;
    for (int l = 0; l <= h->opt.n_labels; ++l) {
      const double c = (double)cnt[l];
      double m = 0.0, sg = 0.0;
      if (c > 0.0) {
        const double mbar = s1[l] / (N * c);                  // per decay
        m = mbar * A;
        if (h->n_batches >= 2) {
          const double var = std::max(s2[l] / (c * c) - N * mbar * mbar, 0.0) / ((h->n_batches - 1.0) * N);
          sg = std::sqrt(var) * A;
        }
      }
      if (mean) mean[l] = m;
      if (sigma_mean) sigma_mean[l] = sg;
      if (voxels) voxels[l] = cnt[l];
    }
    return NM_OK;
  }
  nm_status st = finalize(h, nullptr, nullptr, true);
  if (st != NM_OK) return st;
  std::vector<double> out(4 * kLabelSlots);
  NM_CUDA(cudaMemcpyAsync(out.data(), h->organ_out, out.size() * sizeof(double), cudaMemcpyDeviceToHost, h->stream), "organ copy");
  NM_CUDA(cudaStreamSynchronize(h->stream), "nm_dose_get_organs");
  const int n = h->opt.n_labels + 1;
  for (int l = 0; l < n; ++l) {
    if (mean) mean[l] = out[l];
    if (eps_rms) eps_rms[l] = out[kLabelSlots + l];
    if (sigma_mean) sigma_mean[l] = out[2 * kLabelSlots + l];
    if (voxels) voxels[l] = (int64_t)out[3 * kLabelSlots + l];
  }
  return NM_OK;
}

nm_status nm_dose_get_history_sigma(nm_dose* h, float* sigma) {
  if (!h || !sigma) return fail(NM_ERR_ARG, "bad arguments");
  const nm_status ws = check_whole(h);
  if (ws != NM_OK) return ws;
  if (!h->s2h_lo) return fail(NM_ERR_STATE, "the handle was created without history_sigma");
  if (h->hist_next < 2) return fail(NM_ERR_STATE, "need at least 2 histories");
  cudaStream_t s = h->stream;
  const bool dev = is_device_ptr(sigma);
  if (!dev && !h->out_sigma) NM_CUDA(dalloc(&h->out_sigma, h->V), "output buffer");
  float* out = dev ? sigma : h->out_sigma;
  NM_CUDA(launch_history_sigma(h->tsum, h->s2h_lo, h->s2h_hi, h->density, h->V, (double)h->hist_next,
                               h->gy_per_unit_vol() * h->opt.activity_bq, out, s),
          "history sigma");
  if (!dev) NM_CUDA(cudaMemcpyAsync(sigma, out, h->V * sizeof(float), cudaMemcpyDeviceToHost, s), "sigma copy");
  NM_CUDA(cudaStreamSynchronize(s), "nm_dose_get_history_sigma");
  return NM_OK;
}

nm_status nm_dose_map_organs(nm_dose* h, const float* dose, double* mean) {
  if (!h || !dose || !mean) return fail(NM_ERR_ARG, "bad arguments");
  if (!h->labels) return fail(NM_ERR_STATE, "the handle has no label map");
  cudaStream_t s = h->stream;
  const float* d = dose;
  if (!is_device_ptr(dose)) {
    if (!h->out_dose) NM_CUDA(dalloc(&h->out_dose, h->V), "output buffer");
    NM_CUDA(cudaMemcpyAsync(h->out_dose, dose, h->V * sizeof(float), cudaMemcpyHostToDevice, s), "map copy");
    d = h->out_dose;
  }
  NM_CUDA(launch_map_organ_means(d, h->labels, h->V, h->organ_partial, h->organ_count, h->organ_out, s),
          "organ means");
  NM_CUDA(cudaMemcpyAsync(mean, h->organ_out, (h->opt.n_labels + 1) * sizeof(double), cudaMemcpyDefault, s),
          "organ copy");
  NM_CUDA(cudaStreamSynchronize(s), "nm_dose_map_organs");
  return NM_OK;
}

nm_status nm_time_integrated_activity(const float* const* act, const double* t_h, int32_t n, int64_t V,
                                      double half_life_h, float* out, double* total, void* stream) {
  if (!act || !t_h || !out || n < 1 || n > 16 || V < 1 || V >= ((int64_t)1 << 31))
    return fail(NM_ERR_ARG, "nm_time_integrated_activity: 1..16 maps of 1..2^31-1 voxels and an output");
  if (!(half_life_h > 0.0) || !std::isfinite(half_life_h))
    return fail(NM_ERR_ARG, "nm_time_integrated_activity: the half-life must be finite and > 0");
  double t_s[16];
  for (int k = 0; k < n; ++k) {
    if (!act[k]) return fail(NM_ERR_ARG, "nm_time_integrated_activity: map %d is NULL", k);
    if (!std::isfinite(t_h[k]) || !(t_h[k] >= 0.0) || (k > 0 && !(t_h[k] > t_h[k - 1])))
      return fail(NM_ERR_ARG, "nm_time_integrated_activity: times must be finite, >= 0 and increasing");
    t_s[k] = 3600.0 * t_h[k];
  }
  cudaStream_t s = (cudaStream_t)stream;
  int dev = 0, sms = 0;
  NM_CUDA(cudaGetDevice(&dev), "cudaGetDevice");
  NM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "cudaDeviceGetAttribute");
  const int blocks = (int)std::min<int64_t>((V + 255) / 256, (int64_t)sms * 8);
  // host maps and a host output go through device copies
  std::vector<float*> staged;
  auto cleanup = [&]() {
    for (float* q : staged) cudaFree(q);
  };
  const float* dmaps[16];
  for (int k = 0; k < n; ++k) {
    if (is_device_ptr(act[k])) {
      dmaps[k] = act[k];
    } else {
      float* d = nullptr;
      cudaError_t e = dalloc(&d, V);
      if (!e) {
        staged.push_back(d);
        e = cudaMemcpyAsync(d, act[k], V * sizeof(float), cudaMemcpyHostToDevice, s);
      }
      if (e) { cleanup(); return cuda_fail(e, "nm_time_integrated_activity: staging"); }
      dmaps[k] = d;
    }
  }
  float* dout = out;
  if (!is_device_ptr(out)) {
    float* d = nullptr;
    cudaError_t e = dalloc(&d, V);
    if (e) { cleanup(); return cuda_fail(e, "nm_time_integrated_activity: staging"); }
    staged.push_back(d);
    dout = d;
  }
  double* sums = nullptr;
  cudaError_t e = dalloc(&sums, (size_t)blocks + 1);   // + the status word
  if (e) { cleanup(); return cuda_fail(e, "nm_time_integrated_activity: sums"); }
  std::vector<double> hs(blocks);
  uint32_t st = 0;
  e = cudaMemsetAsync(sums + blocks, 0, sizeof(double), s);
  if (!e) e = launch_time_integral(dmaps, t_s, n, V, 3600.0 * half_life_h / std::log(2.0), dout, sums, blocks, s);
  if (!e) e = cudaMemcpyAsync(hs.data(), sums, blocks * sizeof(double), cudaMemcpyDeviceToHost, s);
  if (!e) e = cudaMemcpyAsync(&st, sums + blocks, sizeof st, cudaMemcpyDeviceToHost, s);
  if (!e && dout != out) e = cudaMemcpyAsync(out, dout, V * sizeof(float), cudaMemcpyDeviceToHost, s);
  if (!e) e = cudaStreamSynchronize(s);
  dfree_now(sums);
  cleanup();
  if (e) return cuda_fail(e, "nm_time_integrated_activity");
  if (st & NM_DEV_BAD_ACTIVITY) return fail(NM_ERR_ARG, "nm_time_integrated_activity: activities must be finite and >= 0");
  if (total) {
    double acc = 0.0;
    for (double x : hs) acc += x;
    *total = acc;
  }
  return NM_OK;
}

nm_status nm_dose_get_tally(nm_dose* h, int64_t* tally) {
  if (!h || !tally) return fail(NM_ERR_ARG, "bad arguments");
  const nm_status ws = check_whole(h);
  if (ws != NM_OK) return ws;
  NM_CUDA(cudaMemcpyAsync(tally, h->tsum, h->V * sizeof(int64_t), cudaMemcpyDefault, h->stream), "tally copy");
  NM_CUDA(cudaStreamSynchronize(h->stream), "nm_dose_get_tally");
  return NM_OK;
}

// ---------------------------------------------------------------------------
// Checkpoints: a flat byte image of a handle's statistics, host or device.
//   header (kCkptHeader bytes, below), then tsum[V] (int64), s2[V] (FP64),
//   org_s1, org_s2 [kLabelSlots] (FP64), counters [kCtrCount] (uint64) and,
//   with history statistics, s2h_lo[V], s2h_hi[V] (uint64).
// ---------------------------------------------------------------------------
namespace {

struct CkptHeader {
  char magic[8];
  int64_t nx, ny, nz, V, label_slots, ctr_count, history;
  uint64_t hist_next, id_next, n_batches, status_seen;
};
constexpr char kCkptMagic[8] = {'N', 'M', 'D', 'O', 'S', 'E', '1', 0};
static_assert(sizeof(CkptHeader) % 16 == 0, "checkpoint arrays stay 16-byte aligned");

uint64_t ckpt_bytes(const nm_dose* h) {
  const uint64_t V = (uint64_t)h->V;
  return sizeof(CkptHeader) + 16 * V + 16 * (uint64_t)kLabelSlots + 8 * (uint64_t)kCtrCount +
         (h->s2h_lo ? 16 * V : 0);
}

// Offsets of the arrays within the image.
struct CkptOffsets {
  uint64_t tsum, s2, org_s1, org_s2, counters, lo, hi;
};
CkptOffsets ckpt_offsets(int64_t V) {
  CkptOffsets o;
  o.tsum = sizeof(CkptHeader);
  o.s2 = o.tsum + 8 * (uint64_t)V;
  o.org_s1 = o.s2 + 8 * (uint64_t)V;
  o.org_s2 = o.org_s1 + 8 * (uint64_t)kLabelSlots;
  o.counters = o.org_s2 + 8 * (uint64_t)kLabelSlots;
  o.lo = o.counters + 8 * (uint64_t)kCtrCount;
  o.hi = o.lo + 8 * (uint64_t)V;
  return o;
}

// Reads and checks the header of an image meant for handle h.
nm_status ckpt_read_header(nm_dose* h, const void* buf, uint64_t bytes, CkptHeader* hd) {
  if (!buf) return fail(NM_ERR_ARG, "checkpoint buffer is NULL");
  if (bytes < sizeof(CkptHeader)) return fail(NM_ERR_ARG, "checkpoint buffer too small");
  NM_CUDA(cudaMemcpyAsync(hd, buf, sizeof *hd, cudaMemcpyDefault, h->stream), "checkpoint header");
  NM_CUDA(cudaStreamSynchronize(h->stream), "checkpoint header");
  if (memcmp(hd->magic, kCkptMagic, 8) != 0) return fail(NM_ERR_ARG, "not a dose checkpoint");
  if (hd->nx != h->nx || hd->ny != h->ny || hd->nz != h->nz || hd->V != h->V ||
      hd->label_slots != kLabelSlots || hd->ctr_count != kCtrCount ||
      hd->history != (h->s2h_lo ? 1 : 0))
    return fail(NM_ERR_ARG, "checkpoint of a different grid or options");
  if (bytes < ckpt_bytes(h)) return fail(NM_ERR_ARG, "checkpoint buffer too small");
  return NM_OK;
}

}  // namespace

nm_status nm_dose_seek(nm_dose* h, uint64_t next_history_id) {
  if (!h) return fail(NM_ERR_ARG, "handle is NULL");
  if (next_history_id > (1ull << 62)) return fail(NM_ERR_ARG, "history id above 2^62");
  h->id_next = next_history_id;
  return NM_OK;
}

nm_status nm_dose_checkpoint_size(const nm_dose* h, uint64_t* bytes) {
  if (!h || !bytes) return fail(NM_ERR_ARG, "bad arguments");
  *bytes = ckpt_bytes(h);
  return NM_OK;
}

nm_status nm_dose_checkpoint(nm_dose* h, void* buf, uint64_t bytes) {
  if (!h || !buf) return fail(NM_ERR_ARG, "bad arguments");
  if (bytes < ckpt_bytes(h)) return fail(NM_ERR_ARG, "checkpoint buffer too small");
  const nm_status ws = check_whole(h);
  if (ws != NM_OK) return ws;
  CkptHeader hd;
  memset(&hd, 0, sizeof hd);
  memcpy(hd.magic, kCkptMagic, 8);
  hd.nx = h->nx; hd.ny = h->ny; hd.nz = h->nz; hd.V = h->V;
  hd.label_slots = kLabelSlots; hd.ctr_count = kCtrCount; hd.history = h->s2h_lo ? 1 : 0;
  hd.hist_next = h->hist_next; hd.id_next = h->id_next; hd.n_batches = h->n_batches;
  hd.status_seen = h->status_seen;
  const CkptOffsets o = ckpt_offsets(h->V);
  uint8_t* b = static_cast<uint8_t*>(buf);
  cudaStream_t s = h->stream;
  const size_t V8 = 8 * (size_t)h->V;
  NM_CUDA(cudaMemcpyAsync(b, &hd, sizeof hd, cudaMemcpyDefault, s), "checkpoint");
  NM_CUDA(cudaMemcpyAsync(b + o.tsum, h->tsum, V8, cudaMemcpyDefault, s), "checkpoint");
  NM_CUDA(cudaMemcpyAsync(b + o.s2, h->s2, V8, cudaMemcpyDefault, s), "checkpoint");
  NM_CUDA(cudaMemcpyAsync(b + o.org_s1, h->org_s1, 8 * kLabelSlots, cudaMemcpyDefault, s), "checkpoint");
  NM_CUDA(cudaMemcpyAsync(b + o.org_s2, h->org_s2, 8 * kLabelSlots, cudaMemcpyDefault, s), "checkpoint");
  NM_CUDA(cudaMemcpyAsync(b + o.counters, h->counters, 8 * kCtrCount, cudaMemcpyDefault, s), "checkpoint");
  if (h->s2h_lo) {
    NM_CUDA(cudaMemcpyAsync(b + o.lo, h->s2h_lo, V8, cudaMemcpyDefault, s), "checkpoint");
    NM_CUDA(cudaMemcpyAsync(b + o.hi, h->s2h_hi, V8, cudaMemcpyDefault, s), "checkpoint");
  }
  NM_CUDA(cudaStreamSynchronize(s), "nm_dose_checkpoint");
  return NM_OK;
}

nm_status nm_dose_restore(nm_dose* h, const void* buf, uint64_t bytes) {
  if (!h) return fail(NM_ERR_ARG, "handle is NULL");
  CkptHeader hd;
  nm_status st = ckpt_read_header(h, buf, bytes, &hd);
  if (st != NM_OK) return st;
  const CkptOffsets o = ckpt_offsets(h->V);
  const uint8_t* b = static_cast<const uint8_t*>(buf);
  cudaStream_t s = h->stream;
  const size_t V8 = 8 * (size_t)h->V;
  NM_CUDA(cudaMemcpyAsync(h->tsum, b + o.tsum, V8, cudaMemcpyDefault, s), "restore");
  NM_CUDA(cudaMemcpyAsync(h->s2, b + o.s2, V8, cudaMemcpyDefault, s), "restore");
  NM_CUDA(cudaMemcpyAsync(h->org_s1, b + o.org_s1, 8 * kLabelSlots, cudaMemcpyDefault, s), "restore");
  NM_CUDA(cudaMemcpyAsync(h->org_s2, b + o.org_s2, 8 * kLabelSlots, cudaMemcpyDefault, s), "restore");
  NM_CUDA(cudaMemcpyAsync(h->counters, b + o.counters, 8 * kCtrCount, cudaMemcpyDefault, s), "restore");
  if (h->s2h_lo) {
    NM_CUDA(cudaMemcpyAsync(h->s2h_lo, b + o.lo, V8, cudaMemcpyDefault, s), "restore");
    NM_CUDA(cudaMemcpyAsync(h->s2h_hi, b + o.hi, V8, cudaMemcpyDefault, s), "restore");
  }
  if (h->broken) NM_CUDA(clear_tallies(h, h->tb, 1, s), "restore");
  if (h->broken) NM_CUDA(cudaMemsetAsync(h->status, 0, 4, s), "restore");
  NM_CUDA(cudaStreamSynchronize(s), "nm_dose_restore");
  h->broken = false;
  h->hist_next = hd.hist_next;
  h->id_next = hd.id_next;
  h->n_batches = hd.n_batches;
  h->status_seen = (uint32_t)hd.status_seen;
  return NM_OK;
}

nm_status nm_dose_merge(nm_dose* h, const void* buf, uint64_t bytes) {
  NvtxRange range("nm_dose_merge");
  if (!h) return fail(NM_ERR_ARG, "handle is NULL");
  CkptHeader hd;
  nm_status st = ckpt_read_header(h, buf, bytes, &hd);
  if (st == NM_OK) st = check_whole(h);
  if (st != NM_OK) return st;
  const uint64_t per = h->units_per_history();
  const uint64_t lim = (uint64_t)INT64_MAX / (per ? per : 1);
  if (h->hist_next > lim || hd.hist_next > lim - h->hist_next)
    return fail(NM_ERR_OVERFLOW, "the merged tally could overflow int64");
  cudaStream_t s = h->stream;
  const uint64_t total = ckpt_bytes(h);
  const uint8_t* b = static_cast<const uint8_t*>(buf);
  uint8_t* tmp = nullptr;
  if (!is_device_ptr(buf)) {
    NM_CUDA(cudaMalloc(&tmp, total), "merge staging");
    cudaError_t e = cudaMemcpyAsync(tmp, buf, total, cudaMemcpyDefault, s);
    if (e != cudaSuccess) {
      cudaFree(tmp);
      return cuda_fail(e, "merge staging copy");
    }
    b = tmp;
  }
  const CkptOffsets o = ckpt_offsets(h->V);
  MergeParams m;
  m.tsum = h->tsum; m.s2 = h->s2; m.s2h_lo = h->s2h_lo; m.s2h_hi = h->s2h_hi;
  m.org_s1 = h->org_s1; m.org_s2 = h->org_s2; m.counters = h->counters;
  m.o_tsum = reinterpret_cast<const ull*>(b + o.tsum);
  m.o_s2 = reinterpret_cast<const double*>(b + o.s2);
  m.o_lo = h->s2h_lo ? reinterpret_cast<const ull*>(b + o.lo) : nullptr;
  m.o_hi = h->s2h_lo ? reinterpret_cast<const ull*>(b + o.hi) : nullptr;
  m.o_org_s1 = reinterpret_cast<const double*>(b + o.org_s1);
  m.o_org_s2 = reinterpret_cast<const double*>(b + o.org_s2);
  m.o_counters = reinterpret_cast<const ull*>(b + o.counters);
  m.V = h->V;
  cudaError_t e = launch_merge_stats(m, h->sms, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (tmp) cudaFree(tmp);
  if (e != cudaSuccess) return cuda_fail(e, "nm_dose_merge");
  h->hist_next += hd.hist_next;
  h->n_batches += hd.n_batches;
  h->id_next = h->id_next > hd.id_next ? h->id_next : hd.id_next;
  h->status_seen |= (uint32_t)hd.status_seen;
  return NM_OK;
}

nm_status nm_dose_counters(nm_dose* h, nm_counters* c) {
  if (!h || !c) return fail(NM_ERR_ARG, "bad arguments");
  ull v[kCtrCount];
  NM_CUDA(cudaMemcpyAsync(v, h->counters, sizeof v, cudaMemcpyDeviceToHost, h->stream), "counters");
  NM_CUDA(cudaStreamSynchronize(h->stream), "nm_dose_counters");
  memset(c, 0, sizeof *c);
  c->histories = h->hist_next;
  c->batches = h->n_batches;
  c->emitted = h->emitted(v);
  c->deposited = (int64_t)v[kCtrDepositedUnits];
  c->escaped = (int64_t)v[kCtrEscapedUnits];
  c->killed = (int64_t)v[kCtrKilledUnits];
  c->steps = v[kCtrSteps];
  c->compton = v[kCtrCompton];
  c->photo = v[kCtrPhoto];
  c->rayleigh = v[kCtrRayleigh];
  c->cutoff = v[kCtrCutoff];
  c->escapes = v[kCtrEscapes];
  c->transport_ms = h->transport_ms;
  c->fold_ms = h->fold_ms;
  c->device_status = h->status_seen;
  c->block_threads = h->block;
  c->chunk = h->chunk;
  c->warp_aggregate = h->warp_agg;
  c->regroup = h->regroup;
  c->regroup_lanes = h->regroup_lanes;
  c->grid_blocks = h->grid;
  c->history_splits = v[kCtrHistSplits];
  return NM_OK;
}

nm_status nm_dose_reset(nm_dose* h) {
  if (!h) return fail(NM_ERR_ARG, "handle is NULL");
  cudaStream_t s = h->stream;
  if (h->broken) NM_CUDA(clear_tallies(h, h->tb, 1, s), "reset");
  if (h->broken) NM_CUDA(cudaMemsetAsync(h->status, 0, 4, s), "reset");
  NM_CUDA(cudaMemsetAsync(h->tsum, 0, h->V * sizeof(ull), s), "reset");
  NM_CUDA(cudaMemsetAsync(h->s2, 0, h->V * sizeof(double), s), "reset");
  NM_CUDA(cudaMemsetAsync(h->counters, 0, kCtrCount * sizeof(ull), s), "reset");
  NM_CUDA(cudaMemsetAsync(h->org_s1, 0, kLabelSlots * sizeof(double), s), "reset");
  NM_CUDA(cudaMemsetAsync(h->org_s2, 0, kLabelSlots * sizeof(double), s), "reset");
  if (h->s2h_lo) {
    NM_CUDA(cudaMemsetAsync(h->s2h_lo, 0, h->V * sizeof(ull), s), "reset");
    NM_CUDA(cudaMemsetAsync(h->s2h_hi, 0, h->V * sizeof(ull), s), "reset");
  }
  NM_CUDA(cudaStreamSynchronize(s), "reset");
  h->broken = false;
  h->hist_next = 0;
  h->id_next = 0;
  h->n_batches = 0;
  h->status_seen = 0;
  h->transport_ms = h->fold_ms = 0;
  return NM_OK;
}

void nm_dose_destroy(nm_dose* h) {
  if (!h) return;
  cudaStreamSynchronize(h->stream);
  delete h;
}

nm_status nm_check_philox(const uint32_t* ctr, const uint32_t* key, int64_t n, uint32_t* out) {
  if (n < 0 || (n > 0 && (!ctr || !key || !out))) return fail(NM_ERR_ARG, "bad arguments");
  if (n == 0) return NM_OK;
  uint4 *dc = nullptr, *dout = nullptr;
  uint2* dk = nullptr;
  cudaError_t e = dalloc(&dc, n);
  if (!e) e = dalloc(&dk, n);
  if (!e) e = dalloc(&dout, n);
  if (!e) e = cudaMemcpy(dc, ctr, n * 16, cudaMemcpyHostToDevice);
  if (!e) e = cudaMemcpy(dk, key, n * 8, cudaMemcpyHostToDevice);
  if (!e) e = launch_check_philox(dc, dk, n, dout, 0);
  if (!e) e = cudaMemcpy(out, dout, n * 16, cudaMemcpyDeviceToHost);
  dfree_now(dc); dfree_now(dk); dfree_now(dout);
  return e ? cuda_fail(e, "nm_check_philox") : NM_OK;
}

nm_status nm_check_kahn(double e_mev, int64_t n, uint64_t seed, float* cos_out) {
  if (n < 0 || (n > 0 && !cos_out) || !(e_mev > 0)) return fail(NM_ERR_ARG, "bad arguments");
  if (n == 0) return NM_OK;
  float* d = nullptr;
  uint32_t* st = nullptr;
  cudaError_t e = dalloc(&d, n);
  if (!e) e = dalloc(&st, 1);
  if (!e) e = cudaMemset(st, 0, 4);
  if (!e) e = launch_check_kahn((float)e_mev, n, (uint32_t)seed, (uint32_t)(seed >> 32), d, st, 0);
  if (!e) e = cudaMemcpy(cos_out, d, n * 4, cudaMemcpyDeviceToHost);
  uint32_t flags = 0;
  if (!e) e = cudaMemcpy(&flags, st, 4, cudaMemcpyDeviceToHost);
  dfree_now(d); dfree_now(st);
  if (e) return cuda_fail(e, "nm_check_kahn");
  if (flags) return fail(NM_ERR_DEVICE, "Kahn trial limit hit");
  return NM_OK;
}

void nm_debug_fail_alloc(int32_t n) { g_fail_alloc.store(n > 0 ? n : 0); }
int32_t nm_debug_batch_slots(int64_t voxels, uint64_t n_decays, int32_t batches, uint64_t free_bytes,
                             uint64_t total_bytes, uint64_t held_bytes) {
  if (voxels < 1 || batches < 1) return 0;
  return batch_slots(voxels, n_decays, batches, free_bytes, total_bytes, held_bytes);
}
void nm_debug_fail_enqueue(int32_t n) { g_fail_enqueue.store(n > 0 ? n : 0); }

void nm_release_cached_memory(void) {
  {
    BufferCache& c = buffer_cache();
    std::lock_guard<std::mutex> lock(c.mu);
    release_cache_locked(c);
  }
  StreamPools& sp = stream_pools();
  std::lock_guard<std::mutex> lock(sp.mu);
  for (auto& kv : sp.pool) cudaMemPoolDestroy(kv.second);   // lives on until its last buffer is freed
  sp.pool.clear();
}

nm_status nm_check_wait_timeout(int64_t max_cycles) {
  if (max_cycles < 0) return fail(NM_ERR_ARG, "max_cycles must be >= 0");
  uint32_t* st = nullptr;
  uint32_t flags = 0;
  cudaError_t e = dalloc(&st, 1);
  if (!e) e = cudaMemset(st, 0, 4);
  if (!e) e = launch_check_wait(max_cycles, st, 0);
  if (!e) e = cudaMemcpy(&flags, st, 4, cudaMemcpyDeviceToHost);
  dfree_now(st);
  if (e) return cuda_fail(e, "nm_check_wait_timeout");
  if (flags & NM_DEV_TIMEOUT) return fail(NM_ERR_TIMEOUT, "a bounded device wait gave up after %lld cycles",
                                          (long long)max_cycles);
  return NM_OK;
}

nm_status nm_check_kn_table(double e_mev, double cut_mev, double e0_mev, int64_t n, uint64_t seed,
                            float* cos_out) {
  if (n < 0 || (n > 0 && !cos_out) || !(cut_mev > 0.0 && cut_mev < e0_mev && e0_mev <= 20.0) ||
      !(e_mev >= cut_mev && e_mev <= e0_mev))
    return fail(NM_ERR_ARG, "bad arguments");
  if (n == 0) return NM_OK;
  const std::vector<float>& kt = kn_inverse_cdf(cut_mev, e0_mev);
  TransportParams p;
  memset(&p, 0, sizeof p);
  p.key = philox_key((uint32_t)seed, (uint32_t)(seed >> 32));
  p.kn_inv_lo = (float)std::log(cut_mev);
  p.kn_inv_idln = (float)((kKnInvE - 1) / (std::log(e0_mev) - std::log(cut_mev)));
  float* d = nullptr;
  float* dt = nullptr;
  cudaError_t e = dalloc(&d, n);
  if (!e) e = dalloc(&dt, kt.size());
  if (!e) e = cudaMemcpy(dt, kt.data(), kt.size() * sizeof(float), cudaMemcpyHostToDevice);
  p.kn_inv = dt;
  if (!e) e = launch_check_kn_table(p, (float)e_mev, n, d, 0);
  if (!e) e = cudaMemcpy(cos_out, d, n * sizeof(float), cudaMemcpyDeviceToHost);
  dfree_now(d);
  dfree_now(dt);
  if (e) return cuda_fail(e, "nm_check_kn_table");
  return NM_OK;
}

nm_status nm_check_beta(double t_max_mev, int32_t z, int64_t n, uint64_t seed, float* t_out) {
  if (n < 0 || (n > 0 && !t_out) || !(t_max_mev > 0.0 && t_max_mev < 20.0) || z < 0 || z > 100)
    return fail(NM_ERR_ARG, "bad arguments");
  if (n == 0) return NM_OK;
  const std::vector<float> tab = beta_inverse_cdf(t_max_mev, z);
  float* d = nullptr;
  float* dt = nullptr;
  cudaError_t e = dalloc(&d, n);
  if (!e) e = dalloc(&dt, kBetaTable + 1);
  if (!e) e = cudaMemcpy(dt, tab.data(), (kBetaTable + 1) * sizeof(float), cudaMemcpyHostToDevice);
  if (!e) e = launch_check_beta(dt, n, (uint32_t)seed, (uint32_t)(seed >> 32), d, 0);
  if (!e) e = cudaMemcpy(t_out, d, n * sizeof(float), cudaMemcpyDeviceToHost);
  dfree_now(d);
  dfree_now(dt);
  if (e) return cuda_fail(e, "nm_check_beta");
  return NM_OK;
}

nm_status nm_dose_alias_table(nm_dose* h, int64_t* n_active, float* prob, int32_t* voxel,
                              int32_t* alias_voxel) {
  if (!h || !n_active) return fail(NM_ERR_ARG, "bad arguments");
  *n_active = h->n_active;
  if (!prob && !voxel && !alias_voxel) return NM_OK;
  if (h->n_active == 0) return NM_OK;
  std::vector<uint4> t(h->n_active);
  NM_CUDA(cudaMemcpy(t.data(), h->alias, h->n_active * sizeof(uint4), cudaMemcpyDeviceToHost), "alias copy");
  for (int64_t i = 0; i < h->n_active; ++i) {
    if (prob) memcpy(&prob[i], &t[i].x, 4);
    if (voxel) voxel[i] = (int32_t)t[i].y;
    if (alias_voxel) alias_voxel[i] = (int32_t)t[i].z;
  }
  return NM_OK;
}

nm_status nm_check_source(nm_dose* h, uint64_t first, int64_t n, uint64_t seed, int32_t* voxel,
                          float* pos, float* dir) {
  if (!h || n < 0 || (n > 0 && (!voxel || !pos || !dir))) return fail(NM_ERR_ARG, "bad arguments");
  if (n == 0) return NM_OK;
  int32_t* dv = nullptr;
  float *dp = nullptr, *dd = nullptr;
  cudaError_t e = dalloc(&dv, n);
  if (!e) e = dalloc(&dp, 3 * n);
  if (!e) e = dalloc(&dd, 3 * n);
  const TransportParams p = h->params(first, (uint64_t)n, seed);
  if (!e) e = launch_check_source(p, first, n, dv, dp, dd, h->stream);
  if (!e) e = cudaMemcpyAsync(voxel, dv, n * 4, cudaMemcpyDeviceToHost, h->stream);
  if (!e) e = cudaMemcpyAsync(pos, dp, 3 * n * 4, cudaMemcpyDeviceToHost, h->stream);
  if (!e) e = cudaMemcpyAsync(dir, dd, 3 * n * 4, cudaMemcpyDeviceToHost, h->stream);
  if (!e) e = cudaStreamSynchronize(h->stream);
  dfree_now(dv); dfree_now(dp); dfree_now(dd);
  return e ? cuda_fail(e, "nm_check_source") : NM_OK;
}

}  // extern "C"
