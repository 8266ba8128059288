// Photon transport for ARCHER-NM's method (§2.1): decay sampling, two
// back-to-back 0.511 MeV photons, Woodcock delta tracking through the voxel
// grid, Klein-Nishina Compton (Kahn's sampler), photoelectric absorption,
// optional Rayleigh, 10 keV photon cutoff, int64 fixed-point tally.
//
// One persistent launch for all batches of a run, each with a tally of its own
// (a launch's last photons then leave SMs idle once, not once per batch), in
// two kernels.  In transport_ring_kernel (the default: a point source, and
// decays with annihilation photons, from the decay site or the end of a
// positron's track, or with gamma lines) a warp's lanes hand photons on to each
// other through a ring in shared memory.  In transport_kernel (history
// statistics, decays with both annihilation photons and gamma lines, or
// `regroup` off) each lane owns one photon; a lane whose photon ends takes the
// decay's second photon or, with the rest of its warp, refills from a
// warp-private pool of history ids that one lane grabs from a global counter
// in chunks.  Every iteration of the loop is one flight step for every live
// lane, so lanes stay converged on the flight; the interaction work is
// regrouped (see the `regroup` variant) so that a warp runs Compton sampling
// for a batch of lanes at once instead of once per step.  Both give the same
// bits.
//
// A history's random numbers come from Philox4x32-10 keyed by the seed with
// counter (block index, stream, history id), so which lane or SM simulates it
// does not matter, and integer atomics make the tally order-independent: a
// fixed seed gives bit-identical tallies.
#include <cstddef>
#include <type_traits>

#include "nm_internal.cuh"

namespace nm {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kKahnTrialLimit = 1000;

struct Energy {
  float s_c, s_pe, s_r;   // per-unit-density factors: mu/rho = za s_c + zp s_pe + zr s_r
  float inv_mubar;        // 1 / majorant (cm) of the lane's tracking region
};

// Energy-dependent factors, computed once per energy change.  s_c is
// interpolated in ln E from the Klein-Nishina table; the majorant is constant
// over a table bin and taken at the bin's lower edge, which bounds every
// material's mu on the whole bin because all three mu/rho decrease with E.
template <bool RAYLEIGH>
__device__ __forceinline__ Energy energy_factors(float e, const float* __restrict__ kn,
                                                 const float* __restrict__ minv, float ln_lo,
                                                 float inv_dln) {
  Energy f;
  float x = (__logf(e) - ln_lo) * inv_dln;
  x = fminf(fmaxf(x, 0.0f), (float)(kKnTable - 1) - 0x1p-10f);
  const int i = (int)x;
  const float w = x - (float)i;
  const float a = kn[i], b = kn[i + 1];
  f.s_c = fmaf(w, b - a, a);
  const float ie = __fdividef(1.0f, e);
  const float ie2 = ie * ie;
  f.s_pe = ie2 * ie;
  f.s_r = RAYLEIGH ? ie2 : 0.0f;
  f.inv_mubar = minv[i];
  return f;
}

__device__ __forceinline__ uint4 draw(uint32_t& ctr, uint32_t stream, uint32_t hlo, uint32_t hhi,
                                      const PhiloxKey& key) {
  return philox4x32_10(make_uint4(ctr++, stream, hlo, hhi), key);
}

// Kahn's rejection sampler for the Klein-Nishina distribution (Kahn 1954).
// With k = E/m_e c^2, eta = E/E' in [1, 1 + 2k] and x = (eta - 1)/k = 1 - cos θ:
//   branch 1 (prob. (1+2k)/(9+2k)): eta uniform, accept with 4(eta-1)/eta^2;
//   branch 2: eta = (1+2k)/(1+2k r), accept with (cos^2 θ + 1/eta)/2.
// x is formed directly from the uniforms so that cos θ keeps full precision
// at low energy.  One Philox block per trial; its 4th word is the azimuth.
__device__ __forceinline__ float kahn_x(float k, uint32_t& ctr, uint32_t stream, uint32_t hlo,
                                        uint32_t hhi, const PhiloxKey& key, uint32_t& r_phi,
                                        uint32_t& flags) {
  const float two_k = 2.0f * k;
  const float thr = __fdividef(1.0f + two_k, 9.0f + two_k);
  for (int trial = 0;; ++trial) {
    const uint4 r = draw(ctr, stream, hlo, hhi, key);
    const float r1 = u01(r.x), r2 = u01(r.y), r3 = u01(r.z);
    float x;
    bool acc;
    if (r1 <= thr) {
      x = 2.0f * r2;
      const float eta = fmaf(k, x, 1.0f);
      acc = r3 * eta * eta <= 4.0f * k * x;
    } else {
      x = __fdividef(2.0f * (1.0f - r2), fmaf(two_k, r2, 1.0f));
      const float eta = fmaf(k, x, 1.0f);
      const float c = 1.0f - x;
      acc = 2.0f * r3 <= fmaf(c, c, __fdividef(1.0f, eta));
    }
    if (acc || trial + 1 >= kKahnTrialLimit) {
      if (!acc) flags |= NM_DEV_KAHN_LIMIT;
      r_phi = r.w;
      return x;
    }
  }
}

// Klein-Nishina x = 1 - cos(theta) at photon energy e from one uniform word:
// the inverse CDF tabulated (in FP64, on the host) at kKnInvE log-spaced
// energies x kKnInvU + 1 cumulative probabilities, interpolated linearly in
// ln E and in the probability (CDF error below 2e-5 everywhere).  One draw,
// no rejection loop, so the lanes of a warp never wait for each other.
__device__ __forceinline__ float kn_table_x(const TransportParams& p, float e, uint32_t r) {
  float t = (__logf(e) - p.kn_inv_lo) * p.kn_inv_idln;
  t = fminf(fmaxf(t, 0.0f), (float)(kKnInvE - 1) - 0x1p-10f);
  const int i = (int)t;
  const float w = t - (float)i;
  const float sv = u01(r) * (float)kKnInvU;
  const int j = min((int)sv, kKnInvU - 1);
  const float v = sv - (float)j;
  const float* a = p.kn_inv + i * (kKnInvU + 1) + j;
  const float* b = a + (kKnInvU + 1);
  const float a0 = __ldg(a), a1 = __ldg(a + 1), b0 = __ldg(b), b1 = __ldg(b + 1);
  const float x0 = fmaf(v, a1 - a0, a0), x1 = fmaf(v, b1 - b0, b0);
  return fmaf(w, x1 - x0, x0);
}

// New direction at polar cosine c and azimuth phi about (u, v, w).
__device__ __forceinline__ void rotate(float& u, float& v, float& w, float c, float phi) {
  const float s2 = fmaf(-c, c, 1.0f);
  const float s = s2 > 0.0f ? s2 * rsqrtf(s2) : 0.0f;
  float sp, cp;
  __sincosf(phi, &sp, &cp);
  const float t2 = fmaf(-w, w, 1.0f);
  float nu, nv, nw;
  if (t2 > 1e-10f) {
    const float it = rsqrtf(t2);
    const float t = t2 * it;
    nu = fmaf(c, u, s * (u * w * cp - v * sp) * it);
    nv = fmaf(c, v, s * (v * w * cp + u * sp) * it);
    nw = fmaf(c, w, -s * cp * t);
  } else {
    nu = s * cp;
    nv = s * sp;
    nw = w > 0.0f ? c : -c;
  }
  const float n = rsqrtf(fmaf(nu, nu, fmaf(nv, nv, nw * nw)));
  u = nu * n;
  v = nv * n;
  w = nw * n;
}

// Two-region Woodcock tracking.  Inside the tracking box the majorant is the
// grid's; outside it only air-like voxels remain and the majorant is far
// smaller, so a photon leaving the body crosses the surrounding air in one
// step instead of several.  A flight is cut at the box boundary: by the
// memorylessness of the exponential, restarting the flight there with the
// other region's majorant leaves the free-path distribution unchanged.
//
// Slab parameters of the ray (x, y, z) + t (u, v, w), t in cm, against the
// box: it is inside the box for tn < t < tf.
__device__ __forceinline__ void region_slabs(const PatientGeom& G, float x, float y, float z, float u, float v,
                                             float w, float& tn, float& tf) {
  // approximate reciprocals: the box has a one-voxel margin, so a distance
  // off by a few ulp cannot reach a voxel the region's majorant does not cover
  const float iu = __fdividef(1.0f, u * G.inv_dx), iv = __fdividef(1.0f, v * G.inv_dy),
              iw = __fdividef(1.0f, w * G.inv_dz);
  const float ax = (G.blo[0] - x) * iu, bx = (G.bhi[0] - x) * iu;
  const float ay = (G.blo[1] - y) * iv, by = (G.bhi[1] - y) * iv;
  const float az = (G.blo[2] - z) * iw, bz = (G.bhi[2] - z) * iw;
  // fminf/fmaxf drop the NaN of 0 * inf (a ray in a box face, parallel to it)
  tf = fminf(fmaxf(ax, bx), fminf(fmaxf(ay, by), fmaxf(az, bz)));
  tn = fmaxf(fminf(ax, bx), fmaxf(fminf(ay, by), fminf(az, bz)));
}

constexpr float kInf = __builtin_huge_valf();

// Distance (cm) from (x, y, z) along (u, v, w) to the boundary of the lane's
// region: from inside, to the box's far side; from outside, to its near side,
// or +inf when the ray misses the box (a ray that has left the convex box
// never meets it again).
__device__ __forceinline__ float region_distance(const PatientGeom& G, bool out, float x, float y, float z,
                                                 float u, float v, float w) {
  float tn, tf;
  region_slabs(G, x, y, z, u, v, w, tn, tf);
  if (!out) return tf;
  return tn <= tf && tf > 0.0f ? fmaxf(tn, 0.0f) : kInf;
}

// The same for the ray and for its reverse (photon B leaves the decay site
// opposite to photon A): reversing the ray maps (tn, tf) to (-tf, -tn).
__device__ __forceinline__ void region_distance_pair(const PatientGeom& G, bool out, float x, float y, float z,
                                                     float u, float v, float w, float& fwd, float& rev) {
  float tn, tf;
  region_slabs(G, x, y, z, u, v, w, tn, tf);
  if (!out) {
    fwd = tf;
    rev = -tn;
  } else {
    fwd = tn <= tf && tf > 0.0f ? fmaxf(tn, 0.0f) : kInf;
    rev = tn <= tf && tn < 0.0f ? fmaxf(-tf, 0.0f) : kInf;
  }
}

__device__ __forceinline__ bool outside_box(const PatientGeom& G, float x, float y, float z) {
  return !(x >= G.blo[0] && x < G.bhi[0] && y >= G.blo[1] && y < G.bhi[1] && z >= G.blo[2] && z < G.bhi[2]);
}

// 1 / majorant at energy e from a region's table (same bin as energy_factors).
__device__ __forceinline__ float inv_majorant_at(float e, const float* __restrict__ minv, float ln_lo,
                                                 float inv_dln) {
  float x = (__logf(e) - ln_lo) * inv_dln;
  x = fminf(fmaxf(x, 0.0f), (float)(kKnTable - 1) - 0x1p-10f);
  return minv[(int)x];
}

// Decay site and first-photon direction of history (hlo, hhi).
struct Site {
  int v;              // decay voxel (-1 in point mode)
  float x, y, z;      // voxel units
  float u, v_, w;     // direction of photon A
};

__device__ __forceinline__ Site sample_site(const PatientGeom& G, const PhiloxKey& key,
                                           uint32_t hlo, uint32_t hhi) {
  Site s;
  uint32_t ctr = 0;
  uint4 r = draw(ctr, kStreamSource, hlo, hhi, key);
  uint32_t rc, rphi;
  if (G.source_mode == NM_SOURCE_DECAY) {
    // Alias table: 64 random bits pick a column uniformly, one more the side.
    const uint64_t r64 = ((uint64_t)r.y << 32) | r.x;
    const uint64_t col = __umul64hi(r64, G.n_active);
    const uint4 a = __ldg(G.alias + col);
    s.v = (u01(r.z) < __uint_as_float(a.x)) ? (int)a.y : (int)a.z;
    const int nxy = G.nx * G.ny;
    const int iz = s.v / nxy;
    const int rem = s.v - iz * nxy;
    const int iy = rem / G.nx;
    const int ix = rem - iy * G.nx;
    const uint32_t rx = r.w;
    r = draw(ctr, kStreamSource, hlo, hhi, key);
    // Uniform inside the voxel; keep ix + u below ix + 1 after rounding.
    s.x = fminf((float)ix + u01(rx), __int_as_float(__float_as_int((float)(ix + 1)) - 1));
    s.y = fminf((float)iy + u01(r.x), __int_as_float(__float_as_int((float)(iy + 1)) - 1));
    s.z = fminf((float)iz + u01(r.y), __int_as_float(__float_as_int((float)(iz + 1)) - 1));
    rc = r.z;
    rphi = r.w;
  } else {
    s.v = -1;
    s.x = G.px;
    s.y = G.py;
    s.z = G.pz;
    rc = r.x;
    rphi = r.y;
  }
  // Isotropic: cos θ uniform on (-1, 1), azimuth uniform.
  const float c = fmaf(2.0f, u01(rc), -1.0f);
  const float sn = sqrtf(fmaxf(0.0f, fmaf(-c, c, 1.0f)));
  float sp, cp;
  __sincosf(fmaf(kTwoPi, u01(rphi), -3.14159265f), &sp, &cp);
  s.u = sn * cp;
  s.v_ = sn * sp;
  s.w = c;
  return s;
}

// Katz-Penfold range of a positron of kinetic energy t (MeV), g/cm^2:
// R = 0.412 t^(1.265 - 0.0954 ln t); and its inverse, the lower root of
// 0.0954 L^2 - 1.265 L + ln(R / 0.412) = 0 in L = ln t.
__device__ __forceinline__ float kp_range(float t) {
  const float l = logf(t);
  return 0.412f * expf((1.265f - 0.0954f * l) * l);
}
__device__ __forceinline__ float kp_energy(float r) {
  if (!(r > 0.0f)) return 0.0f;
  const float c = logf(r * (1.0f / 0.412f));
  const float disc = fmaxf(fmaf(-4.0f * 0.0954f, c, 1.265f * 1.265f), 0.0f);
  return expf((1.265f - sqrtf(disc)) * (1.0f / (2.0f * 0.0954f)));
}

// Positron kinetic energy (MeV) for the uniform word r: linear interpolation
// in the inverse-CDF table of the beta+ spectrum.
__device__ __forceinline__ float beta_energy(const float* __restrict__ tab, uint32_t r) {
  const float sv = u01(r) * (float)kBetaTable;
  const int i = min((int)sv, kBetaTable - 1);
  const float ta = __ldg(tab + i), tb = __ldg(tab + i + 1);
  return fmaf(sv - (float)i, tb - ta, ta);
}

// The positron of a decay, beta+ spectrum mode: kinetic energy from the
// inverse-CDF table (linear between nodes), an isotropic straight track from
// the decay site (x, y, z, voxel units; in voxel v0) walked voxel by voxel,
// each voxel using up rho x (path in it) of the mass range and keeping the
// energy lost there, q(T before) - q(T at the range left), until the range
// is spent.  On return (x, y, z) is the end of the track, where the pair
// annihilates, and q0 the positron's energy in tally units.  Returns false if
// the track left the grid; q_left is then the energy it carried out.
template <class Dep>
__device__ __forceinline__ bool positron_track(const PatientGeom& G, const PhiloxKey& key, uint32_t hlo,
                                               uint32_t hhi, int v0, float& x, float& y, float& z,
                                               uint32_t& q0, uint32_t& q_left, Dep&& dep) {
  uint32_t ctr = 0;
  const uint4 r = draw(ctr, kStreamPositron, hlo, hhi, key);
  const float t0 = beta_energy(G.beta_tab, r.x);
  q0 = (uint32_t)q_units(t0);
  const float cz = fmaf(2.0f, u01(r.y), -1.0f);
  const float sn = sqrtf(fmaxf(0.0f, fmaf(-cz, cz, 1.0f)));
  float sp, cp;
  __sincosf(fmaf(kTwoPi, u01(r.z), -3.14159265f), &sp, &cp);
  const float ux = sn * cp, uy = sn * sp, uz = cz;
  const int nxy = G.nx * G.ny;
  int iz = v0 / nxy;
  int iy = (v0 - iz * nxy) / G.nx;
  int ix = v0 - iz * nxy - iy * G.nx;
  // per axis: track length (cm) to the next voxel plane and between planes
  const float dx = 1.0f / G.inv_dx, dy = 1.0f / G.inv_dy, dz = 1.0f / G.inv_dz;
  const int sx = ux > 0.0f ? 1 : -1, sy = uy > 0.0f ? 1 : -1, sz = uz > 0.0f ? 1 : -1;
  float tnx = ux != 0.0f ? ((float)(ix + (ux > 0.0f)) - x) * dx / ux : kInf;
  float tny = uy != 0.0f ? ((float)(iy + (uy > 0.0f)) - y) * dy / uy : kInf;
  float tnz = uz != 0.0f ? ((float)(iz + (uz > 0.0f)) - z) * dz / uz : kInf;
  const float dtx = ux != 0.0f ? dx / fabsf(ux) : kInf;
  const float dty = uy != 0.0f ? dy / fabsf(uy) : kInf;
  const float dtz = uz != 0.0f ? dz / fabsf(uz) : kInf;
  float r_left = kp_range(t0), tcur = 0.0f;
  uint32_t q_cur = q0;
  int v = v0;
  // a straight line crosses at most nx + ny + nz voxels
  const int limit = G.nx + G.ny + G.nz + 2;
  for (int it = 0;; ++it) {
    const bool bx = tnx <= tny && tnx <= tnz;
    const bool by = !bx && tny <= tnz;
    const float tn = bx ? tnx : by ? tny : tnz;
    const float rho = __uint_as_float(__ldg(G.vox + v) & ~7u);
    const float seg = fmaxf(tn - tcur, 0.0f);
    if (rho * seg >= r_left || it + 1 >= limit) {
      // the range ends in this voxel: it keeps the rest of the energy
      if (q_cur) dep(v, q_cur);
      const float send = tcur + fminf(r_left / rho, seg);
      x = fminf(fmaxf(fmaf(send * G.inv_dx, ux, x), (float)ix), __int_as_float(__float_as_int((float)(ix + 1)) - 1));
      y = fminf(fmaxf(fmaf(send * G.inv_dy, uy, y), (float)iy), __int_as_float(__float_as_int((float)(iy + 1)) - 1));
      z = fminf(fmaxf(fmaf(send * G.inv_dz, uz, z), (float)iz), __int_as_float(__float_as_int((float)(iz + 1)) - 1));
      return true;
    }
    r_left -= rho * seg;
    const uint32_t q_new = min((uint32_t)q_units(kp_energy(r_left)), q_cur);
    if (q_cur > q_new) dep(v, q_cur - q_new);
    q_cur = q_new;
    tcur = tn;
    bool left;
    if (bx) {
      ix += sx; v += sx; tnx += dtx; left = (unsigned)ix >= (unsigned)G.nx;
    } else if (by) {
      iy += sy; v += sy * G.nx; tny += dty; left = (unsigned)iy >= (unsigned)G.ny;
    } else {
      iz += sz; v += sz * nxy; tnz += dtz; left = (unsigned)iz >= (unsigned)G.nz;
    }
    if (left) {
      q_left = q_cur;
      return false;
    }
  }
}

// Adds dq units to *cell.  With WARP_AGG the lanes that hit the same cell
// (same address, so lanes of different batches never merge) add their
// deposits with one warp reduction and one atomic.
template <bool WARP_AGG>
__device__ __forceinline__ void tally_flush(ull* cell, bool has, uint32_t dq, uint32_t lane) {
  if (WARP_AGG) {
    const unsigned m = __ballot_sync(kFull, has);
    if (has) {
      const unsigned g = __match_any_sync(m, (unsigned long long)cell);
      const unsigned sum = __reduce_add_sync(g, dq);
      if (lane == (unsigned)(__ffs(g) - 1)) atomicAdd(cell, (ull)sum);
    }
  } else if (has) {
    atomicAdd(cell, (ull)dq);
  }
}

// The tally of the batch that history idx of the launch belongs to.
__device__ __forceinline__ ull* batch_tally(const PatientGeom& G, uint32_t idx) {
  return G.split.slots > 1 ? G.tally + batch_of(G.split, idx) * G.slot_stride : G.tally;
}

__device__ __forceinline__ ull warp_sum(ull x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
  return x;
}

// Compton event at energy e: Kahn-sampled angle, new energy and direction, and
// the local deposit (the electron's energy, or everything below the cutoff).
// With the tabulated sampler (always with TABLE) the angle takes the two words
// (rk, rp) that the flight step which found the event drew but did not use;
// Kahn's sampler draws its own blocks.
template <bool RAYLEIGH, bool TABLE = false>
__device__ __forceinline__ void compton(const TransportParams& p, const float* s_kn,
                                        const float* s_minv, float& e, int32_t& qe, Energy& f,
                                        float& ux, float& uy, float& uz, uint32_t& ctr,
                                        uint32_t stream, uint32_t hlo, uint32_t hhi,
                                        bool& alive, uint32_t& dq, uint32_t& flags,
                                        unsigned long long* s_cnt, uint32_t rk, uint32_t rp) {
  uint32_t rphi;
  const float k = e * kInvElectronMassMeV;
  float x;
  if (TABLE || p.kn_inv) {
    x = kn_table_x(p, e, rk);
    rphi = rp;
  } else {
    x = kahn_x(k, ctr, stream, hlo, hhi, p.key, rphi, flags);
  }
  const float e2 = __fdividef(e, fmaf(k, x, 1.0f));
  rotate(ux, uy, uz, 1.0f - x, fmaf(kTwoPi, u01(rphi), -3.14159265f));
  if (e2 < p.cut) {
    dq = (uint32_t)qe;
    alive = false;
    atomicAdd(&s_cnt[kCtrCutoff], 1ull);
  } else {
    const int32_t q2 = q_units(e2);
    dq = (uint32_t)(qe - q2);
    e = e2;
    qe = q2;
    f = energy_factors<RAYLEIGH>(e, s_kn, s_minv, p.ln_e_lo, p.inv_dln_e);
  }
}

// History statistics: a lane lists its current history's deposits per voxel
// (kHistVoxels entries in shared memory, structure of arrays over the CTA) and
// adds them to the tally, with their squares' halves to two 64-bit sums, when
// the history ends (the lane takes its next history, or the kernel ends).  The
// halves' sums hold a launch's histories (each below 2^32) without overflow and
// go into the 128-bit sums afterwards (launch_fold_history), so that no lane
// waits for an old value to see a carry.  The list loops stay rolled: unrolled
// they spill 220 bytes of the tracked variant's photon.  4 mm phantom, 2e7
// decays: 7.5 -> 6.8 ms, with tracked positrons 18.2 -> 11.9.
struct HistList {
  uint32_t* v;   // voxel of entry i at v[i * stride]
  uint32_t* q;   // units
  int stride;
};

__device__ __forceinline__ void hist_flush(const HistList& L, int& n, ull* tally, ull* lo, ull* hi) {
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const uint32_t v = L.v[i * L.stride], t = L.q[i * L.stride];
    const ull t2 = (ull)t * t;
    atomicAdd(tally + v, (ull)t);
    atomicAdd(lo + v, t2 & 0xffffffffull);
    atomicAdd(hi + v, t2 >> 32);
  }
  n = 0;
}

__device__ __forceinline__ void hist_add(const HistList& L, int& n, uint32_t v, uint32_t dq, ull* tally, ull* lo,
                                         ull* hi, ull* splits) {
#pragma unroll 1
  for (int i = 0; i < n; ++i)
    if (L.v[i * L.stride] == v) {
      L.q[i * L.stride] += dq;
      return;
    }
  if (n == kHistVoxels) {
    // more voxels than a lane keeps: the totals so far are squared now
    hist_flush(L, n, tally, lo, hi);
    atomicAdd(splits, 1ull);
  }
  L.v[n * L.stride] = v;
  L.q[n * L.stride] = dq;
  ++n;
}

template <bool WARP_AGG, bool RAYLEIGH, bool REGROUP, bool HIST, bool BETA>
__global__ void __launch_bounds__(512, 2) transport_kernel(const TransportParams p) {
  static_assert(!HIST || !WARP_AGG, "history statistics: lane-wise deposits");
  static_assert(!BETA || !WARP_AGG, "beta+ spectrum: lane-wise deposits");
  __shared__ float s_kn[kKnTable];
  __shared__ float s_minv[kKnTable];
  __shared__ float s_minv_out[kKnTable];
  __shared__ MaterialCoef s_mat[NM_MAX_MATERIALS];
  __shared__ Energy s_f0;
  __shared__ float s_inv0_out;              // 1 / majorant outside the box at e0
  // Indexed by CounterSlot: the rare events (photo, cutoff, rayleigh, killed units).
  __shared__ unsigned long long s_cnt[10];  // [8]: positron, [9]: gamma units
  extern __shared__ float s_site[];         // [9][blockDim]: decay site, photon A direction, photon B's
                                            // distance to its region boundary, a pending Compton's two words;
                                            // then the history lists (HIST) and the gamma origin (BETA)
  for (int i = threadIdx.x; i < kKnTable; i += blockDim.x) {
    s_kn[i] = p.kn[i];
    s_minv[i] = p.minv[i];
    s_minv_out[i] = p.minv_out[i];
  }
  if (threadIdx.x < NM_MAX_MATERIALS) s_mat[threadIdx.x] = p.mat[threadIdx.x];
  if (threadIdx.x < 10) s_cnt[threadIdx.x] = 0;
  __syncthreads();
  if (threadIdx.x == 0) {
    s_f0 = energy_factors<RAYLEIGH>(p.e0, s_kn, s_minv, p.ln_e_lo, p.inv_dln_e);
    s_inv0_out = inv_majorant_at(p.e0, s_minv_out, p.ln_e_lo, p.inv_dln_e);
  }
  __syncthreads();
  float* site = s_site + threadIdx.x;
  const int nb = blockDim.x;
  const HistList hl{reinterpret_cast<uint32_t*>(s_site + 9 * nb) + threadIdx.x,
                    reinterpret_cast<uint32_t*>(s_site + (9 + kHistVoxels) * nb) + threadIdx.x, nb};
  int hn = 0;                            // entries in this lane's history list
  // nuclide variant: the decay site (origin of the gamma lines) and the lines
  // of this decay still to be emitted
  float* gsite = s_site + (9 + (HIST ? 2 * kHistVoxels : 0)) * nb + threadIdx.x;
  uint32_t gmask = 0;

  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t lt_mask = (1u << lane) - 1u;
  // Warp-uniform work pool [pool_next, pool_end).
  uint32_t pool_next = 0, pool_end = 0;
  const PatientGeom& G = p.g;
  bool done = false, alive = false, pending_b = false, pending_c = false;
  float px = 0.f, py = 0.f, pz = 0.f, ux = 0.f, uy = 0.f, uz = 0.f;
  float e = 0.f;
  Energy f = s_f0;
  int32_t qe = 0;
  int cv = 0;                            // voxel of a pending Compton event
  ull* tal = p.g.tally;                  // tally of this lane's history's batch
  uint32_t hlo = 0, hhi = 0, stream = 0, ctr = 0;
  bool out = false;                      // outside the tracking box
  float rem = 0.f;                       // cm to the region boundary along (ux, uy, uz)
  int steps = 0;
  uint32_t n_steps = 0, n_compton = 0, n_esc = 0, flags = 0;
  ull escaped = 0;

  for (;;) {
    // ---- second photon of the decay: same site, opposite direction ----------
    if (!alive && pending_b) {
      pending_b = false;
      alive = true;
      px = site[0]; py = site[nb]; pz = site[2 * nb];
      ux = -site[3 * nb]; uy = -site[4 * nb]; uz = -site[5 * nb];
      e = p.e0; qe = p.q_e0; f = s_f0;
      stream = kStreamPhotonB; ctr = 0; steps = 0;
      out = outside_box(G, px, py, pz);
      rem = site[6 * nb];
      if (out) f.inv_mubar = s_inv0_out;
    } else if (BETA && !alive && gmask) {
      // ---- next gamma line of the decay: from the decay site, isotropic ------
      const int j = __ffs(gmask) - 1;
      gmask &= gmask - 1;
      alive = true;
      px = gsite[0]; py = gsite[nb]; pz = gsite[2 * nb];
      stream = kStreamGamma0 + (uint32_t)j; ctr = 0; steps = 0;
      const uint4 rd = draw(ctr, stream, hlo, hhi, p.key);
      const float c = fmaf(2.0f, u01(rd.x), -1.0f);
      const float sn = sqrtf(fmaxf(0.0f, fmaf(-c, c, 1.0f)));
      float sp, cp;
      __sincosf(fmaf(kTwoPi, u01(rd.y), -3.14159265f), &sp, &cp);
      ux = sn * cp; uy = sn * sp; uz = c;
      e = p.gamma_e[j]; qe = p.gamma_q[j];
      atomicAdd(&s_cnt[9], (ull)(uint32_t)qe);
      out = outside_box(p.g, px, py, pz);
      f = energy_factors<RAYLEIGH>(e, s_kn, out ? s_minv_out : s_minv, p.ln_e_lo, p.inv_dln_e);
      rem = region_distance(p.g, out, px, py, pz, ux, uy, uz);
    }
    // ---- refill: lanes without a photon take new histories from the pool ----
    const unsigned need = __ballot_sync(kFull, !alive && !done);
    bool refill = need != 0;
    if (REGROUP && refill) {
      // Start new histories for many lanes at once, once enough lanes wait or
      // nothing else can fly.
      const unsigned flying = __ballot_sync(kFull, alive && !pending_c);
      refill = __popc(need) >= (unsigned)p.regroup_refill || flying == 0;
    }
    if (refill) {
      const uint32_t cnt = __popc(need);
      const uint32_t avail = pool_end - pool_next;
      uint32_t fresh = 0, fresh_end = 0;
      if (avail < cnt) {
        if (lane == 0) {
          const unsigned f0 = atomicAdd(G.work, (unsigned)p.chunk);
          if ((uint64_t)f0 < G.n_hist) {
            fresh = f0;
            fresh_end = (uint32_t)min((uint64_t)f0 + (uint64_t)p.chunk, G.n_hist);
          }
        }
        fresh = __shfl_sync(kFull, fresh, 0);
        fresh_end = __shfl_sync(kFull, fresh_end, 0);
      }
      bool has = false;
      ull* cell = nullptr;
      if (!alive && !done) {
        const uint32_t rank = __popc(need & lt_mask);
        uint32_t idx = 0;
        bool got = true;
        if (rank < avail) {
          idx = pool_next + rank;
        } else if (fresh + (rank - avail) < fresh_end) {
          idx = fresh + (rank - avail);
        } else {
          got = false;
          if (fresh_end == 0) done = true;   // every history has been handed out
        }
        if (got) {
          if (HIST && hn) hist_flush(hl, hn, tal, p.s2h_lo, p.s2h_hi);   // the previous history ends
          tal = batch_tally(G, idx);
          const uint64_t h = G.hist_begin + idx;
          hlo = (uint32_t)h;
          hhi = (uint32_t)(h >> 32);
          Site st = sample_site(G, p.key, hlo, hhi);
          bool pair = true;                  // the annihilation photons start inside the grid
          if (BETA && G.source_mode == NM_SOURCE_DECAY) {
            // another radionuclide: gamma lines of this decay, emitted later
            // from the decay site (the nucleus), one photon at a time
            gsite[0] = st.x; gsite[nb] = st.y; gsite[2 * nb] = st.z;
            uint32_t m = 0, gc = 0;
            for (int j0 = 0; j0 < p.n_gamma; j0 += 4) {
              const uint4 rg = draw(gc, kStreamGammaSelect, hlo, hhi, p.key);
              const uint32_t w4[4] = {rg.x, rg.y, rg.z, rg.w};
              for (int k = 0; k < 4 && j0 + k < p.n_gamma; ++k)
                if (u01(w4[k]) < p.gamma_y[j0 + k]) m |= 1u << (j0 + k);
            }
            gmask = m;
          }
          if (BETA && G.beta_tab) {
            uint32_t q0 = 0, q_left = 0;
            pair = positron_track(G, p.key, hlo, hhi, st.v, st.x, st.y, st.z, q0, q_left,
                                  [&](int v, uint32_t dq) {
                                    if (HIST)
                                      hist_add(hl, hn, (uint32_t)v, dq, tal, p.s2h_lo, p.s2h_hi,
                                               p.g.counters + kCtrHistSplits);
                                    else
                                      atomicAdd(tal + v, (ull)dq);
                                  });
            atomicAdd(&s_cnt[8], (ull)q0);
            if (!pair) escaped += (ull)q_left + (p.annihilate ? 2ull * (ull)(uint32_t)p.q_e0 : 0ull);
          }
          if (BETA && G.source_mode == NM_SOURCE_DECAY && G.q_positron > 0 && !p.annihilate) {
            // no annihilation photon to carry the local deposit: tally it here
            if (HIST)
              hist_add(hl, hn, (uint32_t)st.v, (uint32_t)G.q_positron, tal, p.s2h_lo, p.s2h_hi,
                       p.g.counters + kCtrHistSplits);
            else
              atomicAdd(tal + st.v, (ull)(uint32_t)G.q_positron);
          }
          if (BETA && !p.annihilate && G.source_mode == NM_SOURCE_DECAY) pair = false;
          if (pair) {
          px = st.x; py = st.y; pz = st.z;
          ux = st.u; uy = st.v_; uz = st.w;
          e = p.e0; qe = p.q_e0; f = s_f0;
          stream = kStreamPhotonA; ctr = 0; steps = 0;
          alive = true;
          out = outside_box(G, px, py, pz);
          if (out) f.inv_mubar = s_inv0_out;
          float rem_b;
          region_distance_pair(G, out, px, py, pz, ux, uy, uz, rem, rem_b);
          if (G.source_mode == NM_SOURCE_DECAY) {
            site[0] = st.x; site[nb] = st.y; site[2 * nb] = st.z;
            site[3 * nb] = st.u; site[4 * nb] = st.v_; site[5 * nb] = st.w;
            site[6 * nb] = rem_b;
            pending_b = true;
            if (HIST) {
              if (G.q_positron > 0)
                hist_add(hl, hn, (uint32_t)st.v, (uint32_t)G.q_positron, tal, p.s2h_lo, p.s2h_hi,
                         p.g.counters + kCtrHistSplits);
            } else {
              has = G.q_positron > 0;
              cell = tal + st.v;
            }
          }
          }
        }
      }
      if (avail < cnt) {
        pool_next = min(fresh + (cnt - avail), fresh_end);
        pool_end = fresh_end;
      } else {
        pool_next += cnt;
      }
      tally_flush<WARP_AGG>(cell, has, (uint32_t)G.q_positron, lane);
    }
    if (!__any_sync(kFull, alive || !done)) break;

    bool has = false;
    int dv = 0;
    uint32_t dq = 0;
    // ---- Compton passes (regrouped: run when enough lanes wait) -------------
    if (REGROUP) {
      const unsigned waiting = __ballot_sync(kFull, pending_c);
      const unsigned flying = __ballot_sync(kFull, alive && !pending_c);
      if (waiting && (__popc(waiting) >= (unsigned)p.regroup_compton || flying == 0)) {
        if (pending_c) {
          pending_c = false;
          const uint32_t* words = reinterpret_cast<const uint32_t*>(site);
          compton<RAYLEIGH>(p, s_kn, out ? s_minv_out : s_minv, e, qe, f, ux, uy, uz, ctr, stream, hlo, hhi,
                            alive, dq, flags, s_cnt, words[7 * nb], words[8 * nb]);
          rem = region_distance(G, out, px, py, pz, ux, uy, uz);
          has = true;
          dv = cv;
        }
        // The scattered photons tally their deposit now and take their next
        // flight step in this same iteration instead of idling through it.
        if (HIST) {
          if (has) hist_add(hl, hn, (uint32_t)dv, dq, tal, p.s2h_lo, p.s2h_hi, p.g.counters + kCtrHistSplits);
        } else {
          tally_flush<WARP_AGG>(tal + dv, has, dq, lane);
        }
        has = false;
        dq = 0;
        dv = 0;
      }
    }
    // ---- one Woodcock flight step per live lane -------------------------------
    if (alive && !pending_c && !has) {
      // A fresh Philox block every step (words x and y; z and w serve the
      // Compton angle if the step finds one): keeping them for the next step
      // would save draws per lane but not per warp, where lanes
      // are out of phase, and costs registers.
      const uint4 rr = draw(ctr, stream, hlo, hhi, p.key);
      const uint32_t r0 = rr.x, r1 = rr.y;
      const float imaj = f.inv_mubar;
      float s = -__logf(u01(r0)) * imaj;   // cm
      const bool cross = s >= rem;         // flight cut at the region boundary
      if (cross) s = rem;
      rem -= s;
      px = fmaf(s * G.inv_dx, ux, px);
      py = fmaf(s * G.inv_dy, uy, py);
      pz = fmaf(s * G.inv_dz, uz, pz);
      ++n_steps;
      ++steps;
      // floor once: the same integers test the grid bounds (negative or past
      // the end, as unsigned) and index the voxel (positions are finite)
      const int ix = __float2int_rd(px), iy = __float2int_rd(py), iz = __float2int_rd(pz);
      if ((unsigned)ix >= (unsigned)G.nx || (unsigned)iy >= (unsigned)G.ny || (unsigned)iz >= (unsigned)G.nz) {
        escaped += (ull)qe;
        ++n_esc;
        alive = false;
      } else if (cross) {
        out = !out;
        rem = out ? kInf : region_distance(G, false, px, py, pz, ux, uy, uz);
        f.inv_mubar = inv_majorant_at(e, out ? s_minv_out : s_minv, p.ln_e_lo, p.inv_dln_e);
      } else {
        const int v = (iz * G.ny + iy) * G.nx + ix;
        const uint32_t wv = __ldg(G.vox + v);
        const MaterialCoef c = s_mat[wv & 7u];
        // real event with probability mu(voxel)/mubar; the same uniform picks the type
        const float scale = __uint_as_float(wv & ~7u) * imaj;
        const float ic = c.za * f.s_c;
        const float icp = fmaf(c.zp, f.s_pe, ic);
        const float t = u01(r1);
        if (t < scale * ic) {
          ++n_compton;
          if (REGROUP) {
            pending_c = true;
            cv = v;
            // the step's two unused words wait in the stash for the Compton pass
            uint32_t* words = reinterpret_cast<uint32_t*>(site);
            words[7 * nb] = rr.z;
            words[8 * nb] = rr.w;
          } else {
            compton<RAYLEIGH>(p, s_kn, out ? s_minv_out : s_minv, e, qe, f, ux, uy, uz, ctr, stream, hlo,
                              hhi, alive, dq, flags, s_cnt, rr.z, rr.w);
            rem = region_distance(G, out, px, py, pz, ux, uy, uz);
            has = true;
            dv = v;
          }
        } else if (t < scale * icp) {
          atomicAdd(&s_cnt[kCtrPhoto], 1ull);
          has = true;
          dv = v;
          dq = (uint32_t)qe;
          alive = false;
        } else if (RAYLEIGH && t < scale * fmaf(c.zr, f.s_r, icp)) {
          atomicAdd(&s_cnt[kCtrRayleigh], 1ull);
          // Thomson angular shape (1 + cos^2)/2 by rejection; one block per trial.
          for (int trial = 0;; ++trial) {
            const uint4 r = draw(ctr, stream, hlo, hhi, p.key);
            const float cth = fmaf(2.0f, u01(r.x), -1.0f);
            const bool acc = 2.0f * u01(r.y) <= fmaf(cth, cth, 1.0f);
            if (acc || trial + 1 >= kKahnTrialLimit) {
              if (!acc) flags |= NM_DEV_RAYLEIGH_LIMIT;
              rotate(ux, uy, uz, cth, fmaf(kTwoPi, u01(r.z), -3.14159265f));
              rem = region_distance(G, out, px, py, pz, ux, uy, uz);
              break;
            }
          }
        }
      }
      if (alive && steps >= p.max_steps) {
        atomicAdd(&s_cnt[kCtrKilledUnits], (ull)qe);
        flags |= NM_DEV_STEP_LIMIT;
        alive = false;
        pending_c = false;
      }
    }
    if (HIST) {
      if (has) hist_add(hl, hn, (uint32_t)dv, dq, tal, p.s2h_lo, p.s2h_hi, p.g.counters + kCtrHistSplits);
    } else {
      tally_flush<WARP_AGG>(tal + dv, has, dq, lane);
    }
  }
  if (HIST && hn) hist_flush(hl, hn, tal, p.s2h_lo, p.s2h_hi);

  // ---- counters ---------------------------------------------------------------
  {
    // warp sums, one atomic per warp per counter
    ull sm = warp_sum((ull)n_steps);
    if (lane == 0 && sm) atomicAdd(p.g.counters + kCtrSteps, sm);
    sm = warp_sum((ull)n_compton);
    if (lane == 0 && sm) atomicAdd(p.g.counters + kCtrCompton, sm);
    sm = warp_sum((ull)n_esc);
    if (lane == 0 && sm) atomicAdd(p.g.counters + kCtrEscapes, sm);
    sm = warp_sum(escaped);
    if (lane == 0 && sm) atomicAdd(p.g.counters + kCtrEscapedUnits, sm);
  }
  const unsigned fl = __reduce_or_sync(kFull, flags);
  if (lane == 0 && fl) atomicOr(p.status, fl);
  __syncthreads();
  if (threadIdx.x < 10 && s_cnt[threadIdx.x]) {
    const int k = threadIdx.x;           // the CounterSlot; 8 the positron and 9 the gamma units
    atomicAdd(p.g.counters + (k < 8 ? k : k == 8 ? (int)kCtrPositronUnits : (int)kCtrGammaUnits), s_cnt[k]);
  }
}

// ---------------------------------------------------------------------------
// The default transport: photons handed from lane to lane.
//
// Bound by instruction issue.  A flight step finds a scatter or ends a photon
// about every second time, so a warp whose lanes keep their photon through a
// scatter flies with half its lanes.  Here a lane that finds a Compton event
// parks its photon in the warp's ring in shared memory and, in the same
// exchange, takes a photon that is ready to fly; once 32 are parked the whole
// warp scatters them at once, one per lane, in place.
//
// The ring holds kRing photons and is always full: [head - n_parked, head) are
// parked, the others, from head on, are ready (or empty, energy 0, which hands
// the lane on to the site queue).  An exchange at the head turns a ready slot
// into the youngest parked one; a Compton pass over the 32 oldest parked slots
// makes them the ring's last ready ones.  So the only bookkeeping is head and
// n_parked (warp-uniform), and all accesses go to consecutive slots (no bank
// conflicts).  A lane without a photon takes the next of the site queue (32
// decays sampled at once, two photons each); when every decay has been
// started, it exchanges an empty slot instead, which turns the ring; and once
// the lanes can hold all photons left, each scatters its own, so that the last
// photons of a launch do not wait in the ring (5e6 decays 1.15 -> 1.10 ms, 1e6
// point-source histories in ten launches 0.76 -> 0.50 ms).
//
// Benchmark phantom, 1e9 decays: 234.6 -> 136 ms; per decay 238.8 -> 128.7
// warp instructions at 16.2 -> 25 active lanes.  Of that, the ring itself
// with one word per access 234.6 -> 197.7; slots as 16-byte words, the uniform
// variates without a conversion and no denormals -> 171.7; branches folded into
// predicates, both regions' majorants kept with the photon, escapes counted
// from what is left over -> 150.5; a loop of its own for the end, the region
// and photon B as signs -> 137.8; shared-memory addresses formed once -> 135.9;
// the lanes' own scatters at the end -> 137.3; all batches in one launch -> 136.
// A FIFO that pushes to and pops from different slots (fewer register moves,
// more bookkeeping) measured 148-160.
// ---------------------------------------------------------------------------
constexpr int kRing = 64;       // photons: 31 parked at most before an exchange, 32 lanes more
constexpr int kSiteQueue = 32;  // decays
// A ring slot is three 16-byte words and one of eight bytes, each an array
// over the slots, so that a lane moves its photon with a few wide accesses and
// the warp's accesses have no bank conflicts:
//   pos: position (voxel units), energy (0: empty; negative: photon B);
//   dir: direction, low word of the history id;
//   mid: ready: s_c, s_pe, 1 / majorant of the photon's region, distance to the
//        region's boundary; parked: the Compton pass's two Philox words, the
//        voxel, 1 / majorant;
//   aux: next Philox counter, 1 / majorant of the other region.
// A majorant outside the tracking box carries a minus sign, so that the sign
// tells the region.
// The site queue: position and history id; photon A's direction and its
// distance to the region boundary; photon B's distance, and -1 outside the box.
struct WarpStore {
  float4 pos[kRing], dir[kRing], mid[kRing];
  float4 site_pos[kSiteQueue], site_dir[kSiteQueue];
  uint2 aux[kRing];
  float2 site_rem[kSiteQueue];
};
struct GenStore {
  uint2 gen[kRing];             // flight steps (the counter also counts other draws), Rayleigh factor
};
// Gamma lines (kGammas): the queue holds single photons, which differ in
// energy: s_c, s_pe and the majorants of each, and in the place of site_rem
// its energy and its counter word.  More photons than the queue holds wait as
// (history, lines still to be emitted).
struct GammaStore {
  float4 site_mid[kSiteQueue];
  uint2 defer[kSiteQueue];
};

// What a decay gives (nuclide_kind): the annihilation pair of a positron that
// stays where it is (or a point source's photon), of one that is tracked, or
// gamma lines (and a tracked or local beta particle).
enum Nuclide { kPair = 0, kTracked = 1, kGammas = 2 };

// Layout of a warp's store: the parts its variant needs, one after the other.
template <bool GENERAL, int NUC>
struct StoreOf {
  static constexpr uint32_t kGen = sizeof(WarpStore);
  static constexpr uint32_t kGamma = kGen + (GENERAL ? sizeof(GenStore) : 0);
  static constexpr uint32_t kBytes = kGamma + (NUC == kGammas ? sizeof(GammaStore) : 0);
  static_assert(kBytes % 16 == 0 && kGamma % 16 == 0, "warps' stores stay 16-byte aligned");
};
// The Philox counter word of a gamma line's photon: its stream above the counter.
constexpr int kStreamShift = 27;
constexpr uint32_t kCtrMask = (1u << kStreamShift) - 1u;

// Shared-memory accesses by 32-bit address (the compiler forms the address of
// a shared array anew at every use).
__device__ __forceinline__ float4 lds4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ float2 lds2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ float lds1(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts4(uint32_t a, float x, float y, float z, float w) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}
__device__ __forceinline__ void sts2(uint32_t a, float x, float y) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ void sts1(uint32_t a, float x) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(x) : "memory");
}

// Cross sections at energy e: bins of {kn, next - this, 1 / majorant inside,
// - 1 / majorant outside the tracking box} (energy_factors, both regions).
struct RingEnergy {
  float s_c, s_pe, s_r, maj_in, maj_out;
};
template <bool RAYLEIGH>
__device__ __forceinline__ RingEnergy ring_energy(float e, uint32_t tab, float ln_lo, float inv_dln) {
  RingEnergy f;
  float x = (__logf(e) - ln_lo) * inv_dln;
  x = fminf(fmaxf(x, 0.0f), (float)(kKnTable - 1) - 0x1p-10f);
  const int i = (int)x;
  const float4 t = lds4(tab + 16 * i);
  f.s_c = fmaf(x - (float)i, t.y, t.x);
  const float ie = __fdividef(1.0f, e);
  const float ie2 = ie * ie;
  f.s_pe = ie2 * ie;
  f.s_r = RAYLEIGH ? ie2 : 0.0f;
  f.maj_in = t.z;
  f.maj_out = t.w;
  return f;
}

// Tables of a CTA, at the start of its dynamic shared memory; a store per warp
// follows.
struct RingTables {
  float4 tab[kKnTable];
  float2 mat[NM_MAX_MATERIALS];   // za, zp
  float zr[NM_MAX_MATERIALS];
  uint32_t next[kMaxSlots];       // first history of the launch past batch b
};
static_assert(sizeof(RingTables) % 16 == 0, "the warps' stores follow");

// GENERAL: Rayleigh scattering and Kahn's sampler, whose trials draw from the
// photon's counter; otherwise the counter is the number of flight steps.
template <bool WARP_AGG, bool GENERAL, int NUC>
__global__ void __launch_bounds__(512, 2) transport_ring_kernel(const TransportParams p) {
  typedef StoreOf<GENERAL, NUC> Store;
  static_assert(NUC == kPair || !WARP_AGG, "tracks deposit lane by lane");
  constexpr bool GAMMAS = NUC == kGammas;
  __shared__ RingEnergy s_f0;                  // at the source energy
  // [0..7]: CounterSlot; photons started, killed; energy they deposited; of
  // decays: energy of the beta particles, of the gamma lines, taken out of the
  // grid by tracks (with the photons that then do not start)
  __shared__ unsigned long long s_cnt[14];
  extern __shared__ __align__(16) unsigned char s_dyn[];   // tables, then a Store per warp
  RingTables& tb = *reinterpret_cast<RingTables*>(s_dyn);
  for (int i = threadIdx.x; i < kKnTable; i += blockDim.x) {
    const float a = p.kn[i];
    tb.tab[i] = make_float4(a, p.kn[min(i + 1, kKnTable - 1)] - a, p.minv[i], -p.minv_out[i]);
  }
  if (threadIdx.x < NM_MAX_MATERIALS) {
    const MaterialCoef m = p.mat[threadIdx.x];
    tb.mat[threadIdx.x] = make_float2(m.za, m.zp);
    tb.zr[threadIdx.x] = m.zr;
  }
  if (threadIdx.x < kMaxSlots)
    tb.next[threadIdx.x] = threadIdx.x + 1 < p.g.split.slots ? p.g.split.start(threadIdx.x + 1) : 0xffffffffu;
  if (threadIdx.x < 14) s_cnt[threadIdx.x] = 0;
  __syncthreads();
  uint32_t tables, store;                // volatile: kept, not formed again at every use
  asm volatile("mov.u32 %0, %1;" : "=r"(tables) : "r"((uint32_t)__cvta_generic_to_shared(s_dyn)));
  asm volatile("mov.u32 %0, %1;"
               : "=r"(store)
               : "r"(tables + (uint32_t)sizeof(RingTables) + (threadIdx.x >> 5) * Store::kBytes));
  const uint32_t tab = tables + offsetof(RingTables, tab), mat = tables + offsetof(RingTables, mat),
                 zr = tables + offsetof(RingTables, zr), next = tables + offsetof(RingTables, next);
  if (threadIdx.x == 0) s_f0 = ring_energy<GENERAL>(p.e0, tab, p.ln_e_lo, p.inv_dln_e);
  __syncthreads();
  constexpr int kBorn = 8, kKilled = 9, kDeposit = 10, kBeta = 11, kGamma = 12, kLost = 13;

  const uint32_t lane = threadIdx.x & 31u;
  uint32_t lt_mask;                      // volatile: kept, not fetched again at every use
  asm volatile("mov.u32 %0, %%lanemask_lt;" : "=r"(lt_mask));
#define RING_AT(word, slot) (store + (uint32_t)offsetof(WarpStore, word) + 16u * (slot))
#define RING_AT8(word, slot) (store + (uint32_t)offsetof(WarpStore, word) + 8u * (slot))
#define RING_GEN(slot) (store + Store::kGen + 8u * (slot))
#define GAMMA_MID(slot) (store + Store::kGamma + (uint32_t)offsetof(GammaStore, site_mid) + 16u * (slot))
#define GAMMA_DEFER(slot) (store + Store::kGamma + (uint32_t)offsetof(GammaStore, defer) + 8u * (slot))
  sts1(RING_AT(pos, lane) + 12, 0.0f);   // every slot starts empty
  sts1(RING_AT(pos, 32 + lane) + 12, 0.0f);
  __syncwarp();

  // History ids of the launch span less than 2^32: the low word tells the high one.
  const uint32_t h0 = (uint32_t)p.g.hist_begin, h0_hi = (uint32_t)(p.g.hist_begin >> 32);
  // warp-uniform state
  uint32_t head = 0, n_parked = 0;       // ring
  uint32_t s_next = 0, s_left = 0;       // photons of the site queue
  uint32_t pool_next = 0, pool_end = 0;  // histories of the launch grabbed and not yet sampled
  bool drained = false;                  // every history has been handed out
  uint32_t n_born = 0, n_compton = 0;
  const bool pairs = NUC == kTracked || (NUC == kPair && p.g.source_mode == NM_SOURCE_DECAY);   // two photons per entry
  bool deferred = false;                 // lines of sampled decays are still to be emitted
  // this lane's photon (none while e = 0; photon B while e < 0)
  float px = 0.f, py = 0.f, pz = 0.f, ux = 0.f, uy = 0.f, uz = 0.f, e = 0.f, rem = 0.f;
  float s_c = 0.f, s_pe = 0.f, s_r = 0.f, maj = 1.f, maj2 = 1.f;
  uint32_t hlo = h0, ctr = 0, steps = 0;
  uint32_t flags = 0;
  uint32_t n_steps = 0;                  // flight steps of the photons this lane saw end
  ull deposit = 0;                       // energy of the deposits this lane made

  // Flight steps from the counter word: a gamma line's photon drew its direction first.
  auto steps_of = [](uint32_t c) -> uint32_t { return GAMMAS ? (c & kCtrMask) - 1u : c; };
  // Tally cell of voxel v in the batch of history idx of the launch (batch_of,
  // from the table of batch ends; all batches' voxels count below 2^32).
  auto tally_cell = [&](uint32_t idx, uint32_t v) -> ull* {
    uint32_t b = __umulhi(idx, p.g.split.est);
    if (idx >= __float_as_uint(lds1(next + 4u * b))) ++b;
    return p.g.tally + (b * p.g.slot_stride + v);
  };
  // The Compton event of a photon of signed energy ce with direction and
  // history cd, drawn with the flight step's words rk and rp: its deposit dq,
  // its new direction; returns its new energy, 0 below the cutoff.
  auto scatter = [&](float ce, float4& cd, uint32_t& cctr, uint32_t rk, uint32_t rp, uint32_t& dq) -> float {
    const float e1 = fabsf(ce);
    float x;
    if (!GENERAL || p.kn_inv) {
      x = kn_table_x(p, e1, rk);
    } else {
      const uint32_t clo = __float_as_uint(cd.w);
      uint32_t cnt = GAMMAS ? cctr & kCtrMask : cctr;
      const uint32_t stream = GAMMAS ? cctr >> kStreamShift : ce < 0.0f ? kStreamPhotonB : kStreamPhotonA;
      x = kahn_x(e1 * kInvElectronMassMeV, cnt, stream, clo, h0_hi + (clo < h0 ? 1u : 0u), p.key, rp, flags);
      cctr = GAMMAS ? (cctr & ~kCtrMask) | cnt : cnt;
    }
    const float e2 = __fdividef(e1, fmaf(e1 * kInvElectronMassMeV, x, 1.0f));
    rotate(cd.x, cd.y, cd.z, 1.0f - x, fmaf(kTwoPi, u01(rp), -3.14159265f));
    const int32_t q1 = q_units(e1);
    if (e2 < p.cut) {
      atomicAdd(&s_cnt[kCtrCutoff], 1ull);
      dq = (uint32_t)q1;
      deposit += dq;
      return 0.0f;
    }
    dq = (uint32_t)(q1 - q_units(e2));
    deposit += dq;
    return copysignf(e2, ce);
  };

  // ---- Compton pass: the 32 oldest parked photons (all, if fewer), one per
  // lane; returns the number that fell below the cutoff
  auto compton_pass = [&]() -> uint32_t {
    const uint32_t i = (head - n_parked + lane) & (kRing - 1);
    const float4 cp = lds4(RING_AT(pos, i));
    uint32_t dq = 0;
    ull* cell = nullptr;
    bool gone = false;
    if (cp.w != 0.0f && lane < n_parked) {
      float4 cd = lds4(RING_AT(dir, i));
      const float4 cm = lds4(RING_AT(mid, i));
      cell = tally_cell(__float_as_uint(cd.w) - h0, __float_as_uint(cm.z));
      uint32_t cctr = 0;
      if constexpr (GENERAL) cctr = __float_as_uint(lds1(RING_AT8(aux, i)));
      const float ce = scatter(cp.w, cd, cctr, __float_as_uint(cm.x), __float_as_uint(cm.y), dq);
      sts1(RING_AT(pos, i) + 12, ce);
      if (ce == 0.0f) {
        gone = true;
        if constexpr (GENERAL) n_steps += __float_as_uint(lds1(RING_GEN(i)));
        else n_steps += steps_of(__float_as_uint(lds1(RING_AT8(aux, i))));
      } else {
        const RingEnergy f = ring_energy<GENERAL>(fabsf(ce), tab, p.ln_e_lo, p.inv_dln_e);
        const bool cout = cm.w < 0.0f;
        sts4(RING_AT(dir, i), cd.x, cd.y, cd.z, cd.w);
        sts4(RING_AT(mid, i), f.s_c, f.s_pe, cout ? f.maj_out : f.maj_in,
             region_distance(p.g, cout, cp.x, cp.y, cp.z, cd.x, cd.y, cd.z));
        sts1(RING_AT8(aux, i) + 4, cout ? f.maj_in : f.maj_out);
        if constexpr (GENERAL) {
          sts1(RING_AT8(aux, i), __uint_as_float(cctr));
          sts1(RING_GEN(i) + 4, f.s_r);
        }
      }
    }
    tally_flush<WARP_AGG>(cell, cell != nullptr, dq, lane);
    n_parked -= min(n_parked, 32u);
    const uint32_t n_gone = __popc(__ballot_sync(kFull, gone));
    __syncwarp();
    return n_gone;
  };

  // Takes the ready photon of ring slot i.
  auto take = [&](uint32_t i) {
    const float4 np = lds4(RING_AT(pos, i)), nd = lds4(RING_AT(dir, i)), nm = lds4(RING_AT(mid, i));
    const float2 na = lds2(RING_AT8(aux, i));
    px = np.x; py = np.y; pz = np.z; e = np.w;
    ux = nd.x; uy = nd.y; uz = nd.z; hlo = __float_as_uint(nd.w);
    s_c = nm.x; s_pe = nm.y; maj = nm.z; rem = nm.w;
    ctr = __float_as_uint(na.x); maj2 = na.y;
    if constexpr (GENERAL) {
      const float2 g = lds2(RING_GEN(i));
      steps = __float_as_uint(g.x);
      s_r = g.y;
    }
  };

  // ---- site queue: 32 new decays, one per lane --------------------------------
  // Adds the warp's q (below 2^31 each) to a shared counter.
  auto add_units = [&](int slot, uint32_t q) {
    const ull sum = (ull)__reduce_add_sync(kFull, q & 0xffffu) + ((ull)__reduce_add_sync(kFull, q >> 16) << 16);
    if (lane == 0 && sum) atomicAdd(&s_cnt[slot], sum);
  };
  auto sample_sites = [&]() {
    uint32_t idx = 0, lines = 0;
    bool got = true;
    if (!(GAMMAS && deferred)) {
      const uint32_t avail = pool_end - pool_next;
      uint32_t fresh = 0, fresh_end = 0;
      if (avail < 32) {
        if (lane == 0) {
          const unsigned f = atomicAdd(p.g.work, (unsigned)p.chunk);
          if ((uint64_t)f < p.g.n_hist) {
            fresh = f;
            fresh_end = (uint32_t)min((uint64_t)f + (uint64_t)p.chunk, p.g.n_hist);
          }
        }
        fresh = __shfl_sync(kFull, fresh, 0);
        fresh_end = __shfl_sync(kFull, fresh_end, 0);
      }
      if (lane < avail) {
        idx = pool_next + lane;
      } else if (fresh + (lane - avail) < fresh_end) {
        idx = fresh + (lane - avail);
      } else {
        got = false;
      }
      if (avail < 32) {
        pool_next = min(fresh + (32u - avail), fresh_end);
        pool_end = fresh_end;
        drained = fresh_end == 0;
      } else {
        pool_next += 32;
      }
    } else {
      const float2 d = lds2(GAMMA_DEFER(lane));
      idx = __float_as_uint(d.x);
      lines = __float_as_uint(d.y);
      got = lines != 0u;
    }
    const uint64_t h = p.g.hist_begin + idx;
    const uint32_t slo = (uint32_t)h, shi = (uint32_t)(h >> 32);
    bool has = false;
    ull* cell = nullptr;
    Site st{};
    if (got) {
      st = sample_site(p.g, p.key, slo, shi);
      if (pairs) {
        has = p.g.q_positron > 0;
        cell = tally_cell(idx, (uint32_t)st.v);
      }
    }
    float sx = st.x, sy = st.y, sz = st.z;   // where the photons start: the decay, or the end of the positron's track
    if constexpr (NUC != kPair) {
      uint32_t q0 = 0, q_left = 0;
      bool stays = true;
      if (got && !(GAMMAS && deferred)) {
        if constexpr (GAMMAS) {
          uint32_t gc = 0;
          for (int j0 = 0; j0 < p.n_gamma; j0 += 4) {
            const uint4 rg = draw(gc, kStreamGammaSelect, slo, shi, p.key);
            const uint32_t w4[4] = {rg.x, rg.y, rg.z, rg.w};
#pragma unroll
            for (int k = 0; k < 4; ++k)
              if (j0 + k < p.n_gamma && u01(w4[k]) < p.gamma_y[j0 + k]) lines |= 1u << (j0 + k);
          }
          has = p.g.q_positron > 0;
          cell = tally_cell(idx, (uint32_t)st.v);
        }
        if (NUC == kTracked || p.g.beta_tab) {
          ull* const tal = tally_cell(idx, 0u);
          float tx = st.x, ty = st.y, tz = st.z;
          stays = positron_track(p.g, p.key, slo, shi, st.v, tx, ty, tz, q0, q_left,
                                 [&](int v, uint32_t dq) { atomicAdd(tal + v, (ull)dq); });
          if (NUC == kTracked) {
            sx = tx; sy = ty; sz = tz;
          }
        }
      }
      add_units(kBeta, q0);
      if (!stays) atomicAdd(&s_cnt[kLost], (ull)q_left + (NUC == kTracked ? 2ull * (ull)(uint32_t)p.q_e0 : 0ull));
      if (NUC == kTracked) got = got && stays;
    }
    tally_flush<WARP_AGG>(cell, has, (uint32_t)p.g.q_positron, lane);
    const bool o = outside_box(p.g, sx, sy, sz);
    s_next = 0;
    if constexpr (GAMMAS) {
      // one photon per lane and round, as far as the queue goes
      s_left = 0;
      for (;;) {
        const unsigned m = __ballot_sync(kFull, lines != 0u);
        if (m == 0u || s_left == kSiteQueue) break;
        const uint32_t slot = s_left + __popc(m & lt_mask);
        uint32_t q = 0;
        if (lines && slot < kSiteQueue) {
          const int j = __ffs(lines) - 1;
          lines &= lines - 1;
          uint32_t c = 0;
          const uint4 rd = draw(c, kStreamGamma0 + (uint32_t)j, slo, shi, p.key);
          const float cz = fmaf(2.0f, u01(rd.x), -1.0f);
          const float sn = sqrtf(fmaxf(0.0f, fmaf(-cz, cz, 1.0f)));
          float sp, cp;
          __sincosf(fmaf(kTwoPi, u01(rd.y), -3.14159265f), &sp, &cp);
          const float gx = sn * cp, gy = sn * sp, ge = p.gamma_e[j];
          q = (uint32_t)p.gamma_q[j];
          const RingEnergy f = ring_energy<GENERAL>(ge, tab, p.ln_e_lo, p.inv_dln_e);
          sts4(RING_AT(site_pos, slot), sx, sy, sz, __uint_as_float(slo));
          sts4(RING_AT(site_dir, slot), gx, gy, cz, region_distance(p.g, o, sx, sy, sz, gx, gy, cz));
          sts2(RING_AT8(site_rem, slot), ge, __uint_as_float(((kStreamGamma0 + (uint32_t)j) << kStreamShift) | c));
          sts4(GAMMA_MID(slot), f.s_c, f.s_pe, o ? f.maj_out : f.maj_in, o ? f.maj_in : f.maj_out);
        }
        add_units(kGamma, q);
        s_left = min(s_left + (uint32_t)__popc(m), (uint32_t)kSiteQueue);
      }
      deferred = __any_sync(kFull, lines != 0u);
      if (deferred) sts2(GAMMA_DEFER(lane), __uint_as_float(idx), __uint_as_float(lines));
    } else {
      const unsigned m = __ballot_sync(kFull, got);
      if (got) {
        const uint32_t slot = __popc(m & lt_mask);
        float ra, rb;
        region_distance_pair(p.g, o, sx, sy, sz, st.u, st.v_, st.w, ra, rb);
        sts4(RING_AT(site_pos, slot), sx, sy, sz, __uint_as_float(slo));
        sts4(RING_AT(site_dir, slot), st.u, st.v_, st.w, ra);
        sts2(RING_AT8(site_rem, slot), rb, o ? -1.0f : 1.0f);
      }
      s_left = (uint32_t)__popc(m) << (pairs ? 1 : 0);
    }
    n_born += s_left;
    __syncwarp();
  };

  // ---- one Woodcock flight step per photon, then the exchanges.  ENDING: the
  // site queue is empty for good, and lanes without a photon look for one in
  // the ring, which holds n_ring; returns the new n_ring.  LAST: the ring is
  // empty for good, and lanes scatter their own photons.
  auto flight = [&](auto mode, uint32_t n_ring) -> uint32_t {
    constexpr bool ENDING = decltype(mode)::value == 1, LAST = decltype(mode)::value == 2;
    const bool fly = e != 0.0f;
    // words x and y of the step's block; z and w serve the Compton angle if
    // the step finds a scatter
    const uint32_t hhi = h0_hi + (hlo < h0 ? 1u : 0u);
    const uint32_t stream = GAMMAS ? ctr >> kStreamShift : kStreamPhotonA + (__float_as_uint(e) >> 31);
    const uint4 rr = philox4x32_10(make_uint4(GAMMAS ? ctr & kCtrMask : ctr, stream, hlo, hhi), p.key);
    ++ctr;
    const float imaj = fabsf(maj);
    float s = -__logf(u01(rr.x)) * imaj;   // cm
    const bool cross = s >= rem;           // flight cut at the region boundary
    if (cross) s = rem;
    rem -= s;
    px = fmaf(s * p.g.inv_dx, ux, px);
    py = fmaf(s * p.g.inv_dy, uy, py);
    pz = fmaf(s * p.g.inv_dz, uz, pz);
    if (GENERAL) ++steps;
    // floor once: the same integers test the grid bounds (negative or past
    // the end, as unsigned) and index the voxel (positions are finite)
    const int ix = __float2int_rd(px), iy = __float2int_rd(py), iz = __float2int_rd(pz);
    const bool in_grid = fly && (unsigned)ix < (unsigned)p.g.nx && (unsigned)iy < (unsigned)p.g.ny &&
                         (unsigned)iz < (unsigned)p.g.nz;
    const int v = (iz * p.g.ny + iy) * p.g.nx + ix;
    uint32_t wv = 0;
    if (in_grid && !cross) wv = __ldg(p.g.vox + v);
    if (in_grid && cross) {
      const float t = maj;
      maj = maj2;
      maj2 = t;
      rem = kInf;
      if (maj > 0.0f) rem = region_distance(p.g, false, px, py, pz, ux, uy, uz);
    }
    if (fly && !in_grid) {                 // escapes
      n_steps += GENERAL ? steps : steps_of(ctr);
      e = 0.0f;
    }
    const float2 c = lds2(mat + 8u * (wv & 7u));
    // real event with probability mu(voxel)/mubar; the same uniform picks the type
    const float scale = __uint_as_float(wv & ~7u) * imaj;   // 0 where no voxel was met
    const float ic = c.x * s_c;
    const float icp = fmaf(c.y, s_pe, ic);
    const float t = u01(rr.y);
    bool park = t < scale * ic;
    if constexpr (GENERAL) {
      if (!(t < scale * icp) && t < scale * fmaf(lds1(zr + 4u * (wv & 7u)), s_r, icp)) {
        atomicAdd(&s_cnt[kCtrRayleigh], 1ull);
        // Thomson angular shape (1 + cos^2)/2 by rejection; one block per trial.
        for (int trial = 0;; ++trial) {
          const uint4 r = philox4x32_10(make_uint4(GAMMAS ? ctr & kCtrMask : ctr, stream, hlo, hhi), p.key);
          ++ctr;
          const float cth = fmaf(2.0f, u01(r.x), -1.0f);
          const bool acc = 2.0f * u01(r.y) <= fmaf(cth, cth, 1.0f);
          if (acc || trial + 1 >= kKahnTrialLimit) {
            if (!acc) flags |= NM_DEV_RAYLEIGH_LIMIT;
            rotate(ux, uy, uz, cth, fmaf(kTwoPi, u01(r.z), -3.14159265f));
            rem = region_distance(p.g, maj < 0.0f, px, py, pz, ux, uy, uz);
            break;
          }
        }
      }
    }
    // the rare ends of a photon: absorbed, or stopped by the step limit
    const bool limit = (GENERAL ? steps : steps_of(ctr)) >= (uint32_t)p.max_steps;
    const bool photo = !park && t < scale * icp;
    uint32_t dq = 0;
    if (photo || limit) {
      if (photo) {
        atomicAdd(&s_cnt[kCtrPhoto], 1ull);
        dq = (uint32_t)q_units(fabsf(e));
        deposit += dq;
        n_steps += GENERAL ? steps : steps_of(ctr);
        if (!WARP_AGG) atomicAdd(tally_cell(hlo - h0, (uint32_t)v), (ull)dq);
      } else if (e != 0.0f) {
        atomicAdd(&s_cnt[kCtrKilledUnits], (ull)q_units(fabsf(e)));
        atomicAdd(&s_cnt[kKilled], 1ull);
        if (park) atomicAdd(&s_cnt[kCtrCompton], 1ull);
        flags |= NM_DEV_STEP_LIMIT;
        n_steps += GENERAL ? steps : steps_of(ctr);
      }
      e = 0.0f;
      park = false;
    }
    if (WARP_AGG) tally_flush<true>(photo ? tally_cell(hlo - h0, (uint32_t)v) : nullptr, photo, dq, lane);
    if constexpr (LAST) {
      n_compton += __popc(__ballot_sync(kFull, park));
      uint32_t dq2 = 0;
      if (park) {
        float4 cd = make_float4(ux, uy, uz, __uint_as_float(hlo));
        e = scatter(e, cd, ctr, rr.z, rr.w, dq2);
        ux = cd.x; uy = cd.y; uz = cd.z;
        if (e == 0.0f) {
          n_steps += GENERAL ? steps : steps_of(ctr);
        } else {
          const RingEnergy f = ring_energy<GENERAL>(fabsf(e), tab, p.ln_e_lo, p.inv_dln_e);
          s_c = f.s_c; s_pe = f.s_pe; s_r = f.s_r;
          const bool o = maj < 0.0f;
          maj = o ? f.maj_out : f.maj_in;
          maj2 = o ? f.maj_in : f.maj_out;
          rem = region_distance(p.g, o, px, py, pz, ux, uy, uz);
        }
      }
      tally_flush<WARP_AGG>(park ? tally_cell(hlo - h0, (uint32_t)v) : nullptr, park, dq2, lane);
      return 0u;
    }
    // exchanges: scattered photons, and near the end lanes without one
    const bool swap = park || (ENDING && n_ring != 0 && e == 0.0f);
    const unsigned sm = __ballot_sync(kFull, swap);
    const uint32_t n_swap = __popc(sm), n_park = ENDING ? __popc(__ballot_sync(kFull, park)) : n_swap;
    if (swap) {
      const uint32_t i = (head + __popc(sm & lt_mask)) & (kRing - 1);
      const float4 np = lds4(RING_AT(pos, i)), nd = lds4(RING_AT(dir, i)), nm = lds4(RING_AT(mid, i));
      const float2 na = lds2(RING_AT8(aux, i));
      sts4(RING_AT(pos, i), px, py, pz, e);
      sts4(RING_AT(dir, i), ux, uy, uz, __uint_as_float(hlo));
      sts4(RING_AT(mid, i), __uint_as_float(rr.z), __uint_as_float(rr.w), __int_as_float(v), maj);
      sts1(RING_AT8(aux, i), __uint_as_float(ctr));
      px = np.x; py = np.y; pz = np.z; e = np.w;
      ux = nd.x; uy = nd.y; uz = nd.z; hlo = __float_as_uint(nd.w);
      s_c = nm.x; s_pe = nm.y; maj = nm.z; rem = nm.w;
      ctr = __float_as_uint(na.x); maj2 = na.y;
      if constexpr (GENERAL) {
        const float2 g = lds2(RING_GEN(i));
        sts1(RING_GEN(i), __uint_as_float(steps));
        steps = __float_as_uint(g.x);
        s_r = g.y;
      }
    }
    n_compton += n_park;
    if (ENDING) n_ring += n_park - __popc(__ballot_sync(kFull, swap && e != 0.0f));
    head += n_swap;
    n_parked += n_swap;
    __syncwarp();
    return n_ring;
  };

  for (;;) {
    if (n_parked >= 32) compton_pass();
    if (s_left == 0) {
      if (drained && !(GAMMAS && deferred)) break;
      sample_sites();
    }
    // lanes without a photon take the site queue's next ones
    const unsigned want = __ballot_sync(kFull, e == 0.0f);
    const uint32_t rank = __popc(want & lt_mask);
    if (e == 0.0f && rank < s_left) {
      const uint32_t k = s_next + rank, j = pairs ? k >> 1 : k;
      const uint32_t sign = pairs ? k << 31 : 0u;      // photon B (odd) flies opposite to A
      const float4 sp = lds4(RING_AT(site_pos, j)), sd = lds4(RING_AT(site_dir, j));
      const float2 sr = lds2(RING_AT8(site_rem, j));
      px = sp.x; py = sp.y; pz = sp.z;
      hlo = __float_as_uint(sp.w);
      ux = __uint_as_float(__float_as_uint(sd.x) ^ sign);
      uy = __uint_as_float(__float_as_uint(sd.y) ^ sign);
      uz = __uint_as_float(__float_as_uint(sd.z) ^ sign);
      if constexpr (GAMMAS) {
        const float4 m = lds4(GAMMA_MID(j));
        rem = sd.w;
        e = sr.x;
        s_c = m.x; s_pe = m.y; maj = m.z; maj2 = m.w;
        ctr = __float_as_uint(sr.y);
        if (GENERAL) {
          const float ie = __fdividef(1.0f, e);
          s_r = ie * ie;
        }
      } else {
        rem = sign ? sr.x : sd.w;
        e = __uint_as_float(__float_as_uint(p.e0) ^ sign);
        s_c = s_f0.s_c;
        s_pe = s_f0.s_pe;
        maj = s_f0.maj_in;
        maj2 = s_f0.maj_out;
        if (sr.y < 0.0f) {
          maj = s_f0.maj_out;
          maj2 = s_f0.maj_in;
        }
        ctr = 0;
        if (GENERAL) s_r = s_f0.s_r;
      }
      if (GENERAL) steps = 0;
    }
    const uint32_t n_pop = min((uint32_t)__popc(want), s_left);
    s_next += n_pop;
    s_left -= n_pop;
    flight(std::integral_constant<int, 0>(), 0u);
  }
  // Every photon has been started: lanes without one take what the ring holds.
  // Once the lanes can hold all that is left, they keep their photons and
  // scatter them themselves: the last photons fly without waiting in the ring.
  uint32_t n_ring = __popc(__ballot_sync(kFull, lds1(RING_AT(pos, lane) + 12) != 0.0f)) +
                    __popc(__ballot_sync(kFull, lds1(RING_AT(pos, 32 + lane) + 12) != 0.0f));
  while (n_ring + __popc(__ballot_sync(kFull, e != 0.0f)) > 32) {
    if (n_parked >= 32) n_ring -= compton_pass();
    n_ring = flight(std::integral_constant<int, 1>(), n_ring);
  }
  while (n_parked) compton_pass();
  {
    const unsigned lo = __ballot_sync(kFull, lds1(RING_AT(pos, lane) + 12) != 0.0f),
                   hi = __ballot_sync(kFull, lds1(RING_AT(pos, 32 + lane) + 12) != 0.0f);
    const uint32_t rank = __popc(__ballot_sync(kFull, e == 0.0f) & lt_mask), n_lo = __popc(lo);
    if (e == 0.0f && rank < n_lo + __popc(hi))
      take(rank < n_lo ? __fns(lo, 0, rank + 1) : 32 + __fns(hi, 0, rank - n_lo + 1));
  }
  while (__any_sync(kFull, e != 0.0f)) flight(std::integral_constant<int, 2>(), 0u);
#undef RING_AT
#undef RING_AT8
#undef RING_GEN
#undef GAMMA_MID
#undef GAMMA_DEFER

  // ---- counters ---------------------------------------------------------------
  const ull dep_sum = warp_sum(deposit), step_sum = warp_sum((ull)n_steps);
  if (lane == 0) {
    atomicAdd(&s_cnt[kCtrSteps], step_sum);
    atomicAdd(&s_cnt[kCtrCompton], (ull)n_compton);
    atomicAdd(&s_cnt[kBorn], (ull)n_born);
    atomicAdd(&s_cnt[kDeposit], dep_sum);
  }
  const unsigned fl = __reduce_or_sync(kFull, flags);
  if (lane == 0 && fl) atomicOr(p.status, fl);
  __syncthreads();
  if (threadIdx.x == 0) {
    // every photon that started was absorbed, cut off, killed or escaped, and
    // what it did not deposit went with it
    s_cnt[kCtrEscapes] = s_cnt[kBorn] - s_cnt[kCtrPhoto] - s_cnt[kCtrCutoff] - s_cnt[kKilled];
    s_cnt[kCtrEscapedUnits] = (GAMMAS ? s_cnt[kGamma] : s_cnt[kBorn] * (ull)(uint32_t)p.q_e0) - s_cnt[kDeposit] -
                              s_cnt[kCtrKilledUnits] + s_cnt[kLost];
    if (NUC != kPair && s_cnt[kBeta]) atomicAdd(p.g.counters + kCtrPositronUnits, s_cnt[kBeta]);
    if (GAMMAS && s_cnt[kGamma]) atomicAdd(p.g.counters + kCtrGammaUnits, s_cnt[kGamma]);
  }
  __syncthreads();
  if (threadIdx.x < 8 && s_cnt[threadIdx.x]) atomicAdd(p.g.counters + threadIdx.x, s_cnt[threadIdx.x]);
}

// Scattering cosines at energy e as the transport's table sampler draws them
// (counters 0..n-1 of stream 7, key k0 k1).
__global__ void check_kn_table_kernel(const TransportParams p, float e, int64_t n, float* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t ctr = 0;
  const uint4 r = draw(ctr, 7u, (uint32_t)i, (uint32_t)(i >> 32), p.key);
  out[i] = 1.0f - kn_table_x(p, e, r.x);
}

// Positron energies of histories 0..n-1 as the transport draws them.
__global__ void check_beta_kernel(const float* tab, int64_t n, uint32_t k0, uint32_t k1, float* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t ctr = 0;
  const uint4 r = draw(ctr, kStreamPositron, (uint32_t)i, (uint32_t)(i >> 32), philox_key(k0, k1));
  out[i] = beta_energy(tab, r.x);
}

__global__ void check_philox_kernel(const uint4* ctr, const uint2* key, int64_t n, uint4* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  // the transport's own path: round keys from philox_key, then the rounds
  if (i < n) out[i] = philox4x32_10(ctr[i], philox_key(key[i].x, key[i].y));
}

__global__ void check_kahn_kernel(float e, int64_t n, uint32_t k0, uint32_t k1, float* out,
                                  uint32_t* status) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t ctr = 0, rphi, flags = 0;
  const float x = kahn_x(e * kInvElectronMassMeV, ctr, 7u, (uint32_t)i, (uint32_t)(i >> 32), philox_key(k0, k1),
                         rphi, flags);
  out[i] = 1.0f - x;
  if (flags) atomicOr(status, flags);
}

__global__ void check_source_kernel(const TransportParams p, uint64_t first, int64_t n,
                                    int32_t* voxel, float* pos, float* dir) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t h = first + (uint64_t)i;
  const Site s = sample_site(p.g, p.key, (uint32_t)h, (uint32_t)(h >> 32));
  voxel[i] = s.v;
  pos[3 * i + 0] = s.x / p.g.inv_dx;
  pos[3 * i + 1] = s.y / p.g.inv_dy;
  pos[3 * i + 2] = s.z / p.g.inv_dz;
  dir[3 * i + 0] = s.u;
  dir[3 * i + 1] = s.v_;
  dir[3 * i + 2] = s.w;
}

// Dynamic shared memory: the site stash, the history lists when kept, and
// (nuclide variant) the origin of the gamma lines.
size_t transport_smem(int block, bool history, bool beta) {
  return ((size_t)9 + (history ? 2 * kHistVoxels : 0) + (beta ? 3 : 0)) * block * sizeof(float);
}

template <bool A, bool R, bool G, bool H, bool B = false>
void* kernel_ptr() {
  return (void*)transport_kernel<A, R, G, H, B>;
}

template <bool H, bool B>
void* pick_lanes(bool r, bool g) {
  if (r) return g ? kernel_ptr<false, true, true, H, B>() : kernel_ptr<false, true, false, H, B>();
  return g ? kernel_ptr<false, false, true, H, B>() : kernel_ptr<false, false, false, H, B>();
}

// The lane kernel.  History statistics and the beta+ spectrum exist only
// without warp aggregation; without either, regrouped launches are the ring
// kernel's.
void* pick(bool a, bool r, bool g, bool h, bool beta) {
  if (beta || h) {
    if (a) return nullptr;
    if (!beta) return pick_lanes<true, false>(r, g);
    return h ? pick_lanes<true, true>(r, g) : pick_lanes<false, true>(r, g);
  }
  if (g) return nullptr;
  if (a) return r ? kernel_ptr<true, true, false, false>() : kernel_ptr<true, false, false, false>();
  return r ? kernel_ptr<false, true, false, false>() : kernel_ptr<false, false, false, false>();
}

// The ring kernel runs every regrouped launch without history statistics but
// that of a nuclide which gives both an annihilation pair and gamma lines: 1e8
// decays on the benchmark phantom take 13.2 ms on it and 30.5 ms on the lane
// kernel; 2e7 on the 4 mm phantom with tracked positrons 3.7 and (regrouped)
// 7.4 ms, of 131I 2.9 and 6.0, of 177Lu 1.4 and 3.0.
bool use_ring(bool regroup, bool history, int nuc) { return regroup && !history && nuc >= 0; }

void* pick_ring(bool a, bool general, int nuc) {
  if (nuc == kTracked)
    return general ? (void*)transport_ring_kernel<false, true, kTracked> : (void*)transport_ring_kernel<false, false, kTracked>;
  if (nuc == kGammas)
    return general ? (void*)transport_ring_kernel<false, true, kGammas> : (void*)transport_ring_kernel<false, false, kGammas>;
  if (a) return general ? (void*)transport_ring_kernel<true, true, kPair> : (void*)transport_ring_kernel<true, false, kPair>;
  return general ? (void*)transport_ring_kernel<false, true, kPair> : (void*)transport_ring_kernel<false, false, kPair>;
}

size_t ring_smem(int block, bool general, int nuc) {
  const uint32_t warp = nuc == kGammas ? (general ? StoreOf<true, kGammas>::kBytes : StoreOf<false, kGammas>::kBytes)
                                       : (general ? StoreOf<true, kPair>::kBytes : StoreOf<false, kPair>::kBytes);
  return sizeof(RingTables) + (size_t)(block / 32) * warp;
}

}  // namespace

int nuclide_kind(bool decay, bool beta_track, bool annihilate, int n_gamma) {
  if (!decay) return kPair;
  if (annihilate) return n_gamma > 0 ? -1 : beta_track ? kTracked : kPair;
  return kGammas;
}

cudaError_t launch_transport(const TransportParams& p, int grid, int block, bool warp_agg,
                             bool rayleigh, bool regroup, cudaStream_t s, bool history) {
  const int nuc = nuclide_kind(p.g.source_mode == NM_SOURCE_DECAY, p.g.beta_tab != nullptr, p.annihilate != 0, p.n_gamma);
  if (nuc != kPair && warp_agg) return cudaErrorInvalidValue;
  const bool ring = use_ring(regroup, history, nuc);
  const bool general = rayleigh || !p.kn_inv;
  void* fn = ring ? pick_ring(warp_agg, general, nuc) : pick(warp_agg, rayleigh, regroup, history, nuc != kPair);
  if (!fn) return cudaErrorInvalidValue;
  void* args[] = {(void*)&p};
  // the history lists and the rings take the static + dynamic total past the
  // 48 KB default
  const size_t smem = ring ? ring_smem(block, general, nuc) : transport_smem(block, history, nuc != kPair);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) e = cudaLaunchKernel(fn, dim3(grid), dim3(block), args, smem, s);
  if (e != cudaSuccess) cudaGetLastError();  // a refused launch must not linger as the last error
  return e;
}

int transport_max_blocks_per_sm(int block, bool warp_agg, bool rayleigh, bool kahn, bool regroup, bool history,
                                int nuc) {
  int n = 0;
  if (nuc != kPair && warp_agg) return 0;
  const bool ring = use_ring(regroup, history, nuc), general = rayleigh || kahn;
  void* fn = ring ? pick_ring(warp_agg, general, nuc) : pick(warp_agg, rayleigh, regroup, history, nuc != kPair);
  const size_t smem = ring ? ring_smem(block, general, nuc) : transport_smem(block, history, nuc != kPair);
  if (!fn || cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, block, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_check_kn_table(const TransportParams& p, float e, int64_t n, float* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  check_kn_table_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(p, e, n, out);
  return cudaGetLastError();
}

cudaError_t launch_check_beta(const float* tab, int64_t n, uint32_t k0, uint32_t k1, float* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  check_beta_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(tab, n, k0, k1, out);
  return cudaGetLastError();
}

cudaError_t launch_check_philox(const uint4* ctr, const uint2* key, int64_t n, uint4* out,
                                cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  check_philox_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(ctr, key, n, out);
  return cudaGetLastError();
}

cudaError_t launch_check_kahn(float e, int64_t n, uint32_t k0, uint32_t k1, float* out,
                              uint32_t* status, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  check_kahn_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(e, n, k0, k1, out, status);
  return cudaGetLastError();
}

cudaError_t launch_check_source(const TransportParams& p, uint64_t first, int64_t n, int32_t* voxel,
                                float* pos, float* dir, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  check_source_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(p, first, n, voxel, pos, dir);
  return cudaGetLastError();
}

}  // namespace nm
